"""Graph mode where the device-counted step runs on whole rows or halves (rows of
more tiles than a batch holds) and on clusters: steps equal ordinary dc_step
calls bit for bit past a window's wrap, eagerly and as one captured step
replayed. Each case asserts the schedule that it is about."""

import pytest

from paper_2608_08878_gb300 import synth

from test_gpu_graph import _same_cache

pytestmark = pytest.mark.gpu


def _caches(wl, stream):
    from paper_2608_08878_gb300 import dc, synth_device
    out = []
    for _ in range(2):
        c = dc.DistillCache(wl.layers, wl.kv_heads, wl.head_dim, wl.prompt_len + 8, wl.budget, batch=wl.batch,
                            q_heads=wl.q_heads, window=wl.window, mlp_hidden=wl.mlp_hidden, layernorm=wl.layernorm,
                            engine=2, seed=wl.policy_seed, stream=stream)
        c.append(*synth_device.prompt(wl, 0, wl.prompt_len))
        out.append(c)
    return out


def _run(rows, group, d, budget, batch_rows, cluster, half_rows):
    import torch
    from paper_2608_08878_gb300 import synth_device
    wl = synth.MISTRAL_1L.with_(layers=1, batch=rows, kv_heads=1, q_heads=group, head_dim=d, prompt_len=budget,
                                budget=budget, window=4)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b = _caches(wl, stream)
        assert b.debug_schedule() == {"batch_rows": batch_rows, "cluster": cluster, "half_rows": half_rows}
        s = 0
        for _ in range(wl.window + 1):  # a full window of decode steps first
            x = synth_device.step_inputs(wl, s)
            a.step(*x)
            b.step(*x)
            s += 1
        b.set_graph_mode(True)
        for _ in range(2 * wl.window + 3):  # past the window: the counted slots wrap
            x = synth_device.step_inputs(wl, s)
            assert torch.equal(a.step(*x), b.step(*x)), s
            s += 1
        x = [t.clone() for t in synth_device.step_inputs(wl, s)]
        out = torch.empty(x[0].shape, dtype=torch.float32, device="cuda")
        graph = torch.cuda.CUDAGraph()
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            b.step(*x, out=out)  # captured, not run
        for _ in range(wl.window + 2):
            for t, new in zip(x, synth_device.step_inputs(wl, s)):
                t.copy_(new)
            graph.replay()
            ref = a.step(*synth_device.step_inputs(wl, s))
            stream.synchronize()
            assert torch.equal(out, ref), s
            s += 1
        b.set_graph_mode(False)
        a.sync()
        b.sync()
        _same_cache(a, b)
        for _ in range(2):  # ordinary steps again from the state the device counted
            x = synth_device.step_inputs(wl, s)
            assert torch.equal(a.step(*x), b.step(*x)), s
            s += 1
        a.sync()
        b.sync()
        _same_cache(a, b)


@pytest.mark.parametrize("extra,group,d,budget", [
    (8, 4, 128, 6200),    # the last wave in halves
    (0, 4, 128, 6200),    # whole rows
    (3, 4, 128, 9000),    # logits through HBM, halves
    (0, 4, 64, 9000),     # and whole rows
    (3, 4, 128, 10500),   # scores through HBM too
    (8, 8, 128, 2400),    # eight query heads, halves
    (0, 8, 64, 3300),     # logits through HBM
    (2, 1, 128, 6144),    # one query head, the newest token alone in its tile
])
def test_device_counted_steps_on_whole_rows_and_halves(extra, group, d, budget):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _run(sms + extra, group, d, budget, 0, 0, extra)


@pytest.mark.parametrize("rows,group,d,budget,cluster", [
    (1, 4, 128, 2047, 8),
    (3, 1, 64, 2100, 8),
    (5, 8, 128, 14000, 8),
    (20, 2, 128, 1100, 4),
    (24, 8, 64, 1500, 4),
    (64, 4, 64, 2047, 2),
    (60, 1, 128, 2100, 2),
    (62, 2, 64, 2300, 2),
])
def test_device_counted_steps_on_clusters(rows, group, d, budget, cluster):
    _run(rows, group, d, budget, 1, cluster, 0)
