"""The fused step's whole rows and halves in their steady state: rows with more
tiles than a batch holds (48, 18 with eight query heads), the last wave's rows or
all rows in halves or none, on chip, with logits through HBM (past 8704 tokens,
24 tiles with eight heads) and with scores there too (past 10240); sampled rows,
the split ones among them, against the oracle, and dc_step's one eviction in the
kernel bit for bit against dc_decode_step and dc_evict. Each case asserts the
schedule that it is about."""

import pytest

from paper_2608_08878_gb300 import synth

from harness import LockStep

pytestmark = pytest.mark.gpu

# rows (more than the SMs by so many, or a number), query heads per KV head, head
# dim, budget, scorer, rows in halves
CASES = [
    ("+8", 4, 128, 6200, 0, 8),        # 49 tiles, the last wave in halves
    ("+8", 4, 128, 6271, 0, 8),        # 49 whole tiles
    ("+5", 2, 64, 6144, 0, 5),         # the newest token alone in the 49th tile
    ("+0", 4, 128, 6200, 0, 0),        # whole rows
    ("+0", 1, 64, 6300, 0, 0),
    ("+3", 4, 128, 9000, 0, 3),        # logits through HBM
    ("+0", 4, 128, 9000, 0, 0),
    ("+3", 4, 128, 10500, 0, 3),       # and scores
    ("+0", 4, 128, 10500, 0, 0),
    (40, 4, 128, 12400, 0, 40),        # few rows, past what clusters of 2 hold: all in halves
    ("+8", 8, 128, 2400, 0, 8),        # eight query heads
    ("+0", 8, 128, 3300, 0, 0),        # logits through HBM
    ("+4", 8, 64, 8500, 0, 4),         # and scores
    ("+8", 4, 128, 6200, 1, 8),        # H2O
    ("+0", 4, 128, 6200, 2, 0),        # StreamingLLM
]


def _rows(rows):
    import torch
    return rows if isinstance(rows, int) else torch.cuda.get_device_properties(0).multi_processor_count + int(rows)


@pytest.mark.parametrize("rows,group,d,budget,scorer,halves", CASES)
def test_long_rows_match_the_oracle_and_the_two_calls(rows, group, d, budget, scorer, halves):
    import torch
    from paper_2608_08878_gb300 import dc
    rows = _rows(rows)
    wl = synth.MISTRAL_1L.with_(layers=1, batch=rows, kv_heads=1, q_heads=group, head_dim=d, prompt_len=budget,
                                budget=budget, steps=3, window=4)
    ls = LockStep(wl, [0, rows - 1], engine=2, device_inputs=True, scorer=scorer)
    ls.load_prompt()
    for _ in range(wl.steps):
        ls.step()
    a, b = (LockStep(wl, [], engine=2, device_inputs=True, scorer=scorer) for _ in range(2))
    for x in (a, b):
        x.load_prompt()
        assert x.cache.debug_schedule() == {"batch_rows": 0, "cluster": 0, "half_rows": halves}
    for s in range(8):
        B = budget if s < 6 else budget - 3 * (s - 5)  # then several evictions
        q, kn, vn = a._inputs(s)
        oa = a.cache.step(q, kn, vn, budget=B)
        ob = b.cache.decode_step(q, kn, vn)
        b.cache.evict(B)
        a.cache.sync()
        b.cache.sync()
        assert torch.equal(oa, ob), s
        n = a.cache.length()[0]
        assert n == b.cache.length()[0]
        for which in (dc.BUF_K, dc.BUF_V, dc.BUF_POS, dc.BUF_S, dc.BUF_Z, dc.BUF_VNORM):
            assert torch.equal(a.cache.buffer(which)[:, :n], b.cache.buffer(which)[:, :n]), (s, which)


def test_the_query_names_the_other_schedules():
    """Batches, clusters and the split engine in the same terms."""
    from paper_2608_08878_gb300 import dc
    batches = dc.DistillCache(32, 8, 128, 500, 410, batch=4)
    s = batches.debug_schedule(411)
    assert s["batch_rows"] > 1 and s["cluster"] == 1 and s["half_rows"] == 0
    few = dc.DistillCache(1, 8, 128, 2100, 2048)
    assert few.debug_schedule(2049) == {"batch_rows": 1, "cluster": 8, "half_rows": 0}
    whole = dc.DistillCache(1, 8, 128, 2100, 2048, tail_split=False)
    assert whole.debug_schedule(2049)["cluster"] == 1 and whole.debug_schedule(2049)["half_rows"] == 0
    split = dc.DistillCache(1, 8, 128, 2100, 2048, engine=1)
    assert split.debug_schedule() == {"batch_rows": 0, "cluster": 0, "half_rows": 0}
