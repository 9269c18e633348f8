"""Few rows, each over a thread-block cluster: clusters of 8, 4 and 2 at the
fewest tiles a rank takes, a last rank whose newest token starts a tile, uneven
shares, the most tiles that fit on chip, every scorer's kernel; rows against the
oracle, dc_step bit for bit against dc_decode_step and dc_evict (with one and
with several evictions), and device-counted steps against ordinary ones."""

import pytest

from paper_2608_08878_gb300 import synth

from harness import LockStep

pytestmark = pytest.mark.gpu


def _workload(rows, group, d, budget):
    return synth.MISTRAL_1L.with_(layers=1, batch=rows, kv_heads=1, q_heads=group, head_dim=d, prompt_len=budget,
                                  budget=budget, steps=3, window=4)


@pytest.mark.parametrize("rows,group,d,budget,scorer", [
    (1, 4, 128, 2047, 0),      # 16 whole tiles over 8 CTAs
    (3, 4, 128, 2048, 0),      # the newest token alone in the last tile
    (6, 1, 64, 2100, 0),       # 17 tiles over 8, one query head of 64 dims
    (16, 4, 128, 2047, 0),     # one cluster of 8 too many, or just as many
    (2, 4, 128, 24000, 0),     # 188 tiles: 23 or 24 a CTA
    (5, 8, 128, 14000, 0),     # 110 tiles, eight query heads
    (20, 2, 128, 1100, 0),     # clusters of 4, 9 tiles
    (64, 4, 64, 1279, 0),      # clusters of 2, 10 tiles
    (9, 8, 64, 2500, 1),       # H2O
    (50, 4, 128, 1400, 2),     # StreamingLLM, clusters of 2
])
def test_clusters_match_the_oracle_and_the_two_calls(rows, group, d, budget, scorer):
    import torch
    from paper_2608_08878_gb300 import dc
    wl = _workload(rows, group, d, budget)
    ls = LockStep(wl, sorted({0, rows - 1}), engine=2, device_inputs=True, scorer=scorer)
    ls.load_prompt()
    for _ in range(wl.steps):
        ls.step()
    a, b, g = (LockStep(wl, [], engine=2, device_inputs=True, scorer=scorer) for _ in range(3))
    for x in (a, b, g):
        x.load_prompt()
    for s in range(8):
        B = budget if s < 6 else budget - 3 * (s - 5)  # then several evictions
        q, kn, vn = a._inputs(s)
        if s == wl.window + 1 and scorer == 0:
            g.cache.set_graph_mode(True)
        oa = a.cache.step(q, kn, vn, budget=B)
        ob = b.cache.decode_step(q, kn, vn)
        b.cache.evict(B)
        og = g.cache.step(q, kn, vn, budget=B) if s < 6 else oa
        a.cache.sync()
        b.cache.sync()
        if s == 5 and scorer == 0:
            g.cache.set_graph_mode(False)
        g.cache.sync()
        assert torch.equal(oa, ob) and torch.equal(oa, og), s
        n = a.cache.length()[0]
        assert n == b.cache.length()[0]
        for which in (dc.BUF_K, dc.BUF_V, dc.BUF_POS, dc.BUF_S, dc.BUF_Z, dc.BUF_VNORM):
            assert torch.equal(a.cache.buffer(which)[:, :n], b.cache.buffer(which)[:, :n]), (s, which)
