"""The fused step on batches of rows: batch sizes from one row to the most a
warpgroup's statistics hold, a second round with smaller batches, an odd row
count, rows of one box, one whole tile, one token past a tile and as many tiles
as fit on chip, every scorer's kernel; sampled rows (the first and last rows of
batches among them) against the oracle, and dc_step bit for bit against
dc_decode_step and dc_evict, with one and with several evictions."""

import pytest

from paper_2608_08878_gb300 import synth

from harness import LockStep

pytestmark = pytest.mark.gpu


def _workload(rows, group, d, budget):
    # one layer, one KV head: the batch size is the row count
    return synth.MISTRAL_1L.with_(layers=1, batch=rows, kv_heads=1, q_heads=group, head_dim=d, prompt_len=budget,
                                  budget=budget, steps=3, window=4)


@pytest.mark.parametrize("rows,group,d,budget,scorer", [
    (1, 4, 128, 411, 0),       # one row, one CTA
    (153, 4, 128, 127, 0),     # one CTA with two rows of one whole tile
    (457, 2, 64, 128, 0),      # four rows a batch, the second tile one token
    (3800, 1, 64, 15, 0),      # 24 rows and one left a CTA, one 16-token box
    (4001, 4, 128, 411, 0),    # two rounds of 12, then of 3, the last one short
    (305, 4, 128, 6143, 0),    # 48 tiles: one row fills the on-chip logits
    (160, 8, 128, 2303, 0),    # 18 tiles, eight query heads
    (471, 8, 64, 300, 1),      # H2O
    (471, 4, 128, 300, 2),     # StreamingLLM
])
def test_batches_match_the_oracle_and_the_two_calls(rows, group, d, budget, scorer):
    import torch
    from paper_2608_08878_gb300 import dc
    wl = _workload(rows, group, d, budget)
    sample = sorted({0, min(11, rows - 1), rows // 2, rows - 1})
    ls = LockStep(wl, sample, engine=2, device_inputs=True, scorer=scorer)
    ls.load_prompt()
    for _ in range(wl.steps):
        ls.step()
    a, b = (LockStep(wl, [], engine=2, device_inputs=True, scorer=scorer) for _ in range(2))
    for x in (a, b):
        x.load_prompt()
    for s in range(5):
        B = budget if s < 3 else budget - 3 * (s - 2)  # then several evictions
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
