"""Handle-free attention with rows split over a thread-block cluster: split
counts from 1 to the cluster limit, ragged last splits, last warps without
tokens, against softmax attention in 64 bits.

Tolerance: a logit is a sum of d products accumulated in fp32, |error| <= d
2^-24 sum |q_i k_i| c (c = 1/sqrt(d)) <= d 2^-24 |q| |k| c, about d 2^-24 sqrt(d)
for N(0, 1) inputs (up to 1.5 x for the longest of a few thousand keys); a
weight's relative error is that, twice for the normalisation; the sums over
tokens add n 2^-24 at most."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n", [(1, 2047), (1, 16385), (3, 300), (10, 2049), (40, 1025), (300, 385), (700, 129)])
@pytest.mark.parametrize("d,group", [(64, 1), (64, 8), (128, 2), (128, 4), (128, 8), (64, 4)])
def test_split_rows_match_attention_in_64_bits(rows, n, d, group):
    import torch
    from paper_2608_08878_gb300 import dc
    g = torch.Generator(device="cuda").manual_seed(rows * n + d + group)
    q, k, v = (torch.randn((rows, m, d), device="cuda", generator=g).bfloat16() for m in (group, n, n))
    out = dc.attend_noalloc(q, k, v)
    p = torch.softmax(torch.einsum("rgd,rnd->rgn", q.double(), k.double()) / d ** 0.5, -1)
    ref = torch.einsum("rgn,rnd->rgd", p, v.double())
    rel = float((out.double() - ref).norm() / ref.norm())
    assert rel <= 2 * 1.5 * d * 2.0 ** -24 * d ** 0.5 + n * 2.0 ** -24
