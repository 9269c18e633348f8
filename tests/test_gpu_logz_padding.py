"""log Z of rows whose scores tie at large numbers where the cut falls (a row
padded with a large negative finite number, B beyond the unpadded count; the
same at large positive numbers), of B equal to the row's length there, and the
sampler's log-probability of such a row.

Live items y_1 .. y_n far above m equal items z, B = n + k: the subsets that
count hold all live items and k of the others, so log Z = sum y + k z + log C(m,
k). Tolerance: the sums are double-float or double, one rounding to fp32 at the
end (2^-24 |log Z|), P(S = B) as elsewhere (L 2^-21 in the documented bound): 2^-22
|log Z| + L 2^-21 + 2^-22 max|s|."""

import math

import pytest

pytestmark = pytest.mark.gpu


def _rows(L, live, scale, sign):
    """[1][L] scores: `live` items above the rest, which all equal sign * scale."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(L + live)
    s = torch.full((1, L), sign * scale, device="cuda")
    s[:, :live] = torch.randn((1, live), device="cuda", generator=g) + (0.0 if sign < 0 else 2.0 * scale)
    return s[:, torch.randperm(L, device="cuda", generator=g)].contiguous()


def _log_binomial(m, k):
    return math.lgamma(m + 1) - math.lgamma(k + 1) - math.lgamma(m - k + 1)


@pytest.mark.parametrize("scale", [1e6, 1e10, 1e13, 1e15, 1e16, 1e25, 1e34])
@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("L,live", [(3, 1), (256, 32), (1025, 1), (8193, 4000)])
def test_ties_at_large_numbers(L, live, sign, scale):
    import torch
    from paper_2608_08878_gb300 import dc
    s = _rows(L, live, scale, sign)
    top = s.double().sort(dim=1, descending=True).values
    for B in sorted({live + 1, live + 2, live + (L - live) // 3, (L + live) // 2, L - 1, L}):
        if B > L or B == live:
            continue
        ref = float(top[0, :B].sum()) + _log_binomial(L - live, B - live)
        got = float(dc.pl_log_partition(s, B))
        tol = 2.0 ** -22 * (abs(ref) + float(s.abs().max())) + L * 2.0 ** -21
        assert abs(got - ref) <= tol, (B, got, ref)


@pytest.mark.parametrize("scale", [1e15, 1e16, 1e25])
def test_every_cut_of_a_padded_row(scale):
    from paper_2608_08878_gb300 import dc
    L, live = 256, 32
    s = _rows(L, live, scale, -1)
    top = s.double().sort(dim=1, descending=True).values
    for B in range(live + 1, L):
        ref = float(top[0, :B].sum()) + _log_binomial(L - live, B - live)
        got = float(dc.pl_log_partition(s, B))
        assert abs(got - ref) <= 2.0 ** -22 * (abs(ref) + scale) + L * 2.0 ** -21, (B, got, ref)


def test_a_padded_batch_of_rows_and_its_sample():
    import torch
    from paper_2608_08878_gb300 import dc
    s = torch.cat([_rows(256, live, 1e16, -1) for live in (32, 40, 100)])
    got = dc.pl_log_partition(s, 90).double()
    # the sampled subset: every live item and the first of the padding
    idx, logp = dc.gumbel_top_b(s, torch.zeros_like(s), 90)
    ref = torch.sort(s, dim=1, descending=True, stable=True).indices[:, :90].sort(dim=1).values
    assert torch.equal(idx.long(), ref) and bool(torch.isfinite(logp).all())
    want = s.gather(1, ref).double().sum(1) - got
    tol = 2.0 ** -22 * (got.abs() + 1e16 * 58) + 256 * 2.0 ** -21
    assert bool(((logp.double() - want).abs() <= tol).all())


def test_a_sum_past_the_fp32_range_is_infinite():
    import torch
    from paper_2608_08878_gb300 import dc
    for sign in (-1.0, 1.0):
        s = torch.full((2, 16), sign * 2e38, device="cuda")
        assert bool((dc.pl_log_partition(s, 16) == sign * math.inf).all())
