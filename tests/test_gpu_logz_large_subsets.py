"""log Z at subset sizes up to all items, and of rows at and past the length that
stays in shared memory (40960 scores; longer rows compute each value again from
global memory), against 64 bits; the sampler's log-probability of such rows.

e_B(x_1 .. x_n) = x_1 ... x_n e_{n - B}(1 / x_1 .. 1 / x_n), so that B close to the
number n of finite items takes a recurrence over n - B terms only.

Tolerance: the sums are double-float, log Z is rounded once (2^-24 |log Z|), the
scores are divided by a power of two; a term log(1 + e^x) or log p of an item is
off by at most 8 ulp of 1 (expf, reciprocal, log1pf, and x rounded where |x| e^-|x|
< 1): 2^-22 (|log Z| + max |s| / tau) + L 2^-21."""

import math

import pytest

from test_gpu_logz_shift import _logz64, _scores

pytestmark = pytest.mark.gpu


def _reference(y, B):
    """log e_B of every row in 64 bits; every row of y has the same finite items."""
    import torch
    fin = y[:, torch.isfinite(y[0])].double()
    n = fin.shape[1]
    if 2 * B <= n:
        return _logz64(fin, B)
    return fin.sum(1) + (_logz64(-fin, n - B) if B < n else 0.0)


def _check(s, B, got):
    import torch
    ref = _reference(s / 0.5, B)
    big = float((s[torch.isfinite(s)] / 0.5).abs().max())
    tol = 2.0 ** -22 * (ref.abs() + big) + s.shape[1] * 2.0 ** -21
    assert bool(((got.double() - ref).abs() <= tol).all()), (B, got, ref)


@pytest.mark.parametrize("kind", ["normal", "constant", "spread", "offset", "clusters", "masked"])
@pytest.mark.parametrize("L", [33, 700, 8192, 8193])
def test_large_subsets(kind, L):
    import torch
    from paper_2608_08878_gb300 import dc
    s = _scores(kind, 2, L)
    n = int(torch.isfinite(s[0]).sum())
    for B in sorted({n // 3, n // 2 + 1, n - 200, n - 2, n - 1, n} - {0}):
        if B >= 1:
            _check(s, B, dc.pl_log_partition(s, B, 0.5))


@pytest.mark.parametrize("kind", ["normal", "spread", "clusters", "masked"])
@pytest.mark.parametrize("L", [40960, 40961])
def test_rows_at_the_shared_memory_limit(kind, L):
    import torch
    from paper_2608_08878_gb300 import dc
    s = _scores(kind, 2, L)
    if kind == "masked":  # 13654 finite items: B up to all of them
        s[:, 1::3] = -math.inf
    n = int(torch.isfinite(s[0]).sum())
    for B in [1, 2, 300] + ([n - 100, n - 1, n] if kind == "masked" else []):
        _check(s, B, dc.pl_log_partition(s, B, 0.5))
    if kind == "masked":
        assert bool((dc.pl_log_partition(s, n + 1, 0.5) == -math.inf).all())


@pytest.mark.parametrize("L", [40960, 40961])
def test_the_sampler_of_long_rows(L):
    import torch
    from paper_2608_08878_gb300 import dc
    s = _scores("normal", 2, L)
    g = torch.Generator(device="cuda").manual_seed(3)
    noise = -torch.log(torch.empty_like(s).exponential_(generator=g))
    idx, logp = dc.gumbel_top_b(s, noise, 257, 0.5)
    kept = torch.sort(s / 0.5 + noise, dim=1, descending=True, stable=True).indices[:, :257].sort(dim=1).values
    assert torch.equal(idx.long(), kept)
    total = (s / 0.5).double().gather(1, kept).sum(1)
    _check(s, 257, total - logp.double())
