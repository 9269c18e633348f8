"""log Z and the sampler at the edges of the shifted characteristic-function
evaluation: near-constant scores, scores so spread that E[S] is a staircase,
large common offsets, masked items (-infinity), every B near 1 and near the
number of unmasked items, rows past the registers' capacity -- against the
recurrence over e_k in 64 bits, and the kept sets against a stable sort.

Tolerance: the documented bound 2 L 2^-24 (|log Z| + max |s| / tau) + L 2^-21."""

import math

import pytest

pytestmark = pytest.mark.gpu


def _logz64(y, B):
    import torch
    e = torch.full((y.shape[0], B + 1), -math.inf, dtype=torch.float64, device=y.device)
    e[:, 0] = 0.0
    for i in range(y.shape[1]):
        e[:, 1:] = torch.logaddexp(e[:, 1:], e[:, :-1] + y[:, i: i + 1])
    return e[:, -1]


def _scores(kind, rows, L):
    import torch
    g = torch.Generator(device="cuda").manual_seed(L)
    s = torch.randn((rows, L), device="cuda", generator=g)
    if kind == "constant":
        s = torch.full_like(s, 0.25)
    elif kind == "spread":
        s = s * 1000.0
    elif kind == "offset":
        s = 1e5 + s
    elif kind == "clusters":
        s = torch.where(s > 0.5, 300.0, 0.0)
    elif kind == "masked":
        s[:, ::3] = -math.inf
    return s


@pytest.mark.parametrize("kind", ["normal", "constant", "spread", "offset", "clusters", "masked"])
@pytest.mark.parametrize("L", [1, 2, 33, 700, 8192, 8193])
def test_log_partition_edges(kind, L):
    import torch
    from paper_2608_08878_gb300 import dc
    s = _scores(kind, 3, L)
    fin = int(torch.isfinite(s[0]).sum())
    for B in sorted({b for b in (1, 2, fin // 3, fin - 1, fin) if 1 <= b <= min(fin, 300)}):
        got = dc.pl_log_partition(s, B, 0.5).double()
        ref = _logz64((s / 0.5).double(), B)
        big = float((s[torch.isfinite(s)] / 0.5).abs().max())
        tol = 2 * L * 2.0 ** -24 * (ref.abs() + big) + L * 2.0 ** -21
        assert bool(((got - ref).abs() <= tol).all()), (B, got, ref)
    if 1 <= fin < L:
        assert bool((dc.pl_log_partition(s, fin + 1) == -math.inf).all())


@pytest.mark.parametrize("L,B", [(1, 1), (33, 32), (513, 100), (4096, 1024), (41000, 9000)])
def test_sampler_keeps_a_stable_sorts_prefix(L, B):
    import torch
    from paper_2608_08878_gb300 import dc
    g = torch.Generator(device="cuda").manual_seed(L)
    s = torch.randint(-3, 4, (3, L), device="cuda", generator=g).float()  # many ties
    idx, logp = dc.gumbel_top_b(s, torch.zeros_like(s), B)
    ref = torch.sort(s, dim=1, descending=True, stable=True).indices[:, :B].sort(dim=1).values
    assert torch.equal(idx.long(), ref)
    lz = dc.pl_log_partition(s, B).double()
    assert torch.allclose(logp.double(), s.gather(1, ref).double().sum(1) - lz, rtol=2.0 ** -22, atol=1e-3)
