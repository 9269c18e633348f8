"""Full-cache attention on CUDA cores (handle-free, and a handle's on the split
engine) with keys and values that are not finite: a NaN key makes the row's
output NaN wherever it stands, a logit of -infinity has no weight, +infinity
makes NaN, an infinite value is an infinite output in its column, and other rows
know nothing of it. The reference is softmax attention in 64 bits: the same
entries NaN, +infinity and -infinity, and the finite ones within the bound that
test_gpu_attend_splits.py derives."""

import math

import pytest

pytestmark = pytest.mark.gpu

CASES = ["NaN in the last key", "NaN in the first keys", "NaN in every key", "infinity in a key",
         "infinity in the first keys", "infinity in the last value", "infinity in a value", "NaN in the last value"]


def _plant(case, q, k, v):
    """Row 1 of three gets what `case` says."""
    n = k.shape[1]
    if case == "NaN in the last key":
        k[1, -1, 3] = math.nan
    elif case == "NaN in the first keys":  # eight tokens or more open a warp's work
        k[1, : min(n, 16), 5] = math.nan
    elif case == "NaN in every key":
        k[1, :, 0] = math.nan
    elif case == "infinity in a key":  # a logit of -infinity for every head, +infinity in row 2
        q[1:, :, 7] = -1.0
        k[1, n // 2, 7] = math.inf
        k[2, n // 2, 7] = -math.inf
    elif case == "infinity in the first keys":
        q[1, :, 7] = -1.0
        k[1, : n - 1, 7][:64] = math.inf
    elif case == "infinity in the last value":
        v[1, -1, 2] = math.inf
    elif case == "infinity in a value":
        v[1, n // 3, 1] = -math.inf
    elif case == "NaN in the last value":
        v[1, -1, 0] = math.nan


def _reference(q, k, v):
    import torch
    d = q.shape[-1]
    p = torch.softmax(torch.einsum("rgd,rnd->rgn", q.double(), k.double()) / d ** 0.5, -1)
    # (weight 0 of an infinite value would be NaN: no case has one)
    return torch.einsum("rgn,rnd->rgd", p, v.double())


def _inputs(case, n, d, group):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n * 1024 + d + group)
    q, k, v = (torch.randn((3, m, d), device="cuda", generator=g).bfloat16() for m in (group, n, n))
    _plant(case, q, k, v)
    return q, k, v


def _check(out, ref, n, d):
    import torch
    assert torch.equal(out.isnan(), ref.isnan())
    assert torch.equal(out == math.inf, ref == math.inf) and torch.equal(out == -math.inf, ref == -math.inf)
    fin = ref.isfinite()
    if bool(fin.any()):
        rel = float((out.double() - ref)[fin].norm() / ref[fin].norm())
        assert rel <= 2 * 1.5 * d * 2.0 ** -24 * d ** 0.5 + n * 2.0 ** -24


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("n", [1, 9, 300, 2049])
@pytest.mark.parametrize("d,group", [(128, 4), (128, 8), (64, 1), (64, 2)])
def test_handle_free_attention(case, n, d, group):
    from paper_2608_08878_gb300 import dc
    q, k, v = _inputs(case, n, d, group)
    _check(dc.attend_noalloc(q, k, v), _reference(q, k, v), n, d)


@pytest.mark.parametrize("case", CASES)
def test_full_decode_on_the_split_engine(case):
    from paper_2608_08878_gb300 import dc
    n, d, group = 777, 128, 4
    q, k, v = _inputs(case, n, d, group)
    cache = dc.DistillCache(1, 1, d, n + 1, 100, batch=3, q_heads=group, engine=1)
    cache.append(k[None, :, None].contiguous(), v[None, :, None].contiguous())
    out = cache.full_decode(q[None].contiguous())
    cache.sync()
    _check(out.view(3, group, d), _reference(q, k, v), n, d)
