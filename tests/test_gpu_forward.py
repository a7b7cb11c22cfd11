"""The forward kernel of cis_token_logprobs at the sizes where its row split
and its ragged ends can go wrong, against fp64 log-softmaxes of the same rows.

Tolerance of log p: 2e-5 plus four fp32 steps of it, as everywhere else; of
the entropy, whose terms are bounded by log V, 2e-5 (1 + log V).
"""
import math

import numpy as np
import pytest
import torch

from paper_2609_32444_gb300 import binding

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

DEV = torch.device("cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


def _check(z, ids):
    """Every output of the forward pass on rows z (a view of any stride)."""
    T, V = z.shape
    mask = torch.ones(T, dtype=torch.uint8, device=DEV)
    mask[T // 2] = 0
    plain = binding.cis_token_logprobs(z, ids, mask=mask)
    lp, lse, ent = binding.cis_token_logprobs(z, ids, mask=mask, want_lse=True,
                                              want_entropy=True)
    on = mask != 0
    x = z.double()
    r = torch.arange(T, device=DEV)
    zy = x[r, ids.long()]
    rest = x.clone()
    rest[r, ids.long()] = -math.inf
    odds = zy - torch.logsumexp(rest, 1)
    want = -torch.nn.functional.softplus(-odds).masked_fill(~on, 0)
    want_lse = torch.logsumexp(x, 1).masked_fill(~on, 0)
    ls = x - torch.logsumexp(x, 1, keepdim=True)
    p = ls.exp()
    want_ent = -torch.where(p > 0, p * ls, torch.zeros_like(p)).sum(1).masked_fill(~on, 0)
    tol = 2e-5 + 2.0 ** -21 * want.abs()
    assert bool(((lp.double() - want).abs() <= tol).all())
    assert bool(((plain.double() - want).abs() <= tol).all())
    assert bool(((lse.double() - want_lse).abs() <= 2e-5 + 2.0 ** -21 * want_lse.abs()).all())
    assert bool(((ent.double() - want_ent).abs() <= 2e-5 * (1 + math.log(V))).all())


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("T,V", [
    (5, 1), (5, 2), (4, 7), (4, 8), (4, 9), (6, 15), (3, 63), (3, 2049),   # 64 threads a row
    (4, 4096), (4, 4097), (3, 4104), (700, 8200),                           # 256 threads a row
    (1217, 4113),                                                           # 128
    (300, 8207), (150, 16391), (3, 16391), (2, 40003)])                     # 2 to 8 CTAs a row
def test_row_splits_and_ragged_ends(dtype, T, V):
    """Rows that start at every offset from a 16-byte boundary (an odd stride
    and an odd first element), the sampled token at either end and inside."""
    g = torch.Generator(device=DEV)
    g.manual_seed(V)
    for pad, off in ((0, 0), (3, 1)):
        buf = torch.randn(T * (V + pad) + off, generator=g, device=DEV).mul_(4).to(dtype)
        z = buf[off:].view(T, V + pad)[:, :V]
        ids = torch.randint(0, V, (T,), generator=g, device=DEV).int()
        ids[0], ids[-1] = 0, V - 1
        ids[T // 3] = min(V - 1, 9)
        _check(z, ids)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("fill", ["lowest", "neg_inf", -1e30, -1e10, -1e9, -1e6, -1e5])
def test_rows_of_masked_entries(dtype, fill):
    """Rows with all but a few entries masked, by any of the usual values:
    whole batches of a thread hold nothing else, and one row holds only its
    sampled token; another is at the lowest value throughout."""
    T, V = 4, 9000
    low = {"lowest": torch.finfo(dtype).min, "neg_inf": -math.inf}.get(fill, fill)
    z = torch.full((T, V), low, dtype=dtype, device=DEV)
    ids = torch.tensor([17, 8999, 5000, 3], dtype=torch.int32, device=DEV)
    z[0, 17:8000:900] = 1.5
    z[1, 8990:] = -2.0
    z[2, 5000] = 3.0
    if fill != "neg_inf":
        lp, lse = binding.cis_token_logprobs(z, ids, want_lse=True)
        want = torch.tensor([-math.log(9), -math.log(10), 0.0, -math.log(V)], device=DEV)
        assert bool(((lp - want).abs() <= 2e-5 + 2.0 ** -21 * want.abs()).all())
        lowest = float(z[3, 0])  # (as rounded to the type)
        assert abs(float(lse[3]) - (lowest + math.log(V))) <= 2.0 ** -22 * abs(lowest)
        return
    z[3, :5] = 0.25
    _check(z, ids)


def _whole_products(lo, hi, n):
    """fp32 values m in [lo, hi) whose product with log2e rounds down to a whole number,
    those with the largest remainder."""
    l2e = np.float32(math.log2(math.e))
    k = np.arange(int(lo * float(l2e)) + 1, int(hi * float(l2e)), dtype=np.float64)
    m = (k / np.float64(l2e)).astype(np.float32)
    best = []
    for c in (m, np.nextafter(m, np.float32(np.inf)), np.nextafter(m, np.float32(0))):
        over = c.astype(np.float64) * np.float64(l2e) - k
        over[(c * l2e).astype(np.float64) != k] = 0
        best += list(zip(over, c))
    return [float(c) for _, c in sorted(best)[-n:]]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_maxima_whose_offset_is_rounded_down(dtype):
    """16 entries share the maximum, the others are out of reach: log p = -log 16,
    whatever the maximum (also as p of the diagnostics)."""
    m = [124928.0, 448512.0]
    if dtype == torch.float32:
        m += _whole_products(100, 1000, 3) + _whole_products(1e5, 9e5, 3)
    V = 2050
    z = torch.tensor(m, device=DEV).view(-1, 1).expand(len(m), V).to(dtype).contiguous()
    z[:, 16:] *= 0.5
    ids = torch.arange(len(m), dtype=torch.int32, device=DEV)
    lp, lse, ent = binding.cis_token_logprobs(z, ids, want_lse=True, want_entropy=True)
    p = binding.cis_mismatch_diagnostics(z, z, ids, binding.cis_default_params("cis"))["p"]
    want = math.log(16)
    assert bool(((lp + want).abs() <= 2e-5).all()) and bool(((16 * p - 1).abs() <= 2e-5).all())
    assert bool(((ent - want).abs() <= 2e-5 * (1 + want)).all())
    x = z[:, 0].double()
    assert bool(((lse.double() - x - want).abs() <= 2e-5 + 2.0 ** -21 * x).all())


@pytest.mark.parametrize("sign", [1, -1])
def test_maxima_on_both_sides_of_the_exponents_two_forms(sign):
    """fp32 rows with entries a step below and above 1e6 (the first or the last part of
    a row, or every other vector): a thread's maxima, and the threads', cross over."""
    T, V = 3, 12000
    lo, hi = (999999.9375, 1000000.0625) if sign > 0 else (-1000000.0625, -999999.9375)
    z = torch.full((T, V), lo, device=DEV)
    z[0, V // 2:] = hi
    z[1, :V // 2] = hi
    z[2].view(-1, 2, 4)[:, 1] = hi
    _check(z, torch.tensor([3, 3, 3], dtype=torch.int32, device=DEV))
    _check(z[:, :1030].contiguous(), torch.tensor([3, 3, 3], dtype=torch.int32, device=DEV))


@pytest.mark.parametrize("dtype,z0", [(torch.bfloat16, -19.375), (torch.float32, -18.715)])
@pytest.mark.parametrize("T", [40, 1300])
def test_small_entries_next_to_a_large_one(dtype, z0, T):
    """One entry is 1 and the others so small that a vector of them rounds away against
    it, but not a batch of four, which is one step of 2^-23 within 3%: a thread's 75
    batches at most (fp32) lose 75 * 0.03 * 2^-23 = 2.7e-7, and as much again is left for
    the exponentials; a thread that loses them all loses 4e-6."""
    V = 151936
    z = torch.full((T, V), z0, dtype=dtype, device=DEV)
    z[:, 5] = 0.0
    ids = torch.full((T,), 9, dtype=torch.int32, device=DEV)
    lp = binding.cis_token_logprobs(z, ids).double()
    x = float(z[0, 9])
    want = x - math.log1p((V - 1) * math.exp(x))
    assert float((lp - want).abs().max()) <= 5.3e-7 + 2.0 ** -24 * abs(want)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_entropy_error_over_many_rows(dtype):
    """Root mean square of the relative error: H is near 6.4 (a step of 2^-21), and log
    s', u'/s', their difference, 1 - p, its product and the sums are each rounded at that
    size or below: 0.29 steps in each of six, 5.3e-8, and what the sums carry.  With
    1 - p from an exponential (up to two steps more) it is 6.0e-8."""
    g = torch.Generator(device=DEV)
    g.manual_seed(7)
    T, V = 8192, 1000
    z = torch.randn((T, V), generator=g, device=DEV).to(dtype)
    ids = z.float().argmax(1).int()
    ids[::2] = torch.randint(0, V, (T,), generator=g, device=DEV).int()[::2]
    _, _, ent = binding.cis_token_logprobs(z, ids, want_entropy=True)
    ls = z.double() - torch.logsumexp(z.double(), 1, keepdim=True)
    H = -(ls.exp() * ls).sum(1)
    assert float(((ent - H) / H).square().mean().sqrt()) <= 5.7e-8
