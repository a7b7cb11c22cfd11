"""The fused pass on rows of any alignment and any V (the cluster kernel's
ragged form), and on rows of masked entries at the type's lowest value, against
fp64 softmaxes of the same rows.

With the weight operator "none" and no mask, dz = c (softmax - onehot) with
c = A / T.  fp32 gradients must be within 1e-6 of |c| (the pass's bound), bf16
ones within that of the value rounded once (bf16 has 8 significant bits: half a
step is at most 2^-8 of the value).
"""
import math

import pytest
import torch

from paper_2609_32444_gb300 import binding

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

DEV = torch.device("cuda")
BF16, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


def _check(z, ids, dz, T, V, entropy=False):
    adv = torch.linspace(-2, 3, T, device=DEV).float()
    out = binding.cis_loss_fwd_bwd(z, ids, torch.full((T,), -1.0, device=DEV), adv,
                                   binding.cis_default_params("none"), dlogits=dz, V=V,
                                   want_entropy=entropy)
    x = z[:, :V].double()
    x = x - x.max(1, keepdim=True).values  # (log V next to 3e38 would be lost)
    r, y = torch.arange(T, device=DEV), ids.long()
    zy = x[r, y]
    rest = x.clone()
    rest[r, y] = -math.inf
    lp = -torch.nn.functional.softplus(torch.logsumexp(rest, 1) - zy)
    assert bool(((out["lp"].double() - lp).abs() <= 2e-5 + 2.0 ** -21 * lp.abs()).all())
    c = (adv.double() / T).view(-1, 1)
    want = torch.softmax(x, 1)
    want[r, y] = torch.expm1(lp)
    want = want * c
    tol = 1e-6 * c.abs() + (2.0 ** -8 * want.abs() if dz.dtype == BF16 else 0.0)
    got = dz[:, :V].double()
    assert bool(((got - want).abs() <= tol).all())
    if entropy:
        ls = torch.log_softmax(x, 1)
        h = -torch.where(ls.exp() > 0, ls.exp() * ls, torch.zeros_like(ls)).sum(1)
        assert bool(((out["entropy"].double() - h).abs() <= 2e-5 * (1 + math.log(V))).all())
    assert binding.device_status(out["workspace"]) == 0


@pytest.mark.parametrize("din,dout", [(BF16, BF16), (BF16, F32), (F32, F32), (F32, BF16)])
@pytest.mark.parametrize("T,V", [(5, 1), (9, 2), (9, 7), (9, 8), (9, 9), (17, 15), (17, 17),
                                 (9, 31), (5, 1001), (9, 2047), (9, 2056), (3, 20483),
                                 (3, 32003), (2, 90005),
                                 (2, 409601), (2, 819201)])  # too long for a cluster: row kernel
def test_any_alignment(din, dout, T, V):
    """Rows that start at every phase of a 16-byte boundary: contiguous odd rows
    in both tensors (whole groups are stored), rows whose strides or first
    entries differ (entries are), and padding columns of dlogits left alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(V)
    for pad_in, off_in, pad_out, off_out in ((0, 0, 0, 0), (0, 1, 0, 1), (5, 0, 0, 0),
                                             (0, 0, 3, 1), (1, 3, 1, 3)):
        src = torch.randn(T * (V + pad_in) + off_in, generator=g, device=DEV).mul_(3).to(din)
        z = src[off_in:].view(T, V + pad_in)[:, :V]
        ids = torch.randint(0, V, (T,), generator=g, device=DEV).int()
        ids[0], ids[-1] = 0, V - 1
        buf = torch.full((T * (V + pad_out) + off_out + 64,), 7.0, dtype=dout, device=DEV)
        dz = buf[off_out:off_out + T * (V + pad_out)].view(T, V + pad_out)
        _check(z, ids, dz, T, V, entropy=pad_in == 0)
        assert bool((dz[:, V:] == 7).all()) and bool((buf[-64:] == 7).all())
        assert bool((buf[:off_out] == 7).all())


@pytest.mark.parametrize("dout", [BF16, F32])
@pytest.mark.parametrize("V", [1001, 40003])
def test_masked_and_bad_rows_are_zeroed_whole(dout, V):
    """Masked rows and rows with an out-of-range id, at every phase."""
    T = 17
    z = torch.randn(T, V, device=DEV).to(BF16)
    ids = torch.zeros(T, dtype=torch.int32, device=DEV)
    ids[3] = V
    mask = torch.ones(T, dtype=torch.uint8, device=DEV)
    mask[::2] = 0
    buf = torch.full((T * V + 64,), 7.0, dtype=dout, device=DEV)
    out = binding.cis_loss_fwd_bwd(z, ids, torch.full((T,), -1.0, device=DEV),
                                   torch.ones(T, device=DEV), binding.cis_default_params("cis"),
                                   mask=mask, dlogits=buf[:T * V].view(T, V))
    dead = (mask == 0) | (ids == V)
    assert torch.count_nonzero(out["dlogits"][dead]).item() == 0
    assert bool((out["dlogits"][~dead] != 7).all()) and bool((buf[-64:] == 7).all())


@pytest.mark.parametrize("dtype", [BF16, F32])
@pytest.mark.parametrize("V", [9000, 9001])
@pytest.mark.parametrize("low", [None, -1e30, -1e10, -1e9, -1e5])
def test_rows_at_the_lowest_value(dtype, V, low):
    """Masked vocabularies: all but a few entries at finfo.min or at a large
    negative number, one row with nothing but the sampled token, on the aligned
    and the ragged form; a row at that value throughout is uniform on the ragged
    form and, below -1.4e9, NaN on the aligned one, which keeps no count of such
    entries."""
    T, low = 4, torch.finfo(dtype).min if low is None else low
    z = torch.full((T, V), low, dtype=dtype, device=DEV)
    z[0, 17:8000:900] = 1.5
    z[1, 8990:] = -2.0
    z[2, 5000] = 3.0
    ids = torch.tensor([17, 8999, 5000, 3], dtype=torch.int32, device=DEV)
    n = T if V % 8 or low >= -1e9 else 3
    for dout in (BF16, F32):
        _check(z[:n], ids[:n], torch.empty((n, V), dtype=dout, device=DEV), n, V, entropy=True)
    if n < T:
        out = binding.cis_loss_fwd_bwd(z[3:], ids[3:], torch.full((1,), -1.0, device=DEV),
                                       torch.ones(1, device=DEV),
                                       binding.cis_default_params("none"))
        assert bool(torch.isnan(out["lp"]).all())


def test_weights_and_sampled_gradients_keep_their_roundings():
    """The weights of likely tokens (p > 0.97) and the sampled entry's gradient of
    unlikely ones (p < 0.02), formed without logarithms, on fp32 rows.  k = p / q: 1 - p
    carries a few fp32 roundings, which count by (1 - p) / p < 0.03, 1 / q is a pair, and
    the product is rounded once: 1.5 roundings.  c (p - 1) with c = 1 / T a power of two:
    the few roundings of p count by 0.02, and 1 - p is rounded once: 1.2."""
    T, V = 4096, 1001
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    z = torch.randn((T, V), generator=g, device=DEV) * 2
    ids = torch.randint(0, V, (T,), generator=g, device=DEV)
    r = torch.arange(T, device=DEV)
    odds = torch.where(r % 2 == 0, 3.6 + 6 * torch.rand(T, generator=g, device=DEV),
                       -4.0 - 6 * torch.rand(T, generator=g, device=DEV))
    rest = z.clone()
    rest[r, ids] = -math.inf
    z[r, ids] = torch.logsumexp(rest, 1) + odds
    d = z.double()
    d[r, ids] = -math.inf
    lp = -torch.nn.functional.softplus(torch.logsumexp(d, 1) - z[r, ids].double())
    linf = (lp + 0.1 * torch.randn(T, generator=g, device=DEV)).clamp(max=-1e-4).float()
    adv = torch.ones(T, device=DEV)
    high, u = r % 2 == 0, 2.0 ** -24
    out = binding.cis_loss_fwd_bwd(z, ids.int(), linf, adv, binding.cis_default_params("exact"))
    k = (lp - linf.double()).exp()
    assert float(((out["w"].double() - k).abs() / k)[high].max()) <= 1.5 * u
    out = binding.cis_loss_fwd_bwd(z, ids.int(), linf, adv, binding.cis_default_params("none"))
    got, want = out["dlogits"][r, ids].double(), torch.expm1(lp) / T
    assert float(((got - want) / want).abs()[~high].max()) <= 1.2 * u


@pytest.mark.parametrize("dtype", [BF16, F32])
@pytest.mark.parametrize("T,V", [(3, 1), (3, 8), (3, 9), (3, 1001)])
def test_nan_sampled_entry_without_others(dtype, T, V):
    """A NaN logit makes its row's outputs NaN, also where every other entry is at -inf
    (or there is none); the rows around it are not touched."""
    z = torch.zeros((T, V), dtype=dtype, device=DEV)
    z[1, 1:] = -math.inf
    z[1, 0] = math.nan
    out = binding.cis_loss_fwd_bwd(z, torch.zeros(T, dtype=torch.int32, device=DEV),
                                   torch.full((T,), -0.5, device=DEV),
                                   torch.ones(T, device=DEV), binding.cis_default_params("none"))
    assert bool(torch.isnan(out["lp"][1])) and bool(torch.isnan(out["dlogits"][1, 0]))
    assert bool(torch.isfinite(out["dlogits"][::2].float()).all())
