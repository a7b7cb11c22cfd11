"""The diagnostics' split kernel (any type and alignment, few rows, short rows)
against fp64 closed forms, and the streaming kernel where short rows no longer
take it by themselves.  Bounds: those of test_gpu_diagnostics.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from _util import logits_for_oracle
from paper_2609_32444_gb300 import binding
from test_gpu_diagnostics import DEV, U, _compare, _rows, diag_error_bounds, n_thread

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


def _closed_forms(z, zi, ids, mode):
    lp, lq = torch.log_softmax(z.double(), 1), torch.log_softmax(zi.double(), 1)
    k = (lp - lq).exp()
    f = torch.minimum(k, 1 + 2.3 * (-torch.expm1(lp)).clamp(min=5e-3)) if mode == "cis" \
        else k.clamp(max=2.0)
    p, q = lp.exp(), lq.exp()
    f = torch.where(q > 0, f, torch.ones_like(f))
    qf = q * f
    r = qf - p
    P2 = p.square().sum(1, keepdim=True)
    g2 = 1 - 2 * p + P2
    F = qf.sum(1)
    y = ids.long().view(-1, 1)
    mean_f = qf.square().sum(1) - 2 * F * (qf * p).sum(1) + F * F * P2.view(-1)
    return {"logk": (lp - lq).gather(1, y).view(-1), "p": p.gather(1, y).view(-1),
            "bias2": (r - p * r.sum(1, keepdim=True)).square().sum(1),
            "dvar": (qf * f * g2).sum(1) - mean_f -
                    ((q * g2).sum(1) - (q - p).square().sum(1))}


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("T,V", [(3, 9), (5, 1001), (200, 1001), (3, 8207), (3, 16391),
                                 (1300, 16403), (3, 20001), (2, 40003), (1, 131077)])
def test_widths_clusters_and_alignments(dtype, T, V):
    """128 and 512 threads, one to eight CTAs a row; rows at every phase of a
    16-byte boundary, at the same one in both tensors (vector loads) and at
    different ones (entry by entry); the sampled token at either end."""
    cpu = [x.to(dtype) for x in _rows(V, T, V, torch.float32, sd=0.5)[:2]]
    ids = _rows(V, T, V, torch.float32)[2]
    ids[0], ids[-1] = 0, V - 1
    for pad_t, pad_i in ((0, 0), (1, 2)):
        if pad_t and T > 100:
            continue
        bufs = []
        for x, pad in zip(cpu, (pad_t, pad_i)):
            b = torch.full((T, V + pad), 50.0, dtype=dtype, device=DEV)  # the padding is not read
            b[:, :V] = x.to(DEV)
            bufs.append(b[:, :V])
        mode = "cis" if pad_t else "tis"
        out = binding.cis_mismatch_diagnostics(bufs[0], bufs[1], ids.to(DEV),
                                               binding.cis_default_params(mode))
        want = _closed_forms(bufs[0], bufs[1], ids.to(DEV), mode)
        rows = slice(0, min(T, 16))
        tol = dict(zip(("bias2", "dvar"), diag_error_bounds(cpu[0][rows], cpu[1][rows], mode, 328)))
        for k, w in want.items():
            w = w.cpu().numpy()[rows]
            d = np.abs(out[k].double().cpu().numpy()[rows] - w)
            t = (tol[k] + 2 * U * np.abs(w) if k in tol
                 else 2e-5 * w if k == "p" else 2 * (2e-5 + 2.0 ** -21 * np.abs(w)))
            assert np.all(d <= t), (k, pad_t)


@pytest.mark.parametrize("kernel", ["row", "stream"])
def test_masked_entries(monkeypatch, kernel):
    """Entries masked in both engines, at -inf and at large negative values: the
    results of the rows without those columns, on both kernels."""
    V, T = 2048, 6
    z, zi, ids = _rows(3, T, V, torch.bfloat16, sd=0.5)
    ids = ids % 500
    P = binding.cis_default_params("cis")
    base = _closed_forms(z[:, :500].to(DEV), zi[:, :500].to(DEV), ids.to(DEV), "cis")
    tol = dict(zip(("bias2", "dvar"), diag_error_bounds(z[:, :500], zi[:, :500], "cis", 328)))
    for low in (-math.inf, torch.finfo(torch.bfloat16).min, -1e30, -1e10, -1e9):
        a, b = z.clone().to(DEV), zi.clone().to(DEV)
        a[:, 500:], b[:, 500:] = low, low
        monkeypatch.setenv("CIS_DIAG_KERNEL", kernel)
        out = binding.cis_mismatch_diagnostics(a, b, ids.to(DEV), P)
        for k in ("bias2", "dvar", "logk"):
            w = base[k].cpu().numpy()
            d = np.abs(out[k].double().cpu().numpy() - w)
            assert np.all(d <= tol.get(k, 4e-5) + 2.0 ** -20 * np.abs(w)), (k, low)
    if kernel == "stream":  # a row at such a value throughout, the sampled entry too
        a, b = z.clone().to(DEV), zi.clone().to(DEV)
        a[0], b[1], a[2] = -1e10, torch.finfo(torch.bfloat16).min, -(2.0 ** 32)
        out = binding.cis_mismatch_diagnostics(a, b, ids.to(DEV), P)
        for k, v in out.items():
            assert bool(torch.isnan(v[:3]).all()) and bool(torch.isfinite(v[3:]).all()), k


@pytest.mark.parametrize("T,V,mode", [(700, 1024, "cis"), (400, 2056, "icepop"), (160, 64, "kpop")])
def test_streaming_kernel_on_short_rows(monkeypatch, T, V, mode):
    """Several short rows per CTA through the streaming kernel."""
    monkeypatch.setenv("CIS_DIAG_KERNEL", "stream")
    z, zi, ids = _rows(14, T, V, torch.bfloat16)
    m = torch.ones(T, dtype=torch.uint8)
    m[::5] = 0
    out = binding.cis_mismatch_diagnostics(z.to(DEV), zi.to(DEV), ids.to(DEV),
                                           binding.cis_default_params(mode), mask=m.to(DEV))
    torch.cuda.synchronize()
    ref = oracle.mismatch_diagnostics(
        logits_for_oracle(z), logits_for_oracle(zi), ids.numpy(),
        oracle.params(mode=getattr(oracle, "MODE_" + mode.upper())), mask=m.numpy())
    _compare(out, ref, z, zi, mode, n_thread(V), m.numpy())


@pytest.mark.parametrize("mode,kw", [("cis", {"lam": math.inf}), ("cis", {"lam": 1e39}),
                                     ("cis", {"lam": math.inf, "kappa": 0.0}),
                                     ("band", {"lam": math.inf}), ("tis", {"tis_cap": math.inf}),
                                     ("exact", {"exact_hi": math.inf})])
@pytest.mark.parametrize("kernel,dtype,V", [("row", torch.float32, 1001), ("row", torch.bfloat16, 1001),
                                            ("row", torch.bfloat16, 1024),
                                            ("stream", torch.bfloat16, 1024)])
def test_operators_without_an_upper_bound(monkeypatch, mode, kw, kernel, dtype, V):
    """f = k (the band lifts it to (1 + p) / 2 at least), also where candidates of an
    odd row are paired with none and where both engines mask entries at -inf; the
    bounds are those of the large finite ones."""
    monkeypatch.setenv("CIS_DIAG_KERNEL", kernel)
    z, zi, ids = (x.to(DEV) for x in _rows(9, 5, V, torch.float32, sd=0.3))
    z, zi, ids = z.to(dtype), zi.to(dtype), ids % 700
    zi[0, 700:750] = -1e4  # q flushes to 0, k does not exist
    for masked in (0, V - 800):
        if masked:
            z[:, 800:], zi[:, 800:] = -math.inf, -math.inf
        out = binding.cis_mismatch_diagnostics(z, zi, ids, binding.cis_default_params(mode, **kw))
        big = {k: min(v, 1e30) if k != "kappa" else 1.0 for k, v in kw.items()}
        if "lam" in kw:
            big["kappa"] = 1.0
        want = binding.cis_mismatch_diagnostics(z, zi, ids, binding.cis_default_params(mode, **big))
        for k in ("bias2", "dvar"):
            assert bool(torch.isfinite(out[k]).all()), (k, masked)
            assert torch.equal(out[k], want[k]), (k, masked)
        if mode != "band":  # q f = p: no bias but rounding, each of 1024 entries' squared
            assert bool((out["bias2"][1:] <= V * (8 * U) ** 2).all())
