"""The LM head with masked tokens left out of its products, and with dH's
contraction in ranges: against the oracle, and against the same tokens as a
batch of their own without a mask (which is multiplied as it is).

Tolerances of the gradients are those of test_gpu_lmhead (dz in bf16, fp32
accumulation over K terms); the products of two runs may differ by the fp32
accumulation alone.
"""
import numpy as np
import pytest
import torch

from paper_2609_32444_gb300 import binding, synth
from test_gpu_lmhead import DEV, _check_grad, _check_tokens, _oracle, _run

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


@pytest.fixture(autouse=True)
def _packed(monkeypatch):
    monkeypatch.setenv("CIS_LMHEAD_PACK", "1")  # these sizes are below the rule's


@pytest.mark.parametrize("grad", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("T,V,H,valid", [
    (129, 1000, 256, 1), (300, 1000, 512, 128), (300, 1000, 512, 129),  # one tile, just over one
    (257, 8192, 256, 200), (640, 8192, 256, 511),                       # split contractions
    (384, 700, 256, 384), (200, 5000, 256, 63)])
def test_masked_tokens_left_out(T, V, H, valid, grad):
    """`valid` of T tokens, anywhere in the batch: every output and gradient
    element; masked rows of dH are exact zeros."""
    b = synth.make_batch(5, T=T, V=V, H=H)
    g = torch.Generator().manual_seed(T + valid)
    b.mask.zero_()
    b.mask[torch.randperm(T, generator=g)[:valid]] = 1
    out = _run(b, grad_dtype=grad)
    torch.cuda.synchronize()
    ref = _oracle(b)
    _check_tokens(out, ref, np.arange(T), b, "cis", full=True)
    _check_grad(out["dhidden"], ref["dhidden"], ref["dhidden_abs"], V, grad == torch.bfloat16)
    _check_grad(out["dweight"], ref["dweight"], ref["dweight_abs"], T, grad == torch.bfloat16)
    off = (b.mask == 0).to(DEV)
    assert torch.count_nonzero(out["dhidden"][off]).item() == 0
    assert binding.decode_stats(out["stats"])["status"] == 0


@pytest.mark.parametrize("grad", [torch.float32, torch.bfloat16])
def test_no_valid_token(grad):
    """All tokens masked: zero gradients, zero loss, whatever the buffers held."""
    b = synth.make_batch(5, T=300, V=1000, H=256)
    b.mask.zero_()
    nan = [torch.full(s, float("nan"), dtype=grad, device=DEV) for s in ((300, 256), (1000, 256))]
    need = binding.cis_lmhead_workspace_size(300, 1000, 256)
    ws = torch.full((need + 1024,), 255, dtype=torch.uint8, device=DEV)  # NaN patterns
    ws = ws[(-ws.data_ptr()) % 1024:][:need]
    out = binding.cis_lmhead_fused(
        b.hidden.to(DEV), b.weight.to(DEV), b.ids.to(DEV), b.lp_infer.to(DEV), b.adv.to(DEV),
        binding.cis_default_params("cis"), mask=b.mask.to(DEV), grad_dtype=grad, workspace=ws,
        dhidden=nan[0], dweight=nan[1])
    torch.cuda.synchronize()
    for k in ("dhidden", "dweight", "lp", "w"):
        assert torch.count_nonzero(out[k]).item() == 0, k
    assert float(out["loss"]) == 0.0


@pytest.mark.parametrize("mode", ["cis", "seq_tis"])
@pytest.mark.parametrize("old", [False, True])
def test_same_as_the_valid_tokens_alone(mode, old):
    """A masked batch against its valid tokens as an unmasked batch, with a
    bad id among them, a NaN workspace, and the sequence operator's two sweeps."""
    T, V, H = 500, 3000, 256
    b = synth.make_batch(5, T=T, V=V, H=H)
    g = torch.Generator().manual_seed(4)
    keep = torch.rand(T, generator=g) < 0.6
    b.ids[int(torch.nonzero(keep)[7])] = V + 5
    cu = torch.tensor([0, 130, 131, 390, T], dtype=torch.int32)
    short = torch.tensor([int(keep[:c].sum()) for c in cu.tolist()], dtype=torch.int32)
    lp_old = b.lp_infer + 0.1 * torch.randn(T, generator=g)
    P = binding.cis_default_params(mode)

    def run(rows, mask, cu_seqlens):
        t = [x[rows].contiguous().to(DEV) for x in (b.hidden, b.ids, b.lp_infer, b.adv, lp_old)]
        n = t[0].shape[0]
        need = binding.cis_lmhead_workspace_size(n, V, H)
        ws = torch.full((need + 1024,), 255, dtype=torch.uint8, device=DEV)
        ws = ws[(-ws.data_ptr()) % 1024:][:need]
        return binding.cis_lmhead_fused(t[0], b.weight.to(DEV), t[1], t[2], t[3], P,
                                        lp_old=t[4] if old else None, mask=mask,
                                        cu_seqlens=cu_seqlens.to(DEV), workspace=ws,
                                        want_entropy=True)

    full = run(torch.arange(T), keep.to(torch.uint8).to(DEV), cu)
    alone = run(torch.nonzero(keep).view(-1), None, short)
    torch.cuda.synchronize()
    on = keep.to(DEV)
    for k in ("lp", "w", "entropy"):
        x, y = full[k][on], alone[k]
        assert torch.equal(torch.isnan(x), torch.isnan(y)), k
        fine = ~torch.isnan(y)
        assert bool(((x - y)[fine].abs() <= 1e-5 * (1 + y[fine].abs())).all()), k
        assert torch.count_nonzero(full[k][~on]).item() == 0, k
    assert torch.equal(full["trunc"][on], alone["trunc"])
    for k, x, n in (("dhidden", full["dhidden"][on], V), ("dweight", full["dweight"], T)):
        y = alone[k]
        scale = y.abs().amax(dim=-1, keepdim=True) + 1e-30
        # dz may round to the neighbouring bf16 value where log p differs by an ulp
        assert bool(((x - y).abs() <= (2.0 ** -8 + n * 2.0 ** -24) * scale).all()), k
    s, r = (binding.decode_stats(o["stats"]) for o in (full, alone))
    assert s["status"] == r["status"] == binding.CIS_ERR_BAD_TOKEN_ID
    assert s["n_valid"] == r["n_valid"] and s["n_truncated"] == r["n_truncated"]
