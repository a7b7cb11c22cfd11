"""The fused pass's kernels overlap one another (programmatic dependent launch)
within a call: back-to-back calls that share one workspace, and calls replayed
from a CUDA graph, give the outputs of calls that were waited for, bit for bit.
"""
import pytest
import torch

from paper_2609_32444_gb300 import binding, synth

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

DEV = torch.device("cuda")
KEYS = ("dlogits", "lp", "w", "trunc", "loss", "stats")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


def _inputs(T, V, seed, all_masked=False):
    b = synth.make_batch(2, T=T, V=V, seed=seed)
    if all_masked:
        b.mask.zero_()
    else:
        b.mask[::3] = 0
    b.ids[5] = V + 1  # a bad id: its status bit must survive the clearing kernel
    return [x.to(DEV) for x in (b.logits, b.ids, b.lp_infer, b.adv, b.mask, b.cu_seqlens)]


def _call(x, P, ws):
    z, ids, lp, adv, mask, cu = x
    return binding.cis_loss_fwd_bwd(z, ids, lp, adv, P, mask=mask, cu_seqlens=cu, workspace=ws)


@pytest.mark.parametrize("mode,agg", [("cis", 0), ("tis", 1), ("seq_tis", 0), ("kpop", 1)])
@pytest.mark.parametrize("T,V", [(33, 1024), (1500, 4096), (700, 2049)])
def test_back_to_back_calls_share_a_workspace(T, V, mode, agg):
    """40 calls on three batches in turn (one of them all masked, so that none
    of its rows needs the normaliser) without a wait between them."""
    P = binding.cis_default_params(mode)
    P.agg = agg
    xs = [_inputs(T, V, 1), _inputs(T, V, 2, all_masked=True), _inputs(T, V, 3)]
    ws = torch.empty(binding.cis_loss_workspace_size(T, V), dtype=torch.uint8, device=DEV)
    want = []
    for x in xs:
        o = _call(x, P, ws)
        torch.cuda.synchronize()
        want.append({k: o[k].clone() for k in KEYS})
    got = [(i % 3, _call(xs[i % 3], P, ws)) for i in range(40)]
    torch.cuda.synchronize()
    for i, o in got:
        for k in KEYS:
            assert torch.equal(o[k].view(torch.uint8), want[i][k].view(torch.uint8)), (i, k)
    assert binding.decode_stats(want[0]["stats"])["status"] == binding.CIS_ERR_BAD_TOKEN_ID
    assert binding.decode_stats(want[1]["stats"])["n_valid"] == 0


@pytest.mark.parametrize("mode", ["cis", "seq_mis"])
def test_graph_replay(mode):
    """A captured call replayed on new values in the captured buffers."""
    T, V = 300, 4096
    P = binding.cis_default_params(mode)
    a, b = _inputs(T, V, 4), _inputs(T, V, 5)
    want = {k: v.clone() for k, v in _call(b, P, None).items() if k in KEYS}
    ws = torch.empty(binding.cis_loss_workspace_size(T, V), dtype=torch.uint8, device=DEV)
    x = [t.clone() for t in a]
    _call(x, P, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        o = _call(x, P, ws)
    for _ in range(3):
        for t, v in zip(x, b):
            t.copy_(v)
        g.replay()
    torch.cuda.synchronize()
    for k in KEYS:
        assert torch.equal(o[k].view(torch.uint8), want[k].view(torch.uint8)), k
