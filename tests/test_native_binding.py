"""The binding's native calls against its Python ones: the same results where
both make the call, and the same refusals (what the native part does not take
goes on to the Python code, whose checks raise).
"""
import contextlib
import ctypes
import threading
import time

import pytest
import torch

from paper_2609_32444_gb300 import binding, synth

DEV = torch.device("cuda")
gpu = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_32444_gb300 import build
    build.build()
    binding.lib()


class _Python:
    """Stands in for the native module: every call goes on in Python."""

    def __getattr__(self, name):
        return lambda *a: None


@contextlib.contextmanager
def _python_only():
    kept = binding._native
    binding._native = _Python()
    try:
        yield
    finally:
        binding._native = kept


def _same(a, b):
    assert type(a) is type(b)
    if isinstance(a, dict):
        assert list(a) == list(b)
        for k in a:
            if k != "workspace":
                _same(a[k], b[k])
    elif isinstance(a, (tuple, list)):
        assert len(a) == len(b)
        for x, y in zip(a, b):
            _same(x, y)
    elif a is not None:
        assert a.dtype == b.dtype and a.shape == b.shape and a.device == b.device
        assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


def _both(f):
    x = f()
    with _python_only():
        y = f()
    torch.cuda.synchronize()
    _same(x, y)


def _args():
    b = synth.make_batch(2, T=200, V=1024)
    b.mask[::3] = 0
    return {k: getattr(b, k).to(DEV) for k in ("logits", "ids", "lp_infer", "adv", "mask",
                                              "cu_seqlens")}


class TestOnGpu:
    pytestmark = gpu

    @pytest.mark.parametrize("kw", [
        {}, {"want_lp": False, "want_trunc": False}, {"want_w": False, "want_entropy": True},
        {"dlogits_dtype": torch.float32}, {"V": 1000}, {"mask": None, "cu_seqlens": None}])
    def test_loss(self, kw):
        x = _args()
        P = binding.cis_default_params("cis")
        kw = dict({"mask": x["mask"], "cu_seqlens": x["cu_seqlens"]}, **kw)
        _both(lambda: binding.cis_loss_fwd_bwd(x["logits"], x["ids"], x["lp_infer"], x["adv"], P,
                                               **kw))
        dz = torch.empty((200, 1030), dtype=torch.float32, device=DEV)
        ws = torch.empty(1 << 20, dtype=torch.uint8, device=DEV)
        _both(lambda: {k: v.clone() if k == "dlogits" else v for k, v in binding.cis_loss_fwd_bwd(
            x["logits"], x["ids"], x["lp_infer"], x["adv"], P, lp_old=x["lp_infer"],
            dlogits=dz.zero_(), workspace=ws, **{k: v for k, v in kw.items()
                                                 if k in ("mask", "cu_seqlens")}).items()})

    def test_other_calls(self):
        x = _args()
        P = binding.cis_default_params("tis")
        lp = binding.cis_token_logprobs(x["logits"], x["ids"])
        for kw in ({}, {"want_lse": True}, {"want_entropy": True, "mask": x["mask"]},
                   {"want_lse": True, "want_entropy": True, "V": 1000}):
            _both(lambda: binding.cis_token_logprobs(x["logits"], x["ids"], **kw))
        for kw in ({}, {"want_trunc": False, "want_eps": True, "mask": x["mask"]}):
            _both(lambda: binding.cis_weights(lp, x["lp_infer"], P, **kw))
        _both(lambda: binding.cis_weights(lp, x["lp_infer"], binding.cis_default_params("seq_mis"),
                                          cu_seqlens=x["cu_seqlens"]))
        for e, v in (([0.0, 0.5, 1.0], (lp, lp)), ((0, 1), ()), ([-50.0, -1, 0.0], [lp])):
            _both(lambda: binding.cis_binned_sums(lp, e, v, mask=x["mask"]))
        _both(lambda: binding.cis_mismatch_diagnostics(x["logits"], x["logits"], x["ids"], P,
                                                       mask=x["mask"]))

    def test_refusals(self):
        """Wrong kinds, types, shapes and strides, and the library's own errors."""
        x = _args()
        P = binding.cis_default_params("cis")
        z, ids, li, adv = x["logits"], x["ids"], x["lp_infer"], x["adv"]
        loss = binding.cis_loss_fwd_bwd
        calls = [
            lambda: loss(z.half(), ids, li, adv, P), lambda: loss(z, ids.long(), li, adv, P),
            lambda: loss(z, ids, li[:-1], adv, P), lambda: loss(z.t(), ids, li, adv, P),
            lambda: loss(z, ids, li, adv, bytes(200)), lambda: loss(z, ids, li, adv.cpu(), P),
            lambda: loss(z, ids, li, adv, P, V=2000), lambda: loss(z, ids, li, adv, P, V=-1),
            lambda: loss(z, ids, li, adv, P, dlogits_dtype=torch.float16),
            lambda: loss(z, ids, li, adv, P, dlogits=torch.empty((200, 8), device=DEV)),
            lambda: loss(z, ids, li, adv, binding.cis_default_params("seq_tis")),
            lambda: loss(z, ids, li, adv, binding.cis_default_params("cis", lam=-1.0)),
            lambda: binding.cis_token_logprobs(z[0], ids), lambda: binding.cis_weights(li, None, P),
            lambda: binding.cis_binned_sums(li, [0.5, 0.5]),
            lambda: binding.cis_binned_sums(li, [0.0, 1.0], (li.double(),)),
            lambda: binding.cis_mismatch_diagnostics(z, z.float(), ids, P)]
        for i, f in enumerate(calls):
            errors = []
            for python in (False, True):
                with _python_only() if python else contextlib.nullcontext():
                    with pytest.raises(Exception) as e:
                        f()
                    errors.append((type(e.value), str(e.value)))
            assert errors[0] == errors[1], (i, errors)

    def test_another_type_of_the_same_name_is_refused(self):
        x = _args()
        other = type("cis_params_t", (ctypes.Structure,),
                     {"_fields_": [("b", ctypes.c_uint8 * ctypes.sizeof(binding.cis_params_t))]})
        for python in (False, True):
            with _python_only() if python else contextlib.nullcontext():
                with pytest.raises(ctypes.ArgumentError):
                    binding.cis_weights(x["lp_infer"], x["lp_infer"], other())

    @pytest.mark.parametrize("call", ["loss", "logprobs", "weights", "bins", "diagnostics"])
    @pytest.mark.parametrize("transform", ["vmap", "grad"])
    def test_tensors_without_storage(self, call, transform):
        """A functorch wrapper passes for a plain tensor and has no data pointer: the
        calls raise what the Python code raises."""
        P = binding.cis_default_params("cis")
        z = torch.randn(3, 4, 8, device=DEV)
        ids, v = torch.zeros(4, dtype=torch.int32, device=DEV), torch.zeros(4, device=DEV)
        f = {"loss": lambda x: binding.cis_loss_fwd_bwd(x, ids, v, v, P)["loss"],
             "logprobs": lambda x: binding.cis_token_logprobs(x, ids),
             "weights": lambda x: binding.cis_weights(x[:, 0].contiguous(), v, P)[0],
             "bins": lambda x: binding.cis_binned_sums(x[:, 0].contiguous(), [0.0, 1.0])[1],
             "diagnostics": lambda x: binding.cis_mismatch_diagnostics(x, x, ids, P)["p"]}[call]
        for python in (False, True):
            with _python_only() if python else contextlib.nullcontext():
                with pytest.raises(RuntimeError, match="doesn't have storage"):
                    if transform == "vmap":
                        torch.vmap(f)(z)
                    else:
                        torch.func.grad(lambda x: f(x).sum())(z[0])


def test_host_tensors_are_refused_as_before():
    z, ids, v = torch.zeros(4, 8), torch.zeros(4, dtype=torch.int32), torch.zeros(4)
    P = binding.cis_default_params("cis")
    for f in (lambda: binding.cis_loss_fwd_bwd(z, ids, v, v, P),
              lambda: binding.cis_token_logprobs(z, ids), lambda: binding.cis_weights(v, v, P),
              lambda: binding.cis_mismatch_diagnostics(z, z, ids, P),
              lambda: binding.cis_binned_sums(v, [0.0, 1.0])):
        with pytest.raises(ValueError, match="libcis takes CUDA tensors"):
            f()


def test_threads_meet_a_whole_library(monkeypatch):
    """Calls from several threads while the library loads: none sees it without its
    native part; after a failed load every call raises the load's error."""
    z, ids = torch.zeros(4, 8), torch.zeros(4, dtype=torch.int32)
    load = binding._load_native

    def slow(path):
        time.sleep(0.2)
        load(path)

    monkeypatch.setattr(binding, "_load_native", slow)
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_native", None)
    errors = []

    def call():
        try:
            binding.cis_token_logprobs(z, ids)
        except Exception as e:
            errors.append((type(e), str(e)))

    threads = [threading.Thread(target=call) for _ in range(3)]
    for t in threads:
        t.start()
        time.sleep(0.02)
    for t in threads:
        t.join()
    assert errors == [(ValueError, "libcis takes CUDA tensors")] * 3

    def fail(path):
        raise ImportError("no native part")

    monkeypatch.setattr(binding, "_load_native", fail)
    monkeypatch.setattr(binding, "_lib", None)
    for _ in range(2):
        with pytest.raises(ImportError, match="no native part"):
            binding.cis_token_logprobs(z, ids)


def test_without_the_native_part(monkeypatch):
    """A tree built for another PyTorch: a warning, and the Python code's calls."""
    monkeypatch.setattr(binding._build, "native_path", lambda: "/nonexistent/_cis_native.so")
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_native", None)
    with pytest.warns(RuntimeWarning, match="is not built"):
        assert binding.lib() is not None
    test_host_tensors_are_refused_as_before()
    assert binding.cis_default_params("tis").mode == binding.CIS_MODE_TIS
