// cis_native.cpp -- the binding's calls in native code: argument checks, output
// tensors and the library call of binding.py's functions, without Python's cost
// per tensor.
//
// Bound: the host.  A fused pass of T=256, V=1024 keeps the GPU busy for 13 us,
// and its call took 45 us of Python (checks of five tensors, seven outputs,
// twenty-six converted arguments); from here it takes 17 us, 7.5 of them the
// library's (three launches).
//
// Every function takes its Python counterpart's arguments by position, and
// answers with that function's result; with an int, the library's error; or with
// None where an argument is not what the plain case expects (a tensor of another
// kind, type, shape or device): then nothing was done, and the counterpart goes
// on in Python, where the checks raise.
//
// Data pointers are taken before the GIL is released: a tensor without storage (a
// functorch wrapper, which passes for a plain tensor) raises there.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <string.h>

#include <algorithm>
#include <initializer_list>
#include <utility>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "cis.h"

namespace {

using at::Tensor;

struct Library {
    decltype(&cis_loss_workspace_size) loss_ws = nullptr;
    decltype(&cis_loss_fwd_bwd) loss = nullptr;
    decltype(&cis_token_logprobs) logprobs = nullptr;
    decltype(&cis_weights) weights = nullptr;
    decltype(&cis_binned_sums_workspace_size) bins_ws = nullptr;
    decltype(&cis_binned_sums) bins = nullptr;
    decltype(&cis_mismatch_diagnostics) diagnostics = nullptr;
} lib;

// A tensor argument: None, or a plain tensor (no subclass) with strides.
bool take(PyObject *o, const Tensor *&t)
{
    t = nullptr;
    if (o == Py_None)
        return true;
    if (!THPVariable_CheckExact(o))
        return false;
    t = &THPVariable_Unpack(o);
    return t->defined() && t->layout() == at::kStrided;
}
bool on_gpu(const Tensor *t) { return t == nullptr || t->is_cuda(); }
// None, or a contiguous vector of T elements on the GPU.
bool vec(const Tensor *t, at::ScalarType dt, int64_t T)
{
    return t == nullptr || (t->is_cuda() && t->scalar_type() == dt && t->dim() == 1 &&
                            t->size(0) == T && t->is_contiguous());
}
// Rows with unit column stride: their number and stride.
bool rows(const Tensor &x, int64_t &T, int64_t &ld)
{
    if (x.dim() != 2 || (x.size(1) > 1 && x.stride(1) != 1))
        return false;
    T = x.size(0);
    ld = T > 1 ? x.stride(0) : x.size(1);
    return true;
}
bool dtype_code(at::ScalarType t, int32_t &code)
{
    if (t != at::kBFloat16 && t != at::kFloat)
        return false;
    code = t == at::kBFloat16 ? CIS_BF16 : CIS_F32;
    return true;
}
bool integer(PyObject *o, int64_t &v)
{
    if (!PyLong_CheckExact(o))
        return false;
    int over = 0;
    v = PyLong_AsLongLongAndOverflow(o, &over);
    return over == 0;
}
bool flag(PyObject *o, bool &v)
{
    v = o == Py_True;
    return PyBool_Check(o);
}
// The parameter struct behind a ctypes object of the binding's own type, copied.
PyObject *params_type = nullptr;
bool params(PyObject *o, cis_params_t &p)
{
    Py_buffer b;
    if (reinterpret_cast<PyObject *>(Py_TYPE(o)) != params_type || !PyObject_CheckBuffer(o) ||
        PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        return false;
    }
    const bool ok = b.len == (Py_ssize_t)sizeof(p);
    if (ok)
        memcpy(&p, b.buf, sizeof(p));
    PyBuffer_Release(&b);
    return ok;
}

template <typename T = void> T *ptr(const Tensor *t)
{
    return t ? static_cast<T *>(t->data_ptr()) : nullptr;
}
template <typename T = void> T *ptr(const Tensor &t)
{
    return t.defined() ? ptr<T>(&t) : nullptr;
}
Tensor fresh(at::IntArrayRef shape, at::ScalarType dt, const at::Device &dev)
{
    return at::empty(shape, at::TensorOptions().dtype(dt).device(dev));
}
Tensor fresh_if(bool want, int64_t n, at::ScalarType dt, const at::Device &dev)
{
    return want ? fresh({n}, dt, dev) : Tensor();
}
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject *none() { Py_RETURN_NONE; }
PyObject *wrap(const Tensor &t) { return t.defined() ? THPVariable_Wrap(t) : none(); }
PyObject *dict(std::initializer_list<std::pair<const char *, Tensor>> items)
{
    PyObject *d = PyDict_New();
    for (const auto &it : items) {
        PyObject *v = d ? wrap(it.second) : nullptr;
        if (v == nullptr || PyDict_SetItemString(d, it.first, v) != 0) {
            Py_XDECREF(v);
            Py_XDECREF(d);
            return nullptr;
        }
        Py_DECREF(v);
    }
    return d;
}

// (logits, ids, lp_infer, adv, params, lp_old, mask, cu_seqlens, dlogits,
//  dlogits_dtype, V, want_lp, want_w, want_trunc, workspace, want_entropy)
PyObject *loss_fwd_bwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const Tensor *z, *ids, *lpi, *adv, *old, *mask, *cu, *dz_in, *ws_in;
    cis_params_t P;
    bool want[3], want_ent;
    if (n != 16 || !take(a[0], z) || !take(a[1], ids) || !take(a[2], lpi) || !take(a[3], adv) ||
        !params(a[4], P) || !take(a[5], old) || !take(a[6], mask) || !take(a[7], cu) ||
        !take(a[8], dz_in) || !flag(a[11], want[0]) || !flag(a[12], want[1]) ||
        !flag(a[13], want[2]) || !take(a[14], ws_in) || !flag(a[15], want_ent))
        return none();
    int64_t T, ld, V, To, ldo;
    int32_t code, code_out;
    if (!z || !ids || !lpi || !adv || !z->is_cuda() || !rows(*z, T, ld) ||
        !dtype_code(z->scalar_type(), code) || !vec(ids, at::kInt, T) ||
        !vec(lpi, at::kFloat, T) || !vec(adv, at::kFloat, T) || !vec(old, at::kFloat, T) ||
        !vec(mask, at::kByte, T) || !on_gpu(cu) || !on_gpu(dz_in))
        return none();
    if (cu && (cu->scalar_type() != at::kInt || cu->dim() != 1))
        return none();
    if (a[10] == Py_None)
        V = z->size(1);
    else if (!integer(a[10], V))
        return none();
    at::ScalarType dt = z->scalar_type();
    if (a[9] != Py_None) {
        if (!THPDtype_Check(a[9]))
            return none();
        dt = reinterpret_cast<THPDtype *>(a[9])->scalar_type;
    }
    if (dz_in)
        dt = dz_in->scalar_type();
    if (!dtype_code(dt, code_out) || V < 0)
        return none();
    if (dz_in && (!rows(*dz_in, To, ldo) || To != T || dz_in->size(1) < V))
        return none();
    size_t need = 0;
    if (lib.loss_ws(T, V, &need) != CIS_OK)
        return none();
    const at::Device dev = z->device();
    const Tensor dz = dz_in ? *dz_in : fresh({T, V}, dt, dev);
    rows(dz, To, ldo);
    const Tensor lp = fresh_if(want[0], T, at::kFloat, dev), w = fresh_if(want[1], T, at::kFloat, dev);
    const Tensor tr = fresh_if(want[2], T, at::kByte, dev);
    const Tensor ent = fresh_if(want_ent, T, at::kFloat, dev);
    const Tensor stats = fresh({(int64_t)sizeof(cis_stats_t)}, at::kByte, dev);
    const Tensor loss = fresh({1}, at::kDouble, dev);
    const Tensor ws = ws_in && ws_in->numel() >= (int64_t)need ? *ws_in
                                                               : fresh({(int64_t)need}, at::kByte, dev);
    const void *pz = ptr(z);
    const int32_t *pids = ptr<int32_t>(ids), *pcu = ptr<int32_t>(cu);
    const float *plpi = ptr<float>(lpi), *pold = ptr<float>(old), *padv = ptr<float>(adv);
    const uint8_t *pmask = ptr<uint8_t>(mask);
    const int64_t nseq = cu ? cu->size(0) - 1 : 0;
    void *pdz = ptr(dz), *pws = ptr(ws);
    float *plp = ptr<float>(lp), *pw = ptr<float>(w), *pent = ptr<float>(ent);
    uint8_t *ptrunc = ptr<uint8_t>(tr);
    cis_stats_t *pstats = ptr<cis_stats_t>(stats);
    double *ploss = ptr<double>(loss);
    const size_t nws = (size_t)ws.numel();
    int rc;
    void *s = stream();
    Py_BEGIN_ALLOW_THREADS
    rc = lib.loss(pz, code, T, V, ld, pids, plpi, pold, padv, pmask, pcu, nseq, &P, pdz, code_out,
                  ldo, plp, pw, ptrunc, pent, pstats, ploss, pws, nws, s);
    Py_END_ALLOW_THREADS
    if (rc != CIS_OK)
        return PyLong_FromLong(rc);
    return dict({{"dlogits", dz}, {"lp", lp}, {"w", w}, {"trunc", tr}, {"entropy", ent},
                 {"loss", loss}, {"stats", stats}, {"workspace", ws}});
    END_HANDLE_TH_ERRORS
}

// (logits, ids, mask, V, want_lse, dev_status, want_entropy)
PyObject *token_logprobs(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const Tensor *z, *ids, *mask, *st;
    bool want_lse, want_ent;
    if (n != 7 || !take(a[0], z) || !take(a[1], ids) || !take(a[2], mask) ||
        !flag(a[4], want_lse) || !take(a[5], st) || !flag(a[6], want_ent))
        return none();
    int64_t T, ld, V;
    int32_t code;
    if (!z || !ids || !z->is_cuda() || !rows(*z, T, ld) || !dtype_code(z->scalar_type(), code) ||
        !vec(ids, at::kInt, T) || !vec(mask, at::kByte, T))
        return none();
    if (a[3] == Py_None)
        V = z->size(1);
    else if (!integer(a[3], V))
        return none();
    const at::Device dev = z->device();
    const Tensor lp = fresh({T}, at::kFloat, dev), lse = fresh_if(want_lse, T, at::kFloat, dev);
    const Tensor ent = fresh_if(want_ent, T, at::kFloat, dev);
    const void *pz = ptr(z);
    const int32_t *pids = ptr<int32_t>(ids);
    const uint8_t *pmask = ptr<uint8_t>(mask);
    float *plp = ptr<float>(lp), *plse = ptr<float>(lse), *pent = ptr<float>(ent);
    int32_t *pst = ptr<int32_t>(st);
    int rc;
    void *s = stream();
    Py_BEGIN_ALLOW_THREADS
    rc = lib.logprobs(pz, code, T, V, ld, pids, pmask, plp, plse, pent, pst, s);
    Py_END_ALLOW_THREADS
    if (rc != CIS_OK)
        return PyLong_FromLong(rc);
    if (want_ent)
        return Py_BuildValue("NNN", wrap(lp), wrap(lse), wrap(ent));
    return want_lse ? Py_BuildValue("NN", wrap(lp), wrap(lse)) : wrap(lp);
    END_HANDLE_TH_ERRORS
}

// (lp_train, lp_infer, params, mask, want_trunc, want_eps, cu_seqlens)
PyObject *weights(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const Tensor *lt, *li, *mask, *cu;
    cis_params_t P;
    bool want_tr, want_eps;
    if (n != 7 || !take(a[0], lt) || !take(a[1], li) || !params(a[2], P) || !take(a[3], mask) ||
        !flag(a[4], want_tr) || !flag(a[5], want_eps) || !take(a[6], cu))
        return none();
    if (!lt || !li || lt->dim() != 1)
        return none();
    const int64_t T = lt->size(0);
    if (!vec(lt, at::kFloat, T) || !vec(li, at::kFloat, T) || !vec(mask, at::kByte, T))
        return none();
    if (cu && (!cu->is_cuda() || cu->scalar_type() != at::kInt || cu->dim() != 1 ||
               !cu->is_contiguous()))
        return none();
    const at::Device dev = lt->device();
    const Tensor w = fresh({T}, at::kFloat, dev), tr = fresh_if(want_tr, T, at::kByte, dev);
    const Tensor eps = fresh_if(want_eps, T, at::kFloat, dev);
    const float *plt = ptr<float>(lt), *pli = ptr<float>(li);
    const uint8_t *pmask = ptr<uint8_t>(mask);
    const int32_t *pcu = ptr<int32_t>(cu);
    const int64_t nseq = cu ? cu->size(0) - 1 : 0;
    float *pw = ptr<float>(w), *peps = ptr<float>(eps);
    uint8_t *ptrunc = ptr<uint8_t>(tr);
    int rc;
    void *s = stream();
    Py_BEGIN_ALLOW_THREADS
    rc = lib.weights(plt, pli, pmask, T, pcu, nseq, &P, pw, ptrunc, peps, s);
    Py_END_ALLOW_THREADS
    if (rc != CIS_OK)
        return PyLong_FromLong(rc);
    return Py_BuildValue("NNN", wrap(w), wrap(tr), wrap(eps));
    END_HANDLE_TH_ERRORS
}

// (key, edges, values, mask): edges a list or tuple of floats or ints, values
// one of tensors
PyObject *binned_sums(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const Tensor *key, *mask, *v;
    if (n != 4 || !take(a[0], key) || !take(a[3], mask) || !key || key->dim() != 1 ||
        !(PyList_CheckExact(a[1]) || PyTuple_CheckExact(a[1])) ||
        !(PyList_CheckExact(a[2]) || PyTuple_CheckExact(a[2])))
        return none();
    const int64_t T = key->size(0);
    const Py_ssize_t ne = PySequence_Fast_GET_SIZE(a[1]), nv = PySequence_Fast_GET_SIZE(a[2]);
    if (!vec(key, at::kFloat, T) || !vec(mask, at::kByte, T) || ne < 2 || ne > CIS_MAX_BINS + 1 ||
        nv > CIS_MAX_BIN_VALUES)
        return none();
    double edges[CIS_MAX_BINS + 1];
    for (Py_ssize_t i = 0; i < ne; ++i) {
        PyObject *e = PySequence_Fast_GET_ITEM(a[1], i);
        if (!PyFloat_CheckExact(e))
            return none();
        edges[i] = PyFloat_AS_DOUBLE(e);
    }
    const float *vals[CIS_MAX_BIN_VALUES] = {};
    for (Py_ssize_t i = 0; i < nv; ++i) {
        if (!take(PySequence_Fast_GET_ITEM(a[2], i), v) || !v || !vec(v, at::kFloat, T))
            return none();
        vals[i] = ptr<float>(v);
    }
    const int32_t nb = (int32_t)ne - 1;
    size_t need = 0;
    if (lib.bins_ws(T, nb, (int32_t)nv, &need) != CIS_OK)
        return none();
    const at::Device dev = key->device();
    const Tensor ws = fresh({(int64_t)need + 256}, at::kByte, dev);
    const Tensor counts = fresh({(int64_t)nb}, at::kLong, dev);
    const Tensor sums = fresh({(int64_t)nv, (int64_t)nb}, at::kDouble, dev);
    uint8_t *w = ptr<uint8_t>(ws);
    w += (256 - (reinterpret_cast<uintptr_t>(w) & 255)) & 255;
    const float *pkey = ptr<float>(key);
    const uint8_t *pmask = ptr<uint8_t>(mask);
    int64_t *pcounts = ptr<int64_t>(counts);
    double *psums = nv ? ptr<double>(sums) : nullptr;
    int rc;
    void *s = stream();
    Py_BEGIN_ALLOW_THREADS
    rc = lib.bins(pkey, pmask, T, edges, nb, nv ? vals : nullptr, (int32_t)nv, pcounts, psums, w,
                  need, s);
    Py_END_ALLOW_THREADS
    if (rc != CIS_OK)
        return PyLong_FromLong(rc);
    return Py_BuildValue("NN", wrap(counts), wrap(sums));
    END_HANDLE_TH_ERRORS
}

// (logits_train, logits_infer, ids, params, mask, V, dev_status)
PyObject *mismatch_diagnostics(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const Tensor *zt, *zi, *ids, *mask, *st;
    cis_params_t P;
    if (n != 7 || !take(a[0], zt) || !take(a[1], zi) || !take(a[2], ids) || !params(a[3], P) ||
        !take(a[4], mask) || !take(a[6], st))
        return none();
    int64_t T, Ti, ldt, ldi, V;
    int32_t code;
    if (!zt || !zi || !ids || !zt->is_cuda() || !zi->is_cuda() ||
        zt->scalar_type() != zi->scalar_type() || !rows(*zt, T, ldt) || !rows(*zi, Ti, ldi) ||
        Ti != T || !dtype_code(zt->scalar_type(), code) || !vec(ids, at::kInt, T) ||
        !vec(mask, at::kByte, T))
        return none();
    if (a[5] == Py_None)
        V = std::min(zt->size(1), zi->size(1));
    else if (!integer(a[5], V))
        return none();
    const at::Device dev = zt->device();
    Tensor o[5];
    for (Tensor &t : o)
        t = fresh({T}, at::kFloat, dev);
    const void *pzt = ptr(zt), *pzi = ptr(zi);
    const int32_t *pids = ptr<int32_t>(ids);
    const uint8_t *pmask = ptr<uint8_t>(mask);
    float *po[5];
    for (int i = 0; i < 5; ++i)
        po[i] = ptr<float>(o[i]);
    int32_t *pst = ptr<int32_t>(st);
    int rc;
    void *s = stream();
    Py_BEGIN_ALLOW_THREADS
    rc = lib.diagnostics(pzt, pzi, code, T, V, ldt, ldi, pids, pmask, &P, po[0], po[1], po[2],
                         po[3], po[4], pst, s);
    Py_END_ALLOW_THREADS
    if (rc != CIS_OK)
        return PyLong_FromLong(rc);
    return dict({{"eps", o[0]}, {"logk", o[1]}, {"p", o[2]}, {"bias2", o[3]}, {"dvar", o[4]}});
    END_HANDLE_TH_ERRORS
}

// init(path, params type): the library's entry points, and the type of `params`.
PyObject *init(PyObject *, PyObject *args)
{
    const char *path;
    PyObject *type;
    if (!PyArg_ParseTuple(args, "sO", &path, &type))
        return nullptr;
    void *h = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (h == nullptr)
        return PyErr_Format(PyExc_ImportError, "%s", dlerror());
    bool ok = true;
    auto get = [&](auto &f, const char *name) {
        f = reinterpret_cast<std::decay_t<decltype(f)>>(dlsym(h, name));
        ok = ok && f != nullptr;
    };
    get(lib.loss_ws, "cis_loss_workspace_size");
    get(lib.loss, "cis_loss_fwd_bwd");
    get(lib.logprobs, "cis_token_logprobs");
    get(lib.weights, "cis_weights");
    get(lib.bins_ws, "cis_binned_sums_workspace_size");
    get(lib.bins, "cis_binned_sums");
    get(lib.diagnostics, "cis_mismatch_diagnostics");
    if (!ok)
        return PyErr_Format(PyExc_ImportError, "%s lacks an entry point", path);
    Py_INCREF(type);
    Py_XSETREF(params_type, type);
    return none();
}

template <typename F> PyCFunction fast(F f)
{
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}
PyMethodDef methods[] = {
    {"init", init, METH_VARARGS, nullptr},
    {"loss_fwd_bwd", fast(loss_fwd_bwd), METH_FASTCALL, nullptr},
    {"token_logprobs", fast(token_logprobs), METH_FASTCALL, nullptr},
    {"weights", fast(weights), METH_FASTCALL, nullptr},
    {"binned_sums", fast(binned_sums), METH_FASTCALL, nullptr},
    {"mismatch_diagnostics", fast(mismatch_diagnostics), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cis_native", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cis_native() { return PyModule_Create(&module); }
