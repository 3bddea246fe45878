// CPython extension behind binding.py: argument checks, output allocation and the call into the C ABI in native code.
//
// A decode step or a short prompt spends a few microseconds on the GPU; marshalling its arguments through ctypes and checking
// them in Python took longer than that (decode step, B = 1: 12 us per call from Python, host-bound).  Each function here
// handles the calls whose arguments pass its checks and returns the outputs.  For anything else it does not call the library and
// returns None, and binding.py runs its checked path, which names the argument that is wrong.  A status of the library is raised
// here: the call may have launched kernels that update state in place, so it must not be made a second time.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "rglru.h"

namespace {

struct ParamsHandle {
    rglru_params_t p;
    int32_t H, D, io;
    at::ScalarType dtype;
    c10::Device device;
};
const char *const HANDLE = "rglru.params";

// A tensor argument or None; `bad` is set for anything else.
const at::Tensor *tensor_arg(PyObject *o, bool &bad) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { bad = true; return nullptr; }
    return &THPVariable_Unpack(o);
}
// Absent, or contiguous with this shape, dtype and device
bool fits(const at::Tensor *t, at::IntArrayRef shape, at::ScalarType dtype, c10::Device dev) {
    return t == nullptr || (t->scalar_type() == dtype && t->device() == dev && t->sizes() == shape && t->is_contiguous());
}
void *ptr(const at::Tensor *t) { return t ? t->data_ptr() : nullptr; }
at::Tensor fresh(at::IntArrayRef shape, at::ScalarType dtype, c10::Device dev) {
    return at::Tensor(at::detail::empty_cuda(shape, dtype, dev, std::nullopt));
}
void *current_stream() { return (void *)c10::cuda::getCurrentCUDAStream().stream(); }
PyObject *wrap(const at::Tensor &t) { return THPVariable_Wrap(t); }

// binding.py's exception type for a status of the library, RglruError(code, where)
PyObject *error_type = nullptr;
PyObject *raise_status(int32_t rc, const char *where) {
    PyObject *e = PyObject_CallFunction(error_type ? error_type : PyExc_RuntimeError, "is", (int)rc, where);
    if (e) { PyErr_SetObject((PyObject *)Py_TYPE(e), e); Py_DECREF(e); }
    return nullptr;
}
PyObject *set_error_type(PyObject *, PyObject *type) {
    Py_INCREF(type);
    Py_XSETREF(error_type, type);
    Py_RETURN_NONE;
}

// Workspace of the call: the caller's, or scratch of this call (the library needs no particular contents)
struct Workspace {
    at::Tensor own;
    void *p = nullptr;
    size_t n = 0;
    bool take(const at::Tensor *given, const rglru_shape_t &s, int op, c10::Device dev) {
        if (given) { p = given->data_ptr(); n = (size_t)given->numel(); return true; }
        n = rglru_workspace_bytes(&s, op);
        if (n == 0) return false;
        own = fresh({(int64_t)n}, at::kByte, dev);
        p = own.data_ptr();
        return true;
    }
};

// The call into the library without the interpreter lock: a launch can block (a full queue, a first use that loads code), and other
// Python threads go on meanwhile.  The tensors stay alive: the caller's arguments hold them.
template <typename F> int32_t unlocked(F &&call) {
    int32_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

struct Call {
    const ParamsHandle *h = nullptr;
    rglru_shape_t s{};
    bool begin(PyObject *handle, PyObject *c, PyObject *flags, const at::Tensor *x, int dims) {
        h = (const ParamsHandle *)PyCapsule_GetPointer(handle, HANDLE);
        if (!h) { PyErr_Clear(); return false; }
        if (!x || x->dim() != dims || x->scalar_type() != h->dtype || x->device() != h->device || !x->is_contiguous()) return false;
        if (!h->device.is_cuda() || x->size(dims - 1) != h->D) return false;
        for (int i = 0; i < dims; ++i)
            if (x->size(i) > INT32_MAX) return false;
        const double cv = PyFloat_AsDouble(c);
        const unsigned long fv = PyLong_AsUnsignedLong(flags);
        if (PyErr_Occurred()) { PyErr_Clear(); return false; }
        s.B = (int32_t)x->size(0); s.T = dims == 3 ? (int32_t)x->size(1) : 1; s.D = h->D; s.H = h->H;
        s.io = h->io; s.c = (float)cv; s.flags = (uint32_t)fv;
        return true;
    }
};

// params_handle(conv_w, conv_b, W_a, b_a, W_x, b_x, lam) of tensors that binding.Params has checked and keeps alive
PyObject *params_handle(PyObject *, PyObject *const *a, Py_ssize_t n) {
    bool bad = n != 7;
    const at::Tensor *t[7] = {};
    for (int i = 0; !bad && i < 7; ++i) t[i] = tensor_arg(a[i], bad);
    if (bad || !t[0] || !t[2] || !t[3] || !t[4] || !t[5] || !t[6] || t[2]->dim() != 3 || t[0]->dim() != 2) Py_RETURN_NONE;
    ParamsHandle *h = new ParamsHandle{{ptr(t[0]), (const float *)ptr(t[1]), ptr(t[2]), (const float *)ptr(t[3]), ptr(t[4]), (const float *)ptr(t[5]),
                                        (const float *)ptr(t[6])},
                                       (int32_t)t[2]->size(0), (int32_t)t[0]->size(1),
                                       t[0]->scalar_type() == at::kBFloat16 ? (int32_t)RGLRU_BF16 : (int32_t)RGLRU_F32, t[0]->scalar_type(), t[0]->device()};
    PyObject *cap = PyCapsule_New(h, HANDLE, [](PyObject *c) { delete (ParamsHandle *)PyCapsule_GetPointer(c, HANDLE); });
    if (!cap) delete h;
    return cap;
}

// prefill(handle, x, h0, conv_state_in, c, flags, y, h_T, conv_state_out, workspace, gate_branch, a_prod) -> (y, h_T, conv_state_out)
PyObject *prefill(PyObject *, PyObject *const *a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 12) Py_RETURN_NONE;
    bool bad = false;
    const at::Tensor *x = tensor_arg(a[1], bad), *h0 = tensor_arg(a[2], bad), *cs = tensor_arg(a[3], bad), *y = tensor_arg(a[6], bad),
                     *hT = tensor_arg(a[7], bad), *cso = tensor_arg(a[8], bad), *ws = tensor_arg(a[9], bad), *gb = tensor_arg(a[10], bad),
                     *ap = tensor_arg(a[11], bad);
    Call k;
    if (bad || !k.begin(a[0], a[4], a[5], x, 3)) Py_RETURN_NONE;
    const c10::Device dev = k.h->device;
    const at::ScalarType io = k.h->dtype;
    const int64_t B = k.s.B, T = k.s.T, D = k.s.D;
    if (!fits(h0, {B, D}, at::kFloat, dev) || !fits(cs, {B, 3, D}, io, dev) || !fits(y, {B, T, D}, io, dev) || !fits(hT, {B, D}, at::kFloat, dev) ||
        !fits(cso, {B, 3, D}, io, dev) || !fits(gb, {B, T, D}, io, dev) || !fits(ap, {B, D}, at::kFloat, dev))
        Py_RETURN_NONE;
    const at::Tensor yt = y ? *y : fresh({B, T, D}, io, dev), ht = hT ? *hT : fresh({B, D}, at::kFloat, dev), ct = cso ? *cso : fresh({B, 3, D}, io, dev);
    Workspace w;
    if (!w.take(ws, k.s, RGLRU_OP_PREFILL, dev)) Py_RETURN_NONE;
    const rglru_prefill_extras_t ex{ptr(gb), (float *)ptr(ap)};
    void *const st = current_stream();
    const int32_t rc = unlocked([&] {
        return rglru_prefill_ex(&k.s, &k.h->p, ptr(x), (const float *)ptr(h0), ptr(cs), yt.data_ptr(), (float *)ht.data_ptr(), ct.data_ptr(),
                                gb || ap ? &ex : nullptr, w.p, w.n, st);
    });
    if (rc != RGLRU_OK) return raise_status(rc, "rglru_prefill");
    PyObject *out = PyTuple_New(3);
    if (!out) return nullptr;
    PyTuple_SET_ITEM(out, 0, wrap(yt)); PyTuple_SET_ITEM(out, 1, wrap(ht)); PyTuple_SET_ITEM(out, 2, wrap(ct));
    return out;
    END_HANDLE_TH_ERRORS
}

// decode_step(handle, x, h, conv_state, c, flags, y, workspace) -> y
PyObject *decode_step(PyObject *, PyObject *const *a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 8) Py_RETURN_NONE;
    bool bad = false;
    const at::Tensor *x = tensor_arg(a[1], bad), *h = tensor_arg(a[2], bad), *cs = tensor_arg(a[3], bad), *y = tensor_arg(a[6], bad), *ws = tensor_arg(a[7], bad);
    Call k;
    if (bad || !h || !cs || !k.begin(a[0], a[4], a[5], x, 2)) Py_RETURN_NONE;
    const c10::Device dev = k.h->device;
    const at::ScalarType io = k.h->dtype;
    const int64_t B = k.s.B, D = k.s.D;
    if (!fits(h, {B, D}, at::kFloat, dev) || !fits(cs, {B, 3, D}, io, dev) || !fits(y, {B, D}, io, dev)) Py_RETURN_NONE;
    const at::Tensor yt = y ? *y : fresh({B, D}, io, dev);
    Workspace w;
    if (!w.take(ws, k.s, RGLRU_OP_DECODE, dev)) Py_RETURN_NONE;
    void *const st = current_stream();
    const int32_t rc = unlocked([&] { return rglru_decode_step(&k.s, &k.h->p, ptr(x), (float *)ptr(h), ptr(cs), yt.data_ptr(), w.p, w.n, st); });
    if (rc != RGLRU_OK) return raise_status(rc, "rglru_decode_step");
    if (y) { Py_INCREF(a[6]); return a[6]; }
    return wrap(yt);
    END_HANDLE_TH_ERRORS
}

// backward(handle, x, dy, h0, conv_state_in, y, c, flags, workspace, dh_T, dconv_state_out, state_grads) -> dict of gradients
PyObject *backward(PyObject *, PyObject *const *a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 12) Py_RETURN_NONE;
    bool bad = false;
    const at::Tensor *x = tensor_arg(a[1], bad), *dy = tensor_arg(a[2], bad), *h0 = tensor_arg(a[3], bad), *cs = tensor_arg(a[4], bad), *y = tensor_arg(a[5], bad),
                     *ws = tensor_arg(a[8], bad), *dhT = tensor_arg(a[9], bad), *dcs = tensor_arg(a[10], bad);
    const int want_state = PyObject_IsTrue(a[11]);
    Call k;
    if (bad || want_state < 0 || !dy || !k.begin(a[0], a[6], a[7], x, 3)) { PyErr_Clear(); Py_RETURN_NONE; }
    const c10::Device dev = k.h->device;
    const at::ScalarType io = k.h->dtype;
    const int64_t B = k.s.B, T = k.s.T, D = k.s.D, H = k.s.H, Dh = D / H;
    if (!fits(dy, {B, T, D}, io, dev) || !fits(h0, {B, D}, at::kFloat, dev) || !fits(cs, {B, 3, D}, io, dev) || !fits(y, {B, T, D}, io, dev) ||
        !fits(dhT, {B, D}, at::kFloat, dev) || !fits(dcs, {B, 3, D}, io, dev))
        Py_RETURN_NONE;
    Workspace w;
    if (!w.take(ws, k.s, RGLRU_OP_BACKWARD, dev)) Py_RETURN_NONE;
    const char *const names[10] = {"x", "conv_w", "conv_b", "W_a", "b_a", "W_x", "b_x", "lam", "h0", "conv_state"};
    const int count = want_state ? 10 : 8;
    at::Tensor g[10] = {fresh({B, T, D}, io, dev), fresh({4, D}, at::kFloat, dev), fresh({D}, at::kFloat, dev), fresh({H, Dh, Dh}, at::kFloat, dev),
                        fresh({D}, at::kFloat, dev), fresh({H, Dh, Dh}, at::kFloat, dev), fresh({D}, at::kFloat, dev), fresh({D}, at::kFloat, dev)};
    if (want_state) { g[8] = fresh({B, D}, at::kFloat, dev); g[9] = fresh({B, 3, D}, io, dev); }
    const rglru_state_grads_t sg{(const float *)ptr(dhT), ptr(dcs), want_state ? (float *)g[8].data_ptr() : nullptr, want_state ? g[9].data_ptr() : nullptr};
    auto f = [&](int i) { return (float *)g[i].data_ptr(); };
    void *const st = current_stream();
    const int32_t rc = unlocked([&] {
        return rglru_backward(&k.s, &k.h->p, ptr(x), (const float *)ptr(h0), ptr(cs), ptr(y), ptr(dy), g[0].data_ptr(), f(1), f(2), f(3), f(4), f(5), f(6), f(7),
                              want_state || dhT || dcs ? &sg : nullptr, w.p, w.n, st);
    });
    if (rc != RGLRU_OK) return raise_status(rc, "rglru_backward");
    PyObject *out = PyDict_New();
    if (!out) return nullptr;
    for (int i = 0; i < count; ++i) {
        PyObject *t = wrap(g[i]);
        PyDict_SetItemString(out, names[i], t);
        Py_DECREF(t);
    }
    return out;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"set_error_type", set_error_type, METH_O, nullptr},
    {"params_handle", (PyCFunction)(void (*)(void))params_handle, METH_FASTCALL, nullptr},
    {"prefill", (PyCFunction)(void (*)(void))prefill, METH_FASTCALL, nullptr},
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, nullptr},
    {"backward", (PyCFunction)(void (*)(void))backward, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host(void) { return PyModule_Create(&module); }
