// The host side of one call, native: checks the tensors, makes the outputs, asks torch for the current
// stream and calls an entry point of libdualdiff.so by its address.  binding.py does the same in Python, at
// 8 to 13 us a call, which is more than the small launches take on the device; it remains for everything
// this file does not take: another stream, host buffers, subclasses of torch.Tensor (FakeTensor among
// them) and tensors without storage, calls under a torch function or dispatch mode, tensors that are not as
// they should be, and whatever throws before the launch (an allocation that fails).  The functions below
// then return None, having launched nothing, and the words of the error are the binding's.
// Marshalling only: no arithmetic of the method.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <cstdint>

namespace {

constexpr int kMaxDims = 4;

struct Shape {
    int64_t d[kMaxDims];
    int n;
};

// A torch.Tensor or torch.nn.Parameter itself: what a subclass makes of a call is decided in Python.
const at::Tensor *tensor_of(PyObject *o) { return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr; }

// No mode that would have a say in what torch.empty or Tensor.data_ptr do here.
bool plain_call() { return !at::impl::torch_function_mode_enabled() && !c10::impl::TorchDispatchModeTLS::any_modes_set(); }

// A contiguous tensor on the given device (device < 0: any, which is then the one to compare with).
bool fits(const at::Tensor *t, at::ScalarType type, const Shape &s, int &device)
{
    if (!t || !t->has_storage() || !t->is_cuda() || t->scalar_type() != type || t->dim() != s.n || !t->is_contiguous()) return false;
    for (int i = 0; i < s.n; ++i)
        if (t->size(i) != s.d[i]) return false;
    if (device < 0) device = t->get_device();
    return t->get_device() == device;
}

// Every size fits the entry points' int.
bool shape_of(const at::Tensor *t, int dims, Shape &s)
{
    if (!t || t->dim() != dims) return false;
    s = Shape{{0, 0, 0, 0}, dims};
    for (int i = 0; i < dims; ++i) {
        s.d[i] = t->size(i);
        if (s.d[i] > INT32_MAX) return false;
    }
    return true;
}

at::Tensor make(const Shape &s, at::ScalarType type, int device)
{
    return at::detail::empty_cuda(at::IntArrayRef(s.d, s.n), type, at::Device(at::kCUDA, device), std::nullopt);
}

void *stream_now() { return c10::cuda::getCurrentCUDAStream().stream(); }

void *ptr(const at::Tensor &t) { return t.data_ptr(); }

// Calls an entry point of the library, which throws nothing, without the GIL.  The arguments are values: whatever
// can throw (data_ptr, the current stream, an allocation) comes before, with the GIL held.
template <typename Fn, typename... Args>
int without_gil(Fn fn, Args... args)
{
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = fn(args...);
    Py_END_ALLOW_THREADS
    return status;
}

bool number(PyObject *o, double &v)
{
    if (PyFloat_Check(o)) v = PyFloat_AS_DOUBLE(o);
    else if (PyLong_Check(o)) v = PyLong_AsDouble(o);
    else return false;
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return true;
}
bool integer(PyObject *o, long &v)
{
    if (!PyLong_Check(o)) return false;
    v = PyLong_AsLong(o);
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return v >= INT32_MIN && v <= INT32_MAX;
}

uintptr_t address(PyObject *o) { return (uintptr_t)PyLong_AsVoidPtr(o); }

bool is_none(PyObject *o) { return o == Py_None; }

// What is thrown before the launch is the Python form's to meet again and to word; behind it (wrapping the
// results) there is nothing to repeat.
#define GUARD_BEGIN bool launched = false; try {
#define GUARD_END                                            \
    }                                                        \
    catch (const std::exception &e)                          \
    {                                                        \
        if (launched) {                                      \
            PyErr_SetString(PyExc_RuntimeError, e.what());   \
            return nullptr;                                  \
        }                                                    \
        PyErr_Clear();                                       \
        Py_RETURN_NONE;                                      \
    }

// The output of an attention call: the one given, or a new one.
bool attention_output(PyObject *given, const Shape &s, int dev, at::Tensor &out)
{
    if (is_none(given)) {
        out = make(s, at::kBFloat16, dev);
        return true;
    }
    const at::Tensor *o = tensor_of(given);
    if (!fits(o, at::kBFloat16, s, dev)) return false;
    out = *o;
    return true;
}
bool scale_of(PyObject *given, int64_t D, double &scale)
{
    scale = D > 0 ? 1.0 / std::sqrt((double)D) : 0.0;
    return is_none(given) || number(given, scale);
}
PyObject *attention_result(int status, PyObject *given, at::Tensor &out)
{
    if (status) return PyLong_FromLong(status);
    if (is_none(given)) return THPVariable_Wrap(std::move(out));
    Py_INCREF(given);
    return given;
}

// attention(address, q, k, v, out or None, scale or None) -> out, or the status if it is not 0, or None
PyObject *attention(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    GUARD_BEGIN
    if (n != 6 || !plain_call()) Py_RETURN_NONE;
    const at::Tensor *q = tensor_of(a[1]), *k = tensor_of(a[2]), *v = tensor_of(a[3]);
    Shape s;
    int dev = -1;
    double scale;
    at::Tensor out;
    if (!shape_of(q, 4, s) || !fits(q, at::kBFloat16, s, dev) || !fits(k, at::kBFloat16, s, dev) || !fits(v, at::kBFloat16, s, dev) ||
        !scale_of(a[5], s.d[3], scale))
        Py_RETURN_NONE;
    const void *pq = ptr(*q), *pk = ptr(*k), *pv = ptr(*v);
    if (!attention_output(a[4], s, dev, out)) Py_RETURN_NONE;
    using Fn = int (*)(const void *, const void *, const void *, void *, int, int, int, int, float, void *);
    const int status = without_gil((Fn)address(a[0]), pq, pk, pv, ptr(out), (int)s.d[0], (int)s.d[1], (int)s.d[2], (int)s.d[3],
                                   (float)scale, stream_now());
    launched = true;
    return attention_result(status, a[4], out);
    GUARD_END
}

// block(address, q, k, v, kv_len or None, layout 0 / 1, out or None, scale or None)
PyObject *block(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    GUARD_BEGIN
    if (n != 8 || !plain_call()) Py_RETURN_NONE;
    const at::Tensor *q = tensor_of(a[1]), *k = tensor_of(a[2]), *v = tensor_of(a[3]);
    long layout;
    Shape s, ks;
    if (!shape_of(q, 4, s) || !shape_of(k, 4, ks) || !integer(a[5], layout)) Py_RETURN_NONE;
    const int at_n = layout ? 1 : 2, at_h = layout ? 2 : 1;           // where the positions and the heads stand
    for (int i = 0; i < 4; ++i)
        if (i != at_n && ks.d[i] != s.d[i]) Py_RETURN_NONE;
    int dev = -1;
    double scale;
    at::Tensor out;
    if (!fits(q, at::kBFloat16, s, dev) || !fits(k, at::kBFloat16, ks, dev) || !fits(v, at::kBFloat16, ks, dev) ||
        !scale_of(a[7], s.d[3], scale))
        Py_RETURN_NONE;
    const int32_t *lens = nullptr;
    if (!is_none(a[4])) {
        const at::Tensor *l = tensor_of(a[4]);
        if (!fits(l, at::kInt, Shape{{s.d[0], 0, 0, 0}, 1}, dev)) Py_RETURN_NONE;
        lens = (const int32_t *)ptr(*l);
    }
    const void *pq = ptr(*q), *pk = ptr(*k), *pv = ptr(*v);
    if (!attention_output(a[6], s, dev, out)) Py_RETURN_NONE;
    using Fn = int (*)(const void *, const void *, const void *, void *, int, int, int, int, int, const int32_t *, int, float, void *);
    const int status = without_gil((Fn)address(a[0]), pq, pk, pv, ptr(out), (int)s.d[0], (int)s.d[at_h], (int)s.d[at_n], (int)ks.d[at_n],
                                   (int)s.d[3], lens, (int)layout, (float)scale, stream_now());
    launched = true;
    return attention_result(status, a[6], out);
    GUARD_END
}

// The outputs [B,P] of a decision: made where they are None, else checked.
struct Decision {
    at::Tensor t[3];                 // tokens, mask, score
    PyObject *given[3];
    int32_t *tokens;
    uint8_t *mask;
    float *score;                    // null: not wanted
};
bool outputs(Decision &o, PyObject *const *a, const Shape &s, int dev, bool want_score)
{
    const at::ScalarType types[3] = {at::kInt, at::kByte, at::kFloat};
    for (int i = 0; i < 3; ++i) {
        o.given[i] = is_none(a[i]) ? nullptr : a[i];
        if (!o.given[i]) continue;
        const at::Tensor *x = tensor_of(a[i]);
        if (!fits(x, types[i], s, dev)) return false;
        o.t[i] = *x;
    }
    for (int i = 0; i < 3; ++i)
        if (!o.given[i] && (i < 2 || want_score)) o.t[i] = make(s, types[i], dev);
    o.tokens = (int32_t *)ptr(o.t[0]);
    o.mask = (uint8_t *)ptr(o.t[1]);
    o.score = o.t[2].defined() ? (float *)ptr(o.t[2]) : nullptr;
    return true;
}
PyObject *result(Decision &o)
{
    PyObject *tuple = PyTuple_New(3);
    for (int i = 0; tuple && i < 3; ++i) {
        PyObject *x = o.given[i] ? o.given[i] : Py_None;
        if (o.given[i] || !o.t[i].defined()) Py_INCREF(x);
        else x = THPVariable_Wrap(std::move(o.t[i]));
        PyTuple_SET_ITEM(tuple, i, x);
    }
    return tuple;
}

// verify(address, drafter or None, verifier, tokens, flags, mode, tau, k, seed, out_tokens, out_mask, out_score, want_score)
PyObject *verify(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    GUARD_BEGIN
    if (n != 13 || !plain_call()) Py_RETURN_NONE;
    const at::Tensor *dra = is_none(a[1]) ? nullptr : tensor_of(a[1]), *ver = tensor_of(a[2]);
    const at::Tensor *tok = tensor_of(a[3]), *fl = tensor_of(a[4]);
    Shape full;
    if (!shape_of(ver, 3, full) || (!is_none(a[1]) && !dra)) Py_RETURN_NONE;
    const Shape s = {{full.d[0], full.d[1], 0, 0}, 2};
    int dev = -1;
    long mode, k;
    double tau;
    if (!fits(ver, at::kBFloat16, full, dev) || (dra && !fits(dra, at::kBFloat16, full, dev)) || !fits(tok, at::kInt, s, dev) ||
        !fits(fl, at::kByte, s, dev) || !integer(a[5], mode) || !number(a[6], tau) || !integer(a[7], k) || !PyLong_Check(a[8]))
        Py_RETURN_NONE;
    const uint64_t seed = PyLong_AsUnsignedLongLongMask(a[8]);
    const int want_score = PyObject_IsTrue(a[12]);
    if (want_score < 0) { PyErr_Clear(); Py_RETURN_NONE; }
    const void *pd = dra ? ptr(*dra) : nullptr, *pv = ptr(*ver);
    const int32_t *pt = (const int32_t *)ptr(*tok);
    const uint8_t *pf = (const uint8_t *)ptr(*fl);
    Decision o;
    if (!outputs(o, a + 9, s, dev, want_score == 1)) Py_RETURN_NONE;
    using Fn = int (*)(const void *, const void *, const int32_t *, const uint8_t *, int, float, int, uint64_t, int32_t *, uint8_t *,
                       float *, int, int, int, void *);
    const int status = without_gil((Fn)address(a[0]), pd, pv, pt, pf, (int)mode, (float)tau, (int)k, seed, o.tokens, o.mask, o.score,
                                   (int)full.d[0], (int)full.d[1], (int)full.d[2], stream_now());
    launched = true;
    if (status) return PyLong_FromLong(status);
    return result(o);
    GUARD_END
}

// unmask(address, logits, tokens, flags, tau, k, out_tokens, out_mask, out_conf)
PyObject *unmask(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    GUARD_BEGIN
    if (n != 9 || !plain_call()) Py_RETURN_NONE;
    const at::Tensor *logits = tensor_of(a[1]), *tok = tensor_of(a[2]), *fl = tensor_of(a[3]);
    Shape full;
    if (!shape_of(logits, 3, full)) Py_RETURN_NONE;
    const Shape s = {{full.d[0], full.d[1], 0, 0}, 2};
    int dev = -1;
    long k;
    double tau;
    if (!fits(logits, at::kBFloat16, full, dev) || !fits(tok, at::kInt, s, dev) || !fits(fl, at::kByte, s, dev) || !number(a[4], tau) ||
        !integer(a[5], k))
        Py_RETURN_NONE;
    const void *pl = ptr(*logits);
    const int32_t *pt = (const int32_t *)ptr(*tok);
    const uint8_t *pf = (const uint8_t *)ptr(*fl);
    Decision o;
    if (!outputs(o, a + 6, s, dev, true)) Py_RETURN_NONE;
    using Fn = int (*)(const void *, const int32_t *, const uint8_t *, float, int, int32_t *, uint8_t *, float *, int, int, int, void *);
    const int status = without_gil((Fn)address(a[0]), pl, pt, pf, (float)tau, (int)k, o.tokens, o.mask, o.score, (int)full.d[0],
                                   (int)full.d[1], (int)full.d[2], stream_now());
    launched = true;
    if (status) return PyLong_FromLong(status);
    return result(o);
    GUARD_END
}

PyMethodDef methods[] = {
    {"attention", (PyCFunction)(void (*)(void))attention, METH_FASTCALL, "dd_bidir_attention on device tensors"},
    {"block", (PyCFunction)(void (*)(void))block, METH_FASTCALL, "dd_block_attention on device tensors"},
    {"verify", (PyCFunction)(void (*)(void))verify, METH_FASTCALL, "dd_verify or dd_verify_static on device tensors"},
    {"unmask", (PyCFunction)(void (*)(void))unmask, METH_FASTCALL, "dd_unmask on device tensors"},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_call", "Native host side of the calls (marshalling only).", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_call(void) { return PyModule_Create(&module); }
