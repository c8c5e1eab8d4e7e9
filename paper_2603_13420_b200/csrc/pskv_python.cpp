// Python face of the hot calls of libpskv: what binding.py did through ctypes -- read the sizes off the tensors, check
// that they are contiguous CUDA tensors, allocate results and scratch, take torch's current stream, call the C entry
// point -- in native code.  Nothing is computed here.
//
// Why native: an attention step of a few candidates is 5 to 15 us of GPU work per call, and marshalling a forward
// call in Python took 22 us (a backward call 26): stream object 3.4, three allocations 7, argument objects 4, the
// foreign call itself 2.  Here it takes 5.5 (9), most of it the launches; forward + backward of 8 candidates of 8
// tokens on 4 heads 50 -> 16 us.
//
// The C entry points are handed over by address at start-up (init), so that the module works with whichever build
// of libpskv binding.py has loaded and has no link-time dependency on it.  A call returns its results, or the
// pskv_status as an int when the library refused; binding.py turns that into an exception.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "pskv.h"

namespace {

struct Api {
    decltype(&pskv_attn_fwd) fwd;
    decltype(&pskv_attn_fwd_workspace_bytes) fwd_ws;
    decltype(&pskv_attn_bwd) bwd;
    decltype(&pskv_attn_bwd_lse) bwd_lse;
    decltype(&pskv_attn_bwd_workspace_bytes) bwd_ws;
    decltype(&pskv_attn_fwd_decode) decode;
    decltype(&pskv_attn_fwd_decode_workspace_bytes) decode_ws;
    decltype(&pskv_attn_fwd_multi) fwd_multi;
    decltype(&pskv_attn_fwd_multi_workspace_bytes) fwd_multi_ws;
    decltype(&pskv_attn_bwd_multi) bwd_multi;
    decltype(&pskv_attn_bwd_multi_workspace_bytes) bwd_multi_ws;
    decltype(&pskv_target_ce_fwd) ce;
    decltype(&pskv_target_ce_fwd_workspace_bytes) ce_ws;
} api;

struct BadArgument {
    PyObject *type;
    const char *what;
};

const at::Tensor &tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) throw BadArgument{PyExc_TypeError, "expected a tensor"};
    return THPVariable_Unpack(o);
}

void *ptr(const at::Tensor &t)
{
    if (!t.is_cuda() || !t.is_contiguous()) throw BadArgument{PyExc_ValueError, "tensors must be contiguous CUDA tensors"};
    return t.data_ptr();
}
void *ptr(PyObject *o) { return o == Py_None ? nullptr : ptr(tensor(o)); }

// q [B, H, S, d], hidden [N, Lr, Dm]
void want_dims(const at::Tensor &t, int n)
{
    if (t.dim() != n) throw BadArgument{PyExc_ValueError, "a tensor has the wrong number of dimensions"};
}
// the other tensors are asked for the sizes the call needs and may have further dimensions, or merged ones, behind them
int64_t size_at(const at::Tensor &t, int i)
{
    if (t.dim() <= i) throw BadArgument{PyExc_IndexError, "a tensor has too few dimensions"};
    return t.size(i);
}

at::Tensor like(const at::Tensor &t) { return at::Tensor(at::detail::empty_cuda(t.sizes(), t.scalar_type(), t.device(), std::nullopt)); }
at::Tensor given_or_like(PyObject *o, const at::Tensor &t) { return o == Py_None ? like(t) : tensor(o); }
at::Tensor floats(PyObject *o, at::IntArrayRef sizes, const at::Tensor &dev)
{
    return o == Py_None ? at::Tensor(at::detail::empty_cuda(sizes, at::kFloat, dev.device(), std::nullopt)) : tensor(o);
}

// The caller's scratch, or as much as the call needs (none where it needs none).
struct Scratch {
    at::Tensor own;
    void *p = nullptr;
    size_t bytes = 0;
    Scratch(PyObject *given, size_t need, const at::Tensor &dev)
    {
        if (given != Py_None) {
            const at::Tensor &t = tensor(given);
            p = ptr(t);
            bytes = (size_t)t.numel() * t.element_size();
        } else if (need > 0) {
            own = at::Tensor(at::detail::empty_cuda({(int64_t)need}, at::kByte, dev.device(), std::nullopt));
            p = own.data_ptr();
            bytes = need;
        }
    }
};

float number(PyObject *o)
{
    PyObject *f = PyNumber_Float(o);  // float(o): also of a string
    if (!f) throw python_error();
    const double v = PyFloat_AsDouble(f);
    Py_DECREF(f);
    return (float)v;
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

template <class Fn>
pskv_status without_gil(Fn fn)
{
    struct Released {  // taken back however fn is left: what turns an exception into a Python one needs it
        PyThreadState *save = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(save); }
    } released;
    return fn();
}

template <class... T>
PyObject *results(pskv_status st, const T &...t)
{
    if (st != PSKV_OK) return PyLong_FromLong((long)st);
    PyObject *tuple = PyTuple_New(sizeof...(t));
    if (!tuple) return nullptr;
    Py_ssize_t i = 0;
    ((PyTuple_SET_ITEM(tuple, i++, THPVariable_Wrap(t))), ...);
    return tuple;
}

// Every entry: fixed number of arguments, C++ exceptions turned into Python ones.
template <int N, PyObject *(*body)(PyObject *const *)>
PyObject *entry(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    if (n != N) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    try {
        return body(a);
    } catch (const BadArgument &e) {
        PyErr_SetString(e.type, e.what);
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

struct Dims {
    int B, Hq, Hkv, S, P, d;
};
// prefix [Hkv, P, d] (p_at = 1) or [Bp, Hkv, P, d] (p_at = 2)
Dims dims_of(const at::Tensor &q, PyObject *prefix_k, const at::Tensor &suffix_k, int p_at)
{
    want_dims(q, 4);
    const int64_t Hkv = size_at(suffix_k, 1), P = prefix_k == Py_None ? 0 : size_at(tensor(prefix_k), p_at);
    ptr(q);  // (before anything is allocated where q is)
    return {(int)q.size(0), (int)q.size(1), (int)Hkv, (int)q.size(2), (int)P, (int)q.size(3)};
}

// (q, prefix_k, prefix_v, suffix_k, suffix_v, scale, out, lse, workspace)
PyObject *fwd(PyObject *const *a)
{
    const at::Tensor &q = tensor(a[0]), &sk = tensor(a[3]);
    const Dims m = dims_of(q, a[1], sk, 1);
    const at::Tensor out = given_or_like(a[6], q), lse = floats(a[7], {m.B, m.Hq, m.S}, q);
    const Scratch ws(a[8], a[8] == Py_None ? api.fwd_ws(m.B, m.Hq, m.Hkv, m.S, m.P, m.d) : 0, q);
    void *qp = ptr(q), *pk = ptr(a[1]), *pv = ptr(a[2]), *skp = ptr(sk), *sv = ptr(a[4]), *op = ptr(out), *lp = ptr(lse), *s = stream();
    const float scale = number(a[5]);
    return results(without_gil([&] {
                       return api.fwd(qp, pk, pv, skp, sv, scale, op, (float *)lp, m.B, m.Hq, m.Hkv, m.S, m.P, m.d, ws.p, ws.bytes, s);
                   }), out, lse);
}

// (dout, dlse or None, q, prefix_k, prefix_v, suffix_k, suffix_v, out, lse, scale, dq, dk_suffix, dv_suffix, workspace)
PyObject *bwd(PyObject *const *a)
{
    const at::Tensor &q = tensor(a[2]), &sk = tensor(a[5]), &sv = tensor(a[6]);
    const Dims m = dims_of(q, a[3], sk, 1);
    const at::Tensor dq = given_or_like(a[10], q), dk = given_or_like(a[11], sk), dv = given_or_like(a[12], sv);
    const Scratch ws(a[13], a[13] == Py_None ? api.bwd_ws(m.B, m.Hq, m.Hkv, m.S, m.P, m.d) : 0, q);
    void *dop = ptr(a[0]), *dl = ptr(a[1]), *qp = ptr(q), *pk = ptr(a[3]), *pv = ptr(a[4]), *skp = ptr(sk), *svp = ptr(sv), *op = ptr(a[7]),
         *lp = ptr(a[8]), *dqp = ptr(dq), *dkp = ptr(dk), *dvp = ptr(dv), *s = stream();
    const float scale = number(a[9]);
    return results(without_gil([&] {
                       return dl ? api.bwd_lse(dop, (const float *)dl, qp, pk, pv, skp, svp, op, (const float *)lp, scale, dqp, dkp, dvp, m.B,
                                               m.Hq, m.Hkv, m.S, m.P, m.d, ws.p, ws.bytes, s)
                                 : api.bwd(dop, qp, pk, pv, skp, svp, op, (const float *)lp, scale, dqp, dkp, dvp, m.B, m.Hq, m.Hkv, m.S, m.P,
                                           m.d, ws.p, ws.bytes, s);
                   }), dq, dk, dv);
}

// (q, prefix_k, prefix_v, suffix_k, suffix_v, suffix_len or None, scale, out, lse, workspace)
PyObject *fwd_decode(PyObject *const *a)
{
    const at::Tensor &q = tensor(a[0]), &sk = tensor(a[3]);
    const Dims m = dims_of(q, a[1], sk, 1);
    const int Skv = (int)size_at(sk, 2);
    if (a[5] != Py_None) {
        const at::Tensor &n = tensor(a[5]);
        if (n.scalar_type() != at::kInt || n.dim() != 1 || n.size(0) != m.B)
            throw BadArgument{PyExc_ValueError, "suffix_len must be an int32 CUDA tensor of shape [B]"};
    }
    const at::Tensor out = given_or_like(a[7], q), lse = floats(a[8], {m.B, m.Hq, m.S}, q);
    const Scratch ws(a[9], a[9] == Py_None ? api.decode_ws(m.B, m.Hq, m.Hkv, m.S, Skv, m.P, m.d) : 0, q);
    void *qp = ptr(q), *pk = ptr(a[1]), *pv = ptr(a[2]), *skp = ptr(sk), *sv = ptr(a[4]), *n = ptr(a[5]), *op = ptr(out), *lp = ptr(lse),
         *s = stream();
    const float scale = number(a[6]);
    return results(without_gil([&] {
                       return api.decode(qp, pk, pv, skp, sv, (const int *)n, scale, op, (float *)lp, m.B, m.Hq, m.Hkv, m.S, Skv, m.P, m.d,
                                         ws.p, ws.bytes, s);
                   }), out, lse);
}

std::vector<int> lengths(PyObject *o)
{
    if (PyObject_Size(o) < 0) throw python_error();  // (an iterator has no length)
    PyObject *seq = PySequence_Fast(o, "prefix_len must be a sequence of integers");
    if (!seq) throw python_error();
    std::vector<int> v;
    bool ok = true;
    for (Py_ssize_t i = 0; ok && i < PySequence_Fast_GET_SIZE(seq); ++i) {
        PyObject *n = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, i));
        const unsigned long x = n ? PyLong_AsUnsignedLongMask(n) : 0;  // the low bits, as a C int of ctypes takes them
        Py_XDECREF(n);
        ok = !PyErr_Occurred();
        v.push_back((int)x);
    }
    Py_DECREF(seq);
    if (!ok) throw python_error();
    return v;
}

// (q, prefix_k, prefix_v, prefix_len, suffix_k, suffix_v, scale, out, lse, workspace)
PyObject *fwd_multi(PyObject *const *a)
{
    const at::Tensor &q = tensor(a[0]), &sk = tensor(a[4]);
    const Dims m = dims_of(q, a[1], sk, 2);
    const std::vector<int> len = lengths(a[3]);
    const int Bp = (int)len.size();
    const at::Tensor out = given_or_like(a[7], q), lse = floats(a[8], {m.B, m.Hq, m.S}, q);
    const Scratch ws(a[9], a[9] == Py_None ? std::max<size_t>(256, api.fwd_multi_ws(m.B, Bp, m.Hq, m.Hkv, m.S, m.P, m.d)) : 0, q);
    void *qp = ptr(q), *pk = ptr(a[1]), *pv = ptr(a[2]), *skp = ptr(sk), *sv = ptr(a[5]), *op = ptr(out), *lp = ptr(lse), *s = stream();
    const float scale = number(a[6]);
    return results(without_gil([&] {
                       return api.fwd_multi(qp, pk, pv, len.data(), skp, sv, scale, op, (float *)lp, m.B, Bp, m.Hq, m.Hkv, m.S, m.P, m.d, ws.p,
                                            ws.bytes, s);
                   }), out, lse);
}

// (dout, q, prefix_k, prefix_v, prefix_len, suffix_k, suffix_v, out, lse, scale, dq, dk_suffix, dv_suffix, workspace)
PyObject *bwd_multi(PyObject *const *a)
{
    const at::Tensor &q = tensor(a[1]), &sk = tensor(a[5]), &sv = tensor(a[6]);
    const Dims m = dims_of(q, a[2], sk, 2);
    const std::vector<int> len = lengths(a[4]);
    const int Bp = (int)len.size();
    const at::Tensor dq = given_or_like(a[10], q), dk = given_or_like(a[11], sk), dv = given_or_like(a[12], sv);
    const Scratch ws(a[13], a[13] == Py_None ? std::max<size_t>(256, api.bwd_multi_ws(m.B, Bp, m.Hq, m.Hkv, m.S, m.P, m.d)) : 0, q);
    void *dop = ptr(a[0]), *qp = ptr(q), *pk = ptr(a[2]), *pv = ptr(a[3]), *skp = ptr(sk), *svp = ptr(sv), *op = ptr(a[7]), *lp = ptr(a[8]),
         *dqp = ptr(dq), *dkp = ptr(dk), *dvp = ptr(dv), *s = stream();
    const float scale = number(a[9]);
    return results(without_gil([&] {
                       return api.bwd_multi(dop, qp, pk, pv, len.data(), skp, svp, op, (const float *)lp, scale, dqp, dkp, dvp, m.B, Bp, m.Hq,
                                            m.Hkv, m.S, m.P, m.d, ws.p, ws.bytes, s);
                   }), dq, dk, dv);
}

// (hidden, weight, target, mask, nll, lse, loss, workspace)
PyObject *target_ce(PyObject *const *a)
{
    const at::Tensor &h = tensor(a[0]), &w = tensor(a[1]), &t = tensor(a[2]), &m = tensor(a[3]);
    want_dims(h, 3);
    ptr(h);
    if (t.scalar_type() != at::kInt || m.scalar_type() != at::kFloat)
        throw BadArgument{PyExc_ValueError, "target must be int32 and mask float32"};
    const int64_t N = h.size(0), Lr = h.size(1), Dm = h.size(2), V = size_at(w, 0);
    if (t.sizes() != at::IntArrayRef({N, Lr}) || m.sizes() != at::IntArrayRef({N, Lr}) || size_at(w, 1) != Dm)
        throw BadArgument{PyExc_ValueError, "shape mismatch"};
    const at::Tensor nll = floats(a[4], {N, Lr}, h), lse = floats(a[5], {N, Lr}, h), loss = floats(a[6], {N}, h);
    const Scratch ws(a[7], a[7] == Py_None ? std::max<size_t>(256, api.ce_ws((int)N, (int)Lr, (int)Dm, (int)V)) : 0, h);
    void *hp = ptr(h), *wp = ptr(w), *tp = ptr(t), *mp = ptr(m), *np = ptr(nll), *lp = ptr(lse), *sp = ptr(loss), *s = stream();
    return results(without_gil([&] {
                       return api.ce(hp, wp, (const int *)tp, (const float *)mp, (float *)np, (float *)lp, (float *)sp, (int)N, (int)Lr, (int)Dm,
                                     (int)V, ws.p, ws.bytes, s);
                   }), nll, lse, loss);
}

// Addresses of the C entry points, in the order of struct Api.
PyObject *init(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    static_assert(sizeof(Api) == 13 * sizeof(void *), "one address per entry");
    if (n != 13) {
        PyErr_SetString(PyExc_TypeError, "wrong number of entry points");
        return nullptr;
    }
    void *p[13];
    for (int i = 0; i < 13; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (!p[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
            return nullptr;
        }
    }
    memcpy(&api, p, sizeof(api));
    Py_RETURN_NONE;
}

#define ENTRY(name, n) {#name, (PyCFunction)(void (*)(void))(entry<n, name>), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, nullptr},
    ENTRY(fwd, 9), ENTRY(bwd, 14), ENTRY(fwd_decode, 10), ENTRY(fwd_multi, 10), ENTRY(bwd_multi, 14), ENTRY(target_ce, 8),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef PSKV_BUILT_FOR
#error "the build passes the interpreter and torch that this module is made for"
#endif

PyMODINIT_FUNC PyInit__native(void)
{
    PyObject *m = PyModule_Create(&module);
    // binding.py refuses a module made for another torch: its C++ interface is not a stable one
    if (m && PyModule_AddStringConstant(m, "built_for", PSKV_BUILT_FOR) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
