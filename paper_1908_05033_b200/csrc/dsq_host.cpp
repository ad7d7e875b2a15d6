// Native side of the Python binding (binding.py): tensors in, tensors out.
//
// Marshalling only - dtype checks, output allocation, the current stream, the
// status turned into DsqError - but on the critical path of every small call:
// done in Python through ctypes it took 13 us a call (26 us with two calls, 270
// us for the 20 calls of the ResNet-18-shaped stack, whose kernels at batch 1
// then took 177 us).  Here a call with one launch and one new output takes 6 us of
// host time, the launch included (quantise and 3x3 convolution of one 56x56x64
// image: 13 us for the two, 7 us on the GPU), a replayed stack 15 us in all.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "../../include/dsq.h"
#include "dsq_plan.h"

namespace {

PyObject *g_error_class = nullptr;      // binding.DsqError

// thrown after a Python error has been set
struct PyFailed { };

[[noreturn]] void fail_type(const char *name, const char *dtype)
{
    PyErr_Format(PyExc_TypeError, "%s: want a contiguous CUDA tensor of %s", name, dtype);
    throw PyFailed();
}

void check(int status, const char *where)
{
    if (status == DSQ_OK) return;
    PyObject *e = PyObject_CallFunction(g_error_class, "is", status, where);
    if (e) {
        PyErr_SetObject(g_error_class, e);
        Py_DECREF(e);
    }
    throw PyFailed();
}

const char *dtype_name(at::ScalarType t)
{
    switch (t) {
    case at::kByte: return "torch.uint8";
    case at::kChar: return "torch.int8";
    case at::kFloat: return "torch.float32";
    case at::kBFloat16: return "torch.bfloat16";
    default: return "another type";
    }
}

// a tensor whose dtype, device and layout are checked
const at::Tensor &need(PyObject *o, at::ScalarType t, const char *name)
{
    if (!THPVariable_Check(o)) fail_type(name, dtype_name(t));
    const at::Tensor &v = THPVariable_Unpack(o);
    if (!v.is_cuda() || v.scalar_type() != t || !v.is_contiguous()) fail_type(name, dtype_name(t));
    return v;
}

// any tensor's (or None's) address
const at::Tensor *maybe(PyObject *o, const char *name)
{
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: want a tensor or None", name);
        throw PyFailed();
    }
    return &THPVariable_Unpack(o);
}

void *addr(const at::Tensor *t) { return t ? t->data_ptr() : nullptr; }

int64_t as_int(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyFailed();
    return v;
}

float as_float(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyFailed();
    return (float)v;
}

bool as_bool(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw PyFailed();
    return v != 0;
}

// a sequence of exactly n objects
struct Seq {
    PyObject *s;
    Seq(PyObject *o, Py_ssize_t n, const char *name) : s(PySequence_Fast(o, name))
    {
        if (!s) throw PyFailed();
        if (PySequence_Fast_GET_SIZE(s) != n) {
            Py_DECREF(s);
            PyErr_Format(PyExc_ValueError, "%s: want %zd values", name, n);
            throw PyFailed();
        }
    }
    ~Seq() { Py_DECREF(s); }
    PyObject *operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(s, i); }
};

dsq_quant_t as_quant(PyObject *o, const char *name)
{
    const Seq t(o, 3, name);
    return {(int32_t)as_int(t[0]), as_float(t[1]), as_float(t[2])};
}

dsq_nhwc_t as_shape(PyObject *o)
{
    const Seq t(o, 4, "shape");
    return {(int32_t)as_int(t[0]), (int32_t)as_int(t[1]), (int32_t)as_int(t[2]),
            (int32_t)as_int(t[3])};
}

// the bytes of binding.dsq_conv_t (a ctypes structure)
dsq_conv_t as_conv(PyObject *o)
{
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw PyFailed();
    dsq_conv_t c = {};
    const bool ok = b.len == (Py_ssize_t)sizeof(c);
    if (ok) c = *static_cast<const dsq_conv_t *>(b.buf);
    PyBuffer_Release(&b);
    if (!ok) {
        PyErr_SetString(PyExc_TypeError, "conv: want a dsq_conv_t");
        throw PyFailed();
    }
    return c;
}

at::Tensor new_tensor(at::IntArrayRef sizes, at::ScalarType t, const at::Tensor &like)
{
    return at::empty(sizes, at::TensorOptions().dtype(t).device(like.device()));
}

PyObject *wrap(const at::Tensor &t)
{
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}

// the caller's tensor, or a new one (kept alive in `store`)
const at::Tensor &out_or_new(PyObject *o, at::Tensor &store, at::IntArrayRef sizes,
                             at::ScalarType t, const at::Tensor &like)
{
    if (o != Py_None) store = *maybe(o, "out");
    else store = new_tensor(sizes, t, like);
    return store;
}

// Work is enqueued without the interpreter lock (a launch blocks while the
// device's queue is full).
template <class F> int enqueue(F f)
{
    void *stream = (void *)c10::cuda::getCurrentCUDAStream().stream();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = f(stream);
    Py_END_ALLOW_THREADS
    return st;
}

// wraps a function body: C++ exceptions become Python errors
template <class F> PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F f)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "want %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return f();
    } catch (const PyFailed &) {
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

PyObject *set_error_class(PyObject *, PyObject *cls)
{
    Py_XDECREF(g_error_class);
    Py_INCREF(cls);
    g_error_class = cls;
    Py_RETURN_NONE;
}

// (x, bits, lo, hi, out | None) -> codes
PyObject *quantize_act(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 5, [&]() -> PyObject * {
        const at::Tensor &x = need(a[0], at::kFloat, "x");
        const dsq_quant_t q = {(int32_t)as_int(a[1]), as_float(a[2]), as_float(a[3])};
        if (x.dim() != 4) {
            PyErr_SetString(PyExc_ValueError, "x: want NHWC");
            throw PyFailed();
        }
        const int64_t N = x.size(0), H = x.size(1), W = x.size(2), C = x.size(3);
        const dsq_nhwc_t shape = {(int32_t)N, (int32_t)H, (int32_t)W, (int32_t)C};
        at::Tensor store;
        const at::Tensor &out =
            out_or_new(a[4], store, {N, H, W, (int64_t)dsq_row_pitch(C, q.bits)}, at::kByte, x);
        check(enqueue([&](void *s) {
                  return dsq_quantize_act((const float *)x.data_ptr(), &shape, &q, out.data_ptr(),
                                          (size_t)out.numel(), s);
              }),
              "dsq_quantize_act");
        if (a[4] != Py_None) return Py_NewRef(a[4]);
        return wrap(out);
    });
}

// (depthwise, act, shape, act_q, blob, conv, scale, bias, w_offset, residual,
//  residual_q, requant, want_f32, want_acc, ws | None, out_codes)
// -> (codes | None, y | None, acc | None)
PyObject *conv2d(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 16, [&]() -> PyObject * {
        const bool depthwise = as_bool(a[0]);
        const at::Tensor &act = need(a[1], at::kByte, "act");
        const dsq_nhwc_t shape = as_shape(a[2]);
        const dsq_quant_t act_q = as_quant(a[3], "act_q");
        const at::Tensor &blob = need(a[4], at::kByte, "weights");
        const dsq_conv_t conv = as_conv(a[5]);
        const at::Tensor &scale = need(a[6], at::kFloat, "scale");
        const at::Tensor &bias = need(a[7], at::kFloat, "bias");
        dsq_epilogue_t ep = {};
        ep.scale = (const float *)scale.data_ptr();
        ep.bias = (const float *)bias.data_ptr();
        ep.w_offset = as_float(a[8]);
        ep.residual_codes = addr(maybe(a[9], "residual"));
        if (a[10] != Py_None) ep.residual_q = as_quant(a[10], "residual_q");
        if (a[11] != Py_None) ep.requant = as_quant(a[11], "requant");
        // (a stride of 0 is for the library to reject)
        const int64_t st = conv.stride > 0 ? conv.stride : 1;
        const int64_t N = shape.N, C = conv.Cout;
        const int64_t Ho = (shape.H + 2 * conv.pad - conv.KH) / st + 1;
        const int64_t Wo = (shape.W + 2 * conv.pad - conv.KW) / st + 1;
        at::Tensor y, acc, codes;
        if (as_bool(a[12])) y = new_tensor({N, Ho, Wo, C}, at::kFloat, act);
        if (as_bool(a[13])) acc = new_tensor({N, Ho, Wo, C}, at::kInt, act);
        if (a[11] != Py_None)
            out_or_new(a[15], codes, {N, Ho, Wo, (int64_t)dsq_row_pitch(C, act_q.bits)}, at::kByte,
                       act);
        float *yp = y.defined() ? (float *)y.data_ptr() : nullptr;
        int32_t *accp = acc.defined() ? (int32_t *)acc.data_ptr() : nullptr;
        void *cp = codes.defined() ? codes.data_ptr() : nullptr;
        if (depthwise) {
            check(enqueue([&](void *s) {
                      return dsq_dwconv2d(act.data_ptr(), &shape, &act_q, blob.data_ptr(), &conv,
                                          &ep, yp, cp, accp, s);
                  }),
                  "dsq_dwconv2d");
        } else {
            const at::Tensor *ws = maybe(a[14], "ws");
            check(enqueue([&](void *s) {
                      return dsq_conv2d(act.data_ptr(), &shape, &act_q, blob.data_ptr(), &conv, &ep,
                                        yp, cp, accp, addr(ws), ws ? (size_t)ws->numel() : 0, s);
                  }),
                  "dsq_conv2d");
        }
        PyObject *pc = a[11] != Py_None && a[15] != Py_None ? Py_NewRef(a[15]) : wrap(codes);
        return Py_BuildValue("(NNN)", pc, wrap(y), wrap(acc));
    });
}

// (codes, shape, bits, out | None) -> codes
PyObject *maxpool2x2(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 4, [&]() -> PyObject * {
        const at::Tensor &codes = need(a[0], at::kByte, "codes");
        const dsq_nhwc_t shape = as_shape(a[1]);
        const int bits = (int)as_int(a[2]);
        at::Tensor store;
        const at::Tensor &out = out_or_new(
            a[3], store, {shape.N, shape.H / 2, shape.W / 2, (int64_t)dsq_row_pitch(shape.C, bits)},
            at::kByte, codes);
        check(enqueue([&](void *s) {
                  return dsq_maxpool2x2(codes.data_ptr(), &shape, bits, out.data_ptr(),
                                        (size_t)out.numel(), s);
              }),
              "dsq_maxpool2x2");
        if (a[3] != Py_None) return Py_NewRef(a[3]);
        return wrap(out);
    });
}

// (x, bits, lo, hi, alpha, out | None) -> y
PyObject *soft_fwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 6, [&]() -> PyObject * {
        const at::Tensor &x = need(a[0], at::kFloat, "x");
        const dsq_quant_t q = {(int32_t)as_int(a[1]), as_float(a[2]), as_float(a[3])};
        const float alpha = as_float(a[4]);
        at::Tensor store;
        const at::Tensor &y = out_or_new(a[5], store, x.sizes(), at::kFloat, x);
        check(enqueue([&](void *s) {
                  return dsq_soft_quantize_fwd((const float *)x.data_ptr(), x.numel(), &q, alpha,
                                               (float *)y.data_ptr(), s);
              }),
              "dsq_soft_quantize_fwd");
        if (a[5] != Py_None) return Py_NewRef(a[5]);
        return wrap(y);
    });
}

// (x, grad_y, bits, lo, hi, alpha, out | None, grad_params | None) -> (gx, gp)
PyObject *soft_bwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 8, [&]() -> PyObject * {
        const at::Tensor &x = need(a[0], at::kFloat, "x");
        const at::Tensor &gy = need(a[1], at::kFloat, "grad_y");
        const dsq_quant_t q = {(int32_t)as_int(a[2]), as_float(a[3]), as_float(a[4])};
        const float alpha = as_float(a[5]);
        at::Tensor s0, s1;
        const at::Tensor &gx = out_or_new(a[6], s0, x.sizes(), at::kFloat, x);
        const at::Tensor &gp = out_or_new(a[7], s1, {3}, at::kDouble, x);
        check(enqueue([&](void *s) {
                  return dsq_soft_quantize_bwd((const float *)x.data_ptr(),
                                               (const float *)gy.data_ptr(), x.numel(), &q, alpha,
                                               (float *)gx.data_ptr(), (double *)gp.data_ptr(), s);
              }),
              "dsq_soft_quantize_bwd");
        return Py_BuildValue("(NN)", a[6] != Py_None ? Py_NewRef(a[6]) : wrap(gx),
                             a[7] != Py_None ? Py_NewRef(a[7]) : wrap(gp));
    });
}

// (binary, A, B, M, N, K, bits, ws, row_scale | None, want_i32, out_i32 | None,
//  out_f32 | None) -> (C | None, D | None)
PyObject *gemm(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 12, [&]() -> PyObject * {
        const bool binary = as_bool(a[0]);
        const at::Tensor &A = need(a[1], at::kByte, "A");
        const at::Tensor &B = need(a[2], at::kByte, "B");
        const int64_t M = as_int(a[3]), N = as_int(a[4]), K = as_int(a[5]);
        const int bits = (int)as_int(a[6]);
        const at::Tensor *ws = maybe(a[7], "ws"), *rs = maybe(a[8], "row_scale");
        at::Tensor C, D;
        if (a[10] != Py_None || as_bool(a[9])) out_or_new(a[10], C, {M, N}, at::kInt, A);
        if (a[11] != Py_None || rs) out_or_new(a[11], D, {M, N}, at::kFloat, A);
        int32_t *c = C.defined() ? (int32_t *)C.data_ptr() : nullptr;
        float *d = D.defined() ? (float *)D.data_ptr() : nullptr;
        const size_t wb = ws ? (size_t)ws->numel() : 0;
        check(enqueue([&](void *s) {
                  return binary ? dsq_binary_gemm(A.data_ptr(), B.data_ptr(), M, N, K, c,
                                                  (const float *)addr(rs), d, addr(ws), wb, s)
                                : dsq_gemm(A.data_ptr(), B.data_ptr(), M, N, K, bits, c,
                                           (const float *)addr(rs), d, addr(ws), wb, s);
              }),
              binary ? "dsq_binary_gemm" : "dsq_gemm");
        return Py_BuildValue("(NN)", a[10] != Py_None ? Py_NewRef(a[10]) : wrap(C),
                             a[11] != Py_None ? Py_NewRef(a[11]) : wrap(D));
    });
}

// (X, W, M, N, K, bits, w_offset, col_scale, col_bias | None, ws, out | None) -> Y
PyObject *wgemm(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 11, [&]() -> PyObject * {
        const at::Tensor &X = need(a[0], at::kBFloat16, "X");
        const at::Tensor &W = need(a[1], at::kByte, "W");
        const int64_t M = as_int(a[2]), N = as_int(a[3]), K = as_int(a[4]);
        const int bits = (int)as_int(a[5]);
        const float w_offset = as_float(a[6]);
        const at::Tensor &cs = need(a[7], at::kFloat, "col_scale");
        const at::Tensor *cb = maybe(a[8], "col_bias"), *ws = maybe(a[9], "ws");
        at::Tensor store;
        const at::Tensor &Y = out_or_new(a[10], store, {M, N}, at::kFloat, X);
        check(enqueue([&](void *s) {
                  return dsq_wgemm_bf16(X.data_ptr(), W.data_ptr(), M, N, K, bits, w_offset,
                                        (const float *)cs.data_ptr(), (const float *)addr(cb),
                                        (float *)Y.data_ptr(), addr(ws),
                                        ws ? (size_t)ws->numel() : 0, s);
              }),
              "dsq_wgemm_bf16");
        if (a[10] != Py_None) return Py_NewRef(a[10]);
        return wrap(Y);
    });
}

// ---- recorded call sequences (dsq_plan.h) -----------------------------------
// What a plan was recorded from: everything a caller could exchange or change in
// place between two passes (tensors, ranges, layers).  A plan runs only while all
// of it is as it was.  The parts are walked in one order, each leaving an entry:
//   * a device tensor: the object, its address, size and type - its contents are the
//     kernels' business;
//   * dicts (keys too), lists, tuples and objects that are their attributes (a layer):
//     their type and size, then what they are made of;
//   * an object with a buffer (a ctypes structure, a numpy scalar): its type and a copy
//     of its bytes;
//   * numbers, strings, None: the object.
// Anything else could change unseen, host tensors and device scalars (a range read
// with float()) among them: such a plan runs once and is recorded again.
struct Part {
    PyObject *o = nullptr;                    // held; of a container or buffer: its type
    const void *data = nullptr;               // address of a tensor, or of a buffer now
    int64_t size = 0;                         // elements, members or bytes
    int type = 0;                             // scalar type of a tensor; BUFFER
    static constexpr int BUFFER = -1;
};

struct Recorded {
    dsq_plan *plan = nullptr;
    std::vector<Part> parts;
    std::string bytes;                        // of the buffers, one behind the other
    bool once = false, ran = false;           // holds something that could change unseen
    ~Recorded()
    {
        dsq_plan_free(plan);
        for (Part &p : parts) Py_XDECREF(p.o);
    }
};

bool is_value(PyObject *o)
{
    const PyTypeObject *t = Py_TYPE(o);
    return t == &PyUnicode_Type || t == &PyFloat_Type || t == &PyLong_Type || o == Py_None ||
           t == &PyBool_Type || t == &PyBytes_Type;
}

// whether all an object of this type holds is in its dict (nothing in slots)
bool only_dict(const PyTypeObject *t)
{
    return t->tp_basicsize <= (Py_ssize_t)sizeof(PyObject) +
                                  (Py_ssize_t)sizeof(PyObject *) *
                                      ((t->tp_dictoffset > 0) + (t->tp_weaklistoffset > 0));
}

// Calls f(part) for everything `o` is made of, as above; sets *opaque where a change
// could not be seen; stops when f says so.  (Some 1,500 entries for 52 layers, before
// every pass: the common kinds come first.)
template <class F> bool each_part(PyObject *o, F &f, bool *opaque, int depth = 0)
{
    Part p;
    p.o = o;
    if (is_value(o)) return f(p);
    auto container = [&](Py_ssize_t n) {
        p.o = (PyObject *)Py_TYPE(o);
        p.size = n;
        return f(p);
    };
    auto attributes = [&](PyObject *dict) {
        Py_ssize_t at = 0;
        PyObject *k, *v;
        if (!container(PyDict_GET_SIZE(dict))) return false;
        while (PyDict_Next(dict, &at, &k, &v))
            if (!each_part(k, f, opaque, depth + 1) || !each_part(v, f, opaque, depth + 1)) return false;
        return true;
    };
    if (depth > 32) {                         // (an object that holds itself)
        *opaque = true;
        return f(p);
    }
    if (PyList_Check(o) || PyTuple_Check(o)) {
        const bool list = PyList_Check(o);
        if (!container(Py_SIZE(o))) return false;
        for (Py_ssize_t i = 0; i < Py_SIZE(o); ++i)
            if (!each_part(list ? PyList_GET_ITEM(o, i) : PyTuple_GET_ITEM(o, i), f, opaque, depth + 1))
                return false;
        return true;
    }
    if (PyDict_Check(o)) return attributes(o);
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.dim() == 0 || !t.is_contiguous()) *opaque = true;
        else p.data = t.data_ptr();
        p.size = t.numel();
        p.type = (int)t.scalar_type();
        return f(p);
    }
    if (PyObject_CheckBuffer(o)) {
        Py_buffer b;
        if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) == 0) {
            p.o = (PyObject *)Py_TYPE(o);
            p.type = Part::BUFFER;
            p.data = b.buf;
            p.size = b.len;
            const bool ok = f(p);
            PyBuffer_Release(&b);
            return ok;
        }
        PyErr_Clear();
    } else if (only_dict(Py_TYPE(o))) {
        if (PyObject *dict = PyObject_GenericGetDict(o, nullptr)) {
            const bool ok = attributes(dict);
            Py_DECREF(dict);
            return ok;
        }
        PyErr_Clear();
    }
    *opaque = true;
    return f(p);
}

void free_recorded(PyObject *capsule)
{
    delete static_cast<Recorded *>(PyCapsule_GetPointer(capsule, "dsq_plan"));
}

// (function, parts) -> plan of the calls that function() makes
PyObject *plan_record(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 2, [&]() -> PyObject * {
        std::unique_ptr<Recorded> rec(new Recorded);
        // (before the calls: what they change of it makes the plan invalid)
        rec->parts.reserve(1024);
        auto keep = [&](const Part &p) {
            if (p.type == Part::BUFFER) rec->bytes.append(static_cast<const char *>(p.data), (size_t)p.size);
            rec->parts.push_back(p);
            Py_XINCREF(p.o);
            return true;
        };
        each_part(a[1], keep, &rec->once);
        check(dsq_plan_begin(), "dsq_plan_begin");
        PyObject *r = PyObject_CallNoArgs(a[0]);
        const int st = dsq_plan_end(&rec->plan);
        if (!r) throw PyFailed();
        Py_DECREF(r);
        check(st, "dsq_plan_end");
        PyObject *c = PyCapsule_New(rec.get(), "dsq_plan", free_recorded);
        if (!c) throw PyFailed();
        rec.release();
        return c;
    });
}

// (plan, parts | None) -> True when the plan still stands and was run on the current
// stream; False when it has to be recorded again (None: it has just been recorded)
PyObject *plan_run(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 2, [&]() -> PyObject * {
        Recorded *r = static_cast<Recorded *>(PyCapsule_GetPointer(a[0], "dsq_plan"));
        if (!r) throw PyFailed();
        if ((r->once && r->ran) || !dsq_plan_valid(r->plan)) Py_RETURN_FALSE;
        size_t i = 0, at = 0;
        bool opaque = false;
        auto same = [&](const Part &p) {
            if (i == r->parts.size()) return false;
            const Part &q = r->parts[i++];
            if (q.o != p.o || q.size != p.size || q.type != p.type) return false;
            if (p.type != Part::BUFFER) return q.data == p.data;
            at += (size_t)p.size;
            return std::memcmp(r->bytes.data() + at - (size_t)p.size, p.data, (size_t)p.size) == 0;
        };
        if (a[1] != Py_None && (!each_part(a[1], same, &opaque) || i != r->parts.size())) Py_RETURN_FALSE;
        r->ran = true;
        check(enqueue([&](void *s) { return dsq_plan_run(r->plan, s); }), "dsq_plan_run");
        Py_RETURN_TRUE;
    });
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {{"set_error_class", set_error_class, METH_O, nullptr},
                           FAST(quantize_act), FAST(conv2d), FAST(maxpool2x2), FAST(soft_fwd),
                           FAST(soft_bwd), FAST(gemm), FAST(wgemm), FAST(plan_record),
                           FAST(plan_run), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_dsq_host", nullptr, -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__dsq_host(void) { return PyModule_Create(&g_module); }
