// The calls a layer makes at run time and when it is built, as functions that take torch tensors: reading shapes, strides, pointers and the
// current stream here costs a fraction of what it costs in Python (an eager 256 x 256 -> 768 layer call: 17.9 us with
// ctypes objects, 8.5 us from here; the three calls of a 2048 x 4608 -> 1152 W4A8 layer: 50.6 -> 32.8 us).  Argument
// marshalling only: every check is the C ABI's (include/segquant.h), every function returns its status (with the tensors
// it allocated, where it did), and the GIL is released around the call.  Reading a tensor can throw (a wrapper or sparse
// tensor without storage, a stride of a 0-dimensional one), so everything is read into locals while the GIL is held; what
// runs without it is a call of the C ABI, which does not throw.
#include <Python.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include "segquant.h"

namespace {

struct BadArgument {};           // a Python exception is set

// Positional arguments of one call.
struct Args {
    PyObject *const *a;

    const at::Tensor &tensor(int i) const
    {
        if (!THPVariable_Check(a[i])) {
            PyErr_Format(PyExc_TypeError, "argument %d must be a tensor, not %s", i, Py_TYPE(a[i])->tp_name);
            throw BadArgument();
        }
        return THPVariable_Unpack(a[i]);
    }
    const at::Tensor &matrix(int i) const
    {
        const at::Tensor &t = tensor(i);
        if (t.dim() != 2) {
            PyErr_Format(PyExc_ValueError, "argument %d must be a matrix, not %d-dimensional", i, int(t.dim()));
            throw BadArgument();
        }
        return t;
    }
    bool none(int i) const { return a[i] == Py_None; }
    void *ptr(int i) const { return none(i) ? nullptr : tensor(i).data_ptr(); }
    float *f32(int i) const { return static_cast<float *>(ptr(i)); }
    size_t bytes(int i) const { return size_t(tensor(i).numel()); }       // byte buffers: as many elements
    long long integer(int i) const
    {
        const long long v = PyLong_AsLongLong(a[i]);
        if (v == -1 && PyErr_Occurred()) throw BadArgument();
        return v;
    }
    bool truth(int i) const
    {
        const int v = PyObject_IsTrue(a[i]);
        if (v < 0) throw BadArgument();
        return v != 0;
    }
    const sq_segtable *seg(int i) const { return reinterpret_cast<const sq_segtable *>(integer(i)); }
};

sq_dtype dtype_of(const at::Tensor &t)
{
    if (t.scalar_type() == at::kFloat) return SQ_F32;
    if (t.scalar_type() == at::kBFloat16) return SQ_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(t.scalar_type()));
    throw BadArgument();
}

void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct GilRelease {
    PyThreadState *state = PyEval_SaveThread();
    ~GilRelease() { PyEval_RestoreThread(state); }
};

template <typename F>
sq_status without_gil(F f)
{
    const GilRelease released;
    return f();
}

// What the C ABI takes of a tensor with rows: read while the GIL is held.
struct Rows {
    void *p;
    int64_t rows, cols, ld;           // cols: of the last dimension
    bool on_host;
    explicit Rows(const at::Tensor &t) : p(t.data_ptr()), on_host(!t.is_cuda())
    {
        const at::IntArrayRef sizes = t.sizes(), strides = t.strides();
        if (sizes.empty()) (void)t.size(0);                           // throws the error that t.stride(0) gives in Python
        rows = sizes.front(), cols = sizes.back(), ld = strides.front();
    }
};

template <typename F>
PyObject *guarded(const char *name, Py_ssize_t n, Py_ssize_t want, F f)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, not %zd", name, want, n);
        return nullptr;
    }
    try {
        return f();
    } catch (const BadArgument &) {
        return nullptr;
    } catch (...) {                  // torch's own errors, as torch's Python methods raise them
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

// code matrix [rows, K] with a 128-byte padded row pitch, as binding.new_codes makes it
at::Tensor new_codes(int64_t rows, int64_t K, const at::Tensor &like)
{
    return at::empty({rows, (K + 127) / 128 * 128}, like.options().dtype(at::kByte)).narrow(1, 0, K);
}

// X, Wq, seg, code, s_pos, s_neg, s_w, bias, Y, scratch, workspace, x_stage, y_stage, flags
PyObject *layer_forward(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("layer_forward", n, 14, [&] {
        const Args a{args};
        const sq_dtype dx = dtype_of(a.matrix(0)), dy = dtype_of(a.tensor(8));
        const Rows X(a.matrix(0)), W(a.tensor(1)), Y(a.tensor(8));
        const sq_segtable *seg = a.seg(2);
        const sq_code code = sq_code(a.integer(3));
        const float *sp = a.f32(4), *sn = a.f32(5), *sw = a.f32(6), *bias = a.f32(7);
        const uint32_t flags = uint32_t(a.integer(13));
        void *scratch = a.ptr(9), *ws = a.ptr(10), *xs = a.ptr(11), *ys = a.ptr(12), *stream = current_stream();
        const size_t scratch_bytes = a.bytes(9), ws_bytes = a.bytes(10);
        return PyLong_FromLong(without_gil([&] {
            return segquant_layer_forward(X.p, X.on_host, xs, dx, X.rows, X.cols, X.ld, W.p, W.ld, W.rows, seg, code, sp, sn, sw,
                                          bias, flags, Y.p, Y.on_host, ys, dy, Y.ld, scratch, scratch_bytes, ws, ws_bytes, stream);
        }));
    });
}

// X, seg, s_pos, s_neg, code, flags, c_pos, c_neg
PyObject *quantize_act(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("quantize_act", n, 8, [&] {
        const Args a{args};
        const sq_dtype dx = dtype_of(a.matrix(0));
        const Rows X(a.matrix(0)), C(a.tensor(6));
        const sq_segtable *seg = a.seg(1);
        const float *sp = a.f32(2), *sn = a.f32(3);
        const sq_code code = sq_code(a.integer(4));
        const uint32_t flags = uint32_t(a.integer(5));
        void *cn = a.ptr(7), *stream = current_stream();
        return PyLong_FromLong(without_gil([&] {
            return segquant_quantize_act(X.p, dx, X.rows, X.cols, X.ld, seg, sp, sn, code, flags, C.p, cn, C.ld, stream);
        }));
    });
}

// H, seg, s_pos, s_neg, code, flags, act, mult, c_pos, c_neg
PyObject *quantize_act_fused(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("quantize_act_fused", n, 10, [&] {
        const Args a{args};
        const sq_dtype dh = dtype_of(a.matrix(0));
        const Rows H(a.matrix(0)), C(a.tensor(8));
        const sq_segtable *seg = a.seg(1);
        const float *sp = a.f32(2), *sn = a.f32(3), *mult = a.f32(7);
        const sq_code code = sq_code(a.integer(4));
        const uint32_t flags = uint32_t(a.integer(5));
        const sq_act act = sq_act(a.integer(6));
        const int64_t K = act == SQ_ACT_GEGLU ? H.cols / 2 : H.cols;
        void *cn = a.ptr(9), *stream = current_stream();
        return PyLong_FromLong(without_gil([&] {
            return segquant_quantize_act_fused(H.p, dh, H.rows, K, H.ld, seg, sp, sn, code, flags, act, mult, C.p, cn, C.ld, stream);
        }));
    });
}

// X, seg, number of scales, code, is_weight, dual, workspace, flags -> (status, s_pos, s_neg | None)
PyObject *calib_scales(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("calib_scales", n, 8, [&]() -> PyObject * {
        const Args a{args};
        const at::Tensor &x = a.matrix(0);
        const sq_dtype dx = dtype_of(x);
        const Rows X(x);
        const sq_segtable *seg = a.seg(1);
        const int64_t scales = a.integer(2);
        const sq_code code = sq_code(a.integer(3));
        const bool is_weight = a.truth(4), dual = a.truth(5);
        void *ws = a.ptr(6), *stream = current_stream();
        const size_t ws_bytes = a.bytes(6);
        const uint32_t flags = uint32_t(a.integer(7));
        const auto f32 = x.options().dtype(at::kFloat);
        at::Tensor sp = at::empty({scales}, f32), sn;
        if (dual && !is_weight) sn = at::empty({scales}, f32);
        float *s_pos = sp.data_ptr<float>(), *s_neg = sn.defined() ? sn.data_ptr<float>() : nullptr;
        const sq_status st = without_gil([&] {
            return segquant_calib_scales(X.p, dx, X.rows, X.cols, X.ld, seg, code, is_weight, dual, flags, s_pos, s_neg, ws, ws_bytes, stream);
        });
        return Py_BuildValue("(iNN)", int(st), THPVariable_Wrap(sp), THPVariable_Wrap(sn));
    });
}

// W, seg, s_w, code, flags, Wq | None -> (status, Wq)
PyObject *quantize_weight(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("quantize_weight", n, 6, [&]() -> PyObject * {
        const Args a{args};
        const at::Tensor &w = a.matrix(0);
        const sq_dtype dw = dtype_of(w);
        const Rows W(w);
        const sq_segtable *seg = a.seg(1);
        const float *sw = a.f32(2);
        const sq_code code = sq_code(a.integer(3));
        const uint32_t flags = uint32_t(a.integer(4));
        const at::Tensor q = a.none(5) ? new_codes(W.rows, W.cols, w) : a.tensor(5);
        const Rows C(q);
        void *stream = current_stream();
        const sq_status st = without_gil([&] {
            return segquant_quantize_weight(W.p, dw, W.rows, W.cols, W.ld, seg, sw, code, flags, C.p, C.ld, stream);
        });
        return Py_BuildValue("(iN)", int(st), THPVariable_Wrap(q));
    });
}

// Xq_pos, Xq_neg | None, Wq, seg, code, s_pos, s_neg | None, s_w, bias, Y, acc_dump | None, workspace, kind
enum GemmCall : int { kSeglinear = 0, kDualscale = 1, kW4a8 = 2 };
PyObject *gemm(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("gemm", n, 13, [&] {
        const Args a{args};
        const sq_dtype dy = dtype_of(a.tensor(9));
        const Rows X(a.matrix(0)), W(a.tensor(2)), Y(a.tensor(9));
        const sq_segtable *seg = a.seg(3);
        const sq_code code = sq_code(a.integer(4));
        const float *sp = a.f32(5), *sn = a.f32(6), *sw = a.f32(7), *bias = a.f32(8);
        void *xn = a.ptr(1), *dump = a.ptr(10), *ws = a.ptr(11), *stream = current_stream();
        const size_t ws_bytes = a.bytes(11);
        const int kind = int(a.integer(12));
        const int64_t M = X.rows, K = X.cols, N = W.rows;
        return PyLong_FromLong(without_gil([&] {
            if (kind == kW4a8)
                return segquant_w4a8_gemm(X.p, xn, X.ld, W.p, W.ld, M, N, K, seg, sp, sn, sw, bias, Y.p, dy, Y.ld, dump, ws, ws_bytes,
                                          stream);
            if (kind == kDualscale)
                return segquant_dualscale_gemm(X.p, xn, X.ld, W.p, W.ld, M, N, K, seg, code, sp, sn, sw, bias, Y.p, dy, Y.ld, dump, ws,
                                               ws_bytes, stream);
            return segquant_seglinear_gemm(X.p, X.ld, W.p, W.ld, M, N, K, seg, code, sp, sw, bias, Y.p, dy, Y.ld, dump, ws, ws_bytes,
                                           stream);
        }));
    });
}

// X, seg, P, dual, bits, flags -> (status, s_pos, s_neg | None, c_pos, c_neg | None)
PyObject *quantize_per_row(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("quantize_per_row", n, 6, [&]() -> PyObject * {
        const Args a{args};
        const at::Tensor &x = a.matrix(0);
        const sq_dtype dx = dtype_of(x);
        const Rows X(x);
        const int64_t P = a.integer(2);
        const sq_segtable *seg = a.seg(1);
        const bool dual = a.truth(3);
        const int bits = int(a.integer(4));
        const uint32_t flags = uint32_t(a.integer(5));
        const auto scales = x.options().dtype(at::kFloat);
        at::Tensor sp = at::empty({X.rows, P}, scales), sn, cp = new_codes(X.rows, X.cols, x), cn;
        if (dual) {
            sn = at::empty({X.rows, P}, scales);
            cn = new_codes(X.rows, X.cols, x);
        }
        float *s_pos = sp.data_ptr<float>(), *s_neg = dual ? sn.data_ptr<float>() : nullptr;
        const Rows C(cp);
        void *c_neg = dual ? cn.data_ptr() : nullptr;
        void *stream = current_stream();
        const sq_status st = without_gil([&] {
            return segquant_quantize_per_row(X.p, dx, X.rows, X.cols, X.ld, seg, bits, flags, s_pos, s_neg, C.p, c_neg, C.ld, stream);
        });
        return Py_BuildValue("(iNNNN)", int(st), THPVariable_Wrap(sp), THPVariable_Wrap(sn), THPVariable_Wrap(cp), THPVariable_Wrap(cn));
    });
}

// Wq4, Wq8
PyObject *unpack_w4(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("unpack_w4", n, 2, [&] {
        const Args a{args};
        const Rows W4(a.matrix(0)), W8(a.tensor(1));
        void *stream = current_stream();
        return PyLong_FromLong(without_gil([&] {
            return segquant_unpack_w4(W4.p, W4.ld, W4.rows, 2 * W4.cols, W8.p, W8.ld, stream);
        }));
    });
}

// address of a plan
PyObject *plan_run(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded("plan_run", n, 1, [&] {
        const Args a{args};
        const sq_plan *plan = reinterpret_cast<const sq_plan *>(a.integer(0));
        void *stream = current_stream();
        return PyLong_FromLong(without_gil([&] { return segquant_plan_run(plan, stream); }));
    });
}

#define SQ_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SQ_METHOD(layer_forward), SQ_METHOD(quantize_act), SQ_METHOD(quantize_act_fused), SQ_METHOD(gemm),
                         SQ_METHOD(quantize_per_row), SQ_METHOD(calib_scales), SQ_METHOD(quantize_weight), SQ_METHOD(unpack_w4), SQ_METHOD(plan_run), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module_def); }
