// Host side of the Python binding: the calls of hbfp.h on torch tensors, without the per-argument work of a Python
// marshaller. A small GEMM is three kernels of 2-4 us; ctypes, the format structures and the tensors' attributes cost
// 20 us of Python per call around them, this file about 3 us. Arguments are checked and outputs allocated here; every
// step of the path runs in the CUDA kernels of the library, whose entry points are handed over by address (bind), so
// that whichever build of it the binding has loaded is the one that runs.
//
// Every function returns its result, or the library's status code as a Python int (the binding raises it).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/function.h>
#include <torch/csrc/autograd/functions/utils.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/autograd/saved_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>
#include <ATen/ATen.h>
#include <ATen/core/LegacyTypeDispatch.h>
#include <ATen/cuda/CUDAContext.h>
#include <c10/cuda/CUDACachingAllocator.h>

#include "hbfp.h"

namespace {

// ------------------------------------------------------------------------------ the library

struct Api {
    decltype(&hbfp_packed_layout) packed_layout;
    decltype(&hbfp_quantize) quantize;
    decltype(&hbfp_gemm_q_workspace) gemm_q_workspace;
    decltype(&hbfp_wide_update_value) wide_update;
    decltype(&hbfp_wide_dequantize) wide_dequantize;
    decltype(&hbfp_conv_forward) conv_forward;
    decltype(&hbfp_conv_dgrad_filters) conv_dgrad_filters;
    decltype(&hbfp_im2col_packed_t) im2col_packed_t;
    decltype(&hbfp_im2col_packed) im2col_packed;
    decltype(&hbfp_gemm_q_bias) gemm_q_bias;
    decltype(&hbfp_column_sums) column_sums;
    decltype(&hbfp_fold_taps) fold_taps;
} api;

// ------------------------------------------------------------------------------ arguments

PyObject *n_mant_bits, *n_block, *n_tile, *n_rounding, *n_exp_mode, *n_seed, *n_stream_id, *n_mant, *n_exps, *n_fmt;

struct Fail {};          // a Python error is set

long long as_ll(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Fail{};
    return v;
}
PyObject* attr(PyObject* o, PyObject* name) {
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) throw Fail{};
    return v;
}
uint64_t attr_mask(PyObject* o, PyObject* name) {
    PyObject* v = attr(o, name);
    const unsigned long long r = PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    if (r == (unsigned long long)-1 && PyErr_Occurred()) throw Fail{};
    return r;
}
hbfp_format format_of(PyObject* f) {
    hbfp_format c{};
    c.struct_size = sizeof(c);
    c.mant_bits = (int32_t)attr_mask(f, n_mant_bits);
    c.block = (int32_t)attr_mask(f, n_block);
    c.tile = (int32_t)attr_mask(f, n_tile);
    c.rounding = (int32_t)attr_mask(f, n_rounding);
    c.exp_mode = (int32_t)attr_mask(f, n_exp_mode);
    c.stream_id = (uint32_t)attr_mask(f, n_stream_id);
    c.seed = attr_mask(f, n_seed);
    return c;
}
at::Tensor tensor_of(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
        throw Fail{};
    }
    return THPVariable_Unpack(o);
}
[[noreturn]] void value_error(const char* fmt, const char* name) {
    PyErr_Format(PyExc_ValueError, fmt, name);
    throw Fail{};
}
void check_f32(const at::Tensor& x, const char* name) {
    if (!(x.is_cuda() && x.scalar_type() == at::kFloat && x.dim() == 2 && (x.size(1) <= 1 || x.stride(1) == 1)))
        value_error("%s must be a 2-D float32 CUDA tensor with contiguous rows", name);
}
void check_f32_cpp(const at::Tensor& x) {
    TORCH_CHECK_VALUE(x.is_cuda() && x.scalar_type() == at::kFloat && x.dim() == 2 && (x.size(1) <= 1 || x.stride(1) == 1),
                      "operand must be a 2-D float32 CUDA tensor with contiguous rows");
}
int64_t ld_of(const at::Tensor& x) { return x.size(0) > 1 ? x.stride(0) : std::max<int64_t>(x.size(1), 1); }

// The interpreter lock is let go while memory is allocated and kernels are launched, so that other Python threads run when the
// launch queue is full or the allocator has to wait for the GPU (a call through ctypes lets it go, too). Nothing in there may touch
// a Python object.
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    NoGil() = default;
    NoGil(const NoGil&) = delete;
    ~NoGil() { PyEval_RestoreThread(state); }
};

void* cur_stream() { return at::cuda::getCurrentCUDAStream().stream(); }

at::Tensor empty_f32(at::IntArrayRef sizes, const at::Tensor& like) { return at::empty(sizes, like.options().dtype(at::kFloat).requires_grad(false)); }
at::Tensor empty_i8(int64_t n, const at::Tensor& like) { return at::empty({n}, like.options().dtype(at::kChar).requires_grad(false)); }

// An operand of hbfp_gemm_q: a packed one (an object with mant, exps and fmt) or an FP32 matrix. `keep` holds the tensors.
struct Operand {
    hbfp_operand o{};
    at::Tensor data, exps;
};
Operand operand_of(PyObject* x, long long trans, PyObject* fmt) {
    Operand r;
    r.o.struct_size = sizeof(r.o);
    if (THPVariable_Check(x)) {
        r.data = THPVariable_Unpack(x);
        check_f32(r.data, "operand");
        r.o.kind = HBFP_OPERAND_FP32;
        r.o.data = r.data.data_ptr();
        r.o.ld = ld_of(r.data);
        r.o.trans = (int32_t)trans;
        r.o.fmt = format_of(fmt);
        return r;
    }
    PyObject *m = attr(x, n_mant), *e = nullptr, *f = nullptr;
    try {
        e = attr(x, n_exps);
        f = attr(x, n_fmt);
        r.data = tensor_of(m, "mantissas");
        r.exps = tensor_of(e, "exponents");
        r.o.fmt = format_of(f);
    } catch (...) {
        Py_DECREF(m); Py_XDECREF(e); Py_XDECREF(f);
        throw;
    }
    Py_DECREF(m); Py_DECREF(e); Py_DECREF(f);
    r.o.kind = HBFP_OPERAND_PACKED;
    r.o.data = r.data.data_ptr();
    r.o.exps = (const int8_t*)r.exps.data_ptr();
    return r;
}

// hbfp_gemm_q with the workspace from the caching allocator (stream-ordered, as a temporary tensor's memory is).
int run_gemm(int64_t M, int64_t N, int64_t K, const hbfp_operand& a, const hbfp_operand& b, const at::Tensor& out, const at::Tensor* ws, uint32_t flags,
             const float* bias = nullptr) {
    if (ws) return api.gemm_q_bias(M, N, K, &a, &b, bias, (float*)out.data_ptr(), ld_of(out), ws->data_ptr(), (size_t)ws->numel(), flags, cur_stream());
    size_t bytes = 0;
    const int rc = api.gemm_q_workspace(M, N, K, &a, &b, &bytes);
    if (rc) return rc;
    c10::DataPtr mem;
    if (bytes) mem = c10::cuda::CUDACachingAllocator::get()->allocate(bytes);
    return api.gemm_q_bias(M, N, K, &a, &b, bias, (float*)out.data_ptr(), ld_of(out), mem.get(), bytes, flags, cur_stream());
}

// The exception in flight as torch's own binding raises it: out of memory as torch.OutOfMemoryError, a Python error as itself.
PyObject* python_error_set() {
    torch::translate_exception_to_python(std::current_exception());
    return nullptr;
}
template <class F>
auto without_gil(F f) {
    NoGil free;
    return f();
}
template <class F>
PyObject* guarded(F f) {
    try {
        at::AutoDispatchBelowADInplaceOrView below;          // plain tensors: nothing here is recorded for autograd
        return f();
    } catch (const Fail&) {
        return nullptr;
    } catch (...) {
        return python_error_set();
    }
}
// A layer's forward pass: it records its own node, so nothing is switched off around it; a library error is already a Python one.
template <class F>
PyObject* layer_call(F f) {
    try {
        return f();
    } catch (const Fail&) {
        return nullptr;
    } catch (...) {
        return python_error_set();
    }
}
PyObject* code(int rc) { return PyLong_FromLong(rc); }
bool want(Py_ssize_t n, Py_ssize_t expected) {
    if (n == expected) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", expected, n);
    return false;
}
PyObject* same(PyObject* o) { Py_INCREF(o); return o; }

// ------------------------------------------------------------------------------ calls

// A call's packed result: buffers handed in, or (None) allocated for it.
struct Buffers {
    at::Tensor m, e;
    Buffers(PyObject* mant, PyObject* exps) {
        if (mant == Py_None) return;
        m = tensor_of(mant, "mantissas");
        e = tensor_of(exps, "exponents");
    }
    int make(int64_t rows, int64_t k, const hbfp_format& f, const at::Tensor& like) {
        if (m.defined()) return HBFP_OK;
        hbfp_layout L;
        const int rc = api.packed_layout(rows, k, &f, &L);
        if (rc) return rc;
        m = empty_i8(L.mant_bytes, like);
        e = empty_i8(L.exp_bytes, like);
        return HBFP_OK;
    }
};

// packed_layout(rows, k, fmt) -> the members of hbfp_layout by name
PyObject* packed_layout(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 3)) return nullptr;
    return guarded([&]() -> PyObject* {
        const int64_t rows = as_ll(a[0]), k = as_ll(a[1]);
        const hbfp_format f = format_of(a[2]);
        hbfp_layout L;
        const int rc = api.packed_layout(rows, k, &f, &L);
        if (rc) return code(rc);
        return Py_BuildValue("{sLsLsLsLsLsLsLsLsLsLsL}", "rows", (long long)L.rows, "k", (long long)L.k, "b", (long long)L.b, "bp", (long long)L.bp, "nkb", (long long)L.nkb,
                             "kst", (long long)L.kst, "planes", (long long)L.planes, "plane_stride", (long long)L.plane_stride, "rs", (long long)L.rs,
                             "mant_bytes", (long long)L.mant_bytes, "exp_bytes", (long long)L.exp_bytes);
    });
}

// quantize(x, axis, fmt, mant or None, exps or None) -> (mant, exps)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 5)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor x = tensor_of(a[0], "x");
        check_f32(x, "x");
        const int axis = (int)as_ll(a[1]);
        const hbfp_format f = format_of(a[2]);
        Buffers out(a[3], a[4]);
        const int rc = without_gil([&] {
            const int bad = axis == 1 ? out.make(x.size(0), x.size(1), f, x) : out.make(x.size(1), x.size(0), f, x);
            return bad ? bad : api.quantize((const float*)x.data_ptr(), x.size(0), x.size(1), ld_of(x), axis, &f, out.m.data_ptr(), (int8_t*)out.e.data_ptr(), cur_stream());
        });
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", a[3] == Py_None ? THPVariable_Wrap(out.m) : same(a[3]), a[3] == Py_None ? THPVariable_Wrap(out.e) : same(a[4]));
    });
}

// gemm(transA, transB, A, B, fmtA, fmtB, out or None, workspace or None, flags) -> out
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 9)) return nullptr;
    return guarded([&]() -> PyObject* {
        const int ta = PyObject_IsTrue(a[0]), tb = PyObject_IsTrue(a[1]);
        const at::Tensor A = tensor_of(a[2], "A"), B = tensor_of(a[3], "B");
        check_f32(A, "A");
        check_f32(B, "B");
        const int64_t M = A.size(ta ? 1 : 0), K = A.size(ta ? 0 : 1), K2 = B.size(tb ? 1 : 0), N = B.size(tb ? 0 : 1);
        if (K != K2) value_error("%s", "contraction extents differ");
        hbfp_operand oa{}, ob{};
        oa.struct_size = ob.struct_size = sizeof(oa);
        oa.kind = ob.kind = HBFP_OPERAND_FP32;
        oa.data = A.data_ptr(); oa.ld = ld_of(A); oa.trans = (int32_t)as_ll(a[0]); oa.fmt = format_of(a[4]);
        ob.data = B.data_ptr(); ob.ld = ld_of(B); ob.trans = (int32_t)as_ll(a[1]); ob.fmt = format_of(a[5]);
        const bool fresh = a[6] == Py_None;
        at::Tensor out, ws;
        if (!fresh) out = tensor_of(a[6], "out");
        if (a[7] != Py_None) ws = tensor_of(a[7], "workspace");
        const uint32_t flags = (uint32_t)as_ll(a[8]);
        const int rc = without_gil([&] {
            if (fresh) out = empty_f32({M, N}, A);
            return run_gemm(M, N, K, oa, ob, out, ws.defined() ? &ws : nullptr, flags);
        });
        if (rc) return code(rc);
        return fresh ? THPVariable_Wrap(out) : same(a[6]);
    });
}

// gemm_q(M, N, K, a, b, transA, transB, fmtA or None, fmtB or None, out or None, workspace or None, flags) -> out
PyObject* gemm_q(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 12)) return nullptr;
    return guarded([&]() -> PyObject* {
        const int64_t M = as_ll(a[0]), N = as_ll(a[1]), K = as_ll(a[2]);
        const Operand oa = operand_of(a[3], as_ll(a[5]), a[7]), ob = operand_of(a[4], as_ll(a[6]), a[8]);
        const bool fresh = a[9] == Py_None;
        at::Tensor out, ws;
        if (!fresh) out = tensor_of(a[9], "out");
        if (a[10] != Py_None) ws = tensor_of(a[10], "workspace");
        const uint32_t flags = (uint32_t)as_ll(a[11]);
        const int rc = without_gil([&] {
            if (fresh) out = empty_f32({M, N}, oa.data);
            return run_gemm(M, N, K, oa.o, ob.o, out, ws.defined() ? &ws : nullptr, flags);
        });
        if (rc) return code(rc);
        return fresh ? THPVariable_Wrap(out) : same(a[9]);
    });
}

// wide_update(mant, exps, delta, fmt, c0 or None, c1 or None, whether the FP32 value is wanted) -> None or the value;
// c0, c1: objects with mant and exps
struct ViewPtrs { void* m0 = nullptr; int8_t* e0 = nullptr; void* m1 = nullptr; int8_t* e1 = nullptr; };
void view_of(PyObject* v, void** m, int8_t** e) {
    PyObject* pm = attr(v, n_mant);
    PyObject* pe = PyObject_GetAttr(v, n_exps);
    if (!pe) { Py_DECREF(pm); throw Fail{}; }
    const bool ok = THPVariable_Check(pm) && THPVariable_Check(pe);
    if (ok) { *m = THPVariable_Unpack(pm).data_ptr(); *e = (int8_t*)THPVariable_Unpack(pe).data_ptr(); }
    Py_DECREF(pm); Py_DECREF(pe);
    if (!ok) { PyErr_SetString(PyExc_TypeError, "a view holds tensors"); throw Fail{}; }
}
PyObject* wide_update(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 7)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor m = tensor_of(a[0], "mantissas"), e = tensor_of(a[1], "exponents"), d = tensor_of(a[2], "delta");
        check_f32(d, "delta");
        if (d.dim() != 2 || d.size(0) != m.size(0) || d.size(1) != m.size(1)) value_error("%s must have the shape of the weights", "delta");
        const hbfp_format f = format_of(a[3]);
        ViewPtrs v;
        if (a[4] != Py_None) { view_of(a[4], &v.m0, &v.e0); view_of(a[5], &v.m1, &v.e1); }
        const bool wanted = a[6] == Py_True;
        at::Tensor value;
        const int rc = without_gil([&] {
            if (wanted) value = empty_f32({m.size(0), m.size(1)}, m);
            return api.wide_update((int16_t*)m.data_ptr(), (int8_t*)e.data_ptr(), (const float*)d.data_ptr(), m.size(0), m.size(1), ld_of(d), &f,
                                   v.m0, v.e0, v.m1, v.e1, wanted ? (float*)value.data_ptr() : nullptr, m.size(1), cur_stream());
        });
        return !rc && value.defined() ? THPVariable_Wrap(value) : code(rc);
    });
}

// wide_dequantize(mant, exps, tile, out or None) -> out
PyObject* wide_dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 4)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor m = tensor_of(a[0], "mantissas"), e = tensor_of(a[1], "exponents");
        const bool fresh = a[3] == Py_None;
        const int32_t tile = (int32_t)as_ll(a[2]);
        at::Tensor out;
        if (!fresh) {
            out = tensor_of(a[3], "out");
            check_f32(out, "out");
        }
        const int rc = without_gil([&] {
            if (fresh) out = empty_f32({m.size(0), m.size(1)}, m);
            return api.wide_dequantize((const int16_t*)m.data_ptr(), (const int8_t*)e.data_ptr(), m.size(0), m.size(1), tile, (float*)out.data_ptr(), ld_of(out), cur_stream());
        });
        if (rc) return code(rc);
        return fresh ? THPVariable_Wrap(out) : same(a[3]);
    });
}

// conv_forward(px, filters, n, h, w, c, kh, kw, pad, nf, out or None) -> out
PyObject* conv_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 11)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Operand px = operand_of(a[0], 0, Py_None), fl = operand_of(a[1], 0, Py_None);
        const int64_t nn = as_ll(a[2]), h = as_ll(a[3]), w = as_ll(a[4]), c = as_ll(a[5]), nf = as_ll(a[9]);
        const int kh = (int)as_ll(a[6]), kw = (int)as_ll(a[7]), pad = (int)as_ll(a[8]);
        const bool fresh = a[10] == Py_None;
        at::Tensor out;
        if (!fresh) {
            out = tensor_of(a[10], "out");
            check_f32(out, "out");
        }
        const int rc = without_gil([&] {
            if (fresh) out = empty_f32({nn * h * w, nf}, px.data);
            return api.conv_forward(px.o.data, px.o.exps, nn, h, w, c, kh, kw, pad, &px.o.fmt, &fl.o, nf, (float*)out.data_ptr(), ld_of(out), cur_stream());
        });
        if (rc) return code(rc);
        return fresh ? THPVariable_Wrap(out) : same(a[10]);
    });
}

// conv_dgrad_filters(c1, kh, kw, c_in, c_out, mant or None, exps or None) -> (mant, exps)
PyObject* conv_dgrad_filters(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 7)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Operand c1 = operand_of(a[0], 0, Py_None);
        const int kh = (int)as_ll(a[1]), kw = (int)as_ll(a[2]);
        const int64_t ci = as_ll(a[3]), co = as_ll(a[4]);
        Buffers out(a[5], a[6]);
        const int rc = without_gil([&] {
            const int bad = out.make(ci, (int64_t)kh * kw * co, c1.o.fmt, c1.data);
            return bad ? bad : api.conv_dgrad_filters(c1.o.data, c1.o.exps, kh, kw, ci, co, &c1.o.fmt, out.m.data_ptr(), (int8_t*)out.e.data_ptr(), cur_stream());
        });
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", THPVariable_Wrap(out.m), THPVariable_Wrap(out.e));
    });
}

// im2col_packed_t(x, kh, kw, pad, fmt, mant or None, exps or None) -> (mant, exps)
PyObject* im2col_packed_t(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 7)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor x = tensor_of(a[0], "x");
        if (!(x.is_cuda() && x.scalar_type() == at::kFloat && x.dim() == 4 && x.is_contiguous()))
            value_error("%s must be a contiguous float32 CUDA tensor [n][h][w][c]", "x");
        const int kh = (int)as_ll(a[1]), kw = (int)as_ll(a[2]);
        const int pad = (int)as_ll(a[3]);
        const hbfp_format f = format_of(a[4]);
        Buffers out(a[5], a[6]);
        const int rc = without_gil([&] {
            const int bad = out.make((int64_t)kh * kw * x.size(3), x.size(0) * x.size(1) * x.size(2), f, x);
            return bad ? bad : api.im2col_packed_t((const float*)x.data_ptr(), x.size(0), x.size(1), x.size(2), x.size(3), kh, kw, pad, &f, out.m.data_ptr(),
                                                   (int8_t*)out.e.data_ptr(), cur_stream());
        });
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", THPVariable_Wrap(out.m), THPVariable_Wrap(out.e));
    });
}

// ------------------------------------------------------------------------------ layers

// The two layers as autograd nodes of their own. As Python functions their forward and backward passes spent most of a
// training step in the interpreter: argument marshalling, packed-operand and format objects, one call into the library per
// product and the hand-over between the autograd engine and Python for every layer. A node runs its whole pass here, on the
// engine's thread, without the interpreter.

PyObject* error_type = nullptr;              // HbfpError(code, where)

// Raises HbfpError from code that may hold no interpreter lock.
[[noreturn]] void raise_status(int rc, const char* where) {
    pybind11::gil_scoped_acquire gil;
    PyObject* e = PyObject_CallFunction(error_type, "is", rc, where);
    if (e) {
        PyErr_SetObject(error_type, e);
        Py_DECREF(e);
    }
    python_error err;
    err.persist();
    throw err;
}
void ok_or_raise(int rc, const char* where) {
    if (rc) raise_status(rc, where);
}

struct PackedTensor {
    at::Tensor mant, exps;
    hbfp_format fmt{};
    hbfp_operand operand() const {
        hbfp_operand o{};
        o.struct_size = sizeof(o);
        o.kind = HBFP_OPERAND_PACKED;
        o.data = mant.data_ptr();
        o.exps = (const int8_t*)exps.data_ptr();
        o.fmt = fmt;
        return o;
    }
};
PackedTensor packed_of(PyObject* x) {
    const Operand o = operand_of(x, 0, Py_None);
    if (o.o.kind != HBFP_OPERAND_PACKED) {
        PyErr_SetString(PyExc_TypeError, "a packed operand is expected");
        throw Fail{};
    }
    return {o.data, o.exps, o.o.fmt};
}
hbfp_operand fp32_operand(const at::Tensor& x, int trans, const hbfp_format& f) {
    check_f32_cpp(x);
    hbfp_operand o{};
    o.struct_size = sizeof(o);
    o.kind = HBFP_OPERAND_FP32;
    o.data = x.data_ptr();
    o.ld = ld_of(x);
    o.trans = trans;
    o.fmt = f;
    return o;
}
hbfp_format make_format(int mant_bits, int block, int rounding, uint64_t seed, uint32_t stream_id) {
    hbfp_format f{};
    f.struct_size = sizeof(f);
    f.mant_bits = mant_bits;
    f.block = block;
    f.rounding = rounding;
    f.seed = seed;
    f.stream_id = stream_id;
    return f;
}
PackedTensor alloc_packed(int64_t rows, int64_t k, const hbfp_format& f, const at::Tensor& like, const char* where) {
    hbfp_layout L;
    ok_or_raise(api.packed_layout(rows, k, &f, &L), where);
    return {empty_i8(L.mant_bytes, like), empty_i8(L.exp_bytes, like), f};
}
at::Tensor product(int64_t M, int64_t N, int64_t K, const hbfp_operand& a, const hbfp_operand& b, const at::Tensor& like, const float* bias = nullptr) {
    at::Tensor out = empty_f32({M, N}, like);
    ok_or_raise(run_gemm(M, N, K, a, b, out, nullptr, HBFP_GEMM_AUTO, bias), "hbfp_gemm_q");
    return out;
}
// Whether a pass runs under something that has to see an autograd.Function to record, transform or refuse it: a trace, a functorch
// transform, an input with a forward-mode tangent. A node of this file would vanish from the first (what is left of it there is an
// empty tensor) and drop the tangent; the layer then goes through its Python function (autograd.py).
bool has_tangent(const at::Tensor& t) {
    const torch::autograd::AutogradMeta* meta = t.defined() ? torch::autograd::impl::get_autograd_meta(t) : nullptr;
    return meta && meta->fw_grad_ && t._fw_grad(/*level=*/0).defined();
}
bool needs_function(const at::Tensor& x, const at::Tensor& weight, const at::Tensor& bias = at::Tensor()) {
    return torch::jit::tracer::isTracing() || c10::impl::tls_is_dispatch_key_included(c10::DispatchKey::FuncTorchDynamicLayerFrontMode) ||
           has_tangent(x) || has_tangent(weight) || has_tangent(bias);
}
// Everything a pass computes lies below autograd; gradients come out as plain tensors.
struct Below {
    at::AutoDispatchBelowADInplaceOrView below;
    c10::AutoGradMode off{false};
};
using torch::autograd::SavedVariable;
using torch::autograd::variable_list;

struct LinearNode : public torch::autograd::Node {
    SavedVariable x_;
    PackedTensor c1;
    int mant_bits, tile, batch_block, rounding;
    uint64_t seed;
    uint32_t stream_id;
    int64_t fin, fout;
    // X (which = 0) or dY (which = 2) in blocks along a feature axis or along the batch axis
    hbfp_format act(int which, bool batch_axis) const { return make_format(mant_bits, batch_axis ? batch_block : tile, rounding, seed, stream_id + which); }
    std::string name() const override { return "HbfpLinearBackward"; }
    void release_variables() override {
        std::lock_guard<std::mutex> lock(mutex_);            // backward passes of several threads may meet in a node
        x_.reset_data();
    }
    variable_list apply(variable_list&& grads) override {
        std::lock_guard<std::mutex> lock(mutex_);
        variable_list out(3);
        if (!grads[0].defined()) grads[0] = input_metadata(0).zeros_like();      // as autograd.Function hands it over
        const at::Tensor x0 = x_.unpack(shared_from_this());
        // with create_graph the bias gradient can be differentiated further; the products have no second derivative
        const bool recorded_sum = task_should_compute_output(2) && at::GradMode::is_enabled() && grads[0].requires_grad();
        if (recorded_sum) out[2] = grads[0].sum(0);
        Below guard;
        const at::Tensor dy = grads[0].contiguous(), x = x0.contiguous();
        check_f32_cpp(dy);
        const int64_t batch = x.size(0);
        // backward-data on the shared weight view; backward-weight with blocks down the columns of X and dY
        if (task_should_compute_output(0)) out[0] = product(batch, fin, fout, fp32_operand(dy, 0, act(2, false)), c1.operand(), dy);
        // (of all columns of X: where there are more than the weights have rows, autograd refuses the gradient's shape)
        if (task_should_compute_output(1)) out[1] = product(x.size(1), fout, batch, fp32_operand(x, 1, act(0, true)), fp32_operand(dy, 0, act(2, true)), dy);
        if (task_should_compute_output(2) && !recorded_sum) {
            out[2] = empty_f32({fout}, dy);
            ok_or_raise(api.column_sums((const float*)dy.data_ptr(), batch, fout, ld_of(dy), (float*)out[2].data_ptr(), cur_stream()), "hbfp_column_sums");
        }
        return out;
    }
};

// linear(x, weight, bias or None, c0, c1, mant_bits, tile, batch_block, rounding, seed, stream_id) -> y, or None where the pass
// needs a Python function
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 11)) return nullptr;
    return layer_call([&]() -> PyObject* {
        const at::Tensor x = tensor_of(a[0], "x"), w = tensor_of(a[1], "weight");
        const at::Tensor bias = a[2] != Py_None ? tensor_of(a[2], "bias") : at::Tensor();
        if (needs_function(x, w, bias)) return same(Py_None);
        // a bias of another type, shape or place (a layer cast to half precision, one value for all outputs): the general addition
        if (bias.defined() && !(bias.device() == x.device() && bias.scalar_type() == at::kFloat && bias.dim() == 1 && bias.size(0) == w.size(1)))
            return same(Py_None);
        const PackedTensor c0 = packed_of(a[3]);
        LinearNode proto;
        proto.mant_bits = (int)as_ll(a[5]); proto.tile = (int)as_ll(a[6]); proto.batch_block = (int)as_ll(a[7]); proto.rounding = (int)as_ll(a[8]);
        proto.seed = PyLong_AsUnsignedLongLongMask(a[9]);
        proto.stream_id = (uint32_t)PyLong_AsUnsignedLongLongMask(a[10]);
        if (PyErr_Occurred()) throw Fail{};
        proto.fin = w.size(0);
        proto.fout = w.size(1);
        at::Tensor y;
        {
            Below guard;
            NoGil free;
            const at::Tensor xc = x.contiguous();
            const at::Tensor bc = bias.defined() ? bias.contiguous() : bias;
            y = product(xc.size(0), proto.fout, proto.fin, fp32_operand(xc, 0, proto.act(0, false)), c0.operand(), xc, bc.defined() ? (const float*)bc.data_ptr() : nullptr);
        }
        if (torch::autograd::compute_requires_grad(x, w, bias)) {
            auto node = std::shared_ptr<LinearNode>(new LinearNode(), torch::autograd::deleteNode);
            node->set_next_edges(torch::autograd::collect_next_edges(x, w, bias));
            node->x_ = SavedVariable(x, false);
            node->c1 = packed_of(a[4]);
            node->mant_bits = proto.mant_bits; node->tile = proto.tile; node->batch_block = proto.batch_block; node->rounding = proto.rounding;
            node->seed = proto.seed; node->stream_id = proto.stream_id; node->fin = proto.fin; node->fout = proto.fout;
            torch::autograd::set_history(y, node);
        }
        return THPVariable_Wrap(y);
    });
}

struct ConvNode : public torch::autograd::Node {
    SavedVariable x_;
    PackedTensor c1;
    int mant_bits, pixel_block;
    int64_t c, f;
    hbfp_format pixels(int which) const { return make_format(mant_bits, (int)c, 0, 0, which); }           // blocks of c channels of a pixel
    hbfp_format batch(int which) const { return make_format(mant_bits, pixel_block, 0, 0, which); }       // blocks of consecutive pixels
    std::string name() const override { return "HbfpConv3x3Backward"; }
    void release_variables() override {
        std::lock_guard<std::mutex> lock(mutex_);            // backward passes of several threads may meet in a node
        x_.reset_data();
    }
    static PackedTensor convert(const at::Tensor& x2, const hbfp_format& fmt) {
        PackedTensor p = alloc_packed(x2.size(0), x2.size(1), fmt, x2, "hbfp_quantize");
        ok_or_raise(api.quantize((const float*)x2.data_ptr(), x2.size(0), x2.size(1), ld_of(x2), 1, &fmt, p.mant.data_ptr(), (int8_t*)p.exps.data_ptr(), cur_stream()),
                    "hbfp_quantize");
        return p;
    }
    // 3 x 3 taps, one pixel of padding, as an implicit GEMM: HBFP_ERR_UNSUPPORTED for shapes the kernel does not cover
    static int implicit(const PackedTensor& px, const PackedTensor& filters, int64_t n, int64_t h, int64_t w, int64_t ch, const at::Tensor& y) {
        const hbfp_operand fo = filters.operand();
        const int64_t nf = y.size(-1);
        return api.conv_forward(px.mant.data_ptr(), (const int8_t*)px.exps.data_ptr(), n, h, w, ch, 3, 3, 1, &px.fmt, &fo, nf, (float*)y.data_ptr(), nf, cur_stream());
    }
    at::Tensor forward(const at::Tensor& x, const PackedTensor& c0) const {
        const int64_t n = x.size(0), h = x.size(1), w = x.size(2), px = n * h * w;
        const PackedTensor q = convert(x.view({px, c}), pixels(0));
        at::Tensor y = empty_f32({n, h, w, f}, x);
        const int rc = implicit(q, c0, n, h, w, c, y);
        if (rc != HBFP_ERR_UNSUPPORTED) {
            ok_or_raise(rc, "hbfp_conv_forward");
            return y;
        }
        // gather the packed operand, then the ordinary GEMM (same product)
        const PackedTensor cols = alloc_packed(px, 9 * c, q.fmt, x, "hbfp_im2col_packed");
        ok_or_raise(api.im2col_packed(q.mant.data_ptr(), (const int8_t*)q.exps.data_ptr(), n, h, w, c, 3, 3, 1, &q.fmt, cols.mant.data_ptr(),
                                      (int8_t*)cols.exps.data_ptr(), cur_stream()), "hbfp_im2col_packed");
        ok_or_raise(run_gemm(px, f, 9 * c, cols.operand(), c0.operand(), y.view({px, f}), nullptr, HBFP_GEMM_AUTO), "hbfp_gemm_q");
        return y;
    }
    at::Tensor data_gradient(const at::Tensor& dy2, int64_t n, int64_t h, int64_t w) const {
        // the convolution of the packed output gradient with the forward weights regrouped (taps turned by 180 degrees,
        // feature-map roles swapped) yields dX itself
        hbfp_layout L;
        int rc = api.packed_layout(c, 9 * f, &c1.fmt, &L);
        if (!rc) {
            const PackedTensor turned{empty_i8(L.mant_bytes, dy2), empty_i8(L.exp_bytes, dy2), c1.fmt};
            rc = api.conv_dgrad_filters(c1.mant.data_ptr(), (const int8_t*)c1.exps.data_ptr(), 3, 3, c, f, &c1.fmt, turned.mant.data_ptr(),
                                        (int8_t*)turned.exps.data_ptr(), cur_stream());
            if (!rc) {
                const PackedTensor g = convert(dy2, pixels(2));
                at::Tensor dx = empty_f32({n, h, w, c}, dy2);
                rc = implicit(g, turned, n, h, w, f, dx);
                if (!rc) return dx;
            }
        }
        if (rc != HBFP_ERR_UNSUPPORTED) raise_status(rc, "hbfp_conv_forward");
        // shapes that route does not cover: gradient of the im2col matrix, then its scatter back onto the pixels (FP32)
        const at::Tensor dcols = product(n * h * w, 9 * c, f, fp32_operand(dy2, 0, pixels(2)), c1.operand(), dy2);
        at::Tensor dx = empty_f32({n, h, w, c}, dy2);
        ok_or_raise(api.fold_taps((const float*)dcols.data_ptr(), n, h, w, c, 3, 3, 1, (float*)dx.data_ptr(), cur_stream()), "hbfp_fold_taps");
        return dx;
    }
    variable_list apply(variable_list&& grads) override {
        std::lock_guard<std::mutex> lock(mutex_);
        variable_list out(2);
        if (!grads[0].defined()) grads[0] = input_metadata(0).zeros_like();      // as autograd.Function hands it over
        const at::Tensor x0 = x_.unpack(shared_from_this());
        Below guard;
        const at::Tensor x = x0.contiguous();
        const int64_t n = x.size(0), h = x.size(1), w = x.size(2), px = n * h * w;
        const at::Tensor dy2 = grads[0].contiguous().view({px, f});
        if (task_should_compute_output(0)) out[0] = data_gradient(dy2, n, h, w);
        if (task_should_compute_output(1)) {
            const hbfp_format fx = batch(0);
            const PackedTensor xt = alloc_packed(9 * c, px, fx, x, "hbfp_im2col_packed_t");
            ok_or_raise(api.im2col_packed_t((const float*)x.data_ptr(), n, h, w, c, 3, 3, 1, &fx, xt.mant.data_ptr(), (int8_t*)xt.exps.data_ptr(), cur_stream()),
                        "hbfp_im2col_packed_t");
            out[1] = product(9 * c, f, px, xt.operand(), fp32_operand(dy2, 0, batch(2)), dy2);
        }
        return out;
    }
};

// conv3x3(x, weight, c0, c1, mant_bits, pixel_block, c, f) -> y, or None where the pass needs a Python function
PyObject* conv3x3(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 8)) return nullptr;
    return layer_call([&]() -> PyObject* {
        const at::Tensor x = tensor_of(a[0], "x"), w = tensor_of(a[1], "weight");
        if (needs_function(x, w)) return same(Py_None);
        if (!(x.is_cuda() && x.scalar_type() == at::kFloat && x.dim() == 4)) value_error("%s must be a float32 CUDA tensor [n][h][w][c]", "x");
        auto node = std::shared_ptr<ConvNode>(new ConvNode(), torch::autograd::deleteNode);
        node->mant_bits = (int)as_ll(a[4]);
        node->pixel_block = (int)as_ll(a[5]);
        node->c = as_ll(a[6]);
        node->f = as_ll(a[7]);
        const PackedTensor c0 = packed_of(a[2]);
        at::Tensor y;
        {
            Below guard;
            NoGil free;
            y = node->forward(x.contiguous(), c0);
        }
        if (torch::autograd::compute_requires_grad(x, w)) {
            node->set_next_edges(torch::autograd::collect_next_edges(x, w));
            node->x_ = SavedVariable(x, false);
            node->c1 = packed_of(a[3]);
            torch::autograd::set_history(y, node);
        }
        return THPVariable_Wrap(y);
    });
}

// bind(type of the error to raise, addresses in the order of Api)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    constexpr Py_ssize_t N = sizeof(Api) / sizeof(void*);
    if (!want(n, N + 1)) return nullptr;
    Py_INCREF(a[0]);
    Py_XSETREF(error_type, a[0]);
    ++a;
    void* p[N];
    for (Py_ssize_t i = 0; i < N; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (!p[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
            return nullptr;
        }
    }
    static_assert(sizeof(p) == sizeof(api), "one address per member");
    memcpy(&api, p, sizeof(api));
    Py_RETURN_NONE;
}

#define HBFP_METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {HBFP_METHOD(bind), HBFP_METHOD(packed_layout), HBFP_METHOD(quantize), HBFP_METHOD(gemm), HBFP_METHOD(gemm_q), HBFP_METHOD(wide_update),
                         HBFP_METHOD(wide_dequantize), HBFP_METHOD(conv_forward), HBFP_METHOD(conv_dgrad_filters),
                         HBFP_METHOD(im2col_packed_t), HBFP_METHOD(linear), HBFP_METHOD(conv3x3),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() {
    struct { PyObject** at; const char* name; } names[] = {{&n_mant_bits, "mant_bits"}, {&n_block, "block"}, {&n_tile, "tile"}, {&n_rounding, "rounding"},
        {&n_exp_mode, "exp_mode"}, {&n_seed, "seed"}, {&n_stream_id, "stream_id"}, {&n_mant, "mant"}, {&n_exps, "exps"}, {&n_fmt, "fmt"}};
    for (auto& x : names)
        if (!(*x.at = PyUnicode_InternFromString(x.name))) return nullptr;
    return PyModule_Create(&module);
}
