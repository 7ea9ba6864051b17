// Host side of the Python binding: the calls of hbfp.h on torch tensors, without the per-argument work of a Python
// marshaller. A small GEMM is three kernels of 2-4 us; ctypes, the format structures and the tensors' attributes cost
// 20 us of Python per call around them, this file about 3 us. Arguments are checked and outputs allocated here; every
// step of the path runs in the CUDA kernels of the library, whose entry points are handed over by address (bind), so
// that whichever build of it the binding has loaded is the one that runs.
//
// Every function returns its result, or the library's status code as a Python int (the binding raises it).
#include <torch/csrc/autograd/python_variable.h>
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
    decltype(&hbfp_gemm_q) gemm_q;
    decltype(&hbfp_gemm_q_workspace) gemm_q_workspace;
    decltype(&hbfp_wide_update_value) wide_update;
    decltype(&hbfp_wide_dequantize) wide_dequantize;
    decltype(&hbfp_conv_forward) conv_forward;
    decltype(&hbfp_conv_dgrad_filters) conv_dgrad_filters;
    decltype(&hbfp_im2col_packed_t) im2col_packed_t;
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
int64_t ld_of(const at::Tensor& x) { return x.size(0) > 1 ? x.stride(0) : std::max<int64_t>(x.size(1), 1); }

void* stream() { return at::cuda::getCurrentCUDAStream().stream(); }

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
int run_gemm(int64_t M, int64_t N, int64_t K, const hbfp_operand& a, const hbfp_operand& b, const at::Tensor& out, const at::Tensor* ws, uint32_t flags) {
    if (ws) return api.gemm_q(M, N, K, &a, &b, (float*)out.data_ptr(), ld_of(out), ws->data_ptr(), (size_t)ws->numel(), flags, stream());
    size_t bytes = 0;
    const int rc = api.gemm_q_workspace(M, N, K, &a, &b, &bytes);
    if (rc) return rc;
    c10::DataPtr mem;
    if (bytes) mem = c10::cuda::CUDACachingAllocator::get()->allocate(bytes);
    return api.gemm_q(M, N, K, &a, &b, (float*)out.data_ptr(), ld_of(out), mem.get(), bytes, flags, stream());
}

template <class F>
PyObject* guarded(F f) {
    try {
        at::AutoDispatchBelowADInplaceOrView below;          // plain tensors: nothing here is recorded for autograd
        return f();
    } catch (const Fail&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
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

// quantize(x, axis, fmt, mant or None, exps or None) -> (mant, exps)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 5)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor x = tensor_of(a[0], "x");
        check_f32(x, "x");
        const int axis = (int)as_ll(a[1]);
        const hbfp_format f = format_of(a[2]);
        at::Tensor m, e;
        if (a[3] == Py_None) {
            hbfp_layout L;
            const int rc = axis == 1 ? api.packed_layout(x.size(0), x.size(1), &f, &L) : api.packed_layout(x.size(1), x.size(0), &f, &L);
            if (rc) return code(rc);
            m = empty_i8(L.mant_bytes, x);
            e = empty_i8(L.exp_bytes, x);
        } else {
            m = tensor_of(a[3], "mantissas");
            e = tensor_of(a[4], "exponents");
        }
        const int rc = api.quantize((const float*)x.data_ptr(), x.size(0), x.size(1), ld_of(x), axis, &f, m.data_ptr(), (int8_t*)e.data_ptr(), stream());
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", a[3] == Py_None ? THPVariable_Wrap(m) : same(a[3]), a[3] == Py_None ? THPVariable_Wrap(e) : same(a[4]));
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
        const at::Tensor out = fresh ? empty_f32({M, N}, A) : tensor_of(a[6], "out");
        at::Tensor ws;
        if (a[7] != Py_None) ws = tensor_of(a[7], "workspace");
        const int rc = run_gemm(M, N, K, oa, ob, out, ws.defined() ? &ws : nullptr, (uint32_t)as_ll(a[8]));
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
        const at::Tensor out = fresh ? empty_f32({M, N}, oa.data) : tensor_of(a[9], "out");
        at::Tensor ws;
        if (a[10] != Py_None) ws = tensor_of(a[10], "workspace");
        const int rc = run_gemm(M, N, K, oa.o, ob.o, out, ws.defined() ? &ws : nullptr, (uint32_t)as_ll(a[11]));
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
        const at::Tensor value = a[6] == Py_True ? empty_f32({m.size(0), m.size(1)}, m) : at::Tensor();
        const int rc = api.wide_update((int16_t*)m.data_ptr(), (int8_t*)e.data_ptr(), (const float*)d.data_ptr(), m.size(0), m.size(1), ld_of(d), &f,
                                       v.m0, v.e0, v.m1, v.e1, value.defined() ? (float*)value.data_ptr() : nullptr, m.size(1), stream());
        return !rc && value.defined() ? THPVariable_Wrap(value) : code(rc);
    });
}

// wide_dequantize(mant, exps, tile, out or None) -> out
PyObject* wide_dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 4)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor m = tensor_of(a[0], "mantissas"), e = tensor_of(a[1], "exponents");
        const bool fresh = a[3] == Py_None;
        const at::Tensor out = fresh ? empty_f32({m.size(0), m.size(1)}, m) : tensor_of(a[3], "out");
        check_f32(out, "out");
        const int rc = api.wide_dequantize((const int16_t*)m.data_ptr(), (const int8_t*)e.data_ptr(), m.size(0), m.size(1), (int32_t)as_ll(a[2]),
                                           (float*)out.data_ptr(), ld_of(out), stream());
        if (rc) return code(rc);
        return fresh ? THPVariable_Wrap(out) : same(a[3]);
    });
}

// conv_forward(px, filters, n, h, w, c, kh, kw, pad, nf, out or None) -> out
PyObject* conv_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 11)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Operand px = operand_of(a[0], 0, Py_None), fl = operand_of(a[1], 0, Py_None);
        const int64_t nn = as_ll(a[2]), h = as_ll(a[3]), w = as_ll(a[4]), nf = as_ll(a[9]);
        const bool fresh = a[10] == Py_None;
        const at::Tensor out = fresh ? empty_f32({nn * h * w, nf}, px.data) : tensor_of(a[10], "out");
        check_f32(out, "out");
        const int rc = api.conv_forward(px.o.data, px.o.exps, nn, h, w, as_ll(a[5]), (int)as_ll(a[6]), (int)as_ll(a[7]), (int)as_ll(a[8]), &px.o.fmt, &fl.o,
                                        nf, (float*)out.data_ptr(), ld_of(out), stream());
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
        at::Tensor m, e;
        if (a[5] == Py_None) {
            hbfp_layout L;
            const int rc = api.packed_layout(ci, (int64_t)kh * kw * co, &c1.o.fmt, &L);
            if (rc) return code(rc);
            m = empty_i8(L.mant_bytes, c1.data);
            e = empty_i8(L.exp_bytes, c1.data);
        } else {
            m = tensor_of(a[5], "mantissas");
            e = tensor_of(a[6], "exponents");
        }
        const int rc = api.conv_dgrad_filters(c1.o.data, c1.o.exps, kh, kw, ci, co, &c1.o.fmt, m.data_ptr(), (int8_t*)e.data_ptr(), stream());
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", THPVariable_Wrap(m), THPVariable_Wrap(e));
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
        const hbfp_format f = format_of(a[4]);
        at::Tensor m, e;
        if (a[5] == Py_None) {
            hbfp_layout L;
            const int rc = api.packed_layout((int64_t)kh * kw * x.size(3), x.size(0) * x.size(1) * x.size(2), &f, &L);
            if (rc) return code(rc);
            m = empty_i8(L.mant_bytes, x);
            e = empty_i8(L.exp_bytes, x);
        } else {
            m = tensor_of(a[5], "mantissas");
            e = tensor_of(a[6], "exponents");
        }
        const int rc = api.im2col_packed_t((const float*)x.data_ptr(), x.size(0), x.size(1), x.size(2), x.size(3), kh, kw, (int)as_ll(a[3]), &f, m.data_ptr(),
                                           (int8_t*)e.data_ptr(), stream());
        if (rc) return code(rc);
        return Py_BuildValue("(NN)", THPVariable_Wrap(m), THPVariable_Wrap(e));
    });
}

// linear_forward(x, c0, fmt, fin, fout, bias or None) -> y
PyObject* linear_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 6)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Operand x = operand_of(a[0], 0, a[2]), w = operand_of(a[1], 0, Py_None);
        const int64_t batch = x.data.size(0), fin = as_ll(a[3]), fout = as_ll(a[4]);
        at::Tensor y = empty_f32({batch, fout}, x.data);
        const int rc = run_gemm(batch, fout, fin, x.o, w.o, y, nullptr, HBFP_GEMM_AUTO);
        if (rc) return code(rc);
        if (a[5] != Py_None) y.add_(tensor_of(a[5], "bias"));
        return THPVariable_Wrap(y);
    });
}

// linear_backward(dy, x, c1, fmt of dy, batch-axis fmts of x and dy, fin, fout, need dx, need dw, need db) -> (dx, dw, db)
PyObject* linear_backward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want(n, 11)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor dy = tensor_of(a[0], "dy"), x = tensor_of(a[1], "x");
        check_f32(dy, "dy");
        check_f32(x, "x");
        const int64_t batch = x.size(0), fin = as_ll(a[6]), fout = as_ll(a[7]);
        at::Tensor dx, dw, db;
        if (PyObject_IsTrue(a[8])) {
            const Operand g = operand_of(a[0], 0, a[3]), w = operand_of(a[2], 0, Py_None);
            dx = empty_f32({batch, fin}, dy);
            const int rc = run_gemm(batch, fin, fout, g.o, w.o, dx, nullptr, HBFP_GEMM_AUTO);
            if (rc) return code(rc);
        }
        if (PyObject_IsTrue(a[9])) {
            // contraction over the batch axis: blocks down the columns of X and dY
            const Operand xt = operand_of(a[1], 1, a[4]), g = operand_of(a[0], 0, a[5]);
            dw = empty_f32({fin, fout}, dy);
            const int rc = run_gemm(fin, fout, batch, xt.o, g.o, dw, nullptr, HBFP_GEMM_AUTO);
            if (rc) return code(rc);
        }
        if (PyObject_IsTrue(a[10])) db = dy.sum(0);
        auto wrap = [](const at::Tensor& t) { return t.defined() ? THPVariable_Wrap(t) : same(Py_None); };
        return Py_BuildValue("(NNN)", wrap(dx), wrap(dw), wrap(db));
    });
}

// bind(addresses in the order of Api)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    constexpr Py_ssize_t N = sizeof(Api) / sizeof(void*);
    if (!want(n, N)) return nullptr;
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
PyMethodDef methods[] = {HBFP_METHOD(bind), HBFP_METHOD(quantize), HBFP_METHOD(gemm), HBFP_METHOD(gemm_q), HBFP_METHOD(wide_update),
                         HBFP_METHOD(wide_dequantize), HBFP_METHOD(conv_forward), HBFP_METHOD(conv_dgrad_filters),
                         HBFP_METHOD(im2col_packed_t), HBFP_METHOD(linear_forward), HBFP_METHOD(linear_backward),
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
