// extern "C" entry points of the HBFP library: argument checks, workspace carving, dispatch.
#include "common.cuh"

#include <string.h>

#include <algorithm>
#include <atomic>
#include <utility>

namespace hbfp {

__device__ int32_t g_device_status;

// The address belongs to the device and never changes: asked for once per device (threads that race store the same value).
int32_t* device_status_word() {
    static std::atomic<int32_t*> known[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    int32_t* p = known[dev].load(std::memory_order_acquire);
    if (!p) {
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_device_status) != cudaSuccess) return nullptr;
        known[dev].store(p, std::memory_order_release);
    }
    return p;
}

// Words through which one conversion passes on to the next what it has waited for (see Placing), taken in turn.
constexpr unsigned long long TURN_WORDS = 4096;
__device__ unsigned long long g_turn_words[TURN_WORDS];

unsigned long long* turn_words() {
    static std::atomic<unsigned long long*> known[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    unsigned long long* p = known[dev].load(std::memory_order_acquire);
    if (!p) {
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_turn_words) != cudaSuccess) return nullptr;
        known[dev].store(p, std::memory_order_release);
    }
    return p;
}

// The places of two conversions, the second beside the first or (where it may not be) after it.
struct PlacedPair {
    Placing first, second;
    // second_bytes: loaded by the second conversion
    PlacedPair(bool beside, int64_t second_bytes) {
        static std::atomic<unsigned long long> turns{0};
        unsigned long long* const words = beside ? turn_words() : nullptr;
        if (!words) return;
        const unsigned long long turn = ++turns;
        first = {LEAD, words + turn % TURN_WORDS, turn, second_bytes};
        second = {BESIDE, words + turn % TURN_WORDS, turn, 0};
    }
};

int read_clear_device_status(cudaStream_t st, int32_t* out) {
    HBFP_CUDA_OK(cudaStreamSynchronize(st));
    int32_t v = 0, zero = 0;
    HBFP_CUDA_OK(cudaMemcpyFromSymbol(&v, g_device_status, sizeof(v)));
    HBFP_CUDA_OK(cudaMemcpyToSymbol(g_device_status, &zero, sizeof(zero)));
    *out = v;
    if (v == 0) return HBFP_OK;
    return v >= 900 && v < 1000 ? HBFP_ERR_EXPONENT_RANGE : HBFP_ERR_TIMEOUT;
}

namespace {

// What the calling thread's last hbfp_gemm* call launched: the family's name (hbfp_last_gemm_kernel) and the kernel's own
// (hbfp_last_gemm_launch).
thread_local const char* t_last_gemm_kernel = "";
thread_local const char* t_last_gemm_launch = "";
void ran(const char* kernel, const char* launch = nullptr) {
    t_last_gemm_kernel = kernel;
    t_last_gemm_launch = launch ? launch : kernel;
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct GemmPlan {
    Layout la, lb;
    size_t off_am, off_ae, off_bm, off_be, off_partial, total;
    TensorPlan tp;
    // A call on the floating-point operand forms (gemm_fp.cu) uses the same memory in another way: the forms of A and B, then a
    // packed place for an FP32 operand that cannot be converted straight to its form (weight tiles).
    FpPlan fp;
    size_t off_fa, off_fb, off_fm, off_fe, total_fp;
};

size_t fp_plane_bytes(const Layout& L) { return align_up(2 * (size_t)(L.rows * L.kst), 1024); }
size_t fp_bytes(const Layout& L, const FpPlan& f, bool is_b) {
    return (is_b ? f.planes_b : 1) * fp_plane_bytes(L) + (f.form ? align_up(4 * (size_t)(L.nkb * L.rs), 1024) : 0);
}
FpOperand fp_operand(const Layout& L, const FpPlan& f, bool is_b, char* at) {
    FpOperand o{};
    const int planes = is_b ? f.planes_b : 1;
    o.p0 = at;
    o.p1 = planes > 1 ? at + fp_plane_bytes(L) : nullptr;
    o.scales = f.form ? reinterpret_cast<float*>(at + planes * fp_plane_bytes(L)) : nullptr;
    o.rows = L.rows;
    o.kst = L.kst;
    o.rs = L.rs;
    return o;
}

int check_operand(const hbfp_operand* o) {
    if (!o || o->struct_size != sizeof(hbfp_operand)) return HBFP_ERR_INVALID_ARG;
    if (o->kind != HBFP_OPERAND_FP32 && o->kind != HBFP_OPERAND_PACKED) return HBFP_ERR_INVALID_ARG;
    return HBFP_OK;
}

int make_plan(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b, GemmPlan* g) {
    if (M < 0 || N < 0 || K < 0) return HBFP_ERR_INVALID_ARG;
    int rc = check_operand(a);
    if (rc) return rc;
    rc = check_operand(b);
    if (rc) return rc;
    rc = make_layout(M, K, &a->fmt, &g->la);
    if (rc) return rc;
    rc = make_layout(N, K, &b->fmt, &g->lb);
    if (rc) return rc;
    if (g->la.b != g->lb.b) return HBFP_ERR_INVALID_ARG;   // the blocks of the two operands must coincide
    size_t off = 0;
    g->off_am = off; if (a->kind == HBFP_OPERAND_FP32) off += align_up((size_t)g->la.mant_bytes, 1024);
    g->off_ae = off; if (a->kind == HBFP_OPERAND_FP32) off += align_up((size_t)g->la.exp_bytes, 1024);
    g->off_bm = off; if (b->kind == HBFP_OPERAND_FP32) off += align_up((size_t)g->lb.mant_bytes, 1024);
    g->off_be = off; if (b->kind == HBFP_OPERAND_FP32) off += align_up((size_t)g->lb.exp_bytes, 1024);
    g->tp = plan_gemm_tensor(M, N, K, g->la, g->lb, a->fmt.mant_bits, b->fmt.mant_bits);
    g->off_partial = off;
    g->total = off + align_up(g->tp.partial_bytes, 1024);
    // operands that need a pass of their own to take the form
    const int passes = (a->kind != HBFP_OPERAND_FP32 || a->fmt.tile != 0) + (b->kind != HBFP_OPERAND_FP32 || b->fmt.tile != 0);
    g->fp = plan_gemm_fp(M, N, g->la, g->lb, passes);
    g->off_fa = g->off_fb = g->off_fm = g->off_fe = g->total_fp = 0;
    if (g->fp.use) {
        g->off_fb = fp_bytes(g->la, g->fp, false);
        g->off_fm = g->off_fb + fp_bytes(g->lb, g->fp, true);
        // one place: B is packed after A has been expanded
        size_t mant = 0, exps = 0;
        for (const auto& x : {std::make_pair(a, &g->la), std::make_pair(b, &g->lb)})
            if (x.first->kind == HBFP_OPERAND_FP32 && x.first->fmt.tile != 0) {
                mant = std::max(mant, align_up((size_t)x.second->mant_bytes, 1024));
                exps = std::max(exps, align_up((size_t)x.second->exp_bytes, 1024));
            }
        g->off_fe = g->off_fm + mant;
        g->total_fp = g->off_fe + exps;
    }
    return HBFP_OK;
}

void fill_operand(hbfp_operand* o, const float* data, int64_t ld, int trans, const hbfp_format* f) {
    memset(o, 0, sizeof(*o));
    o->struct_size = sizeof(*o);
    o->kind = HBFP_OPERAND_FP32;
    o->data = data;
    o->ld = ld;
    o->trans = trans;
    if (f) o->fmt = *f;
}

// How an FP32 operand is stored. A: trans 0 = [rows][K] (blocks along rows), trans 1 = [K][rows]; B: trans 0 = [K][rows]
// (blocks down columns), trans 1 = [rows][K].
bool k_contiguous(const hbfp_operand* o, bool is_a) { return is_a ? o->trans == 0 : o->trans != 0; }

int check_fp32(const hbfp_operand* o, bool is_a, int64_t rows, int64_t K) {
    if (!o->data && rows * K > 0) return HBFP_ERR_INVALID_ARG;
    return o->ld < (k_contiguous(o, is_a) ? K : rows) ? HBFP_ERR_INVALID_ARG : HBFP_OK;
}

// Bytes that the conversion of B loads through L1: none where it loads by the copy engine (whole blocks down aligned columns).
int64_t streamed_bytes(const hbfp_operand* b, int64_t N, int64_t K, const Layout& L) {
    if (b->kind == HBFP_OPERAND_PACKED) return L.planes * N * K;
    return !k_contiguous(b, false) && L.b == L.bp && L.b <= 128 && b->ld % 4 == 0 ? 0 : 4 * N * K;
}

// Quantises an FP32 operand into the workspace (or takes a packed one as is).
int resolve_operand(const hbfp_operand* o, bool is_a, int64_t rows, int64_t K, const Layout& L,
                    char* ws, size_t off_m, size_t off_e, Packed* out, const Placing& at, cudaStream_t st) {
    out->L = L;
    out->mant_bits = o->fmt.mant_bits;
    if (o->kind == HBFP_OPERAND_PACKED) {
        if (!o->data || !o->exps) return HBFP_ERR_INVALID_ARG;
        if ((reinterpret_cast<uintptr_t>(o->data) & 255) || (reinterpret_cast<uintptr_t>(o->exps) & 127))
            return HBFP_ERR_ALIGNMENT;
        out->mant = static_cast<const int8_t*>(o->data);
        out->exps = o->exps;
        return HBFP_OK;
    }
    const int rc = check_fp32(o, is_a, rows, K);
    if (rc) return rc;
    int8_t* m = reinterpret_cast<int8_t*>(ws + off_m);
    int8_t* e = reinterpret_cast<int8_t*>(ws + off_e);
    out->mant = m;
    out->exps = e;
    const float* x = static_cast<const float*>(o->data);
    return k_contiguous(o, is_a) ? launch_quantize(x, rows, K, o->ld, 1, &o->fmt, m, e, st, at) : launch_quantize(x, K, rows, o->ld, 0, &o->fmt, m, e, st, at);
}

// An operand in the floating-point form at `f`: converted straight to it where it is an FP32 matrix without weight tiles,
// otherwise packed (or taken packed) and expanded; the place is that of the last launch. The packed place is one for both operands.
int resolve_form(const hbfp_operand* o, bool is_a, int64_t rows, int64_t K, const GemmPlan& g, char* ws, const FpOperand& f, const Placing& at, cudaStream_t st) {
    if (o->kind == HBFP_OPERAND_FP32) {
        const int rc = check_fp32(o, is_a, rows, K);
        if (rc) return rc;
        const float* x = static_cast<const float*>(o->data);
        if (o->fmt.tile == 0)          // always covered where plan_gemm_fp takes the forms; a packed place is not reserved for these
            return k_contiguous(o, is_a) ? launch_quantize_form(x, rows, K, o->ld, 1, &o->fmt, g.fp.form, !is_a, at, f, st)
                                         : launch_quantize_form(x, K, rows, o->ld, 0, &o->fmt, g.fp.form, !is_a, at, f, st);
    }
    Packed p;
    const int rc = resolve_operand(o, is_a, rows, K, is_a ? g.la : g.lb, ws, g.off_fm, g.off_fe, &p, Placing{}, st);
    if (rc) return rc;
    return launch_expand(p, g.fp, !is_a, at, f, st);
}

// bias (may be null) is added in the kernel's own store where it can; *bias_done says so, otherwise the caller adds it.
int gemm_impl(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b, const float* bias, bool* bias_done, float* C,
              int64_t ldc, void* workspace, size_t ws_bytes, uint32_t flags, int32_t* P, cudaStream_t st) {
    *bias_done = false;
    GemmPlan g;
    int rc = make_plan(M, N, K, a, b, &g);
    if (rc) return rc;
    if (flags > HBFP_GEMM_FORCE_SMALL) return HBFP_ERR_INVALID_ARG;
    if (P) {   // the inspection hook never splits K and needs no scratch
        g.total -= align_up(g.tp.partial_bytes, 1024);
        g.tp.partial_bytes = 0;
        g.tp.splits = 1;
        g.tp.kb_per_split = g.la.nkb;
    }
    if (M == 0 || N == 0) return HBFP_OK;
    if ((!C && !P) || ldc < N) return HBFP_ERR_INVALID_ARG;
    if (g.total > 0) {
        if (!workspace || ws_bytes < g.total) return HBFP_ERR_WORKSPACE;
        if (reinterpret_cast<uintptr_t>(workspace) & 255) return HBFP_ERR_ALIGNMENT;
    }
    // A caller whose workspace holds the packed operands only (hbfp_gemm_static) gets the integer kernels.
    const bool use_fp = g.fp.use && !P && workspace && ws_bytes >= g.total_fp && (reinterpret_cast<uintptr_t>(workspace) & 255) == 0 &&
                        (flags == HBFP_GEMM_AUTO || flags == HBFP_GEMM_FORCE_TENSOR) && (reinterpret_cast<uintptr_t>(C) & 3) == 0;
    char* ws = static_cast<char*>(workspace);
    Packed pa{nullptr, nullptr, g.la, a->fmt.mant_bits}, pb{nullptr, nullptr, g.lb, b->fmt.mant_bits};
    // a problem of a few hundred MOPs is over before a tensor-core kernel has filled its pipeline
    const bool small = !P && (flags == HBFP_GEMM_AUTO || flags == HBFP_GEMM_FORCE_SMALL) && small_gemm_eligible(M, N, pa, pb, flags == HBFP_GEMM_FORCE_SMALL);
    if (flags == HBFP_GEMM_FORCE_SMALL && !small) return HBFP_ERR_UNSUPPORTED;
    if (small && small_fused_eligible(a, k_contiguous(a, true), b, k_contiguous(b, false), M, N, g.la)) {
        rc = check_fp32(a, true, M, K);
        if (!rc) rc = check_fp32(b, false, N, K);
        if (rc) return rc;
        ran("gemm_small_kernel", "gemm_small_fused_kernel");
        return launch_gemm_small_fused(M, N, K, a, k_contiguous(a, true), b, k_contiguous(b, false), g.la, C, ldc, st);
    }
    if (!P && flags == HBFP_GEMM_AUTO && a->kind == HBFP_OPERAND_FP32 && a->trans == 0 && a->fmt.tile == 0 &&
        b->kind == HBFP_OPERAND_PACKED && skinny_gemm_eligible(M, N, g.la, g.lb, a->fmt.mant_bits, b->fmt.mant_bits)) {
        rc = check_fp32(a, true, M, K);
        if (rc) return rc;
        rc = resolve_operand(b, false, N, K, g.lb, ws, g.off_bm, g.off_be, &pb, Placing{}, st);
        if (rc) return rc;
        ran("gemm_skinny_kernel");
        *bias_done = true;
        return launch_gemm_skinny(M, N, K, static_cast<const float*>(a->data), a->ld, &a->fmt, pb, bias, C, ldc, st);
    }
    if (use_fp && !small) {
        const FpOperand fa = fp_operand(g.la, g.fp, false, ws + g.off_fa), fb = fp_operand(g.lb, g.fp, true, ws + g.off_fb);
        const bool beside = b->kind == HBFP_OPERAND_PACKED || b->fmt.tile == 0;       // B in one launch
        const PlacedPair at(beside, streamed_bytes(b, N, K, g.lb));
        rc = resolve_form(a, true, M, K, g, ws, fa, at.first, st);
        if (rc) return rc;
        rc = resolve_form(b, false, N, K, g, ws, fb, at.second, st);
        if (rc) return rc;
        ran("gemm_tc_kernel", g.fp.pair ? "gemm_fp_kernel/pair" : g.fp.splits > 1 ? "gemm_fp_kernel/split" : "gemm_fp_kernel");
        *bias_done = true;
        return launch_gemm_fp(M, N, g.la, g.fp, fa, fb, bias, C, ldc, st);
    }
    // two conversions of one launch each (longer blocks and weight tiles may take several, or another kernel)
    const bool beside = a->kind == HBFP_OPERAND_FP32 && b->kind == HBFP_OPERAND_FP32 && a->fmt.tile == 0 && b->fmt.tile == 0 && K > 0 && g.la.b <= 256;
    const PlacedPair at(beside, streamed_bytes(b, N, K, g.lb));
    rc = resolve_operand(a, true, M, K, g.la, ws, g.off_am, g.off_ae, &pa, at.first, st);
    if (rc) return rc;
    rc = resolve_operand(b, false, N, K, g.lb, ws, g.off_bm, g.off_be, &pb, at.second, st);
    if (rc) return rc;
    if (small) {
        ran("gemm_small_kernel");
        *bias_done = true;
        return launch_gemm_small(M, N, pa, pb, bias, C, ldc, st);
    }
    const bool quad_rows = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && (ldc % 4) == 0;
    const bool want_tensor = flags != HBFP_GEMM_FORCE_SIMT && g.tp.supported &&
                             (reinterpret_cast<uintptr_t>(C) & 3) == 0;
    if (want_tensor) {
        // With a short contraction (under 1 KiB of mantissas per row) a tile is bound by the write of
        // its C part, and the single-SM kernel, whose warps own wider row segments, is ~10 % faster.
        const bool long_k = g.la.nkb * g.la.bp >= 1024;
        const bool pair_ok = !P && quad_rows && flags != HBFP_GEMM_FORCE_TENSOR_1SM && pair_gemm_eligible(M, N, pa, pb, g.tp) &&
                             (long_k || flags == HBFP_GEMM_FORCE_TENSOR_2SM);
        if (pair_ok) {
            ran("gemm_tc2_kernel");
            return launch_gemm_tensor_pair(M, N, pa, pb, C, ldc, g.tp, ws ? ws + g.off_partial : nullptr, st);
        }
        if (flags == HBFP_GEMM_FORCE_TENSOR_2SM) return HBFP_ERR_UNSUPPORTED;
        ran("gemm_tc_kernel");
        *bias_done = !P && g.tp.splits > 1;
        return launch_gemm_tensor(M, N, K, pa, pb, bias, C, ldc, P, g.tp, ws ? ws + g.off_partial : nullptr, st);
    }
    if (flags >= HBFP_GEMM_FORCE_TENSOR) return HBFP_ERR_UNSUPPORTED;
    ran("gemm_simt_kernel");
    return launch_gemm_simt(M, N, K, pa, pb, C, ldc, P, st);
}

}  // namespace

int gemm_least_workspace(int transA, int transB, int64_t M, int64_t N, int64_t K, const hbfp_format* fmtA, const hbfp_format* fmtB, size_t* bytes) {
    if (!fmtA || !fmtB) return HBFP_ERR_INVALID_ARG;
    hbfp_operand a, b;
    fill_operand(&a, nullptr, 0, transA, fmtA);
    fill_operand(&b, nullptr, 0, transB, fmtB);
    GemmPlan g;
    int rc = make_plan(M, N, K, &a, &b, &g);
    if (rc) return rc;
    *bytes = g.total;
    return HBFP_OK;
}

}  // namespace hbfp

using namespace hbfp;

extern "C" {

const char* hbfp_last_gemm_kernel(void) { return t_last_gemm_kernel; }
const char* hbfp_last_gemm_launch(void) { return t_last_gemm_launch; }

const char* hbfp_status_string(int status) {
    switch (status) {
        case HBFP_OK: return "ok";
        case HBFP_ERR_INVALID_ARG: return "invalid argument";
        case HBFP_ERR_UNSUPPORTED: return "unsupported format or size";
        case HBFP_ERR_ALIGNMENT: return "buffer not aligned as required";
        case HBFP_ERR_WORKSPACE: return "workspace missing or too small";
        case HBFP_ERR_CUDA: return "CUDA call failed";
        case HBFP_ERR_TIMEOUT: return "bounded device-side wait expired";
        case HBFP_ERR_EXPONENT_RANGE: return "operand exponents outside the tensor-core path's exact range";
        case HBFP_ERR_STATIC_LIMIT: return "problem exceeds the built-in scratch of hbfp_gemm_static";
        default: return "unknown status";
    }
}

int hbfp_packed_layout(int64_t rows, int64_t k, const hbfp_format* fmt, hbfp_layout* out) {
    if (!out) return HBFP_ERR_INVALID_ARG;
    Layout L;
    int rc = make_layout(rows, k, fmt, &L);
    if (rc) return rc;
    out->rows = L.rows; out->k = L.k; out->b = L.b; out->bp = L.bp; out->nkb = L.nkb; out->kst = L.kst;
    out->planes = L.planes; out->plane_stride = L.plane_stride; out->rs = L.rs;
    out->mant_bytes = L.mant_bytes; out->exp_bytes = L.exp_bytes;
    return HBFP_OK;
}

int hbfp_packed_sizes(int64_t rows, int64_t k, const hbfp_format* fmt, size_t* mant_bytes, size_t* exp_bytes) {
    Layout L;
    int rc = make_layout(rows, k, fmt, &L);
    if (rc) return rc;
    if (mant_bytes) *mant_bytes = (size_t)L.mant_bytes;
    if (exp_bytes) *exp_bytes = (size_t)L.exp_bytes;
    return HBFP_OK;
}

int hbfp_quantize(const float* x, int64_t d0, int64_t d1, int64_t ld, int contract_axis,
                  const hbfp_format* fmt, void* mant, int8_t* exps, void* stream) {
    if (d0 < 0 || d1 < 0 || ld < d1 || (contract_axis != 0 && contract_axis != 1)) return HBFP_ERR_INVALID_ARG;
    if (!fmt) return HBFP_ERR_INVALID_ARG;
    if ((!x && d0 * d1 > 0) || !mant || !exps) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant) & 255) || (reinterpret_cast<uintptr_t>(exps) & 127)) return HBFP_ERR_ALIGNMENT;
    return launch_quantize(x, d0, d1, ld, contract_axis, fmt, static_cast<int8_t*>(mant), exps,
                           static_cast<cudaStream_t>(stream));
}

int hbfp_quantize_tiles(const float* w, int64_t d0, int64_t d1, int64_t ld, const hbfp_format* fmt,
                        void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1, int8_t* tile_exps,
                        void* stream) {
    if (d0 < 0 || d1 < 0 || ld < d1 || !fmt) return HBFP_ERR_INVALID_ARG;
    if ((!w && d0 * d1 > 0) || !mant_c0 || !exps_c0 || !mant_c1 || !exps_c1) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant_c0) & 255) || (reinterpret_cast<uintptr_t>(mant_c1) & 255) ||
        (reinterpret_cast<uintptr_t>(exps_c0) & 127) || (reinterpret_cast<uintptr_t>(exps_c1) & 127))
        return HBFP_ERR_ALIGNMENT;
    return launch_quantize_tiles(w, d0, d1, ld, fmt, static_cast<int8_t*>(mant_c0), exps_c0,
                                 static_cast<int8_t*>(mant_c1), exps_c1, tile_exps,
                                 static_cast<cudaStream_t>(stream));
}

int hbfp_quantize_conv_weights(const float* w, int64_t taps, int64_t c_in, int64_t c_out, int64_t ld,
                               const hbfp_format* fmt, void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1,
                               int8_t* tile_exps, void* stream) {
    if (!w || !fmt || taps <= 0 || c_in <= 0 || c_out <= 0 || ld < c_out) return HBFP_ERR_INVALID_ARG;
    if ((mant_c0 && !exps_c0) || (mant_c1 && !exps_c1) || (!mant_c0 && !mant_c1 && !tile_exps)) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant_c0) & 255) || (reinterpret_cast<uintptr_t>(mant_c1) & 255) ||
        (reinterpret_cast<uintptr_t>(exps_c0) & 127) || (reinterpret_cast<uintptr_t>(exps_c1) & 127))
        return HBFP_ERR_ALIGNMENT;
    return launch_quantize_conv_weights(w, taps, c_in, c_out, ld, fmt, static_cast<int8_t*>(mant_c0), exps_c0,
                                        static_cast<int8_t*>(mant_c1), exps_c1, tile_exps, static_cast<cudaStream_t>(stream));
}

static int wide_views_ok(void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1) {
    if (!mant_c0 && !mant_c1 && !exps_c0 && !exps_c1) return HBFP_OK;        // wide storage only
    if (!mant_c0 || !exps_c0 || !mant_c1 || !exps_c1) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant_c0) & 255) || (reinterpret_cast<uintptr_t>(mant_c1) & 255) ||
        (reinterpret_cast<uintptr_t>(exps_c0) & 127) || (reinterpret_cast<uintptr_t>(exps_c1) & 127))
        return HBFP_ERR_ALIGNMENT;
    return HBFP_OK;
}

int hbfp_wide_quantize(const float* w, int64_t d0, int64_t d1, int64_t ld, const hbfp_format* fmt, int16_t* wide,
                       int8_t* wide_exps, void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1, void* stream) {
    if (d0 < 0 || d1 < 0 || ld < d1 || !fmt) return HBFP_ERR_INVALID_ARG;
    if (d0 * d1 > 0 && (!w || !wide || !wide_exps)) return HBFP_ERR_INVALID_ARG;
    int rc = wide_views_ok(mant_c0, exps_c0, mant_c1, exps_c1);
    if (rc) return rc;
    return launch_wide(0, w, ld, d0, d1, fmt, wide, wide_exps, static_cast<int8_t*>(mant_c0), exps_c0,
                       static_cast<int8_t*>(mant_c1), exps_c1, nullptr, 0, static_cast<cudaStream_t>(stream));
}

int hbfp_wide_update(int16_t* wide, int8_t* wide_exps, const float* delta, int64_t d0, int64_t d1, int64_t ldd,
                     const hbfp_format* fmt, void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1, void* stream) {
    return hbfp_wide_update_value(wide, wide_exps, delta, d0, d1, ldd, fmt, mant_c0, exps_c0, mant_c1, exps_c1, nullptr, 0, stream);
}

int hbfp_wide_update_value(int16_t* wide, int8_t* wide_exps, const float* delta, int64_t d0, int64_t d1, int64_t ldd,
                           const hbfp_format* fmt, void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1,
                           float* value, int64_t ldv, void* stream) {
    if (d0 < 0 || d1 < 0 || ldd < d1 || (value && ldv < d1) || !fmt) return HBFP_ERR_INVALID_ARG;
    if (d0 * d1 > 0 && (!delta || !wide || !wide_exps)) return HBFP_ERR_INVALID_ARG;
    int rc = wide_views_ok(mant_c0, exps_c0, mant_c1, exps_c1);
    if (rc) return rc;
    return launch_wide(1, delta, ldd, d0, d1, fmt, wide, wide_exps, static_cast<int8_t*>(mant_c0), exps_c0,
                       static_cast<int8_t*>(mant_c1), exps_c1, value, ldv, static_cast<cudaStream_t>(stream));
}

int hbfp_wide_narrow(const int16_t* wide, const int8_t* wide_exps, int64_t d0, int64_t d1, const hbfp_format* fmt,
                     void* mant_c0, int8_t* exps_c0, void* mant_c1, int8_t* exps_c1, void* stream) {
    if (d0 < 0 || d1 < 0 || !fmt || (d0 * d1 > 0 && (!wide || !wide_exps))) return HBFP_ERR_INVALID_ARG;
    if (!mant_c0 || !mant_c1) return HBFP_ERR_INVALID_ARG;
    int rc = wide_views_ok(mant_c0, exps_c0, mant_c1, exps_c1);
    if (rc) return rc;
    return launch_wide(2, nullptr, d1, d0, d1, fmt, const_cast<int16_t*>(wide), const_cast<int8_t*>(wide_exps),
                       static_cast<int8_t*>(mant_c0), exps_c0, static_cast<int8_t*>(mant_c1), exps_c1, nullptr, 0,
                       static_cast<cudaStream_t>(stream));
}

int hbfp_wide_dequantize(const int16_t* wide, const int8_t* wide_exps, int64_t d0, int64_t d1, int32_t tile, float* out,
                         int64_t ldo, void* stream) {
    if (d0 < 0 || d1 < 0 || tile <= 0 || ldo < d1) return HBFP_ERR_INVALID_ARG;
    if (d0 * d1 > 0 && (!wide || !wide_exps || !out)) return HBFP_ERR_INVALID_ARG;
    return launch_wide_dequantize(wide, wide_exps, d0, d1, tile, out, ldo, static_cast<cudaStream_t>(stream));
}

int hbfp_im2col_packed(const void* mant_x, const int8_t* exps_x, int64_t n, int64_t h, int64_t w, int64_t c, int kh,
                       int kw, int pad, const hbfp_format* fmt, void* mant_out, int8_t* exps_out, void* stream) {
    if (!fmt || n < 0 || h <= 0 || w <= 0 || c <= 0 || kh <= 0 || kw <= 0 || pad < 0) return HBFP_ERR_INVALID_ARG;
    if (!mant_x || !exps_x || !mant_out || !exps_out) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant_x) & 255) || (reinterpret_cast<uintptr_t>(mant_out) & 255) ||
        (reinterpret_cast<uintptr_t>(exps_out) & 127))
        return HBFP_ERR_ALIGNMENT;
    return launch_im2col_packed(static_cast<const int8_t*>(mant_x), exps_x, n, h, w, c, kh, kw, pad, fmt,
                                static_cast<int8_t*>(mant_out), exps_out, static_cast<cudaStream_t>(stream));
}

int hbfp_conv_forward(const void* mant_x, const int8_t* exps_x, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw,
                      int pad, const hbfp_format* fmt_x, const hbfp_operand* filters_op, int64_t filters, float* Y,
                      int64_t ldy, void* stream) {
    if (!fmt_x || !filters_op || n < 0 || h <= 0 || w <= 0 || c <= 0 || kh <= 0 || kw <= 0 || pad < 0 || filters <= 0)
        return HBFP_ERR_INVALID_ARG;
    if (!mant_x || !exps_x || !Y || ldy < filters) return HBFP_ERR_INVALID_ARG;
    if (filters_op->struct_size != sizeof(hbfp_operand) || filters_op->kind != HBFP_OPERAND_PACKED || !filters_op->data ||
        !filters_op->exps)
        return HBFP_ERR_INVALID_ARG;
    if (fmt_x->block <= 0 || c % fmt_x->block != 0 || fmt_x->tile != 0 || filters_op->fmt.block != fmt_x->block) return HBFP_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(mant_x) & 255) || (reinterpret_cast<uintptr_t>(filters_op->data) & 255)) return HBFP_ERR_ALIGNMENT;
    Packed px, pw;
    int rc = make_layout(n * h * w, c, fmt_x, &px.L);
    if (rc) return rc;
    rc = make_layout(filters, (int64_t)kh * kw * c, &filters_op->fmt, &pw.L);
    if (rc) return rc;
    px.mant = static_cast<const int8_t*>(mant_x);
    px.exps = exps_x;
    px.mant_bits = fmt_x->mant_bits;
    pw.mant = static_cast<const int8_t*>(filters_op->data);
    pw.exps = static_cast<const int8_t*>(filters_op->exps);
    pw.mant_bits = filters_op->fmt.mant_bits;
    if (n == 0) return HBFP_OK;
    ran("conv_fwd_kernel");
    return launch_conv_forward(px, pw, n, h, w, c, kh, kw, pad, filters, Y, ldy, static_cast<cudaStream_t>(stream));
}

int hbfp_conv_dgrad_filters(const void* mant_c1, const int8_t* exps_c1, int kh, int kw, int64_t c_in, int64_t c_out,
                            const hbfp_format* fmt, void* mant_out, int8_t* exps_out, void* stream) {
    if (!fmt || kh <= 0 || kw <= 0 || c_in < 0 || c_out <= 0) return HBFP_ERR_INVALID_ARG;
    if (!mant_c1 || !exps_c1 || !mant_out || !exps_out) return HBFP_ERR_INVALID_ARG;
    const int64_t t = fmt->tile;
    if (t <= 0 || fmt->block != t) return HBFP_ERR_INVALID_ARG;
    // whole 16-byte pieces of unpadded blocks: tiles of 32, 64 or 128 output maps
    if ((t != 32 && t != 64 && t != 128) || c_out % t != 0 || c_in % t != 0) return HBFP_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(mant_c1) & 255) || (reinterpret_cast<uintptr_t>(mant_out) & 255)) return HBFP_ERR_ALIGNMENT;
    const int64_t taps = (int64_t)kh * kw;
    Packed c1;
    Layout Lo;
    int rc = make_layout(taps * c_in, c_out, fmt, &c1.L);
    if (rc) return rc;
    rc = make_layout(c_in, taps * c_out, fmt, &Lo);
    if (rc) return rc;
    c1.mant = static_cast<const int8_t*>(mant_c1);
    c1.exps = exps_c1;
    c1.mant_bits = fmt->mant_bits;
    return launch_conv_dgrad_filters(c1, (int)taps, c_in, c_out, (int)t, static_cast<int8_t*>(mant_out), exps_out, Lo,
                                     static_cast<cudaStream_t>(stream));
}

int hbfp_im2col_packed_t(const float* x, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad,
                         const hbfp_format* fmt, void* mant, int8_t* exps, void* stream) {
    if (!fmt || n < 0 || h <= 0 || w <= 0 || c <= 0 || kh <= 0 || kw <= 0 || pad < 0) return HBFP_ERR_INVALID_ARG;
    if ((!x && n > 0) || !mant || !exps) return HBFP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(mant) & 255) || (reinterpret_cast<uintptr_t>(exps) & 127)) return HBFP_ERR_ALIGNMENT;
    return launch_im2col_cols(x, n, h, w, c, kh, kw, pad, fmt, static_cast<int8_t*>(mant), exps,
                              static_cast<cudaStream_t>(stream));
}

int hbfp_unpack(const void* mant, const int8_t* exps, int64_t rows, int64_t k, const hbfp_format* fmt,
                int16_t* q, int8_t* s, void* stream) {
    Packed p;
    int rc = make_layout(rows, k, fmt, &p.L);
    if (rc) return rc;
    if (!mant || !exps) return HBFP_ERR_INVALID_ARG;
    p.mant = static_cast<const int8_t*>(mant);
    p.exps = exps;
    p.mant_bits = fmt->mant_bits;
    return launch_unpack(p, q, s, static_cast<cudaStream_t>(stream));
}

int hbfp_dequantize(const void* mant, const int8_t* exps, int64_t rows, int64_t k, const hbfp_format* fmt,
                    float* out, int64_t ld, void* stream) {
    Packed p;
    int rc = make_layout(rows, k, fmt, &p.L);
    if (rc) return rc;
    if (!mant || !exps || !out || ld < k) return HBFP_ERR_INVALID_ARG;
    p.mant = static_cast<const int8_t*>(mant);
    p.exps = exps;
    p.mant_bits = fmt->mant_bits;
    return launch_dequantize(p, out, ld, static_cast<cudaStream_t>(stream));
}

int hbfp_gemm_q_workspace(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b,
                          size_t* bytes) {
    if (!bytes) return HBFP_ERR_INVALID_ARG;
    GemmPlan g;
    int rc = make_plan(M, N, K, a, b, &g);
    if (rc) return rc;
    *bytes = g.total_fp > g.total ? g.total_fp : g.total;
    return HBFP_OK;
}

int hbfp_gemm_workspace(int transA, int transB, int64_t M, int64_t N, int64_t K, const hbfp_format* fmtA,
                        const hbfp_format* fmtB, size_t* bytes) {
    if (!fmtA || !fmtB) return HBFP_ERR_INVALID_ARG;
    hbfp_operand a, b;
    fill_operand(&a, nullptr, 0, transA, fmtA);
    fill_operand(&b, nullptr, 0, transB, fmtB);
    return hbfp_gemm_q_workspace(M, N, K, &a, &b, bytes);
}

int hbfp_gemm_q(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b, float* C,
                int64_t ldc, void* workspace, size_t workspace_bytes, uint32_t flags, void* stream) {
    return hbfp_gemm_q_bias(M, N, K, a, b, nullptr, C, ldc, workspace, workspace_bytes, flags, stream);
}

int hbfp_gemm_q_bias(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b, const float* bias, float* C,
                     int64_t ldc, void* workspace, size_t workspace_bytes, uint32_t flags, void* stream) {
    if (!C && M * N > 0) return HBFP_ERR_INVALID_ARG;
    bool bias_done = false;
    const int rc = gemm_impl(M, N, K, a, b, bias, &bias_done, C, ldc, workspace, workspace_bytes, flags, nullptr, static_cast<cudaStream_t>(stream));
    if (rc || !bias || bias_done || M == 0 || N == 0) return rc;
    return launch_add_bias(C, M, N, ldc, bias, static_cast<cudaStream_t>(stream));
}

int hbfp_column_sums(const float* x, int64_t rows, int64_t cols, int64_t ld, float* out, void* stream) {
    if (rows < 0 || cols < 0 || ld < cols || (cols > 0 && (!out || (rows > 0 && !x)))) return HBFP_ERR_INVALID_ARG;
    return launch_column_sums(x, rows, cols, ld, out, static_cast<cudaStream_t>(stream));
}

int hbfp_fold_taps(const float* cols, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad, float* out, void* stream) {
    if (n < 0 || h <= 0 || w <= 0 || c <= 0 || kh <= 0 || kw <= 0 || pad < 0 || 2 * pad != kh - 1 || 2 * pad != kw - 1) return HBFP_ERR_INVALID_ARG;
    if (n > 0 && (!cols || !out)) return HBFP_ERR_INVALID_ARG;
    return launch_fold_taps(cols, n, h, w, c, kh, kw, pad, out, static_cast<cudaStream_t>(stream));
}

int hbfp_gemm(int transA, int transB, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda,
              const float* B, int64_t ldb, float* C, int64_t ldc, const hbfp_format* fmtA,
              const hbfp_format* fmtB, void* workspace, size_t workspace_bytes, uint32_t flags, void* stream) {
    if (!fmtA || !fmtB) return HBFP_ERR_INVALID_ARG;
    hbfp_operand a, b;
    fill_operand(&a, A, lda, transA, fmtA);
    fill_operand(&b, B, ldb, transB, fmtB);
    return hbfp_gemm_q(M, N, K, &a, &b, C, ldc, workspace, workspace_bytes, flags, stream);
}

int hbfp_gemm_block_partials(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, const hbfp_operand* b,
                             int32_t* P, uint32_t impl, void* stream) {
    if (!P || !a || !b) return HBFP_ERR_INVALID_ARG;
    if (a->kind != HBFP_OPERAND_PACKED || b->kind != HBFP_OPERAND_PACKED) return HBFP_ERR_INVALID_ARG;
    if (impl != HBFP_GEMM_FORCE_SIMT && impl != HBFP_GEMM_FORCE_TENSOR) return HBFP_ERR_INVALID_ARG;
    bool bias_done;
    return gemm_impl(M, N, K, a, b, nullptr, &bias_done, nullptr, N, nullptr, 0, impl, P, static_cast<cudaStream_t>(stream));
}

int hbfp_selftest_bounded_wait(int64_t limit_cycles, int32_t code, int32_t* outcome, void* stream) {
    return launch_wait_probe((long long)limit_cycles, (int)code, reinterpret_cast<int*>(outcome), static_cast<cudaStream_t>(stream));
}

int hbfp_last_gemm_cycles(uint64_t* cycles) {
    if (!cycles) return HBFP_ERR_INVALID_ARG;
    return pair_gemm_cycles(cycles);
}

int hbfp_device_status(void* stream, int32_t* status) {
    if (!status) return HBFP_ERR_INVALID_ARG;
    return read_clear_device_status(static_cast<cudaStream_t>(stream), status);
}

}  // extern "C"
