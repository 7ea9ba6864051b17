// Internal declarations shared by the CUDA translation units of the HBFP library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hbfp.h"

namespace hbfp {

// ------------------------------------------------------------------------------ layout

struct Layout {
    int64_t rows, k, b, bp, nkb, kst, planes, plane_stride, rs, mant_bytes, exp_bytes;
};

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Validates a format and computes the packed layout (see "Packed operand layout" in hbfp.h).
inline int make_layout(int64_t rows, int64_t k, const hbfp_format* f, Layout* L) {
    if (!f || !L || rows < 0 || k < 0) return HBFP_ERR_INVALID_ARG;
    if (f->struct_size != sizeof(hbfp_format)) return HBFP_ERR_INVALID_ARG;
    if (f->mant_bits < 3 || f->mant_bits > 12) return HBFP_ERR_UNSUPPORTED;
    if (f->block < 0 || f->tile < 0) return HBFP_ERR_INVALID_ARG;
    if (f->tile > 0 && f->tile != f->block) return HBFP_ERR_INVALID_ARG;
    if (f->rounding != 0 && f->rounding != 1) return HBFP_ERR_INVALID_ARG;
    if (f->exp_mode != 0 && f->exp_mode != 1) return HBFP_ERR_INVALID_ARG;
    int64_t b = f->block == 0 ? (k > 0 ? k : 1) : f->block;
    // The per-block integer sum must fit int32 (wide accumulators never overflow, Sec. 5.3).
    int64_t qmax = ((int64_t)1 << (f->mant_bits - 1)) - 1;
    if (qmax * qmax * b > 0x7fffffffll) return HBFP_ERR_UNSUPPORTED;
    L->rows = rows;
    L->k = k;
    L->b = b;
    L->bp = b <= 32 ? 32 : b <= 64 ? 64 : b <= 128 ? 128 : round_up(b, 128);
    L->nkb = (k + b - 1) / b;
    L->kst = round_up(L->nkb * L->bp, 128);
    if (L->kst == 0) L->kst = 128;
    L->planes = f->mant_bits <= 8 ? 1 : 2;
    L->plane_stride = round_up(rows * L->kst, 1024);
    if (L->plane_stride == 0) L->plane_stride = 1024;
    L->rs = round_up(rows > 0 ? rows : 1, 16);
    L->mant_bytes = L->planes * L->plane_stride;
    L->exp_bytes = round_up((L->nkb > 0 ? L->nkb : 1) * L->rs, 128);
    return HBFP_OK;
}

// ------------------------------------------------------------------------------ launch plumbing

#define HBFP_CUDA_OK(expr)                          \
    do {                                            \
        cudaError_t _e = (expr);                    \
        if (_e != cudaSuccess) return HBFP_ERR_CUDA; \
    } while (0)

inline int launch_status() { return cudaGetLastError() == cudaSuccess ? HBFP_OK : HBFP_ERR_CUDA; }

// Chained launches. A call is a chain of kernels of 2 to 20 us each, and between two of them in a stream lie the end of the one,
// the launch of the other and its start. Kernels are launched so that their CTAs may be placed as soon as all CTAs of the kernel
// before have started and an SM has room (programmatic stream serialization); they set up their barriers and tensor memory there
// and then wait for that kernel to end (chain_wait) before they touch global memory. The wait covers the whole stream: the
// kernel before had waited in its turn. Every kernel launched by launch_chained has to wait, in at least one thread. Launched plainly
// are the paired-SM integer GEMM, long launches of the 12-bit operand forms (gemm_fp.cu), long kernels and a few long CTAs behind a
// product (below) and the wait probe.
// It is the gap between launches that shrinks: calls back to back with their conversions, without chains / with them: 256 cube 8.2 / 6.4
// us, 1111 x 777 x 3001 (b = 24, with draws) 46.3 / 34.1, 1024 x 4096 x 4096 (b = 32) 77 / 67.6, 2048 cube (b = 64) 39.3 / 30.1, 16 rows against
// 4096 x 4096 packed weights 11.6 / 8.9. A call of one launch takes by itself what it took.
// A kernel says that its successor may be placed (chain_next) only after it has itself waited and, where it uses tensor memory, has
// allocated it: a successor that took the columns first would wait for a kernel that waits for the columns.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void chain_start() { chain_wait(); chain_next(); }

// How a conversion follows the launch before it on its stream.
//   CHAINED  as above
//   LEAD     chained, and the launch after it may be BESIDE
//   BESIDE   next to the LEAD before it: the conversion of a product's second operand, which reads and writes nothing that the conversion
//            of the first one writes. It waits when it is through, and what follows waits for it and with it for both.
// What a BESIDE kernel reads, a chained kernel before the LEAD may have written (weights updated just before). The LEAD's wait gives
// those writes to the LEAD alone, and that the LEAD's CTAs have said chain_next orders no memory. So the LEAD passes them on: past its
// wait its first thread releases a word of memory, to a value that no other pair of launches has, and every CTA of the BESIDE kernel
// acquires that word before it reads anything: release and acquire at the scope of the GPU are cumulative. A CTA that does not find the
// value waits for the whole LEAD (a word taken over by a later call, a CTA that starts after the word was given back), which is slower
// and as right. The first CTA gives the word back, so that a replayed graph starts without it. Loads of a BESIDE kernel are not .nc.
// Back to back, all three launches chained / so / with a plain launch as the LEAD, which is a kernel boundary by itself (and before the
// word, when nothing passed the writes on): 1111 x 777 x 3001, b = 24, draws 36.3 / 34.2 / 34.8 us (33.7); 1024 x 4096 x 4096, b = 32
// 71.2 / 67.8 / 68.2 (67.0); 512 cube, b = 64 11.0 / 10.4 / 12.4 (9.9). By itself a 512 cube takes 1.13 / 1.02 / 1.00 of what it took,
// over 36 formats and orders.
enum Place : int { CHAINED = 0, LEAD = 1, BESIDE = 2 };
struct Placing {
    int place = CHAINED;
    unsigned long long* word = nullptr;
    unsigned long long turn = 0;
    int64_t more = 0;             // of a LEAD: bytes that the BESIDE launch loads
};
// (The usual place first: with the others in the way rows of 1024 x 1024, b = 32, took 3.3 us instead of 3.1.)
struct Chain {
    const Placing& at;
    __device__ __forceinline__ explicit Chain(const Placing& a) : at(a) {
        if (__builtin_expect(at.place == CHAINED, 1)) {
            chain_wait();
            chain_next();
            return;
        }
        if (at.place == BESIDE) {
            unsigned long long seen = at.turn;
            if (threadIdx.x == 0) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(at.word) : "memory");
            if (__syncthreads_or(seen != at.turn)) chain_wait();
        } else {
            chain_wait();
            if ((blockIdx.x | blockIdx.y | threadIdx.x) == 0) asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(at.word), "l"(at.turn) : "memory");
        }
        chain_next();
    }
    __device__ __forceinline__ ~Chain() {
        if (__builtin_expect(at.place != BESIDE, 1)) return;
        chain_wait();
        if ((blockIdx.x | blockIdx.y | threadIdx.x) == 0) asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(at.word), "l"(0ull) : "memory");
    }
};

// Two kinds of kernels are not chained behind a product, that is where this thread has launched one on the stream since its last launch
// that was not chained (times behind a product, chained / not):
// - Those that load 50 MB and more. The products take most of an SM's memory as shared memory, and an SM keeps its split between that and
//   L1 until it has been idle. A kernel that is placed behind a product never lets it be: it runs with the little L1 that the product had
//   left, which is what its loads in flight are held in. Update of 8192 x 8192, t = 64 156 / 113 us, with its FP32 value 215 / 154, rows of
//   8192 x 8192 converted, b = 32 68 / 56; 4096 x 4096, t = 64 40 / 32, b = 32 17.3 / 14.8, its column sums 18 / 13; 2048 x 4096, t = 64 18.4 /
//   16.9, b = 32 8.4 / 8.6; 2048 x 2048, t = 64 8.8 / 10.7. Kernels that load through the copy engine keep their data in shared memory and
//   are always chained.
// - A few long CTAs (at most two per SM, of thousands of elements): placed as SMs fall free, they crowd on the first of them. Update of
//   1024 x 1024, t = 24, with draws 15.6 / 12.7 us, t = 128 with its FP32 value 11.6 / 8.6.
// Behind other kernels they are chained (rows of 8192 x 8192 back to back 51.2 / 53.1, updates of 1024 x 1024, t = 24 10.7 / 12.5).
constexpr int64_t STREAMED_BYTES = 50 * 1000 * 1000;
constexpr unsigned FEW_CTAS = 2 * 148;
struct LastProduct {
    cudaStream_t st = nullptr;
    bool holds = false;
};
inline thread_local LastProduct t_last_product;
inline void note_product(cudaStream_t st) { t_last_product = {st, true}; }

template <class... Params, class... Args>
inline void launch_one(bool chained, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chained;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);      // launch_status() has the verdict
}
template <class... Params, class... Args>
inline void launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    launch_one(true, kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}
// Whether a kernel that loads so many bytes is chained.
inline bool chain_streamed(int64_t bytes, cudaStream_t st) {
    const bool chained = bytes < STREAMED_BYTES || !t_last_product.holds || t_last_product.st != st;
    if (!chained) t_last_product.holds = false;
    return chained;
}
template <class... Params, class... Args>
inline void launch_streamed(int64_t bytes, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    launch_one(chain_streamed(bytes, st), kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}
// A conversion. A BESIDE launch is always chained, a LEAD counts for both.
template <class... Params, class... Args>
inline void launch_placed(const Placing& at, int64_t bytes, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    launch_one(at.place == BESIDE || chain_streamed(bytes + at.more, st), kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}
// The same as launch_streamed for long CTAs.
template <class... Params, class... Args>
inline void launch_streamed_long(int64_t bytes, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    launch_one(chain_streamed(grid.x * grid.y <= FEW_CTAS ? STREAMED_BYTES : bytes, st), kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}
// The same with clusters of `cluster` CTAs along x; not chained where the kernel's tiles want the order of an empty chip (gemm_fp.cu).
template <class... Params, class... Args>
inline void launch_chained_clusters(void (*kernel)(Params...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool chained, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    unsigned n = 0;
    if (chained) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// A packed operand as the kernels see it.
struct Packed {
    const int8_t* mant;   // plane 0
    const int8_t* exps;   // [nkb][rs]
    Layout L;
    int mant_bits;
};

// Quantiser launchers (quantize.cu).
// place: LEAD or BESIDE for the first and the second of two conversions that share no memory; a conversion of several launches is
// CHAINED in place of BESIDE.
int launch_quantize(const float* x, int64_t d0, int64_t d1, int64_t ld, int contract_axis,
                    const hbfp_format* f, int8_t* mant, int8_t* exps, cudaStream_t st, const Placing& at = Placing{});
int launch_quantize_tiles(const float* w, int64_t d0, int64_t d1, int64_t ld, const hbfp_format* f,
                          int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                          int8_t* tile_exps, cudaStream_t st);
int launch_quantize_conv_weights(const float* w, int64_t taps, int64_t c_in, int64_t c_out, int64_t ld,
                                 const hbfp_format* f, int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                                 int8_t* tile_exps, cudaStream_t st);
// Wide weight storage: mode 0 quantise FP32 weights, 1 apply an FP32 update in place, 2 read only; in every
// mode the packed narrow views are written when their pointers are given, in mode 1 also the FP32 values.
int launch_wide(int mode, const float* src, int64_t ld, int64_t d0, int64_t d1, const hbfp_format* f,
                int16_t* wide, int8_t* wide_exps, int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                float* value, int64_t ldv, cudaStream_t st);
int launch_wide_dequantize(const int16_t* wide, const int8_t* exps, int64_t d0, int64_t d1, int tile, float* out,
                           int64_t ldo, cudaStream_t st);
// Packed convolution operand gathered from the packed per-pixel operand.
int launch_im2col_packed(const int8_t* xm, const int8_t* xe, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw,
                         int pad, const hbfp_format* f, int8_t* om, int8_t* oe, cudaStream_t st);
// Packed transposed convolution operand (blocks along the output pixels) straight from the FP32 activations.
int launch_im2col_cols(const float* x, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad,
                       const hbfp_format* f, int8_t* mant, int8_t* exps, cudaStream_t st);
int launch_unpack(const Packed& p, int16_t* q, int8_t* s, cudaStream_t st);
int launch_dequantize(const Packed& p, float* out, int64_t ld, cudaStream_t st);

// GEMM launchers. P (optional) receives the per-block integer sums [M][N][nkb].
int launch_gemm_simt(int64_t M, int64_t N, int64_t K, const Packed& a, const Packed& b, float* C,
                     int64_t ldc, int32_t* P, cudaStream_t st);

// Tiled dp4a kernel for small problems (gemm_small.cu): one-plane operands, one launch, no split-K.
bool small_gemm_eligible(int64_t M, int64_t N, const Packed& a, const Packed& b, bool any_size);
int launch_gemm_small(int64_t M, int64_t N, const Packed& a, const Packed& b, const float* bias, float* C, int64_t ldc, cudaStream_t st);
// The same from FP32 operands, conversion included (contig: K is contiguous).
bool small_fused_eligible(const hbfp_operand* a, bool a_contig, const hbfp_operand* b, bool b_contig, int64_t M, int64_t N, const Layout& la);
int launch_gemm_small_fused(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, bool a_contig, const hbfp_operand* b, bool b_contig, const Layout& la,
                            float* C, int64_t ldc, cudaStream_t st);

// A few rows of FP32 activations against packed weights, conversion included (gemm_skinny.cu): one launch, no scratch.
bool skinny_gemm_eligible(int64_t M, int64_t N, const Layout& la, const Layout& lb, int bits_a, int bits_b);
int launch_gemm_skinny(int64_t M, int64_t N, int64_t K, const float* x, int64_t ld, const hbfp_format* fx, const Packed& w, const float* bias, float* C,
                       int64_t ldc, cudaStream_t st);

// Workspace of the integer kernels alone (hbfp_gemm_workspace may ask for more).
int gemm_least_workspace(int transA, int transB, int64_t M, int64_t N, int64_t K, const hbfp_format* fmtA,
                         const hbfp_format* fmtB, size_t* bytes);

struct TensorPlan {
    int supported;      // 0: this case has no tensor-core kernel
    int n_tile;         // 64, 128 or 256
    int splits;         // split-K factor (1 = none)
    int64_t kb_per_split;
    size_t partial_bytes;  // split-K scratch
};
TensorPlan plan_gemm_tensor(int64_t M, int64_t N, int64_t K, const Layout& la, const Layout& lb,
                            int mant_bits_a, int mant_bits_b);
// bias: added by the sum of the parts, only where K is split (plan.splits > 1).
int launch_gemm_tensor(int64_t M, int64_t N, int64_t K, const Packed& a, const Packed& b, const float* bias, float* C,
                       int64_t ldc, int32_t* P, const TensorPlan& plan, void* partial,
                       cudaStream_t st);

// Paired-SM variant (two CTAs of a cluster per 256 x 256 tile): 8-bit mantissas, blocks up to 128,
// no split-K, enough tiles to occupy every SM pair.
bool pair_gemm_eligible(int64_t M, int64_t N, const Packed& a, const Packed& b, const TensorPlan& plan);
int launch_gemm_tensor_pair(int64_t M, int64_t N, const Packed& a, const Packed& b, float* C, int64_t ldc,
                            const TensorPlan& plan, void* partial, cudaStream_t st);

// Floating-point operand forms (gemm_fp.cu): short blocks of 8-bit mantissas, and 9 to 12 bits.
struct FpOperand {          // device buffers, rows x kst elements of two bytes
    void* p0;               // form S: bfloat16 q * 2^s; form W: binary16 q (A) or its upper part (B)
    void* p1;               // form W, B: binary16 lower part
    float* scales;          // form W: 2^s [nkb][rs]
    int64_t rows, kst, rs;
};
struct FpPlan {
    int use;                // 0: the integer kernels
    int form, pair, ncol, splits, kb_per_split, planes_b;
};
FpPlan plan_gemm_fp(int64_t M, int64_t N, const Layout& la, const Layout& lb, int passes);
int launch_expand(const Packed& x, const FpPlan& plan, bool is_b, const Placing& at, const FpOperand& out, cudaStream_t st);
// Converts an FP32 operand straight to a form (quantize.cu); HBFP_ERR_UNSUPPORTED for weight tiles.
int launch_quantize_form(const float* x, int64_t d0, int64_t d1, int64_t ld, int contract_axis, const hbfp_format* f, int wide, bool is_b,
                         const Placing& at, const FpOperand& out, cudaStream_t st);
int launch_gemm_fp(int64_t M, int64_t N, const Layout& la, const FpPlan& plan, const FpOperand& a, const FpOperand& b, const float* bias, float* C,
                   int64_t ldc, cudaStream_t st);

// FP32 parts of a layer (layer.cu): the bias added to a stored product, the column sums that are its gradient.
int launch_add_bias(float* C, int64_t M, int64_t N, int64_t ldc, const float* bias, cudaStream_t st);
int launch_column_sums(const float* x, int64_t rows, int64_t cols, int64_t ld, float* out, cudaStream_t st);
int launch_fold_taps(const float* cols, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad, float* out, cudaStream_t st);

// Convolution forward as an implicit GEMM over the packed pixels (gemm_conv.cu).
int launch_conv_forward(const Packed& x, const Packed& wt, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw,
                        int pad, int64_t filters, float* Y, int64_t ldy, cudaStream_t st);

// One warp running the kernels' bounded barrier wait on a barrier nobody arrives on (test hook).
int launch_wait_probe(long long limit_cycles, int code, int* outcome, cudaStream_t st);
int launch_conv_dgrad_filters(const Packed& c1, int taps, int64_t c_in, int64_t c_out, int t, int8_t* mant_out,
                              int8_t* exps_out, const Layout& Lo, cudaStream_t st);
int pair_gemm_cycles(uint64_t* cycles);   // longest CTA of the last paired-SM GEMM launch on the current device, in SM cycles

// Device status word (bounded waits report here).
int32_t* device_status_word();   // device address, per current device
int read_clear_device_status(cudaStream_t st, int32_t* out);

}  // namespace hbfp
