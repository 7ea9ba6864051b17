// BFP GEMM for the smallest problems (a 256 or 512 cube: a few tens to hundreds of MOPs with a contraction of at
// most 512 bytes). The tensor-core kernels need several microseconds to set up their pipeline and, for outputs
// of a few tiles, a second launch to add split-K parts; here a plain tiled kernel finishes first (256 cube: 3.9
// against 6.0 us, 512 cube: 5.3 against 8.7 us), in one launch and without splitting K. It does not scale: on
// this part both dp4a and the warp-level int8 MMA it uses cost about 230 ns per 32-byte step of a 32 x 32 tile
// (the MLP's layers, 33-43 steps, take 10-12 us here against 9.6 us on the tensor-core path), so the dispatch
// keeps it to short contractions and grids of at most two CTAs per SM.
//
// One CTA per 32 x 32 tile of C, 256 threads, a 16 x 8 piece per warp. The packed mantissas of the tile's 32 rows
// of A and 32 rows of B come in 512-byte slices of K by asynchronous 16-byte copies into two shared-memory buffers
// (a slice is in flight while the previous one is multiplied); the exponents of all K-blocks of those rows are
// staged once. Per K-block: the exact int32 sum by mma.sync.m16n8k32 (Eq. 2), converted to binary32 and
// accumulated with one FMA by 2^(sA + sB), blocks in ascending order: bit for bit the sequential definition.
#include "quant_math.cuh"

namespace hbfp {
namespace {

constexpr int SM_TILE = 32;                 // rows of A and rows of B (columns of C) per CTA
constexpr int SM_SLICE = 512;               // bytes of K per slice
constexpr int SM_PITCH = SM_SLICE + 16;     // row pitch in shared memory: rows 4 banks apart
constexpr int SM_BUF = 2 * SM_TILE * SM_PITCH;   // one slice of both operands
constexpr int SM_MAX_NKB = 1024;            // exponents staged per row
constexpr int SM_AUTO_BYTES = 512;          // automatic choice: contractions of at most one slice ...
constexpr int64_t SM_AUTO_CTAS = 2 * 148;   // ... and at most two CTAs per SM

// 2^e for any integer e the sum of two stored exponents can take; outside the normal range the slow exact route
__device__ __forceinline__ float scale_of(int e) {
    return (e >= -126 && e <= 127) ? __int_as_float((e + 127) << 23) : ldexpf(1.0f, e);
}
__device__ __forceinline__ void copy16_async(void* dst_shared, const void* src_global) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_shared)), "l"(src_global) : "memory");
}

__global__ void __launch_bounds__(256)
gemm_small_kernel(int64_t M, int64_t N, int nkb, int bp, const int8_t* __restrict__ mA, int64_t kstA,
                  const int8_t* __restrict__ eA, int64_t rsA, const int8_t* __restrict__ mB, int64_t kstB,
                  const int8_t* __restrict__ eB, int64_t rsB, const float* __restrict__ bias, float* __restrict__ C, int64_t ldc) {
    chain_start();
    extern __shared__ __align__(16) unsigned char smem[];
    int8_t* xA = reinterpret_cast<int8_t*>(smem + 2 * SM_BUF);  // [nkb][32]
    int8_t* xB = xA + (size_t)nkb * SM_TILE;                    // [nkb][32]

    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.y * SM_TILE, j0 = (int64_t)blockIdx.x * SM_TILE;
    const int total_bytes = nkb * bp;                           // a multiple of 32, at most the row pitch of either operand
    const int slices = (total_bytes + SM_SLICE - 1) / SM_SLICE;
    // loader role: per slice, 16-byte pieces t, t + 256, ... of the 32 x 32 pieces of each operand (row = piece / 32)
    const int8_t* rowA[4];
    const int8_t* rowB[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = (tid + 256 * u) >> 5;
        rowA[u] = mA + min(i0 + r, M - 1) * kstA;               // rows beyond the matrix: the last valid row, never stored
        rowB[u] = mB + min(j0 + r, N - 1) * kstB;
    }
    auto issue = [&](int s) {
        unsigned char* buf = smem + (s & 1) * SM_BUF;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = (tid + 256 * u) >> 5, piece = (tid + 256 * u) & 31;
            const int off = s * SM_SLICE + 16 * piece;
            if (off < total_bytes) {
                copy16_async(buf + r * SM_PITCH + 16 * piece, rowA[u] + off);
                copy16_async(buf + SM_TILE * SM_PITCH + r * SM_PITCH + 16 * piece, rowB[u] + off);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    issue(0);
    // exponents of every K-block of the tile's rows
    for (int t = tid; t < nkb * SM_TILE; t += 256) {
        const int kb = t >> 5, r = t & 31;
        xA[t] = eA[(int64_t)kb * rsA + min(i0 + r, M - 1)];
        xB[t] = eB[(int64_t)kb * rsB + min(j0 + r, N - 1)];
    }

    // compute role: warp w owns the 16 x 8 piece of C at rows 16 (w & 1), columns 8 (w >> 1): one
    // mma.sync.m16n8k32 (s8 x s8 -> s32, exact) per 32-byte step. Fragment layout: this lane holds rows g and g + 8
    // of A (g = lane / 4) at k bytes 4 (lane % 4) and + 16, row g of B at the same bytes, and of C rows g, g + 8 at
    // columns 2 (lane % 4), + 1.
    const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, kq = 4 * (lane & 3);
    const int ra = 16 * (warp & 1) + g, rb = 8 * (warp >> 1) + g;
    const int cr0 = 16 * (warp & 1) + g, cc0 = 8 * (warp >> 1) + 2 * (lane & 3);
    const int steps_per_block = bp >> 5;                        // 32-byte steps per K-block
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    int p0 = 0, p1 = 0, p2 = 0, p3 = 0;
    int step_in_block = 0, kb = 0;
    for (int s = 0; s < slices; ++s) {
        if (s + 1 < slices) {
            issue(s + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();                                        // slice s (and, first, the exponents) visible to all
        const unsigned char* sA = smem + (s & 1) * SM_BUF + ra * SM_PITCH + kq;
        const unsigned char* sB = smem + (s & 1) * SM_BUF + SM_TILE * SM_PITCH + rb * SM_PITCH + kq;
        const int steps = min(SM_SLICE / 32, (total_bytes - s * SM_SLICE) >> 5);
        for (int q = 0; q < steps; ++q) {
            const uint32_t a0 = *reinterpret_cast<const uint32_t*>(sA + 32 * q);
            const uint32_t a1 = *reinterpret_cast<const uint32_t*>(sA + 8 * SM_PITCH + 32 * q);
            const uint32_t a2 = *reinterpret_cast<const uint32_t*>(sA + 32 * q + 16);
            const uint32_t a3 = *reinterpret_cast<const uint32_t*>(sA + 8 * SM_PITCH + 32 * q + 16);
            const uint32_t b0 = *reinterpret_cast<const uint32_t*>(sB + 32 * q);
            const uint32_t b1 = *reinterpret_cast<const uint32_t*>(sB + 32 * q + 16);
            asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                         : "+r"(p0), "+r"(p1), "+r"(p2), "+r"(p3) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
            if (++step_in_block == steps_per_block) {
                const int ea0 = xA[kb * SM_TILE + cr0], ea1 = xA[kb * SM_TILE + cr0 + 8];
                const int eb0 = xB[kb * SM_TILE + cc0], eb1 = xB[kb * SM_TILE + cc0 + 1];
                acc[0] = fmaf((float)p0, scale_of(ea0 + eb0), acc[0]);
                acc[1] = fmaf((float)p1, scale_of(ea0 + eb1), acc[1]);
                acc[2] = fmaf((float)p2, scale_of(ea1 + eb0), acc[2]);
                acc[3] = fmaf((float)p3, scale_of(ea1 + eb1), acc[3]);
                p0 = p1 = p2 = p3 = 0;
                step_in_block = 0;
                ++kb;
            }
        }
        __syncthreads();                                        // the buffer is free for the slice after the next
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int64_t i = i0 + cr0 + 8 * a, j = j0 + cc0 + b;
            if (i < M && j < N) C[i * ldc + j] = bias ? __fadd_rn(acc[2 * a + b], __ldg(bias + j)) : acc[2 * a + b];
        }
}

// ------------------------------------------------------------------------------ both operands FP32

// The same 32 x 32 tiles from FP32 operands, conversion included: one launch instead of three. A 256 cube is a few microseconds
// of anything, and what its three kernels cost was their launches and starts (8.5 us of device time, 14.3 as a call; here 6.7 and 8.2). Half of
// the 16 warps convert the tile's 32 rows of A and half the 32 columns of B to binary16 mantissas in shared memory; every tile of
// a row of tiles repeats that, which bounds it to short contractions (one slice) and few tiles. Mantissas of 8 bits and block
// sums below 2^24 are exact in binary16 MMAs with FP32 accumulators, which this part issues four times as often per K as the
// int8 ones; a lane takes eight consecutive K of both operands, so fragments are 16-byte loads.
constexpr int SF_THREADS = 512, SF_HALF = 256;
constexpr int SF_MAX_GROUPS = SM_AUTO_BYTES / 8;

struct SmallOperand {
    const float* x;
    int64_t ld, lines;              // lines: rows of A or columns of B
    int contig, vec;                // contig: blocks along contiguous rows; vec: pieces of eight are 16-byte aligned
    QParams q;
};
struct SmallProblem {
    SmallOperand a, b;
    int K, blk, bp, lg_bp, nkb, pitch;     // pitch of a converted line in bytes
    float* C;
    int64_t ldc;
};

template <bool SR>
__device__ __forceinline__ void sf_store(const float (&e8)[8], int s, const QParams& q, uint4 w, unsigned char* at) {
    uint4 h, unused;
    if (SR && q.rounding == 1) quantize_form8<true, FORM_WIDE_A>(e8, s, q, w, h, unused);
    else quantize_form8<false, FORM_WIDE_A>(e8, s, q, w, h, unused);
    *reinterpret_cast<uint4*>(at) = h;
}

// 32 lines from `line0` on whose K is contiguous: a thread keeps its piece of eight packed positions and walks down the lines.
template <bool SR>
__device__ __forceinline__ void sf_convert_rows(const SmallOperand& o, const SmallProblem& p, int64_t line0, int t, unsigned char* dst, int8_t* exps) {
    constexpr int UNR = 4;
    const int gpr = p.nkb * p.bp / 8, rpp = SF_HALF / gpr, r0 = t / gpr, pos = 8 * (t - r0 * gpr);
    const int kb = pos >> p.lg_bp, within = pos & (p.bp - 1), k = kb * p.blk + within, lpb = p.bp / 8;
    const int n = r0 < rpp ? min(p.blk - within, p.K - k) : 0;
    for (int rb = 0; rb < SM_TILE; rb += UNR * rpp) {
        float e8[UNR][8];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int r = rb + u * rpp + r0;
            const int nr = r < SM_TILE && line0 + r < o.lines ? n : 0;
            const float* src = o.x + (line0 + r) * o.ld + k;
            if (nr >= 8 && o.vec) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(src)), c = __ldg(reinterpret_cast<const float4*>(src) + 1);
                e8[u][0] = a.x; e8[u][1] = a.y; e8[u][2] = a.z; e8[u][3] = a.w;
                e8[u][4] = c.x; e8[u][5] = c.y; e8[u][6] = c.z; e8[u][7] = c.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) e8[u][j] = j < nr ? __ldg(src + j) : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            if (rb + u * rpp >= SM_TILE) break;                       // all threads alike
            const int r = rb + u * rpp + r0;
            uint32_t am = amax8_bits(e8[u]);
            for (int off = 1; off < lpb; off <<= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
            const int s = block_exponent(am, o.q.m, o.q.exp_mode);
            if (r < SM_TILE && r0 < rpp) {
                const uint4 w = SR && o.q.rounding == 1 ? draws_of_eight(o.q, (uint64_t)((line0 + r) * p.K + k)) : make_uint4(0u, 0u, 0u, 0u);
                sf_store<SR>(e8[u], s, o.q, w, dst + r * p.pitch + 2 * pos);
                if (within == 0) exps[kb * SM_TILE + r] = (int8_t)s;
            }
        }
    }
}

// 32 lines that are columns of x [K][lines]: lane = line, a warp takes every eighth group of eight K, so that its loads are 128
// consecutive bytes; the groups stay in registers between the block maximum (through shared memory) and the rounding.
template <bool SR, int PER>
__device__ __forceinline__ void sf_convert_cols(const SmallOperand& o, const SmallProblem& p, int64_t line0, int t, int barrier, uint32_t (*amax)[SM_TILE],
                                                unsigned char* dst, int8_t* exps) {
    const int lane = t & 31, warp = t >> 5, groups = p.nkb * p.bp / 8, lpb = p.bp / 8;
    const bool in = line0 + lane < o.lines;
    float e8[PER][8];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int g = warp + 8 * i, kb = g >> (p.lg_bp - 3), within = 8 * (g & (lpb - 1)), k = kb * p.blk + within;
        const int n = g < groups && in ? min(p.blk - within, p.K - k) : 0;
        const float* src = o.x + (int64_t)k * o.ld + line0 + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) e8[i][j] = j < n ? __ldg(src + j * o.ld) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (warp + 8 * i < groups) amax[warp + 8 * i][lane] = amax8_bits(e8[i]);
    asm volatile("bar.sync %0, %1;" ::"r"(barrier), "n"(SF_HALF) : "memory");
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int g = warp + 8 * i, kb = g >> (p.lg_bp - 3), within = 8 * (g & (lpb - 1)), k = kb * p.blk + within;
        if (g >= groups) break;                                       // the whole warp
        uint32_t am = 0;
        for (int j = 0; j < lpb; ++j) am = max(am, amax[kb * lpb + j][lane]);
        const int s = block_exponent(am, o.q.m, o.q.exp_mode);
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (SR && o.q.rounding == 1) {
            // Eight neighbouring columns share the draws of a row (the pitch of the draws is a multiple of eight): lane i of an
            // octet makes those of row k + i, column c takes halfword c of each.
            const int c = lane & 7;
            const uint4 mine = draws_of_group(o.q, (uint64_t)((int64_t)(k + c) * o.lines + line0 + (lane & ~7)) >> 3);
            uint32_t d[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int from = (lane & ~7) + j;
                const uint32_t x = __shfl_sync(0xffffffffu, mine.x, from), y = __shfl_sync(0xffffffffu, mine.y, from);
                const uint32_t z = __shfl_sync(0xffffffffu, mine.z, from), v = __shfl_sync(0xffffffffu, mine.w, from);
                d[j] = draw_from(make_uint4(x, y, z, v), (uint32_t)c);
            }
            w = make_uint4(d[0] | d[1] << 16, d[2] | d[3] << 16, d[4] | d[5] << 16, d[6] | d[7] << 16);
        }
        sf_store<SR>(e8[i], s, o.q, w, dst + lane * p.pitch + 16 * g);
        if (within == 0) exps[kb * SM_TILE + lane] = (int8_t)s;
    }
}

// SR: either operand rounds stochastically. PER: groups of eight K per warp of a column conversion (4: up to 256 K). Both keep the
// code of a launch short: it runs once from top to bottom, and fetching it is a good part of so short a kernel.
template <bool SR, int PER>
__global__ void __launch_bounds__(SF_THREADS)
gemm_small_fused_kernel(const SmallProblem p) {
    chain_start();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t amax[2][SF_MAX_GROUPS][SM_TILE];
    __shared__ int8_t xA[SF_MAX_GROUPS / 4 * SM_TILE], xB[SF_MAX_GROUPS / 4 * SM_TILE];      // [block][32]
    unsigned char *fA = smem, *fB = smem + SM_TILE * p.pitch;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t i0 = (int64_t)blockIdx.y * SM_TILE, j0 = (int64_t)blockIdx.x * SM_TILE;
    if (tid < SF_HALF) {
        if (p.a.contig) sf_convert_rows<SR>(p.a, p, i0, tid, fA, xA);
        else sf_convert_cols<SR, PER>(p.a, p, i0, tid, 1, amax[0], fA, xA);
    } else {
        if (p.b.contig) sf_convert_rows<SR>(p.b, p, j0, tid - SF_HALF, fB, xB);
        else sf_convert_cols<SR, PER>(p.b, p, j0, tid - SF_HALF, 2, amax[1], fB, xB);
    }
    __syncthreads();
    if (warp >= 8) return;
    // warp w: rows 16 (w & 1), columns 8 (w >> 1) of the tile; fragments as in gemm_small_kernel
    const int g = lane >> 2, q = lane & 3, cr0 = 16 * (warp & 1) + g, cc0 = 8 * (warp >> 1) + 2 * q;
    const unsigned char *sA = fA + cr0 * p.pitch + 16 * q, *sB = fB + (8 * (warp >> 1) + g) * p.pitch + 16 * q;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int kb = 0; kb < p.nkb; ++kb) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        for (int o = 0; o < p.bp; o += 32, sA += 64, sB += 64) {
            const uint4 a = *reinterpret_cast<const uint4*>(sA), a8 = *reinterpret_cast<const uint4*>(sA + 8 * p.pitch), b = *reinterpret_cast<const uint4*>(sB);
            asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                         : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a.x), "r"(a8.x), "r"(a.y), "r"(a8.y), "r"(b.x), "r"(b.y));
            asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                         : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a.z), "r"(a8.z), "r"(a.w), "r"(a8.w), "r"(b.z), "r"(b.w));
        }
        const int ea0 = xA[kb * SM_TILE + cr0], ea1 = xA[kb * SM_TILE + cr0 + 8], eb0 = xB[kb * SM_TILE + cc0], eb1 = xB[kb * SM_TILE + cc0 + 1];
        acc[0] = fmaf(d[0], scale_of(ea0 + eb0), acc[0]);
        acc[1] = fmaf(d[1], scale_of(ea0 + eb1), acc[1]);
        acc[2] = fmaf(d[2], scale_of(ea1 + eb0), acc[2]);
        acc[3] = fmaf(d[3], scale_of(ea1 + eb1), acc[3]);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int64_t i = i0 + cr0 + 8 * a, j = j0 + cc0 + b;
            if (i < p.a.lines && j < p.b.lines) p.C[i * p.ldc + j] = acc[2 * a + b];
        }
}

}  // namespace

// One-plane operands, at most SM_MAX_NKB K-blocks; unless any_size, a problem small enough that the tensor-core
// kernels' set-up time would dominate.
bool small_gemm_eligible(int64_t M, int64_t N, const Packed& a, const Packed& b, bool any_size) {
    if (a.L.planes != 1 || b.L.planes != 1) return false;
    if (a.L.bp != b.L.bp || a.L.nkb != b.L.nkb || a.L.b != b.L.b) return false;
    if (a.L.bp % 32 != 0 || a.L.nkb > SM_MAX_NKB || a.L.nkb * a.L.bp > (1 << 20)) return false;
    if (M <= 0 || N <= 0 || (M + SM_TILE - 1) / SM_TILE > 65535) return false;
    // the per-block sum must convert to binary32 exactly, as on the tensor-core path
    const int64_t qa = (1ll << (a.mant_bits - 1)) - 1, qb = (1ll << (b.mant_bits - 1)) - 1;
    if (qa * qb * a.L.b >= (1ll << 24)) return false;
    const int64_t ctas = ((M + SM_TILE - 1) / SM_TILE) * ((N + SM_TILE - 1) / SM_TILE);
    return any_size || (a.L.nkb * a.L.bp <= SM_AUTO_BYTES && ctas <= SM_AUTO_CTAS);
}

int launch_gemm_small(int64_t M, int64_t N, const Packed& a, const Packed& b, const float* bias, float* C, int64_t ldc, cudaStream_t st) {
    const int nkb = (int)a.L.nkb;
    const size_t smem = 2 * SM_BUF + 2 * (size_t)nkb * SM_TILE;          // at most 132 KB
    // the attribute belongs to the device: set once per device (same value from any thread)
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HBFP_ERR_CUDA;
    if (!attr_set[dev]) {
        HBFP_CUDA_OK(cudaFuncSetAttribute(gemm_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * SM_BUF + 2 * SM_MAX_NKB * SM_TILE));
        attr_set[dev] = true;
    }
    const dim3 grid((unsigned)((N + SM_TILE - 1) / SM_TILE), (unsigned)((M + SM_TILE - 1) / SM_TILE));
    launch_chained(gemm_small_kernel, grid, 256, smem, st, M, N, nkb, (int)a.L.bp, a.mant, a.L.kst, a.exps, a.L.rs, b.mant, b.L.kst,
                                               b.exps, b.L.rs, bias, C, ldc);
    note_product(st);
    return launch_status();
}

namespace {
template <bool SR, int PER>
int sf_launch(const SmallProblem& p, dim3 grid, cudaStream_t st) {
    static bool attr_set[64] = {};                                      // the attribute belongs to the device (same value from any thread)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HBFP_ERR_CUDA;
    if (!attr_set[dev]) {
        HBFP_CUDA_OK(cudaFuncSetAttribute(gemm_small_fused_kernel<SR, PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * SM_TILE * (2 * SM_AUTO_BYTES + 64)));
        attr_set[dev] = true;
    }
    launch_chained(gemm_small_fused_kernel<SR, PER>, grid, SF_THREADS, 2 * (size_t)SM_TILE * p.pitch, st, p);      // at most 68 KB
    note_product(st);
    return launch_status();
}
}  // namespace

// Where the small kernel would be chosen, both operands are FP32 without weight tiles and no draw straddles two groups.
bool small_fused_eligible(const hbfp_operand* a, bool a_contig, const hbfp_operand* b, bool b_contig, int64_t M, int64_t N, const Layout& la) {
    if (a->kind != HBFP_OPERAND_FP32 || b->kind != HBFP_OPERAND_FP32 || a->fmt.tile != 0 || b->fmt.tile != 0) return false;
    if (la.bp > 128 || la.nkb * la.bp > SM_AUTO_BYTES || la.nkb <= 0) return false;
    // (Times of both sides before launches were chained.)
    // A CTA's registers fill an SM when a column conversion holds 512 K; a second round of tiles then costs more than two launches
    // (512 cube 18.6 against 10.7 us of device time; 512 x 512 x 256, two CTAs per SM, 10.5 against 14.3 as a call).
    const int64_t ctas = ((M + SM_TILE - 1) / SM_TILE) * ((N + SM_TILE - 1) / SM_TILE);
    if (la.nkb * la.bp > 256 && ctas > 148) return false;
    // Draws are made again in every tile of a row of tiles: with more tiles than SMs or long columns on both sides two launches
    // win (device time / as a call: 512 x 512 x 256 19.4 against 11.1, 20.7 / 16.3; 384 cube from columns 21.5 / 10.8, 22.7 / 16.5;
    // 128 x 1792 x 209 18.4 against 12.1).
    if (a->fmt.rounding || b->fmt.rounding) {
        if (la.nkb * la.bp > 128 && ctas > 148) return false;
        if (la.nkb * la.bp > 384 && ctas > 74 && !a_contig && !b_contig) return false;
    }
    return (a_contig || a->fmt.rounding == 0 || M % 8 == 0) && (b_contig || b->fmt.rounding == 0 || N % 8 == 0);
}

int launch_gemm_small_fused(int64_t M, int64_t N, int64_t K, const hbfp_operand* a, bool a_contig, const hbfp_operand* b, bool b_contig, const Layout& la,
                            float* C, int64_t ldc, cudaStream_t st) {
    SmallProblem p{};
    p.K = (int)K;
    p.blk = (int)la.b;
    p.bp = (int)la.bp;
    p.lg_bp = la.bp == 32 ? 5 : la.bp == 64 ? 6 : 7;
    p.nkb = (int)la.nkb;
    p.pitch = (int)round_up(2 * la.nkb * la.bp, 128) + 64;              // rows half a line of banks apart
    p.C = C;
    p.ldc = ldc;
    auto fill = [&](SmallOperand& o, const hbfp_operand* h, bool contig, int64_t lines) {
        o.x = static_cast<const float*>(h->data);
        o.ld = h->ld;
        o.lines = lines;
        o.contig = contig;
        o.vec = (reinterpret_cast<uintptr_t>(o.x) & 15) == 0 && (h->ld & 3) == 0 && (p.blk & 3) == 0;
        o.q = make_params(&h->fmt);
    };
    fill(p.a, a, a_contig, M);
    fill(p.b, b, b_contig, N);
    const dim3 grid((unsigned)((N + SM_TILE - 1) / SM_TILE), (unsigned)((M + SM_TILE - 1) / SM_TILE));
    const bool sr = a->fmt.rounding == 1 || b->fmt.rounding == 1, shallow = la.nkb * la.bp <= 256;
    if (shallow) return sr ? sf_launch<true, 4>(p, grid, st) : sf_launch<false, 4>(p, grid, st);
    return sr ? sf_launch<true, 8>(p, grid, st) : sf_launch<false, 8>(p, grid, st);
}

}  // namespace hbfp
