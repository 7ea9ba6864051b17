// FP32 -> block-floating-point conversion kernels (the FP-to-BFP step of Sec. 4.1 / Sec. 5.3)
// and the inverse helpers used for inspection. HBM-bound: every FP32 element is read once,
// one (or two) mantissa bytes and 1/b exponent bytes are written.
//
// Kernels
//   quant_row_fast   blocks along contiguous rows, b in {32,64,128,256}: 8 elements per
//                    thread (two 128-bit loads, one Philox call in stochastic mode), block
//                    max by warp shuffles, exponents staged in shared memory so that the
//                    [kb][row] exponent array is written in full 32-byte sectors.
//   quant_row_flat   the same for row lengths that are not a multiple of 512 (K % b == 0): 8-element
//                    groups numbered through the whole matrix, no ragged last tile.
//   quant_col_tma    blocks down the columns, b in {32,64,128}, 16-byte aligned pitch: persistent
//                    CTAs stream 128 x 64 FP32 tiles through a TMA pipeline and write the packed,
//                    transposed tile with a swizzled TMA store (full lines in both directions).
//   quant_col_block  blocks down the columns, any b <= 128 and any pitch: 32 columns of four, two or one K-blocks (by their length)
//                    per CTA, a lane per column.
//   quant_row_ragged blocks along rows, any b <= 128, row length, pitch and alignment, in one pass.
//   tile_strip_kernel, tile_kernel, tile_kernel_full   t x t weight tiles (t <= 128): one pass writes both packed views and
//                    the tile exponent grid.
//   exps_* / mant_generic   two-pass path for every other geometry (any b, any alignment).
#include "quant_math.cuh"

#include <type_traits>

// This file is compiled twice. Part 1 (default) is the library's quantiser; part 2 holds only the launches of the
// full-tile kernel for tiles of 32 and 64, built with another ptxas level (see build.py): measured on 8192 x 8192,
// t = 64, the in-place update takes 111 instead of 129 us and the narrow views 48 instead of 56 us that way, while the
// same level costs tiles of 128 and the other kernels of this file time.
#ifndef HBFP_QUANT_PART
#define HBFP_QUANT_PART 1
#endif

namespace hbfp {
namespace {

// ------------------------------------------------------------------------------ quant_row_fast

// LPB = lanes per block (b = 8 * LPB). CTA: 256 threads, tile 32 rows x 512 columns.
// Three CTAs per SM with draws, four without: left to itself the compiler took 88 to 98 registers for the former and so two
// CTAs (3186 x 12360 and 265 x 12360, b = 128, stochastic: 54.2 us, now 47.5; the 12-bit form of a 4096 x 4096 operand 22.4, now 20.6).
template <int LPB, bool SR, int PLANES>
__global__ void __launch_bounds__(256, SR ? 3 : 4)
quant_row_fast(const float* __restrict__ x, int64_t rows, int64_t K, int64_t ld, QParams p,
               int8_t* __restrict__ mant, int64_t kst, int64_t plane_stride,
               int8_t* __restrict__ exps, int64_t rs, int64_t nkb, const int8_t* __restrict__ given, const FormArgs fa) {
    const Chain chain(p.at);
    // given != nullptr: one exponent per row for the whole axis, computed beforehand (a block longer than the
    // tile); the kernel then only rounds and packs
    constexpr int B = 8 * LPB;
    constexpr int KB_PER_SPAN = 256 / B;            // blocks in one warp span of 256 columns
    constexpr int KB_PER_TILE = 512 / B;
    __shared__ int8_t s_exps[KB_PER_TILE][32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.y * 32;
    const int64_t c0 = (int64_t)blockIdx.x * 512;

    for (int i = tid; i < KB_PER_TILE * 32; i += 256) (&s_exps[0][0])[i] = 0;
    __syncthreads();

    // warp w owns rows r0 + 4w .. +3, both spans: 8 items, in two batches of 4 rows.
#pragma unroll
    for (int span = 0; span < 2; ++span) {
        float4 v[4][2];
        const int64_t col = c0 + span * 256 + lane * 8;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t r = r0 + warp * 4 + i;
            if (r < rows && col < K) {
                const float4* src = reinterpret_cast<const float4*>(x + r * ld + col);
                v[i][0] = __ldcs(src);
                v[i][1] = __ldcs(src + 1);
            } else {
                v[i][0] = make_float4(0.f, 0.f, 0.f, 0.f);
                v[i][1] = v[i][0];
            }
        }
        // the draws do not depend on the data: they are made while the loads are in flight
        uint4 wd[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            wd[i] = make_uint4(0u, 0u, 0u, 0u);
            if (SR) wd[i] = draws_of_group(p, (uint64_t)((r0 + warp * 4 + i) * K + col) >> 3);   // a multiple of 8 on this path
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t r = r0 + warp * 4 + i;
            const float e8[8] = {v[i][0].x, v[i][0].y, v[i][0].z, v[i][0].w,
                                 v[i][1].x, v[i][1].y, v[i][1].z, v[i][1].w};
            uint32_t am = amax8_bits(e8);
#pragma unroll
            for (int off = 1; off < LPB; off <<= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
            const int s = given ? (r < rows ? (int)given[r] : -63) : block_exponent(am, p.m, p.exp_mode);
            const uint4 w = wd[i];
            if constexpr (is_form(PLANES)) {
                round_and_store8<SR, PLANES>(e8, s, p, w, mant, r * kst + col, plane_stride, r < rows && col < kst);
                check_exponent<PLANES>(s, fa);
            } else {
                // written out: with the address formed before the branch, as the call above does, the kernel with draws no longer fits
                // 80 registers and spills (4096 x 4096, b = 256: 18.8 -> 19.5 us)
                uint2 hi, lo;
                quantize_pack8<SR, PLANES>(e8, s, p, w, hi, lo);
                if (r < rows && col < kst) {
                    *reinterpret_cast<uint2*>(mant + r * kst + col) = hi;
                    if (PLANES == 2) *reinterpret_cast<uint2*>(mant + plane_stride + r * kst + col) = lo;
                }
            }
            if ((lane % LPB) == 0 && r < rows && col < K)
                s_exps[span * KB_PER_SPAN + lane / LPB][warp * 4 + i] = (int8_t)s;
        }
    }
    __syncthreads();
    if (given || PLANES == FORM_SCALED) return;
    // exponents: [kb][row], 32 rows of one block are 32 contiguous bytes.
    const int64_t kb0 = c0 / B;
    for (int i = tid; i < KB_PER_TILE * 8; i += 256) {
        const int kbl = i >> 3, part = i & 7;
        const int64_t kb = kb0 + kbl, r = r0 + part * 4;
        if (kb < nkb && r < rs) {
            const uint32_t e4 = *reinterpret_cast<const uint32_t*>(&s_exps[kbl][part * 4]);
            if (is_form(PLANES))
                *reinterpret_cast<float4*>(reinterpret_cast<float*>(exps) + kb * rs + r) =
                    make_float4(pow2f((int8_t)e4), pow2f((int8_t)(e4 >> 8)), pow2f((int8_t)(e4 >> 16)), pow2f((int8_t)(e4 >> 24)));
            else *reinterpret_cast<uint32_t*>(exps + kb * rs + r) = e4;
        }
    }
}

// ------------------------------------------------------------------------------ quant_col_block

// Blocks down the columns of x [K][R] (contract axis 0); output rows are the columns of x. Any block length up to 128, any
// pitch and alignment (the paper's tile of 24 among them). A lane takes one column and up to NV of a block's rows, so that every load
// is a warp's 128 consecutive bytes of one row, all of a thread's loads are in flight together, the values stay in registers between
// the maximum and the rounding, and the packed bytes of a thread are one whole sector of its output row: nothing passes through shared
// memory but the draws. Blocks of up to 32 belong to one warp and need no barrier, longer ones to two or four. A block's rows over
// four warps of eight, through shared memory both ways, left a quarter of the threads idle at b = 24 and waited at two barriers.
// Before / now: 10000 x 10000, b = 24 154 / 93 us (4.3 / 5.4 TB/s with the padding written), with draws 268 / 110; 20000 x 3001, b = 64,
// with draws 107 / 69; 5001 x 4999, b = 32 33 / 20; the 12-bit form of 2373 x 4352, b = 24 20.6 / 10.2.
constexpr int COLT = 32, COL_WARPS = 4;

template <int PLANES, int NV, int WPB, bool SR>      // WPB: warps per block; the padded block length is 32 WPB
__global__ void __launch_bounds__(32 * COL_WARPS)
quant_col_block(const float* __restrict__ x, int64_t K, int64_t R, int64_t ld, int b, QParams p,
                int8_t* __restrict__ mant, int64_t kst, int64_t plane_stride,
                int8_t* __restrict__ exps, int64_t rs, int64_t nkb, unsigned tiles_n, const FormArgs fa, const int8_t* __restrict__ given) {
    const Chain chain(p.at);
    // given != nullptr: one exponent per column for the whole axis, computed beforehand; the blocks are then pieces of it
    constexpr int BP = 32 * WPB, BPC = COL_WARPS / WPB;                // BPC: blocks of a CTA
    __shared__ uint32_t pmax[WPB > 1 ? COL_WARPS : 1][COLT];
    __shared__ __align__(16) uint4 rnd[SR ? COL_WARPS : 1][SR ? NV : 1][5];      // draws of a row: its 32 columns lie in at most five groups of eight
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned kg = blockIdx.x / tiles_n;
    const int64_t kb = (int64_t)kg * BPC + warp / WPB, c0 = (int64_t)(blockIdx.x - kg * tiles_n) * COLT, col = c0 + lane;
    if (WPB == 1 && kb >= nkb) return;
    const int part = warp % WPB;
    const int64_t k0 = kb * b + part * 32;
    const int n = kb < nkb ? max(0, (int)min((int64_t)min(NV, b - part * 32), K - k0)) : 0;     // rows of this warp
    const float* src = x + k0 * ld + col;
    const bool full = n == NV && c0 + COLT <= R;
    float v[NV];
    if (full) {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = __ldcs(src + (int64_t)j * ld);
    } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = j < n && col < R ? __ldcs(src + (int64_t)j * ld) : 0.f;
    }
    // the draws do not depend on the data: they are made while the loads are in flight, one Philox call per group of eight
    // consecutive source elements (rows that all start with a group touch four of them)
    if (SR) {
        auto draw = [&](auto count) {
            constexpr int N = decltype(count)::value;
            for (int i = lane; i < n * N; i += 32) {
                const int kk = i / N, g = i - kk * N;
                rnd[warp][kk][g] = draws_of_group(p, ((uint64_t)((k0 + kk) * R + c0) >> 3) + g);
            }
            __syncwarp();
        };
        if ((R & 7) == 0) draw(std::integral_constant<int, 4>{});
        else draw(std::integral_constant<int, 5>{});
    }
    uint32_t am = 0;
#pragma unroll
    for (int j = 0; j < NV; j += 2) am = max3_abs_bits(am, v[j], v[j + 1]);
    if (WPB > 1) {
        pmax[warp][lane] = am;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WPB; ++w) am = max(am, pmax[warp - part + w][lane]);
        if (kb >= nkb) return;
    }
    const int s = given ? (col < R ? (int)given[col] : -63) : block_exponent(am, p.m, p.exp_mode);
    check_exponent<PLANES>(s, fa);
    if constexpr (is_form(PLANES)) { if (part == 0 && col < R) store_exponent<PLANES>(exps, kb * rs + col, s); }
    else if (!given && part == 0 && col < rs) exps[kb * rs + col] = col < R ? (int8_t)s : (int8_t)0;      // lines beyond the matrix are documented as zero
    const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
    const float sc = pow2f(SR ? 16 - s : -s);
    const uint16_t* rnd16 = reinterpret_cast<const uint16_t*>(rnd[SR ? warp : 0]) + lane;
    const uint32_t first = SR ? (uint32_t)((uint64_t)(k0 * R + c0) & 7) : 0u, row_step = (uint32_t)(R & 7);
    uint32_t hi[8], lo[8];
    uint32_t fo[is_form(PLANES) ? 2 : 1][16];
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint32_t h[2] = {0u, 0u};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int j = 4 * w + 2 * k;
            if (j >= NV) continue;                                     // the block's padding
            if (SR) {
                // zeros below the block or the matrix stay zero whatever the draw (their table rows hold anything)
                const uint32_t r0 = rnd16[j * 40 + ((first + (uint32_t)j * row_step) & 7)], r1 = rnd16[(j + 1) * 40 + ((first + (uint32_t)(j + 1) * row_step) & 7)];
                h[k] = round_sr_pair2(v[j], v[j + 1], sc, r0, r1, qm, nqm);
            } else {
                h[k] = round_rne_pair(v[j], v[j + 1], sc, qm, nqm);
            }
        }
        if constexpr (is_form(PLANES)) {
            form_pair<PLANES>(h[0], pow2f(s), fo[0][2 * w], fo[1][2 * w]);
            form_pair<PLANES>(h[1], pow2f(s), fo[0][2 * w + 1], fo[1][2 * w + 1]);
        } else {
            pack4<PLANES>(h[0], h[1], hi[w], lo[w]);
        }
    }
    if (col >= R) return;
    if constexpr (is_form(PLANES)) {
#pragma unroll
        for (int pl = 0; pl < (PLANES == FORM_WIDE_B ? 2 : 1); ++pl) {
            int8_t* row = mant + 2 * (pl * plane_stride + col * kst);
            store_sector(row + 2 * (kb * BP + part * 32), &fo[pl][0]);
            store_sector(row + 2 * (kb * BP + part * 32) + 32, &fo[pl][8]);
            if (kb == nkb - 1 && part == 0)                            // the row tail [nkb * bp, kst)
                for (int64_t o = nkb * BP; o < kst; o += 8) *reinterpret_cast<uint4*>(row + 2 * o) = make_uint4(0, 0, 0, 0);
        }
    } else {
#pragma unroll
        for (int pl = 0; pl < PLANES; ++pl) {
            int8_t* row = mant + pl * plane_stride + col * kst;
            store_sector(row + kb * BP + part * 32, pl ? lo : hi);
            if (kb == nkb - 1 && part == 0)
                for (int64_t o = nkb * BP; o < kst; o += 16) *reinterpret_cast<uint4*>(row + o) = make_uint4(0, 0, 0, 0);
        }
    }
}

// One launch for blocks of b (padded to bp): OUT is 1 or 2 planes or a form.
template <int OUT>
int launch_col_block(const float* x, int64_t K, int64_t rows, int64_t ld, int b, int64_t bp, int64_t nkb, const QParams& p, const Layout& L, int8_t* mant, int8_t* exps,
                     cudaStream_t st, const FormArgs& fa, const int8_t* given) {
    const unsigned tiles_n = (unsigned)((rows + COLT - 1) / COLT);
    const int64_t per = 128 / bp, grid = (int64_t)tiles_n * ((nkb + per - 1) / per);
#define HBFP_QCOL(NV, WPB, SRV) launch_placed(p.at, 4 * K * rows, quant_col_block<OUT, NV, WPB, SRV>, (unsigned)grid, 32 * COL_WARPS, 0, st, x, K, rows, ld, b, p, mant, L.kst, L.plane_stride, exps, L.rs, nkb, tiles_n, fa, given)
#define HBFP_QCOL_SR(NV, WPB) do { if (p.rounding) HBFP_QCOL(NV, WPB, true); else HBFP_QCOL(NV, WPB, false); } while (0)
    if (bp == 32) { if (b <= 24) HBFP_QCOL_SR(24, 1); else HBFP_QCOL_SR(32, 1); }
    else if (bp == 64) HBFP_QCOL_SR(32, 2);
    else if constexpr (!is_form(OUT)) HBFP_QCOL_SR(32, 4);
    else return HBFP_ERR_UNSUPPORTED;
#undef HBFP_QCOL_SR
#undef HBFP_QCOL
    return launch_status();
}

// ------------------------------------------------------------------------------ weight tiles

// Writes one quantised t x t tile (qt: [tp][tp] int16, zero padded) into both packed views, with the
// tile's exponent s replicated over its rows and columns, and zeroes the row tails beyond the last tile.
// (u, v) = tile row / tile column; the tile covers hi x wj elements from (i0, j0).
struct TileViews {
    int8_t* mant_c0; int64_t kst0, ps0; int8_t* exps_c0; int64_t rs0, nkb0;
    int8_t* mant_c1; int64_t kst1, ps1; int8_t* exps_c1; int64_t rs1, nkb1;
    float* value; int64_t ldv;      // FP32 value of the wide words (modes that write them), or null
};

// Bytes that the modes below load: FP32 and words.
template <int MODE>
constexpr int64_t tile_bytes(int64_t d0, int64_t d1) { return d0 * d1 * (MODE == 1 || MODE == 4 ? 6 : MODE == 2 ? 2 : 4); }

// 2^e for every stored exponent: below -126 the power itself is subnormal, and its product with a mantissa is exact.
__device__ __forceinline__ float pow2f_stored(int e) {
    return __uint_as_float(e >= -126 ? (uint32_t)(e + 127) << 23 : 0x00400000u >> (-127 - e));
}
// The values of two packed 16-bit mantissas.
__device__ __forceinline__ float2 wide_values(uint32_t q2, float scale) {
    return make_float2(__fmul_rn((float)(int16_t)(q2 & 0xFFFFu), scale), __fmul_rn((float)((int32_t)q2 >> 16), scale));
}
__device__ __forceinline__ void store_wide_values(float* dst, const uint32_t h[4], float scale) {
    const float2 a = wide_values(h[0], scale), b = wide_values(h[1], scale), c = wide_values(h[2], scale), d = wide_values(h[3], scale);
    reinterpret_cast<float4*>(dst)[0] = make_float4(a.x, a.y, b.x, b.y);
    reinterpret_cast<float4*>(dst)[1] = make_float4(c.x, c.y, d.x, d.y);
}

// Stochastic rounding to 16 bits: floor((floor(y) + r) / 2^16) of y = x * 2^(16-s), which reaches 2^31, in 32 bits: the upper half of
// floor(y) plus the carry of the lower one. (Saturated at +-2^31 the conversion leaves what the clamp makes of the value itself; a
// NaN ends at the lower bound, as a conversion to 64 bits has it.)
__device__ __forceinline__ int floor_wide(float y, uint32_t r) {
    const int t = __float2int_rd(y);
    const int q = (t >> 16) + (int)((((uint32_t)t & 0xFFFFu) + r) >> 16);
    return y != y ? -32767 : clampq(q, 32767);
}
__device__ __forceinline__ int round_sr_wide(float x, int s, uint32_t r) { return floor_wide(__fmul_rn(x, pow2f(16 - s)), r); }

// qt rows have a pitch of tp + 2 halfwords, so that the column reads of view c0 spread over the banks.
// sh: the views take the top bits of the words in qt (an arithmetic shift by sh bits); for wide storage qt
// holds the stored words, i.e. the mantissas plus half a narrow unit (see tile_kernel); sh = 0 copies.
template <int PLANES>
__device__ __forceinline__ void write_tile_views(const int16_t* qt, int tp, int hi, int wj, int64_t i0, int64_t j0,
                                                 int64_t u, int64_t v, int s, int sh, const TileViews& tv, int tid) {
    const int qp = tp + 2;
    const int lg = 31 - __clz(tp >> 2), gmask = (tp >> 2) - 1;       // tp is 32, 64 or 128
    int8_t* const mant_c0 = tv.mant_c0; int8_t* const mant_c1 = tv.mant_c1;
    int8_t* const exps_c0 = tv.exps_c0; int8_t* const exps_c1 = tv.exps_c1;
    const int64_t kst0 = tv.kst0, ps0 = tv.ps0, rs0 = tv.rs0, nkb0 = tv.nkb0;
    const int64_t kst1 = tv.kst1, ps1 = tv.ps1, rs1 = tv.rs1, nkb1 = tv.nkb1;
    // view c1: row i0+ii gets bytes [v*tp, v*tp+tp) = qt[ii][0..tp)
    if (mant_c1) for (int e = tid; e < hi * (tp / 4); e += 256) {
        const int ii = e >> lg, g = (e & gmask) * 4;
        uint32_t h = 0, l = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = qt[ii * qp + g + j] >> sh;
            if (PLANES == 1) h |= (uint32_t)(q & 0xff) << (8 * j);
            else { h |= (uint32_t)((q >> 4) & 0xff) << (8 * j); l |= (uint32_t)(q & 15) << (8 * j); }
        }
        int8_t* dst = mant_c1 + (i0 + ii) * kst1 + v * tp + g;
        *reinterpret_cast<uint32_t*>(dst) = h;
        if (PLANES == 2) *reinterpret_cast<uint32_t*>(dst + ps1) = l;
    }
    // view c0: row j0+jj gets bytes [u*tp, u*tp+tp) = qt[0..tp)[jj]
    // (neighbouring threads write neighbouring words of one output row)
    if (mant_c0) for (int e = tid; e < wj * (tp / 4); e += 256) {
        const int jj = e >> lg, g = (e & gmask) * 4;
        uint32_t h = 0, l = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = qt[(g + j) * qp + jj] >> sh;
            if (PLANES == 1) h |= (uint32_t)(q & 0xff) << (8 * j);
            else { h |= (uint32_t)((q >> 4) & 0xff) << (8 * j); l |= (uint32_t)(q & 15) << (8 * j); }
        }
        int8_t* dst = mant_c0 + (j0 + jj) * kst0 + u * tp + g;
        *reinterpret_cast<uint32_t*>(dst) = h;
        if (PLANES == 2) *reinterpret_cast<uint32_t*>(dst + ps0) = l;
    }
    // replicated exponents: exps_c1[v][i0+ii], exps_c0[u][j0+jj]
    // (lines beyond the matrix, at most 15 after the last tile, are documented as zero)
    const int pad1 = u == nkb0 - 1 ? (int)(rs1 - i0) : hi, pad0 = v == nkb1 - 1 ? (int)(rs0 - j0) : wj;
    if (exps_c1) for (int e = tid; e < pad1; e += 256) exps_c1[v * rs1 + i0 + e] = e < hi ? (int8_t)s : (int8_t)0;
    if (exps_c0) for (int e = tid; e < pad0; e += 256) exps_c0[u * rs0 + j0 + e] = e < wj ? (int8_t)s : (int8_t)0;
    // row tails beyond the last tile: zero them (last tile column / last tile row only)
    if (mant_c1 && v == nkb1 - 1)
        for (int64_t e = tid; e < (int64_t)hi * ((kst1 - nkb1 * tp) / 4); e += 256) {
            const int64_t per = (kst1 - nkb1 * tp) / 4, ii = e / per, o = nkb1 * tp + (e % per) * 4;
            *reinterpret_cast<uint32_t*>(mant_c1 + (i0 + ii) * kst1 + o) = 0;
            if (PLANES == 2) *reinterpret_cast<uint32_t*>(mant_c1 + ps1 + (i0 + ii) * kst1 + o) = 0;
        }
    if (mant_c0 && u == nkb0 - 1)
        for (int64_t e = tid; e < (int64_t)wj * ((kst0 - nkb0 * tp) / 4); e += 256) {
            const int64_t per = (kst0 - nkb0 * tp) / 4, jj = e / per, o = nkb0 * tp + (e % per) * 4;
            *reinterpret_cast<uint32_t*>(mant_c0 + (j0 + jj) * kst0 + o) = 0;
            if (PLANES == 2) *reinterpret_cast<uint32_t*>(mant_c0 + ps0 + (j0 + jj) * kst0 + o) = 0;
        }
}

// The same (modes below) with one CTA of 256 threads per tile, the FP32 tile and the words in shared memory: the tile_strip_kernel's strips
// leave most of the chip idle where the tiles are few, and its 32-bit accesses cost more than this kernel's sixteen bytes on tiles of
// whole eights that its strips are wide for one of (rule and both sides measured in launch_tiles).
// FAST: t, d1 multiples of 8, pitches and bases 16-byte aligned: a thread handles eight consecutive
// weights of a row at a time (two 128-bit loads, one Philox call, 128-bit store of the int16 mantissas).
template <int MODE, int PLANES, bool FAST>
__global__ void __launch_bounds__(256)
tile_kernel(const float* __restrict__ src, int64_t ld, int64_t d0, int64_t d1, int t, int tp, QParams p,
            int16_t* __restrict__ wide, int8_t* __restrict__ grid, int64_t grid_ld, TileViews tv) {
    chain_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int fp = FAST ? t + 4 : t + 1;                                   // pitch of the FP32 tile
    float* tile = reinterpret_cast<float*>(smem_raw);                      // [t][fp]
    const int qp = tp + 2;
    int16_t* qt = reinterpret_cast<int16_t*>(tile + (size_t)t * fp);       // [tp][tp + 2], zero padded
    __shared__ uint32_t s_am[8];
    __shared__ int s_exp;

    const int tid = threadIdx.x, lane = tid & 31, wrow = tid >> 5;
    const int64_t u = blockIdx.y, v = blockIdx.x;       // tile row (along d0), tile column (along d1)
    const int64_t i0 = u * t, j0 = v * t;
    const int hi = (int)min((int64_t)t, d0 - i0), wj = (int)min((int64_t)t, d1 - j0);
    const int G = wj >> 3;                              // FAST: groups of eight per tile row
    constexpr bool UPDATE = MODE == 1 || MODE == 4;
    const int wbits = MODE == 3 ? p.m : 16, wqmax = MODE == 3 ? p.qmax : 32767;
    // Wide modes: qt holds the stored word the views are cut from: the mantissa plus half a narrow unit,
    // held inside the range whose top bits stay within +-qmax (so the shift alone rounds to nearest and
    // saturates symmetrically). MODE 3 copies (sh = 0).
    const int sh = MODE == 3 ? 0 : 16 - p.m;
    const int half = sh > 0 ? 1 << (sh - 1) : 0;
    const int w_hi = ((p.qmax + 1) << sh) - half - 1, w_lo = -(p.qmax << sh) - half;
    const uint32_t w_hi2 = ((uint32_t)w_hi & 0xFFFFu) * 0x10001u, w_lo2 = ((uint32_t)w_lo & 0xFFFFu) * 0x10001u;
    const uint32_t half2 = (uint32_t)half * 0x10001u;
    auto stored_pair = [&](uint32_t h) { return MODE == 3 ? h : __vadd2(__vmaxs2(__vmins2(h, w_hi2), w_lo2), half2); };
    auto stored_one = [&](int q) { return MODE == 3 ? q : max(w_lo, min(w_hi, q)) + half; };
    for (int e = tid; e < tp * qp / 2; e += 256) reinterpret_cast<uint32_t*>(qt)[e] = 0;
    int s;
    if (MODE == 2) {
        __syncthreads();
        s = grid[u * grid_ld + v];
        if (FAST) {
            for (int item = tid; item < hi * G; item += 256) {
                const int ii = item / G, gj = item - ii * G;
                const uint4 q8 = *reinterpret_cast<const uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj);
                uint32_t* dst = reinterpret_cast<uint32_t*>(qt + ii * qp + 8 * gj);
                dst[0] = stored_pair(q8.x); dst[1] = stored_pair(q8.y); dst[2] = stored_pair(q8.z); dst[3] = stored_pair(q8.w);
            }
        } else {
            for (int ii = wrow; ii < hi; ii += 8)
                for (int jj = lane; jj < wj; jj += 32) qt[ii * qp + jj] = (int16_t)stored_one(wide[(i0 + ii) * d1 + j0 + jj]);
        }
    } else {
        const float old_scale = UPDATE ? pow2f(grid[u * grid_ld + v]) : 0.f;
        uint32_t am = 0;
        if (FAST) {
            for (int item = tid; item < hi * G; item += 256) {
                const int ii = item / G, gj = item - ii * G;
                const float4* sp = reinterpret_cast<const float4*>(src + (i0 + ii) * ld + j0 + 8 * gj);
                float4 a = __ldcs(sp), b = __ldcs(sp + 1);
                if (UPDATE) {
                    const uint4 q8 = *reinterpret_cast<const uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj);
                    a.x = __fadd_rn(__fmul_rn((float)(int16_t)(q8.x & 0xFFFFu), old_scale), a.x);
                    a.y = __fadd_rn(__fmul_rn((float)(int16_t)(q8.x >> 16), old_scale), a.y);
                    a.z = __fadd_rn(__fmul_rn((float)(int16_t)(q8.y & 0xFFFFu), old_scale), a.z);
                    a.w = __fadd_rn(__fmul_rn((float)(int16_t)(q8.y >> 16), old_scale), a.w);
                    b.x = __fadd_rn(__fmul_rn((float)(int16_t)(q8.z & 0xFFFFu), old_scale), b.x);
                    b.y = __fadd_rn(__fmul_rn((float)(int16_t)(q8.z >> 16), old_scale), b.y);
                    b.z = __fadd_rn(__fmul_rn((float)(int16_t)(q8.w & 0xFFFFu), old_scale), b.z);
                    b.w = __fadd_rn(__fmul_rn((float)(int16_t)(q8.w >> 16), old_scale), b.w);
                }
                float4* tp4 = reinterpret_cast<float4*>(tile + ii * fp + 8 * gj);
                tp4[0] = a; tp4[1] = b;
                const float e8[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                am = max(am, amax8_bits(e8));
            }
        } else {
            for (int ii = wrow; ii < hi; ii += 8)
                for (int jj = lane; jj < wj; jj += 32) {
                    float val = src[(i0 + ii) * ld + j0 + jj];
                    if (UPDATE) val = __fadd_rn(__fmul_rn((float)wide[(i0 + ii) * d1 + j0 + jj], old_scale), val);
                    tile[ii * fp + jj] = val;
                    am = max(am, abs_bits(val));
                }
        }
        for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
        if (lane == 0) s_am[wrow] = am;
        __syncthreads();
        if (tid == 0) {
            uint32_t a = 0;
            for (int i = 0; i < 8; ++i) a = max(a, s_am[i]);
            s_exp = block_exponent(a, wbits, p.exp_mode);
            if (grid) grid[u * grid_ld + v] = (int8_t)s_exp;
        }
        __syncthreads();
        s = s_exp;
        if (FAST) {
            const uint32_t qm = qmax_pair(wqmax), nqm = neg_qmax_pair(wqmax);
            for (int item = tid; item < hi * G; item += 256) {
                const int ii = item / G, gj = item - ii * G;
                const float4* tp4 = reinterpret_cast<const float4*>(tile + ii * fp + 8 * gj);
                const float4 a = tp4[0], b = tp4[1];
                const float e8[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                if (p.rounding == 1) w = draws_of_group(p, (uint64_t)((i0 + ii) * d1 + j0 + 8 * gj) >> 3);
                const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                uint32_t h[4];
                if (MODE == 3) {
                    // at most 12 bits: the packed halfword forms
                    const float sc = pow2f(p.rounding == 1 ? 16 - s : -s);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        h[j] = p.rounding == 1 ? round_sr_pair(e8[2 * j], e8[2 * j + 1], sc, ww[j], qm, nqm)
                                               : round_rne_pair(e8[2 * j], e8[2 * j + 1], sc, qm, nqm);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        int q0, q1;
                        if (p.rounding == 0) {
                            q0 = round_rne(e8[2 * j], s, 32767);
                            q1 = round_rne(e8[2 * j + 1], s, 32767);
                        } else {
                            q0 = round_sr_wide(e8[2 * j], s, ww[j] & 0xFFFFu);
                            q1 = round_sr_wide(e8[2 * j + 1], s, ww[j] >> 16);
                        }
                        h[j] = ((uint32_t)q0 & 0xFFFFu) | ((uint32_t)q1 << 16);
                    }
                }
                uint32_t* dst = reinterpret_cast<uint32_t*>(qt + ii * qp + 8 * gj);
                dst[0] = stored_pair(h[0]); dst[1] = stored_pair(h[1]); dst[2] = stored_pair(h[2]); dst[3] = stored_pair(h[3]);
                if (MODE != 3) *reinterpret_cast<uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj) = make_uint4(h[0], h[1], h[2], h[3]);
                if (MODE == 4) store_wide_values(tv.value + (i0 + ii) * tv.ldv + j0 + 8 * gj, h, pow2f_stored(s));
            }
        } else {
            for (int ii = wrow; ii < hi; ii += 8)
                for (int jj = lane; jj < wj; jj += 32) {
                    const float val = tile[ii * fp + jj];
                    const uint64_t L = (uint64_t)((i0 + ii) * d1 + j0 + jj);
                    int q;
                    if (MODE == 3) q = quantize_one(val, s, p, L);
                    else if (p.rounding == 0) q = round_rne(val, s, 32767);
                    else q = round_sr_wide(val, s, draw_of_element(p, L));
                    qt[ii * qp + jj] = (int16_t)stored_one(q);
                    if (MODE != 3) wide[(i0 + ii) * d1 + j0 + jj] = (int16_t)q;
                    if (MODE == 4) tv.value[(i0 + ii) * tv.ldv + j0 + jj] = __fmul_rn((float)q, pow2f_stored(s));
                }
        }
    }
    if (tv.mant_c0 == nullptr && tv.mant_c1 == nullptr) return;
    __syncthreads();
    write_tile_views<PLANES>(qt, tp, hi, wj, i0, j0, u, v, s + sh, sh, tv, tid);
}

// Weight matrices with one exponent per t x t tile (Sec. 4.2 "Tiling", t <= 128) and their wide storage
// (Sec. 4.2 "Wide weight storage"), for every tile geometry, alignment and width
// that neither tile_kernel_full nor tile_kernel takes.
//   MODE 3  quantise FP32 weights src (pitch ld) straight to p.m bits (no wide copy)
//   MODE 0  quantise FP32 weights src to wide storage: int16 mantissas `wide` (row-major, pitch d1) and
//           one exponent per tile in grid [tiles along d0][tiles along d1]
//   MODE 1  update: w = fl32(wide * 2^s + src) with src the FP32 update, re-quantised to 16 bits in place
//   MODE 4  the same, and the FP32 value of the new words to tv.value (a mode of its own: a runtime test in mode 1
//           cost the plain update of 8192 x 8192 weights 1.5 us of 110); 4 bytes per weight more instead of a second
//           pass that reads the words again, 12.1 -> 13.1 us against 12.1 + 5.5 for 1024 x 4096 weights
//   MODE 2  read wide storage only
// In every mode, when view pointers are given, the tile goes to the two packed views
//   c1: rows = d0, contraction along d1 (the stored orientation);  c0: rows = d1, contraction along d0
// with, for the wide modes, the top p.m bits of the stored 16-bit words (the mantissa plus half a narrow
// unit: rounded to nearest, clamped to the symmetric range) under the exponent s + 16 - p.m.
//
// Bound by HBM in the limit and by instructions and the latency of its phases before it. A CTA takes a strip of 2^lg_rv x cv tiles, up
// to 64 rows x 32 KC columns (128 x 128 for tiles above 64): with a CTA per tile, 576 weights of a 24 x 24 tile had 256 threads, five
// barriers and a start of their own. A warp owns whole rows of one tile row, its lanes consecutive columns, so that every load and
// store of an unaligned matrix is 32 neighbours; the values stay in registers between the maxima and the rounding. The narrow
// mantissas go to shared memory in padded coordinates (tile columns and rows tp apart, zeros between), from which view c1 leaves as
// words of whole rows and view c0 as byte-transposed blocks of 4 columns x 16 rows. Draws are made once per eight weights, into a
// table per warp. What a thread does once has to be little, it holds only 16 to 32 weights: the counts of tiles and the reciprocal of
// t come from the host (with 64-bit divisions, predicates on every access and a row of view c1 per warp the same strips took 116
// instructions per weight of a lane instead of 50). Updates, a CTA per tile before / this: 8192 x 8191, t = 64 355 / 169 us, with draws
// 504 / 240; 2000 x 3001, t = 24, with draws 96 / 28; 6000 x 6000, t = 24, 12 bits, with draws 279 / 159; 500 x 500, t = 32 8.3 / 6.6.
struct StripShape {
    int t, tp, lg_tp, cv, lg_rv, rpw;             // cv * t <= 32 KC, cv * tp <= 160, rpw: rows of a warp
    int recip, recip_per;                         // ceil(2^16 / t), ceil(2^20 / (cv * tp / 8)): exact for the indices of a strip
    int nu, nv;                                   // tiles along d0 and d1
};

// NW warps of up to RPW rows, KC columns per lane.
template <int MODE, int PLANES, int NW, int RPW, int KC, bool SR>
__global__ void __launch_bounds__(32 * NW, NW == 16 ? 1 : 4)
tile_strip_kernel(const float* __restrict__ src, int64_t ld, int64_t d0, int64_t d1, const StripShape sh, QParams p,
                  int16_t* __restrict__ wide, int8_t* __restrict__ grid, int64_t grid_ld, TileViews tv) {
    chain_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool UPDATE = MODE == 1 || MODE == 4;
    constexpr int GROUPS = 4 * KC + 1, NT = 32 * NW, LG_NW = NW == 16 ? 4 : 3;      // GROUPS: eights of draws that a row's columns touch
    const int t = sh.t, tp = sh.tp, cv = sh.cv, rv = 1 << sh.lg_rv, lw = LG_NW - sh.lg_rv;      // 2^lw warps per tile row
    const int qp = cv * tp + 8;                                            // halfword pitch of qt
    int16_t* qt = reinterpret_cast<int16_t*>(smem_raw);                    // [rv * tp][qp]
    uint4* rnd = reinterpret_cast<uint4*>(smem_raw + (size_t)rv * tp * qp * 2);               // [NW][RPW][GROUPS] (SR)
    __shared__ uint32_t pm[NW][32 * KC];
    __shared__ int s_exp[64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int u0 = (int)blockIdx.y << sh.lg_rv, v0 = (int)blockIdx.x * cv;
    const int64_t i00 = (int64_t)u0 * t, j0 = (int64_t)v0 * t;             // first row and column of the strip
    const int wj = (int)min((int64_t)(cv * t), d1 - j0), tiles = min(cv, sh.nv - v0);          // columns and tile columns of the strip
    // this warp's rows: nrow from row0 on, in tile row u0 + ur
    const int ur = warp >> lw, rb = (warp & ((1 << lw) - 1)) * sh.rpw;
    const int64_t row0 = i00 + ur * t + rb;
    const int nrow = u0 + ur < sh.nu ? max(0, (int)min((int64_t)min(sh.rpw, t - rb), d0 - row0)) : 0;
    int tile_of[KC], qcol[KC];
    bool in[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        const int c = lane + 32 * k;
        in[k] = c < wj;
        tile_of[k] = in[k] ? (c * sh.recip) >> 16 : 0;
        qcol[k] = in[k] ? tile_of[k] * (tp - t) + c : 0;
    }
    const int nsh = MODE == 3 ? 0 : 16 - p.m, half = nsh > 0 ? 1 << (nsh - 1) : 0;
    // the top bits of the stored word plus half a narrow unit, held inside the symmetric range
    auto narrow = [&](int q) { return MODE == 3 ? q : clampq((q + half) >> nsh, p.qmax); };
    const bool views = tv.mant_c0 != nullptr || tv.mant_c1 != nullptr;
    if (views && (t != tp || wj < cv * t || (int64_t)(u0 + rv) * t > d0))
        for (int e = tid; e < rv * tp * qp / 8; e += NT) reinterpret_cast<uint4*>(qt)[e] = make_uint4(0u, 0u, 0u, 0u);
    int16_t* const qrow = qt + (ur * tp + rb) * qp;
    const float* const srow = src + row0 * ld + j0 + lane;
    int16_t* const wrow = wide + row0 * d1 + j0 + lane;
    if (MODE == 2) {
        if (tid < rv * cv) {
            const int uu = u0 + tid / cv, vv = v0 + tid % cv;
            s_exp[tid] = uu < sh.nu && vv < sh.nv ? grid[uu * grid_ld + vv] : 0;
        }
        __syncthreads();                                                   // the zeros are written
        int w[RPW][KC];
#pragma unroll
        for (int r = 0; r < RPW; ++r)
#pragma unroll
            for (int k = 0; k < KC; ++k) w[r][k] = r < nrow && in[k] ? wrow[r * d1 + 32 * k] : 0;
#pragma unroll
        for (int r = 0; r < RPW; ++r)
            if (r < nrow)
#pragma unroll
                for (int k = 0; k < KC; ++k)
                    if (in[k]) qrow[r * qp + qcol[k]] = (int16_t)narrow(w[r][k]);
    } else {
        // FULL: no row or column of the strip is missing, and nothing asks
        auto convert = [&](auto is_full) {
            constexpr bool FULL = decltype(is_full)::value;
            float x[RPW][KC];
#pragma unroll
            for (int r = 0; r < RPW; ++r)
#pragma unroll
                for (int k = 0; k < KC; ++k) x[r][k] = FULL || (r < nrow && in[k]) ? __ldcs(srow + r * ld + 32 * k) : 0.f;
            uint4* const my_rnd = rnd + warp * (RPW * GROUPS);
            // while the loads are in flight; rows that all start with an eight of draws touch one less of them
            auto draw_eights = [&](auto count) {
                constexpr int N = decltype(count)::value;
                for (int i = lane; i < nrow * N; i += 32) {
                    const int r = i / N, g = i - r * N;
                    const uint64_t L0 = (uint64_t)((row0 + r) * d1 + j0);
                    if (8 * g < (int)(L0 & 7) + wj) my_rnd[r * GROUPS + g] = draws_of_group(p, (L0 >> 3) + g);
                }
            };
            auto draw = [&]() {
                if ((((uint32_t)d1 | (uint32_t)j0) & 7) == 0) draw_eights(std::integral_constant<int, GROUPS - 1>{});
                else draw_eights(std::integral_constant<int, GROUPS>{});
            };
            if (UPDATE) {
                // the wide words of (at most) eighteen weights at a time, requested together
                constexpr int RW = RPW * KC <= 18 ? RPW : RPW / 2;
#pragma unroll
                for (int r0 = 0; r0 < RPW; r0 += RW) {
                    int w[RW][KC];
#pragma unroll
                    for (int r = 0; r < RW; ++r)
#pragma unroll
                        for (int k = 0; k < KC; ++k) w[r][k] = FULL || (r0 + r < nrow && in[k]) ? wrow[(r0 + r) * d1 + 32 * k] : 0;
                    if (SR && r0 == 0) draw();
#pragma unroll
                    for (int k = 0; k < KC; ++k) {
                        const float old_scale = FULL || nrow > 0 ? pow2f(grid[(u0 + ur) * grid_ld + v0 + tile_of[k]]) : 0.f;
                        // the product is exact: one rounding
#pragma unroll
                        for (int r = 0; r < RW; ++r) x[r0 + r][k] = __fmaf_rn((float)w[r][k], old_scale, x[r0 + r][k]);
                    }
                }
            } else if (SR) {
                draw();
            }
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                uint32_t am = 0;
#pragma unroll
                for (int r = 0; r < RPW; r += 2) am = max3_abs_bits(am, x[r][k], x[r + 1][k]);
                pm[warp][lane + 32 * k] = am;
            }
            __syncthreads();
            // a warp per tile
            for (int i = warp; i < rv * cv; i += NW) {
                const int uu = i / cv, vv = i - uu * cv;
                uint32_t am = 0;
                for (int c = vv * t + lane; c < (vv + 1) * t; c += 32)
                    for (int w = 0; w < 1 << lw; ++w) am = max(am, pm[(uu << lw) + w][c]);
                am = __reduce_max_sync(0xffffffffu, am);
                if (lane == 0) {
                    const int s = block_exponent(am, MODE == 3 ? p.m : 16, p.exp_mode);
                    s_exp[i] = s;
                    if (grid && u0 + uu < sh.nu && vv < tiles) grid[(u0 + uu) * grid_ld + v0 + vv] = (int8_t)s;
                }
            }
            __syncthreads();
            const uint16_t* drow = reinterpret_cast<const uint16_t*>(my_rnd) + lane;
            const uint32_t first = SR ? (uint32_t)((uint64_t)(row0 * d1 + j0) & 7) : 0u, row_step = (uint32_t)(d1 & 7);
            float scale[KC];
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                const int s = s_exp[ur * cv + tile_of[k]];
                scale[k] = SR ? pow2f(16 - s) : pow2f(-s);
            }
#pragma unroll
            for (int r = 0; r < RPW; ++r)
                if (FULL || r < nrow) {
                    const uint16_t* dr = drow + r * (8 * GROUPS) + ((first + r * row_step) & 7);
#pragma unroll
                    for (int k = 0; k < KC; ++k) {
                        const float y = __fmul_rn(x[r][k], scale[k]);
                        int q;
                        if (!SR) {
                            q = clampq(__float2int_rn(y), MODE == 3 ? p.qmax : 32767);
                        } else if (MODE == 3) {
                            q = clampq((__float2int_rd(y) + (int)dr[32 * k]) >> 16, p.qmax);
                        } else {
                            q = floor_wide(y, dr[32 * k]);
                        }
                        if (FULL || in[k]) {
                            if (MODE != 3) wrow[r * d1 + 32 * k] = (int16_t)q;
                            if (MODE == 4) tv.value[(row0 + r) * tv.ldv + j0 + lane + 32 * k] = __fmul_rn((float)q, pow2f_stored(s_exp[ur * cv + tile_of[k]]));
                            qrow[r * qp + qcol[k]] = (int16_t)narrow(q);
                        }
                    }
                }
        };
        if (wj == 32 * KC && sh.rpw == RPW && t == RPW << lw && u0 + rv <= sh.nu && i00 + rv * t <= d0) convert(std::true_type{});
        else convert(std::false_type{});
    }
    if (!views) return;
    __syncthreads();
    // bytes of a view from pairs of narrow mantissas: plane 0 the upper (or only) eight bits, plane 1 the four below
    auto upper = [](uint2 q) {
        return PLANES == 2 ? __byte_perm((q.x >> 4) & 0x00ff00ffu, (q.y >> 4) & 0x00ff00ffu, 0x6420) : __byte_perm(q.x, q.y, 0x6420);
    };
    auto lower = [](uint2 q) { return __byte_perm(q.x & 0x000f000fu, q.y & 0x000f000fu, 0x6420); };
    // view c1: row i gets bytes [v0 tp, (v0 + tiles) tp) in pieces of eight, and zeros beyond the last tile
    if (tv.mant_c1) {
        int8_t* const base = tv.mant_c1 + i00 * tv.kst1 + (int64_t)v0 * tp;
        const int per = cv * tp / 8;
        for (int e = tid; e < rv * tp * per; e += NT) {
            const int r = (int)((uint32_t)(e * sh.recip_per) >> 20), w = 8 * (e - r * per), uu = r >> sh.lg_tp, ii = r & (tp - 1), i = uu * t + ii;
            if (ii >= t || i00 + i >= d0 || w >= tiles * tp) continue;
            const uint4 q = *reinterpret_cast<const uint4*>(qt + r * qp + w);
            int8_t* dst = base + i * tv.kst1 + w;
            *reinterpret_cast<uint2*>(dst) = make_uint2(upper(make_uint2(q.x, q.y)), upper(make_uint2(q.z, q.w)));
            if (PLANES == 2) *reinterpret_cast<uint2*>(dst + tv.ps1) = make_uint2(lower(make_uint2(q.x, q.y)), lower(make_uint2(q.z, q.w)));
        }
        if (v0 + tiles == sh.nv && (int64_t)sh.nv * tp < tv.kst1)
            for (int i = warp; i < rv * t && i00 + i < d0; i += NW)
                for (int64_t o = (int64_t)sh.nv * tp + 4 * lane; o < tv.kst1; o += 128) {
                    *reinterpret_cast<uint32_t*>(tv.mant_c1 + (i00 + i) * tv.kst1 + o) = 0u;
                    if (PLANES == 2) *reinterpret_cast<uint32_t*>(tv.mant_c1 + tv.ps1 + (i00 + i) * tv.kst1 + o) = 0u;
                }
    }
    // view c0: row j gets bytes [u0 tp, ...): blocks of 4 columns x 16 rows of qt, byte-transposed
    if (tv.mant_c0) {
        const int ncol4 = tiles * tp / 4;
        for (int e = tid; e < ncol4 * (rv * tp / 16); e += NT) {
            const int g = (int)((uint32_t)e / (uint32_t)ncol4), c = 4 * (e - g * ncol4), vv = c >> sh.lg_tp, jin = c & (tp - 1);
            if (u0 + ((16 * g) >> sh.lg_tp) >= sh.nu) continue;
            const int64_t j = j0 + vv * t + jin;
            const int cols = (int)min((int64_t)(t - jin), d1 - j);         // of the four that exist
            if (cols <= 0) continue;
            uint32_t out[PLANES][4][4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                uint2 q[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const uint2*>(qt + (16 * g + 4 * b + i) * qp + c);
#pragma unroll
                for (int pl = 0; pl < PLANES; ++pl) {
                    const uint32_t R0 = pl ? lower(q[0]) : upper(q[0]), R1 = pl ? lower(q[1]) : upper(q[1]);
                    const uint32_t R2 = pl ? lower(q[2]) : upper(q[2]), R3 = pl ? lower(q[3]) : upper(q[3]);
                    const uint32_t t0 = __byte_perm(R0, R1, 0x5140), t1 = __byte_perm(R2, R3, 0x5140);
                    const uint32_t t2 = __byte_perm(R0, R1, 0x7362), t3 = __byte_perm(R2, R3, 0x7362);
                    out[pl][0][b] = __byte_perm(t0, t1, 0x5410);
                    out[pl][1][b] = __byte_perm(t0, t1, 0x7632);
                    out[pl][2][b] = __byte_perm(t2, t3, 0x5410);
                    out[pl][3][b] = __byte_perm(t2, t3, 0x7632);
                }
            }
            int8_t* dst = tv.mant_c0 + j * tv.kst0 + (int64_t)u0 * tp + 16 * g;
#pragma unroll
            for (int pl = 0; pl < PLANES; ++pl)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < cols)
                        *reinterpret_cast<uint4*>(dst + pl * tv.ps0 + i * tv.kst0) = make_uint4(out[pl][i][0], out[pl][i][1], out[pl][i][2], out[pl][i][3]);
        }
        if (u0 + rv >= sh.nu && (int64_t)sh.nu * tp < tv.kst0)             // the row tails
            for (int c = warp; c < wj; c += NW)
                for (int64_t o = (int64_t)sh.nu * tp + 4 * lane; o < tv.kst0; o += 128) {
                    *reinterpret_cast<uint32_t*>(tv.mant_c0 + (j0 + c) * tv.kst0 + o) = 0u;
                    if (PLANES == 2) *reinterpret_cast<uint32_t*>(tv.mant_c0 + tv.ps0 + (j0 + c) * tv.kst0 + o) = 0u;
                }
    }
    // replicated exponents: exps_c1[v][i], exps_c0[u][j] (lines beyond the matrix, at most 15 after the last tile, are documented as zero)
    for (int i = warp; i < rv * cv; i += NW) {
        const int uu = i / cv, vv = i - uu * cv;
        if (u0 + uu >= sh.nu || vv >= tiles) continue;
        const int8_t se = (int8_t)(s_exp[i] + nsh);
        const int64_t ia = i00 + uu * t, ja = j0 + vv * t;
        if (tv.exps_c1) {
            const int64_t end = u0 + uu == sh.nu - 1 ? tv.rs1 : ia + t;
            for (int64_t r = ia + lane; r < end; r += 32) tv.exps_c1[(v0 + vv) * tv.rs1 + r] = r < d0 ? se : (int8_t)0;
        }
        if (tv.exps_c0) {
            const int64_t end = v0 + vv == sh.nv - 1 ? tv.rs0 : ja + t;
            for (int64_t c = ja + lane; c < end; c += 32) tv.exps_c0[(u0 + uu) * tv.rs0 + c] = c < d1 ? se : (int8_t)0;
        }
    }
}

// Tiles of 32, 64 or 128 (the tile is its own padded width), aligned rows of whole eights: the same arithmetic as
// tile_strip_kernel with fewer instructions per weight. A thread keeps its groups of eight weights in registers
// between the maximum and the rounding pass (no FP32 tile in shared memory); the rounded words go to a 16-bit
// tile in shared memory once, from which view c1 leaves as 8-byte pieces cut by byte permutes and view c0 as
// the byte-transposes of 4 x 4 blocks (eight permutes per block) instead of one shared-memory load, shift and
// mask per byte. ROWS4 = 4 x 4 blocks stacked per thread for view c0 (wider stores per output row).
// GENERAL: the last tile of a row or column of tiles is smaller (its missing groups are zeros), or the width is one that is cut early;
// a parameter, so that whole tiles ask nothing (8192 x 8192, t = 64: 113 us, 115 with the question). Updates, the kernel for any tile
// before / this: 1111 x 5000, t = 64, draws 20.6 / 14.2 us, 3000 x 3000, t = 128 28.8 / 23.8, 4096 x 4096, t = 64, 4 bits 51.3 / 34.2.
template <int MODE, int PLANES, int TP, bool GENERAL>
__global__ void __launch_bounds__(256)
tile_kernel_full(const float* __restrict__ src, int64_t ld, int64_t d0, int64_t d1, QParams p,
                 int16_t* __restrict__ wide, int8_t* __restrict__ grid, int64_t grid_ld, TileViews tv) {
    chain_start();
    constexpr int G = TP / 8;                          // groups of eight per tile row
    constexpr int NITEMS = TP * G;                     // groups per tile
    constexpr int ITEMS = (NITEMS + 255) / 256;        // per thread
    constexpr int QP = TP + 8;                         // halfword pitch of qt: rows stay 16-byte aligned
    __shared__ __align__(16) int16_t qt[TP * QP];
    __shared__ uint32_t s_am[8];
    __shared__ int s_exp;
    const int tid = threadIdx.x, lane = tid & 31, wrow = tid >> 5;
    const int64_t u = blockIdx.y, v = blockIdx.x;
    const int64_t i0 = u * TP, j0 = v * TP;
    const int hi = GENERAL ? (int)min((int64_t)TP, d0 - i0) : TP, wj = GENERAL ? (int)min((int64_t)TP, d1 - j0) : TP;
    auto there = [&](int ii, int gj) { return !GENERAL || (ii < hi && 8 * gj < wj); };
    constexpr bool UPDATE = MODE == 1 || MODE == 4;
    const int wbits = MODE == 3 ? p.m : 16, wqmax = MODE == 3 ? p.qmax : 32767;
    const int sh = MODE == 3 ? 0 : 16 - p.m;
    const int half = sh > 0 ? 1 << (sh - 1) : 0;
    const int w_hi = ((p.qmax + 1) << sh) - half - 1, w_lo = -(p.qmax << sh) - half;
    const uint32_t w_hi2 = ((uint32_t)w_hi & 0xFFFFu) * 0x10001u, w_lo2 = ((uint32_t)w_lo & 0xFFFFu) * 0x10001u;
    const uint32_t half2 = (uint32_t)half * 0x10001u;
    // A 32-bit shift may drag the upper halfword's bits into the lower one's byte: widths too narrow for that are shifted here.
    const bool early = GENERAL && MODE != 3 && sh + (PLANES == 2 ? 4 : 0) > 8;
    auto stored_pair = [&](uint32_t h) {
        if (MODE == 3) return h;
        const uint32_t w = __vadd2(__vmaxs2(__vmins2(h, w_hi2), w_lo2), half2);
        return early ? __byte_perm((uint32_t)((int)(int16_t)w >> sh), (uint32_t)((int)w >> (16 + sh)), 0x5410) : w;
    };
    int s;
    if (MODE == 2) {
        s = grid[u * grid_ld + v];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int item = tid + 256 * k;
            if (NITEMS % 256 == 0 || item < NITEMS) {
                const int ii = item / G, gj = item - ii * G;
                const uint4 q8 = there(ii, gj) ? *reinterpret_cast<const uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj) : make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4*>(qt + ii * QP + 8 * gj) = make_uint4(stored_pair(q8.x), stored_pair(q8.y), stored_pair(q8.z), stored_pair(q8.w));
            }
        }
    } else {
        const float old_scale = UPDATE ? pow2f(grid[u * grid_ld + v]) : 0.f;
        // the FP32 groups of the tile are requested before anything waits for them; for an update the wide
        // words follow, combined as fl32(wide * 2^s + delta) with one rounding
        float4 a[ITEMS], b[ITEMS];
        uint32_t am = 0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int item = tid + 256 * k;
            a[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            b[k] = a[k];
            if (NITEMS % 256 == 0 || item < NITEMS) {
                const int ii = item / G, gj = item - ii * G;
                const float4* sp = reinterpret_cast<const float4*>(src + (i0 + ii) * ld + j0 + 8 * gj);
                if (there(ii, gj)) {
                    a[k] = __ldcs(sp);
                    b[k] = __ldcs(sp + 1);
                }
            }
        }
        if (UPDATE) {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const int item = tid + 256 * k;
                if (NITEMS % 256 == 0 || item < NITEMS) {
                    const int ii = item / G, gj = item - ii * G;
                    const uint4 q8 = there(ii, gj) ? *reinterpret_cast<const uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj) : make_uint4(0u, 0u, 0u, 0u);
                    a[k].x = __fadd_rn(__fmul_rn((float)(int16_t)(q8.x & 0xFFFFu), old_scale), a[k].x);
                    a[k].y = __fadd_rn(__fmul_rn((float)(int16_t)(q8.x >> 16), old_scale), a[k].y);
                    a[k].z = __fadd_rn(__fmul_rn((float)(int16_t)(q8.y & 0xFFFFu), old_scale), a[k].z);
                    a[k].w = __fadd_rn(__fmul_rn((float)(int16_t)(q8.y >> 16), old_scale), a[k].w);
                    b[k].x = __fadd_rn(__fmul_rn((float)(int16_t)(q8.z & 0xFFFFu), old_scale), b[k].x);
                    b[k].y = __fadd_rn(__fmul_rn((float)(int16_t)(q8.z >> 16), old_scale), b[k].y);
                    b[k].z = __fadd_rn(__fmul_rn((float)(int16_t)(q8.w & 0xFFFFu), old_scale), b[k].z);
                    b[k].w = __fadd_rn(__fmul_rn((float)(int16_t)(q8.w >> 16), old_scale), b[k].w);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const float e8[8] = {a[k].x, a[k].y, a[k].z, a[k].w, b[k].x, b[k].y, b[k].z, b[k].w};
            am = max(am, amax8_bits(e8));
        }
        for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
        if (lane == 0) s_am[wrow] = am;
        __syncthreads();
        if (tid == 0) {
            uint32_t m8 = 0;
            for (int i = 0; i < 8; ++i) m8 = max(m8, s_am[i]);
            s_exp = block_exponent(m8, wbits, p.exp_mode);
            if (grid) grid[u * grid_ld + v] = (int8_t)s_exp;
        }
        __syncthreads();
        s = s_exp;
        const uint32_t qm = qmax_pair(wqmax), nqm = neg_qmax_pair(wqmax);
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int item = tid + 256 * k;
            if (NITEMS % 256 == 0 || item < NITEMS) {
                const int ii = item / G, gj = item - ii * G;
                uint32_t h[4] = {0u, 0u, 0u, 0u};
                if (there(ii, gj)) {                                   // (a missing group of eight is zero whatever its draws)
                    const float e8[8] = {a[k].x, a[k].y, a[k].z, a[k].w, b[k].x, b[k].y, b[k].z, b[k].w};
                    uint4 w = make_uint4(0u, 0u, 0u, 0u);
                    if (p.rounding == 1) w = draws_of_group(p, (uint64_t)((i0 + ii) * d1 + j0 + 8 * gj) >> 3);
                    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
                    if (MODE == 3) {
                        const float sc = pow2f(p.rounding == 1 ? 16 - s : -s);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            h[j] = p.rounding == 1 ? round_sr_pair(e8[2 * j], e8[2 * j + 1], sc, ww[j], qm, nqm)
                                                   : round_rne_pair(e8[2 * j], e8[2 * j + 1], sc, qm, nqm);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            int q0, q1;
                            if (p.rounding == 0) {
                                q0 = round_rne(e8[2 * j], s, 32767);
                                q1 = round_rne(e8[2 * j + 1], s, 32767);
                            } else {
                                q0 = round_sr_wide(e8[2 * j], s, ww[j] & 0xFFFFu);
                                q1 = round_sr_wide(e8[2 * j + 1], s, ww[j] >> 16);
                            }
                            h[j] = ((uint32_t)q0 & 0xFFFFu) | ((uint32_t)q1 << 16);
                        }
                    }
                }
                *reinterpret_cast<uint4*>(qt + ii * QP + 8 * gj) = make_uint4(stored_pair(h[0]), stored_pair(h[1]), stored_pair(h[2]), stored_pair(h[3]));
                if (MODE != 3 && there(ii, gj)) *reinterpret_cast<uint4*>(wide + (i0 + ii) * d1 + j0 + 8 * gj) = make_uint4(h[0], h[1], h[2], h[3]);
                if (MODE == 4 && there(ii, gj)) store_wide_values(tv.value + (i0 + ii) * tv.ldv + j0 + 8 * gj, h, pow2f_stored(s));
            }
        }
    }
    if (tv.mant_c0 == nullptr && tv.mant_c1 == nullptr) return;
    __syncthreads();
    // Bytes of the views from pairs of stored halfwords: plane 0 takes bits [sh + 4 (PLANES - 1), + 8) of each
    // halfword, plane 1 the four bits below; the masks remove what a 32-bit shift drags across the halfwords.
    const int sh_lo = early ? 0 : sh, sh_hi = sh_lo + (PLANES == 2 ? 4 : 0);
    auto bytes4 = [&](uint32_t w0, uint32_t w1, int k, uint32_t mask) {
        return __byte_perm((w0 >> k) & mask, (w1 >> k) & mask, 0x6420);
    };
    const int s_view = s + sh;
    // view c1: row i0 + ii, bytes [v TP + 8 gj, + 8)
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int item = tid + 256 * k;
        if (NITEMS % 256 == 0 || item < NITEMS) {
            const int ii = item / G, gj = item - ii * G;
            if (GENERAL && ii >= hi) continue;
            const uint4 q8 = *reinterpret_cast<const uint4*>(qt + ii * QP + 8 * gj);
            int8_t* dst = tv.mant_c1 + (i0 + ii) * tv.kst1 + v * TP + 8 * gj;
            *reinterpret_cast<uint2*>(dst) = make_uint2(bytes4(q8.x, q8.y, sh_hi, 0x00ff00ffu), bytes4(q8.z, q8.w, sh_hi, 0x00ff00ffu));
            if (PLANES == 2)
                *reinterpret_cast<uint2*>(dst + tv.ps1) = make_uint2(bytes4(q8.x, q8.y, sh_lo, 0x000f000fu), bytes4(q8.z, q8.w, sh_lo, 0x000f000fu));
        }
    }
    // view c0: row j0 + jj, bytes [u TP + g, ...): blocks of 4 columns x (4 ROWS4) rows of qt, byte-transposed
    constexpr int ROWS4 = TP >= 64 ? 4 : 1;                            // 16- or 4-byte stores
    constexpr int NBLK = (TP / 4) * (TP / (4 * ROWS4));
#pragma unroll
    for (int k = 0; k < (NBLK + 255) / 256; ++k) {
        const int e = tid + 256 * k;
        if (NBLK % 256 == 0 || e < NBLK) {
            const int jj = (e % (TP / 4)) * 4, g = (e / (TP / 4)) * 4 * ROWS4;
            if (GENERAL && jj >= wj) continue;
            uint32_t out[PLANES][4][ROWS4];
#pragma unroll
            for (int rb = 0; rb < ROWS4; ++rb) {
                uint2 r[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) r[i] = *reinterpret_cast<const uint2*>(qt + (g + 4 * rb + i) * QP + jj);
#pragma unroll
                for (int pl = 0; pl < PLANES; ++pl) {
                    const int kk = pl == 0 ? sh_hi : sh_lo;
                    const uint32_t mask = pl == 0 ? 0x00ff00ffu : 0x000f000fu;
                    const uint32_t R0 = bytes4(r[0].x, r[0].y, kk, mask), R1 = bytes4(r[1].x, r[1].y, kk, mask);
                    const uint32_t R2 = bytes4(r[2].x, r[2].y, kk, mask), R3 = bytes4(r[3].x, r[3].y, kk, mask);
                    const uint32_t t0 = __byte_perm(R0, R1, 0x5140), t1 = __byte_perm(R2, R3, 0x5140);
                    const uint32_t t2 = __byte_perm(R0, R1, 0x7362), t3 = __byte_perm(R2, R3, 0x7362);
                    out[pl][0][rb] = __byte_perm(t0, t1, 0x5410);
                    out[pl][1][rb] = __byte_perm(t0, t1, 0x7632);
                    out[pl][2][rb] = __byte_perm(t2, t3, 0x5410);
                    out[pl][3][rb] = __byte_perm(t2, t3, 0x7632);
                }
            }
#pragma unroll
            for (int pl = 0; pl < PLANES; ++pl)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int8_t* dst = tv.mant_c0 + pl * tv.ps0 + (j0 + jj + c) * tv.kst0 + u * TP + g;
                    if (ROWS4 == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(out[pl][c][0], out[pl][c][1], out[pl][c][2 % ROWS4], out[pl][c][3 % ROWS4]);
                    else if (ROWS4 == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(out[pl][c][0], out[pl][c][1 % ROWS4]);
                    else *reinterpret_cast<uint32_t*>(dst) = out[pl][c][0];
                }
        }
    }
    // replicated exponents, and the row tails beyond the last tile
    if (tid < TP) {                                                    // lines beyond the matrix are documented as zero
        if (!GENERAL || i0 + tid < tv.rs1) tv.exps_c1[v * tv.rs1 + i0 + tid] = tid < hi ? (int8_t)s_view : (int8_t)0;
        if (!GENERAL || j0 + tid < tv.rs0) tv.exps_c0[u * tv.rs0 + j0 + tid] = tid < wj ? (int8_t)s_view : (int8_t)0;
    }
    if (v == tv.nkb1 - 1)
        for (int64_t e = tid; e < (int64_t)hi * ((tv.kst1 - tv.nkb1 * TP) / 4); e += 256) {
            const int64_t per = (tv.kst1 - tv.nkb1 * TP) / 4, ii = e / per, o = tv.nkb1 * TP + (e % per) * 4;
            *reinterpret_cast<uint32_t*>(tv.mant_c1 + (i0 + ii) * tv.kst1 + o) = 0;
            if (PLANES == 2) *reinterpret_cast<uint32_t*>(tv.mant_c1 + tv.ps1 + (i0 + ii) * tv.kst1 + o) = 0;
        }
    if (u == tv.nkb0 - 1)
        for (int64_t e = tid; e < (int64_t)wj * ((tv.kst0 - tv.nkb0 * TP) / 4); e += 256) {
            const int64_t per = (tv.kst0 - tv.nkb0 * TP) / 4, jj = e / per, o = tv.nkb0 * TP + (e % per) * 4;
            *reinterpret_cast<uint32_t*>(tv.mant_c0 + (j0 + jj) * tv.kst0 + o) = 0;
            if (PLANES == 2) *reinterpret_cast<uint32_t*>(tv.mant_c0 + tv.ps0 + (j0 + jj) * tv.kst0 + o) = 0;
        }
}

// ------------------------------------------------------------------------------ generic two-pass path

// Element (r, kk) of the operand view: r = line, kk = position along the contraction axis.
__device__ __forceinline__ float view_at(const float* x, int64_t ld, int axis, int64_t r, int64_t kk) {
    return axis == 1 ? x[r * ld + kk] : x[kk * ld + r];
}

// Pass 1a, blocks along rows: one warp per (line, block).
__global__ void exps_axis1(const float* __restrict__ x, int64_t rows, int64_t K, int64_t ld, int64_t b,
                           int64_t nkb, QParams p, int8_t* __restrict__ exps, int64_t rs) {
    chain_start();
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t item = warp; item < rows * nkb; item += nwarps) {
        const int64_t r = item / nkb, kb = item % nkb;
        const int64_t k1 = min(K, (kb + 1) * b);
        uint32_t am = 0;
        for (int64_t kk = kb * b + lane; kk < k1; kk += 32) am = max(am, abs_bits(x[r * ld + kk]));
        for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
        if (lane == 0) exps[kb * rs + r] = (int8_t)block_exponent(am, p.m, p.exp_mode);
    }
}

// One exponent per whole row (block = 0, "BFP without tiles", Sec. 6) for rows of 2048 G elements: a CTA per row
// keeps the row in registers (eight elements per thread and step, G steps) between the maximum and the rounding,
// so the tensor is read once.
template <int G, bool SR, int PLANES>
__global__ void __launch_bounds__(256)
quant_row_whole(const float* __restrict__ x, int64_t ld, int64_t d1, QParams p, int8_t* __restrict__ mant, int64_t kst,
                int64_t plane_stride, int8_t* __restrict__ exps) {
    chain_start();
    __shared__ uint32_t part[8];
    const int tid = threadIdx.x;
    const int64_t r = blockIdx.x;
    const float4* src = reinterpret_cast<const float4*>(x + r * ld);
    float e[G][8];
    uint32_t am = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int g = tid + 256 * i;
        const float4 a = __ldg(src + 2 * g), b = __ldg(src + 2 * g + 1);
        e[i][0] = a.x; e[i][1] = a.y; e[i][2] = a.z; e[i][3] = a.w;
        e[i][4] = b.x; e[i][5] = b.y; e[i][6] = b.z; e[i][7] = b.w;
    }
#pragma unroll
    for (int i = 0; i < G; ++i) am = max(am, amax8_bits(e[i]));
    for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
    if ((tid & 31) == 0) part[tid >> 5] = am;
    __syncthreads();
    am = part[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) am = max(am, part[i]);
    const int s = block_exponent(am, p.m, p.exp_mode);
    if (tid == 0) exps[r] = (int8_t)s;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int g = tid + 256 * i;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (SR) w = draws_of_group(p, (uint64_t)(r * d1 + 8 * (int64_t)g) >> 3);
        uint2 hi, lo;
        quantize_pack8<SR, PLANES>(e[i], s, p, w, hi, lo);
        *reinterpret_cast<uint2*>(mant + r * kst + 8 * g) = hi;
        if (PLANES == 2) *reinterpret_cast<uint2*>(mant + plane_stride + r * kst + 8 * g) = lo;
    }
}

// Pass 1b, blocks down columns: one thread per (block, line); neighbouring threads read
// neighbouring addresses.
__global__ void exps_axis0(const float* __restrict__ x, int64_t rows, int64_t K, int64_t ld, int64_t b,
                           int64_t nkb, QParams p, int8_t* __restrict__ exps, int64_t rs) {
    chain_start();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * nkb) return;
    const int64_t kb = i / rows, r = i % rows;
    const int64_t k1 = min(K, (kb + 1) * b);
    uint32_t am = 0;
    for (int64_t kk = kb * b; kk < k1; ++kk) am = max(am, abs_bits(x[kk * ld + r]));
    exps[kb * rs + r] = (int8_t)block_exponent(am, p.m, p.exp_mode);
}

// Pass 1c, t x t tiles of the stored matrix [d0][d1]: one warp per tile computes the tile's
// exponent and repeats it for every line of the view that crosses the tile.
__global__ void exps_tiles(const float* __restrict__ x, int64_t d0, int64_t d1, int64_t ld, int64_t t,
                           QParams p, int axis, int8_t* __restrict__ exps, int64_t rs, int64_t nu, int64_t nv) {
    chain_start();
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp >= nu * nv) return;
    const int64_t u = warp / nv, v = warp % nv;
    const int64_t i1 = min(d0, (u + 1) * t), j1 = min(d1, (v + 1) * t);
    uint32_t am = 0;
    for (int64_t i = u * t; i < i1; ++i)
        for (int64_t j = v * t + lane; j < j1; j += 32) am = max(am, abs_bits(x[i * ld + j]));
    for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
    const int8_t s = (int8_t)block_exponent(am, p.m, p.exp_mode);
    // axis 1: lines are stored rows, block index is the tile column. axis 0: the transpose.
    if (axis == 1) for (int64_t i = u * t + lane; i < i1; i += 32) exps[v * rs + i] = s;
    else for (int64_t j = v * t + lane; j < j1; j += 32) exps[u * rs + j] = s;
}

// Pass 1d, convolution weights [taps * c_in][c_out] (Sec. 5.1: the two feature-map dimensions are tiled, the
// filter taps are not): one CTA per (input-map tile u, output-map tile v) takes the maximum over every tap
// (a warp per weight row, lanes along the output maps) and repeats the tile's exponent for every line and
// K-block of the two views that cross the tile.
constexpr int CONVW_THREADS = 512;
__global__ void __launch_bounds__(CONVW_THREADS)
exps_conv_tiles(const float* __restrict__ x, int64_t taps, int64_t c_in, int64_t c_out, int64_t ld, int64_t t, QParams p,
                int8_t* __restrict__ exps0, int64_t rs0, int8_t* __restrict__ exps1, int64_t rs1, int64_t nu, int64_t nv,
                int8_t* __restrict__ tile_exps, uint32_t* __restrict__ amax, bool fill) {
    chain_start();
    __shared__ uint32_t part[CONVW_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t u = blockIdx.x / nv, v = blockIdx.x % nv;
    const int64_t j1 = min(c_out, (v + 1) * t);
    uint32_t am = 0;
    // with `amax` the rows are split over gridDim.y CTAs that merge their maxima there (exponents come from a
    // second launch with `fill`); without it this CTA scans the whole tile
    for (int64_t r = (int64_t)blockIdx.y * (CONVW_THREADS / 32) + warp; !fill && r < taps * t; r += (int64_t)gridDim.y * (CONVW_THREADS / 32)) {
        const int64_t tap = r / t, ci = u * t + r % t;
        for (int64_t j = v * t + lane; j < j1; j += 32) am = max(am, abs_bits(x[(tap * c_in + ci) * ld + j]));
    }
    for (int off = 16; off > 0; off >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
    if (lane == 0) part[warp] = am;
    __syncthreads();
    am = part[0];
    for (int i = 1; i < CONVW_THREADS / 32; ++i) am = max(am, part[i]);
    if (amax && !fill) {
        if (threadIdx.x == 0) atomicMax(amax + blockIdx.x, am);
        return;
    }
    if (fill) am = amax[blockIdx.x];
    const int8_t s = (int8_t)block_exponent(am, p.m, p.exp_mode);
    if (tile_exps && threadIdx.x == 0) tile_exps[u * nv + v] = s;
    // view c0 (forward): lines are output maps, K-block (tap, u). view c1: lines are (tap, ci), K-block v.
    if (exps0)
        for (int64_t i = threadIdx.x; i < taps * (j1 - v * t); i += CONVW_THREADS) {
            const int64_t tap = i / (j1 - v * t), j = v * t + i % (j1 - v * t);
            exps0[(tap * nu + u) * rs0 + j] = s;
        }
    if (exps1)
        for (int64_t i = threadIdx.x; i < taps * t; i += CONVW_THREADS) {
            const int64_t tap = i / t, ci = u * t + i % t;
            exps1[v * rs1 + tap * c_in + ci] = s;
        }
}

// Pass 2: one thread per 4 output bytes of a line; reads the exponent written by pass 1.
template <int PLANES>
__global__ void mant_generic(const float* __restrict__ x, int64_t d1, int64_t rows, int64_t K, int64_t ld,
                             int axis, int64_t b, int64_t bp, int64_t nkb, QParams p,
                             const int8_t* __restrict__ exps, int64_t rs, int8_t* __restrict__ mant,
                             int64_t kst, int64_t plane_stride) {
    chain_start();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per = kst / 4;
    if (i >= rows * per) return;
    const int64_t r = i / per, o = (i % per) * 4;
    uint32_t h = 0, l = 0;
    const int64_t kb = o / bp;
    if (kb < nkb) {
        const int s = exps[kb * rs + r];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t within = o % bp + j, kk = kb * b + within;
            int q = 0;
            if (within < b && kk < K) {
                const uint64_t L = axis == 1 ? (uint64_t)(r * d1 + kk) : (uint64_t)(kk * d1 + r);
                q = quantize_one(view_at(x, ld, axis, r, kk), s, p, L);
            }
            if (PLANES == 1) h |= (uint32_t)(q & 0xff) << (8 * j);
            else { h |= (uint32_t)((q >> 4) & 0xff) << (8 * j); l |= (uint32_t)(q & 15) << (8 * j); }
        }
    }
    *reinterpret_cast<uint32_t*>(mant + r * kst + o) = h;
    if (PLANES == 2) *reinterpret_cast<uint32_t*>(mant + plane_stride + r * kst + o) = l;
}

// ------------------------------------------------------------------------------ packed im2col gather

// Convolution operand without the FP32 im2col matrix: with a block of c channels along the contraction
// (taps ordered (i, j, channel)) every block of an im2col row is the quantised channel vector of one input
// pixel, so the packed operand [n ho wo][kh kw c] is a gather of the packed per-pixel operand [n h w][c]:
// bp bytes of mantissas and one exponent per tap, zeros (exponent -63, as an all-zero block has) outside the
// image. One warp per output row, 16 bytes per lane and step (row tails beyond the last tap are zeroed too).
constexpr int IM2COL_MAX_TAPS = 64, IM2COL_ROWS = 64;

__global__ void __launch_bounds__(256)
im2col_gather(const int8_t* __restrict__ xm, const int8_t* __restrict__ xe, int kst_x, int64_t ps_x,
              int h, int w, int ho, int wo, int kh, int kw, int pad, int lg_bp, int planes,
              uint32_t rows_out, int kst_out, int64_t ps_out, int64_t rs_out,
              int8_t* __restrict__ om, int8_t* __restrict__ oe) {
    chain_start();
    // A CTA takes 64 consecutive output rows, a warp eight of them; the lanes sweep a row 16 bytes at a
    // time. The filter offsets of the taps are tabulated once per CTA, the pixel coordinates once per row
    // (32-bit arithmetic: the host checks the sizes), and the exponents of the 64 rows are collected in
    // shared memory so that each tap's bytes leave as whole sectors.
    __shared__ int8_t s_e[IM2COL_MAX_TAPS][IM2COL_ROWS];
    __shared__ int8_t s_dy[IM2COL_MAX_TAPS], s_dx[IM2COL_MAX_TAPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t r0 = blockIdx.x * IM2COL_ROWS;
    const int taps = kh * kw, chunks = kst_out >> 4;
    if ((int)threadIdx.x < taps) {
        s_dy[threadIdx.x] = (int8_t)((int)threadIdx.x / kw - pad);
        s_dx[threadIdx.x] = (int8_t)((int)threadIdx.x % kw - pad);
    }
    __syncthreads();
    const uint32_t per_img = (uint32_t)(ho * wo);
    // four rows at a time, so that four independent loads are in flight per lane (eight were slower)
    for (int k = 0; k < IM2COL_ROWS / 8; k += 4) {
        int oy[4], ox[4];
        int64_t img_base[4];
        bool live[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t r = r0 + warp * (IM2COL_ROWS / 8) + k + q;
            live[q] = r < rows_out;
            const uint32_t rr = live[q] ? r : 0u;
            const uint32_t img = rr / per_img, rem = rr - img * per_img;
            oy[q] = (int)(rem / (uint32_t)wo);
            ox[q] = (int)(rem - (uint32_t)oy[q] * (uint32_t)wo);
            img_base[q] = (int64_t)img * h * w;
        }
        for (int ck = lane; ck < chunks; ck += 32) {
            const int o = ck << 4;                              // byte offset in the output row
            const int tap = o >> lg_bp, within = o - (tap << lg_bp);
            const int dy = tap < taps ? s_dy[tap] : 0, dx = tap < taps ? s_dx[tap] : 0;
            for (int pl = 0; pl < planes; ++pl) {
                int64_t src[4];
                uint4 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int iy = oy[q] + dy, ix = ox[q] + dx;
                    src[q] = (tap < taps && iy >= 0 && iy < h && ix >= 0 && ix < w) ? img_base[q] + iy * w + ix : -1;
                    v[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (src[q] >= 0) v[q] = *reinterpret_cast<const uint4*>(xm + pl * ps_x + src[q] * kst_x + within);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int lr = warp * (IM2COL_ROWS / 8) + k + q;
                    if (live[q]) {
                        *reinterpret_cast<uint4*>(om + pl * ps_out + (int64_t)(r0 + lr) * kst_out + o) = v[q];
                        if (pl == 0 && within == 0 && tap < taps) s_e[tap][lr] = src[q] >= 0 ? xe[src[q]] : (int8_t)-63;
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < taps * IM2COL_ROWS; idx += 256) {
        const int tap = idx / IM2COL_ROWS, j = idx % IM2COL_ROWS;
        if (r0 + j < rows_out) oe[(int64_t)tap * rs_out + r0 + j] = s_e[tap][j];
    }
}

// Backward-weight operand of a convolution without the FP32 im2col matrix: dW = cols^T dY contracts over the
// output pixels, so cols^T [kh kw c][n h w] is quantised with blocks of b consecutive pixels along each
// (tap, channel) row. A block is a window of the image shifted by the tap, so nothing can be shared between
// taps except the loads: a CTA takes one block of b pixels (whole image rows: b % w == 0, h w % b == 0,
// output as large as the input) and stages the b / w + kh - 1 image rows it touches in shared memory once
// (zeros outside the image). Then, tap by tap and 64 channels at a time, thread (channel, quarter) keeps its
// quarter of the block's pixels in registers between the maximum (exchanged through shared memory) and the
// rounding, and writes its b / 4 mantissa bytes with 16-byte stores.
template <int PLANES, int NPX, bool SR>      // NPX = b / 4 pixels per thread: 4, 8, 16 or 32
__global__ void __launch_bounds__(256)
im2col_cols(const float* __restrict__ x, int h, int w, int lg_w, int c, int kh, int kw, int pad, QParams p,
            int64_t kst, int64_t plane_stride, int64_t rs, int8_t* __restrict__ mant, int8_t* __restrict__ exps) {
    chain_start();
    constexpr int B = 4 * NPX;
    constexpr int BP = B <= 32 ? 32 : B <= 64 ? 64 : 128;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* img_rows = reinterpret_cast<float*>(smem_raw);        // [B / w + kh - 1][w][c]
    __shared__ uint32_t pmax[4][64];
    const int tid = threadIdx.x, chl = tid & 63, q = tid >> 6;
    const int64_t pb = blockIdx.x;                               // pixel block
    const int64_t p0 = pb * B;
    const int per_img = h * w;
    const int64_t img = p0 / per_img;
    const int oy0 = (int)((p0 - img * per_img) >> lg_w);
    const int srows = (B >> lg_w) + kh - 1;
    // stage the source rows oy0 - pad .. oy0 + B / w - 1 + (kh - 1 - pad)
    const int row_elems = w * c;
    for (int e = tid * 4; e < srows * row_elems; e += 256 * 4) {
        const int sr = e / row_elems, off = e - sr * row_elems;
        const int iy = oy0 - pad + sr;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (iy >= 0 && iy < h) v = __ldg(reinterpret_cast<const float4*>(x + ((img * h + iy) * (int64_t)w) * c + off));
        *reinterpret_cast<float4*>(img_rows + e) = v;
    }
    __syncthreads();
    const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
    const int taps = kh * kw;
    // this thread's pixels: column in the image row and offset in the staged rows, worked out once
    int ox_of[NPX], off_of[NPX];
#pragma unroll
    for (int j = 0; j < NPX; ++j) {
        const int px = q * NPX + j;
        ox_of[j] = px & (w - 1);
        off_of[j] = px * c;                                      // ((px >> lg_w) * w + ox) * c
    }
    for (int c0 = 0; c0 < c; c0 += 64) {
        const int ch = c0 + chl;
        const bool live = ch < c;
        for (int tap = 0; tap < taps; ++tap) {
            const int dy = tap / kw, dx = tap - dy * kw - pad;   // dy indexes the staged rows directly
            const float* tap_base = img_rows + (dy * w + dx) * c + (live ? ch : 0);
            float v[NPX];
            uint32_t am = 0;
#pragma unroll
            for (int j = 0; j < NPX; ++j)
                v[j] = (live && (unsigned)(ox_of[j] + dx) < (unsigned)w) ? tap_base[off_of[j]] : 0.f;
#pragma unroll
            for (int j = 0; j < NPX; j += 2) am = max3_abs_bits(am, v[j], v[j + 1]);
            pmax[q][chl] = am;
            __syncthreads();
            am = max(max(pmax[0][chl], pmax[1][chl]), max(pmax[2][chl], pmax[3][chl]));
            __syncthreads();                                     // pmax is rewritten by the next tap
            if (!live) continue;
            const int s = block_exponent(am, p.m, p.exp_mode);
            const int64_t row = (int64_t)tap * c + ch;
            if (q == 0) exps[pb * rs + row] = (int8_t)s;
            const float sc = pow2f(SR ? 16 - s : -s);
            uint32_t hi[NPX / 4], lo[NPX / 4];
#pragma unroll
            for (int wi = 0; wi < NPX / 4; ++wi) {
                uint32_t r[4] = {0u, 0u, 0u, 0u};
                if (SR) {
                    // stochastic rounding draws by the element's index in the activation tensor
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int px = q * NPX + 4 * wi + j, ry = px >> lg_w, ix = (px & (w - 1)) + dx;
                        const int iy = oy0 - pad + ry + dy;
                        if (ix >= 0 && ix < w && iy >= 0 && iy < h)
                            r[j] = draw_of_element(p, (uint64_t)(((img * h + iy) * (int64_t)w + ix) * c + ch));
                    }
                }
                uint32_t h01, h23;
                if (SR) {
                    h01 = round_sr_pair2(v[4 * wi], v[4 * wi + 1], sc, r[0], r[1], qm, nqm);
                    h23 = round_sr_pair2(v[4 * wi + 2], v[4 * wi + 3], sc, r[2], r[3], qm, nqm);
                } else {
                    h01 = round_rne_pair(v[4 * wi], v[4 * wi + 1], sc, qm, nqm);
                    h23 = round_rne_pair(v[4 * wi + 2], v[4 * wi + 3], sc, qm, nqm);
                }
                pack4<PLANES>(h01, h23, hi[wi], lo[wi]);
            }
            int8_t* dst = mant + row * kst + pb * BP + q * NPX;
            if (NPX >= 16) {
#pragma unroll
                for (int i = 0; i < NPX / 16; ++i) {
                    *reinterpret_cast<uint4*>(dst + 16 * i) = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
                    if (PLANES == 2) *reinterpret_cast<uint4*>(dst + plane_stride + 16 * i) = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < NPX / 4; ++i) {
                    *reinterpret_cast<uint32_t*>(dst + 4 * i) = hi[i];
                    if (PLANES == 2) *reinterpret_cast<uint32_t*>(dst + plane_stride + 4 * i) = lo[i];
                }
            }
            if (B < BP && q == 0) {                              // block padding (16-pixel blocks in 32 bytes)
#pragma unroll
                for (int px0 = B; px0 < BP; px0 += 4) {
                    *reinterpret_cast<uint32_t*>(mant + row * kst + pb * BP + px0) = 0u;
                    if (PLANES == 2) *reinterpret_cast<uint32_t*>(mant + plane_stride + row * kst + pb * BP + px0) = 0u;
                }
            }
        }
    }
}

// The same operand for filters three columns wide, blocks of 64 pixels and images 8 to 64 pixels wide. A thread takes one
// channel and one filter row: the 64 pixels of the block under that row are 64 loads (lanes along the channels: whole
// 128-byte lines), all in flight together, and stay in registers for the three filter columns, whose operands are the same
// values shifted by one with compile-time indices - no shared memory, no barrier, no index or bounds arithmetic per element
// (im2col_cols spends its time on those). The maxima share their middle columns. Nearest-even rounds with one FMA per value;
// each (tap, channel) row leaves as two whole 32-byte sectors. Bound by the 75 MB it writes for 64 channels at 32 x 32, batch 128:
// 65 -> 26.6 us (17 us at the copy rate); 128 channels at 16 x 16: 38 -> 15.0 us.
// CTAs per SM, and with them the registers of a thread: short rows want all their loads in flight (w = 16: 15.0 us with one or
// two CTAs per SM, 18.5 with three), long rows more warps (w = 32: 46 / 31 / 27 us with one / two / three, 37 with four).
template <int PLANES, int W, bool SR>
constexpr int cols3_ctas() { return SR || PLANES == 2 || W <= 16 ? 1 : 3; }

template <int PLANES, int W, bool SR>
__global__ void __launch_bounds__(192, cols3_ctas<PLANES, W, SR>())
im2col_cols3(const float* __restrict__ x, int h, int c, int kh, int pad, QParams p, int64_t kst, int64_t plane_stride, int64_t rs,
             int8_t* __restrict__ mant, int8_t* __restrict__ exps) {
    chain_start();
    constexpr int B = 64, ROWS = B / W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint16_t* rnd = reinterpret_cast<const uint16_t*>(smem_raw);       // draws of the rows under the filter [ROWS + kh - 1][W][c] (stochastic)
    const int64_t pb = blockIdx.x;
    const int blocks_per_img = h / ROWS;
    const int64_t img = pb / blocks_per_img;
    const int oy0 = (int)(pb - img * blocks_per_img) * ROWS;
    if (SR) {
        // draws by the element's index in the activation tensor: eight consecutive channels share a Philox call
        const int64_t first = ((img * h + oy0 - pad) * W) * c;               // index of the first staged element (a multiple of 8, may lie before the image)
        uint4* t = reinterpret_cast<uint4*>(smem_raw);
        for (int i = threadIdx.x; i < (ROWS + kh - 1) * W * c / 8; i += blockDim.x) t[i] = draws_of_group(p, (uint64_t)(first + 8 * (int64_t)i) >> 3);
        __syncthreads();
    }
    const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
    for (int item = threadIdx.x; item < kh * c; item += blockDim.x) {
        const int dy = item / c, ch = item - dy * c;
        float v[B];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int iy = oy0 + r + dy - pad;
            const float* src = x + ((img * h + iy) * (int64_t)W) * c + ch;
            const bool in = iy >= 0 && iy < h;
#pragma unroll
            for (int q = 0; q < W; ++q) v[r * W + q] = in ? __ldg(src + q * c) : 0.f;
        }
        uint32_t core = 0, left = 0, right = 0;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int q = 1; q < W - 1; q += 2) core = max3_abs_bits(core, v[r * W + q], v[r * W + q + 1]);
            left = max(left, abs_bits(v[r * W]));
            right = max(right, abs_bits(v[r * W + W - 1]));
        }
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
            const int dx = kx - 1;                                           // filter column: pixel q takes the value at q + dx
            uint32_t am = core;
            if (dx <= 0) am = max(am, left);
            if (dx >= 0) am = max(am, right);
            const int s = block_exponent(am, p.m, p.exp_mode);
            const int64_t row = (int64_t)(dy * 3 + kx) * c + ch;
            exps[pb * rs + row] = (int8_t)s;
            const float sc = pow2f(SR ? 16 - s : -s);
            uint32_t hi[B / 4], lo[B / 4];
#pragma unroll
            for (int w4 = 0; w4 < B / 4; ++w4) {
                uint32_t hh[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int e0 = 4 * w4 + 2 * k, e1 = e0 + 1;
                    const bool in0 = (e0 % W) + dx >= 0, in1 = (e1 % W) + dx < W;      // only the outer columns can leave the image
                    const float x0 = in0 ? v[in0 ? e0 + dx : 0] : 0.f, x1 = in1 ? v[in1 ? e1 + dx : 0] : 0.f;
                    if (SR) {
                        const uint32_t r0 = in0 ? rnd[((e0 / W + dy) * W + (e0 % W) + dx) * c + ch] : 0u;
                        const uint32_t r1 = in1 ? rnd[((e1 / W + dy) * W + (e1 % W) + dx) * c + ch] : 0u;
                        hh[k] = round_sr_pair2(x0, x1, sc, r0, r1, qm, nqm);
                    } else {
                        hh[k] = round_rne_pair(x0, x1, sc, qm, nqm);
                    }
                }
                pack4<PLANES>(hh[0], hh[1], hi[w4], lo[w4]);
            }
            int8_t* dst = mant + row * kst + pb * B;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                store_sector(dst + 32 * half, &hi[8 * half]);
                if (PLANES == 2) store_sector(dst + plane_stride + 32 * half, &lo[8 * half]);
            }
        }
    }
}

// Filter operand of the backward-data convolution from view c1 of tiled convolution weights: row ci of the result
// is, tap by tap in reversed order, the c_out packed bytes of c1's row (tap, ci) (Sec. 5.1: backward-data is the
// convolution of the output gradient with the filters turned by 180 degrees and their feature-map roles swapped;
// the mantissas and tile exponents are the forward pass's own). One warp per (ci, tap), 16 bytes per lane.
__global__ void __launch_bounds__(256)
conv_dgrad_filters_kernel(const int8_t* __restrict__ m1, const int8_t* __restrict__ e1, int64_t kst1, int64_t ps1,
                          int64_t rs1, int taps, int64_t c_in, int64_t c_out, int t, int planes,
                          int8_t* __restrict__ mo, int8_t* __restrict__ eo, int64_t ksto, int64_t pso, int64_t rso) {
    chain_start();
    const int lane = threadIdx.x & 31;
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= c_in * taps) return;
    const int64_t ci = item / taps;
    const int tap = (int)(item - ci * taps);
    const int64_t src_row = (int64_t)(taps - 1 - tap) * c_in + ci;
    for (int pl = 0; pl < planes; ++pl)
        for (int64_t o = 16 * lane; o < c_out; o += 512)
            *reinterpret_cast<uint4*>(mo + pl * pso + ci * ksto + (int64_t)tap * c_out + o) =
                *reinterpret_cast<const uint4*>(m1 + pl * ps1 + src_row * kst1 + o);
    const int cb_n = (int)(c_out / t);
    for (int cb = lane; cb < cb_n; cb += 32) eo[((int64_t)tap * cb_n + cb) * rso + ci] = e1[(int64_t)cb * rs1 + src_row];
    // bytes of the row beyond the last tap (the row pitch is a multiple of 128)
    if (tap == taps - 1)
        for (int64_t o = (int64_t)taps * c_out + 16 * lane; o < ksto; o += 512)
            for (int pl = 0; pl < planes; ++pl) *reinterpret_cast<uint4*>(mo + pl * pso + ci * ksto + o) = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------------------------ inverse helpers

__global__ void unpack_kernel(const int8_t* __restrict__ mant, const int8_t* __restrict__ exps, int64_t rows,
                              int64_t K, int64_t b, int64_t bp, int64_t nkb, int64_t kst, int64_t plane_stride,
                              int planes, int64_t rs, int16_t* __restrict__ q, int8_t* __restrict__ s) {
    chain_start();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q && i < rows * K) {
        const int64_t r = i / K, kk = i % K, o = (kk / b) * bp + kk % b;
        int v = mant[r * kst + o];
        if (planes == 2) v = v * 16 + mant[plane_stride + r * kst + o];
        q[i] = (int16_t)v;
    }
    if (s && i < rows * nkb) {
        const int64_t r = i / nkb, kb = i % nkb;
        s[i] = exps[kb * rs + r];
    }
}

__global__ void dequant_kernel(const int8_t* __restrict__ mant, const int8_t* __restrict__ exps, int64_t rows,
                               int64_t K, int64_t b, int64_t bp, int64_t kst, int64_t plane_stride, int planes,
                               int64_t rs, float* __restrict__ out, int64_t ld) {
    chain_start();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * K) return;
    const int64_t r = i / K, kk = i % K, kb = kk / b, o = kb * bp + kk % b;
    int v = mant[r * kst + o];
    if (planes == 2) v = v * 16 + mant[plane_stride + r * kst + o];
    out[r * ld + kk] = ldexpf((float)v, (int)exps[kb * rs + r]);
}

// ------------------------------------------------------------------------------ quant_row_flat

// Blocks along contiguous rows for row lengths that are not a multiple of the 512-column tile of
// quant_row_fast (K % b == 0, e.g. im2col matrices with K = 576 or 1152): the rows are cut into 8-element groups that are
// numbered through the whole matrix, and a warp takes 32 consecutive groups wherever the row boundaries fall, so no lane
// idles on a ragged last tile. The zeros between K and the packed pitch are written by the lanes of the row's first
// groups (numbered like the others, half of the lanes of 64-channel pixels had nothing to
// load: 131072 x 64 12.6 us, now 8.5 = 5.9 TB/s; 10^6 x 32 with stochastic rounding, three quarters idle, 125 -> 42 us; 131072 x 576
// 64.8 -> 61.1).
// CTA: 256 threads x ITEMS groups each (256 ITEMS consecutive groups).
template <int LPB, bool SR, int PLANES, int ITEMS>
__global__ void __launch_bounds__(256)
quant_row_flat(const float* __restrict__ x, int64_t rows, int64_t K, int64_t ld, QParams p,
               int8_t* __restrict__ mant, int64_t kst, int64_t plane_stride,
               int8_t* __restrict__ exps, int64_t rs, uint32_t gpr, uint32_t total_groups, const FormArgs fa) {
    const Chain chain(p.at);
    constexpr int B = 8 * LPB;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t g0 = blockIdx.x * (256u * ITEMS) + tid;
    // (row, group in row) of this thread's first group; the next ones are 256 groups further on each
    uint32_t row = g0 / gpr, cg = g0 - row * gpr;
    const uint32_t q256 = 256u / gpr, r256 = 256u - q256 * gpr;
    float4 v[ITEMS][2];
    uint32_t rw[ITEMS], cc[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        rw[j] = row;
        cc[j] = cg * 8;
        const bool in = g0 + j * 256u < total_groups;
        if (in) {
            const float4* src = reinterpret_cast<const float4*>(x + (int64_t)row * ld + cc[j]);
            v[j][0] = __ldcs(src);
            v[j][1] = __ldcs(src + 1);
        } else {
            v[j][0] = make_float4(0.f, 0.f, 0.f, 0.f);
            v[j][1] = v[j][0];
        }
        row += q256;
        cg += r256;
        if (cg >= gpr) { cg -= gpr; ++row; }
    }
    // the draws do not depend on the data: they are made while the loads are in flight
    uint4 wd[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        wd[j] = make_uint4(0u, 0u, 0u, 0u);
        if (SR) wd[j] = draws_of_group(p, ((uint64_t)rw[j] * (uint64_t)K + cc[j]) >> 3);     // a multiple of 8 on this path
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool live = g0 + j * 256u < total_groups;      // uniform over the LPB lanes of a block
        const float e8[8] = {v[j][0].x, v[j][0].y, v[j][0].z, v[j][0].w, v[j][1].x, v[j][1].y, v[j][1].z, v[j][1].w};
        uint32_t am = amax8_bits(e8);
#pragma unroll
        for (int off = 1; off < LPB; off <<= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
        const int s = block_exponent(am, p.m, p.exp_mode);
        const uint4 w = wd[j];
        round_and_store8<SR, PLANES>(e8, s, p, w, mant, (int64_t)rw[j] * kst + cc[j], plane_stride, live);
        check_exponent<PLANES>(s, fa);
        if (live)
            for (uint32_t o = (uint32_t)K + cc[j]; o < kst; o += 8u * gpr) store_zero8<PLANES>(mant, (int64_t)rw[j] * kst + o, plane_stride);
        if (live && (lane % LPB) == 0) store_exponent<PLANES>(exps, (int64_t)(cc[j] / B) * rs + rw[j], s);
    }
    if (!is_form(PLANES)) zero_padding_lines(exps, rows, rs, K / B);
}

// FORM: 0 for the packed layout (its planes as L says), else the form to write.
template <int LPB, int ITEMS, int FORM>
int launch_row_flat_items(const float* x, int64_t rows, int64_t K, int64_t ld, const QParams& p, const Layout& L,
                          int8_t* mant, int8_t* exps, cudaStream_t st, const FormArgs& fa) {
    const uint32_t gpr = (uint32_t)(K / 8), total = (uint32_t)(rows * (K / 8));
    const unsigned grid = (total + 256u * ITEMS - 1u) / (256u * ITEMS);
#define HBFP_QFLAT(SRV, OUT) launch_placed(p.at, 4 * rows * K, quant_row_flat<LPB, SRV, OUT, ITEMS>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, gpr, total, fa)
    if constexpr (FORM != 0) { if (p.rounding == 1) HBFP_QFLAT(true, FORM); else HBFP_QFLAT(false, FORM); }
    else if (p.rounding == 1) { if (L.planes == 1) HBFP_QFLAT(true, 1); else HBFP_QFLAT(true, 2); }
    else { if (L.planes == 1) HBFP_QFLAT(false, 1); else HBFP_QFLAT(false, 2); }
#undef HBFP_QFLAT
    return launch_status();
}

// Groups per thread: more of them amortise the index arithmetic, fewer keep the register footprint small
// and more loads in flight. Measured on 131072 x 576 (b = 64): eight 68 us, four 58 us, two 61 us with
// nearest-even rounding; 91 / 84 / 82 us with stochastic rounding (the Philox state of every group in flight
// is live). Narrow rows (one or two 128-byte units, e.g. one block of 64 channels per pixel) do as well with two.
template <int LPB, int FORM = 0>
int launch_row_flat(const float* x, int64_t rows, int64_t K, int64_t ld, const QParams& p, const Layout& L,
                    int8_t* mant, int8_t* exps, cudaStream_t st, const FormArgs& fa = FormArgs{}) {
    if (L.kst > 256 && p.rounding == 0) return launch_row_flat_items<LPB, 4, FORM>(x, rows, K, ld, p, L, mant, exps, st, fa);
    return launch_row_flat_items<LPB, 2, FORM>(x, rows, K, ld, p, L, mant, exps, st, fa);
}

// ------------------------------------------------------------------------------ quant_row_ragged

// Quotient and remainder by a divisor known to the host (magic = floor((2^32 - 1) / d)), for numerators below 2^32: the estimate is at
// most one short. A division of 64 bits per piece of eight was half of these kernels' instructions.
struct Divisor { uint32_t d, magic; };
inline Divisor divisor(uint32_t d) { return {d, 0xFFFFFFFFu / d}; }
__device__ __forceinline__ uint32_t divide(uint32_t n, const Divisor& v, uint32_t& rest) {
    uint32_t q = __umulhi(n, v.magic);
    rest = n - q * v.d;
    if (rest >= v.d) { rest -= v.d; ++q; }
    return q;
}

// Blocks along rows for every other block length up to 128, row length, pitch and alignment (24 columns per block, odd row
// lengths). As in quant_row_flat the packed row, padding included, is cut into pieces of eight elements numbered through the
// whole matrix, LPB = bp / 8 lanes per block; a piece that lies in a block's padding loads nothing. Without alignment a lane
// fetches its eight floats one by one (the sectors of a warp's pieces stay in L1 between them), and its eight draws may
// straddle two Philox groups: the second call is made only then. One pass instead of the two of exps_axis1 and
// mant_generic, which index, divide and draw per element: 16384 x 16384, b = 24, nearest-even 2627 -> 287 us. Matrices beyond 2^32
// pieces are launched in parts. With a 64-bit division per piece, before / now: 10000 x 10000, b = 24, draws 168 / 152 us, 8320 x 1708,
// b = 128, draws 24.7 / 20.6, 100 x 16380, b = 24, draws 8.3 / 5.2. (Unaligned rows: a lane per element of 32 neighbours, a warp reduction
// and a byte store per 32 elements, 20000 x 3001, b = 24 210 us against 75; the three aligned quads around the eight floats 85.)
// Pieces of a warp. On unaligned rows with draws, as many whole blocks as 64 Philox groups serve: their elements are consecutive, so two
// calls per lane into a table per warp do for what took two per piece (5001 columns, b = 32, 4999 rows 45.2 -> 39.6 us, 1111 x 3001,
// b = 24 9.7 -> 8.0). Aligned rows mostly start at a group and need one call per piece; the lanes that the table leaves idle cost them
// more (10000 x 10000, b = 24 152 -> 177, 8320 x 1708, b = 128 20.6 -> 25.9).
template <int LPB, bool TABLE>
__host__ __device__ constexpr int ragged_pieces() { return TABLE ? 64 - LPB : 64; }

template <int LPB, bool SR, int PLANES, bool VEC>
__global__ void __launch_bounds__(256)
quant_row_ragged(const float* __restrict__ x, int64_t rows, int64_t K, int64_t ld, int b, QParams p,
                 int8_t* __restrict__ mant, int64_t kst, int64_t plane_stride,
                 int8_t* __restrict__ exps, int64_t rs, int64_t nkb, const Divisor ppr, int64_t row_first, uint32_t total, const FormArgs fa) {
    const Chain chain(p.at);
    constexpr bool TABLE = SR && !VEC;
    constexpr int ITEMS = 2, PIECES = ragged_pieces<LPB, TABLE>();
    __shared__ __align__(16) uint4 rnd[TABLE ? 8 : 1][TABLE ? 65 : 1];         // (the word after the last group is read and not used)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t g0 = (blockIdx.x * 8 + warp) * PIECES;
    float e8[ITEMS][8];
    int64_t row[ITEMS];
    int cb[ITEMS], kk0[ITEMS], pc[ITEMS];             // block of the row; first element of the piece along the row; piece of the row
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t g = g0 + i * 32 + lane;
        uint32_t rest;
        row[i] = row_first + divide(g, ppr, rest);
        pc[i] = (int)rest;
        cb[i] = pc[i] / LPB;
        const int within = 8 * (pc[i] - cb[i] * LPB);
        kk0[i] = cb[i] * b + within;
        const int n = (g < total && i * 32 + lane < PIECES && cb[i] < nkb) ? (int)min((int64_t)(b - within), K - kk0[i]) : 0;    // elements of the piece
        const float* src = x + row[i] * ld + kk0[i];
        if (VEC && n >= 8) {
            const float4 u = __ldcs(reinterpret_cast<const float4*>(src)), w = __ldcs(reinterpret_cast<const float4*>(src) + 1);
            e8[i][0] = u.x; e8[i][1] = u.y; e8[i][2] = u.z; e8[i][3] = u.w;
            e8[i][4] = w.x; e8[i][5] = w.y; e8[i][6] = w.z; e8[i][7] = w.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) e8[i][j] = j < n ? __ldca(src + j) : 0.f;
        }
    }
    // the draws do not depend on the data: they are made while the loads are in flight (the matrix is rows x K as passed)
    uint64_t first = 0;
    if (TABLE) {
        first = __shfl_sync(0xffffffffu, (unsigned long long)(row[0] * K + min((int64_t)kk0[0], K)), 0) >> 3;
        rnd[TABLE ? warp : 0][TABLE ? lane : 0] = draws_of_group(p, first + lane);
        rnd[TABLE ? warp : 0][TABLE ? lane + 32 : 0] = draws_of_group(p, first + lane + 32);
        __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool live = g0 + i * 32 + lane < total && i * 32 + lane < PIECES;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (SR && VEC) w = draws_of_eight(p, (uint64_t)(row[i] * K + kk0[i]));
        if (TABLE) {
            const int at = live && cb[i] < nkb ? (int)((uint64_t)(row[i] * K + min((int64_t)kk0[i], K)) - 8 * first) : 0;     // halfword of the table
            const uint32_t* word = reinterpret_cast<const uint32_t*>(rnd[TABLE ? warp : 0]) + (at >> 1);
            const uint32_t t[5] = {word[0], word[1], word[2], word[3], word[4]};
            w = at & 1 ? make_uint4(__funnelshift_r(t[0], t[1], 16), __funnelshift_r(t[1], t[2], 16), __funnelshift_r(t[2], t[3], 16), __funnelshift_r(t[3], t[4], 16))
                       : make_uint4(t[0], t[1], t[2], t[3]);
        }
        uint32_t am = amax8_bits(e8[i]);
#pragma unroll
        for (int off = 1; off < LPB; off <<= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, off));
        const int s = block_exponent(am, p.m, p.exp_mode);
        round_and_store8<SR, PLANES>(e8[i], s, p, w, mant, row[i] * kst + 8 * (int64_t)pc[i], plane_stride, live);
        check_exponent<PLANES>(s, fa);
        if (live && (lane % LPB) == 0 && cb[i] < nkb) store_exponent<PLANES>(exps, (int64_t)cb[i] * rs + row[i], s);
    }
    if (!is_form(PLANES) && row_first == 0) zero_padding_lines(exps, rows, rs, nkb);
}

// OUT: 1 or 2 planes or a form. vec: pieces of eight start on 16-byte boundaries.
template <int OUT>
int launch_row_ragged(bool vec, const float* x, int64_t rows, int64_t K, int64_t ld, const QParams& p, const Layout& L,
                      int8_t* mant, int8_t* exps, cudaStream_t st, const FormArgs& fa = FormArgs{}) {
    const int64_t ppr = L.kst / 8, rows_per = std::max<int64_t>(1, ((1ll << 32) - 65536) / ppr);       // pieces of a row; rows of a launch
    if (ppr >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    const Divisor d = divisor((uint32_t)ppr);
    QParams q = p;
    for (int64_t r = 0; r < rows; r += rows_per, q.at = Placing{}) {
        const int64_t total = std::min(rows - r, rows_per) * ppr;
#define HBFP_RAGGED(LPB, SRV, VEC) launch_placed(q.at, 4 * rows * K, quant_row_ragged<LPB, SRV, OUT, VEC>, (unsigned)((total + 8 * ragged_pieces<LPB, SRV && !VEC>() - 1) / (8 * ragged_pieces<LPB, SRV && !VEC>())), 256, 0, st, x, rows, K, ld, (int)L.b, q, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, d, r, (uint32_t)total, fa)
#define HBFP_RAGGED_SR(LPB, VEC) do { if (p.rounding) HBFP_RAGGED(LPB, true, VEC); else HBFP_RAGGED(LPB, false, VEC); } while (0)
#define HBFP_RAGGED_VEC(LPB) do { if (vec) HBFP_RAGGED_SR(LPB, true); else HBFP_RAGGED_SR(LPB, false); } while (0)
        if (L.bp == 32) HBFP_RAGGED_VEC(4); else if (L.bp == 64) HBFP_RAGGED_VEC(8); else HBFP_RAGGED_VEC(16);
#undef HBFP_RAGGED_VEC
#undef HBFP_RAGGED_SR
#undef HBFP_RAGGED
    }
    return launch_status();
}

// ------------------------------------------------------------------------------ quant_col_tma

// Blocks down the columns of x [K][R] for b in {32, 64, 128}, the layout of the B operand of a
// forward GEMM. Persistent CTAs stream 128 (k) x 64 (columns) FP32 tiles by TMA, one in flight per CTA and
// five or six CTAs per SM: against two in flight and three CTAs the same bytes are on their way and a warp that waits leaves more
// others to issue (16384^2, b = 64, stochastic 256 -> 236 us; b = 128 nearest-even 215 -> 214; 1000 x 3000 7.8 -> 6.5); thread (column n, quarter q) keeps 32 consecutive k of its column in registers between
// the block maximum and the rounding pass, and the packed tile (64 output rows x 128 mantissa bytes,
// contraction-major) goes back to global memory as one 128B-swizzled TMA store per plane, so both
// directions move full lines whatever the matrix pitch.
constexpr int QC_COLS = 64, QC_ROWS = 128, QC_STAGES = 1, QC_THREADS = 256;
constexpr int QC_IN_BYTES = QC_ROWS * QC_COLS * 4;          // 32 KB
constexpr int QC_OUT_BYTES = QC_COLS * QC_ROWS;             // 8 KB per plane

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int c0, int c1, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1) : "memory");
}

template <int PLANES, int LB, bool SR>      // b = 128 >> LB
__global__ void __launch_bounds__(QC_THREADS)
quant_col_tma(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapM0,
              const __grid_constant__ CUtensorMap mapM1, QParams p, int8_t* __restrict__ exps, int64_t rs,
              int64_t nkb, int64_t K, int64_t R, int tiles_n, int total_tiles, int32_t* status,
              const int8_t* __restrict__ given, int8_t* __restrict__ form_out, int64_t kst, int64_t plane_stride) {
    const Chain chain(p.at);
    // given != nullptr: one exponent per column for the whole axis, computed beforehand (blocks longer than a
    // tile); the kernel then only rounds and packs
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
    // [out planes | in stages | draws (stochastic) | block maxima | barriers]
    // forms leave from registers: a thread's 32 consecutive k are two whole sectors of its output row
    constexpr int OFF_IN = is_form(PLANES) ? 0 : PLANES * QC_OUT_BYTES;
    constexpr int OFF_RND = OFF_IN + QC_STAGES * QC_IN_BYTES;
    constexpr int OFF_PMAX = OFF_RND + (SR ? QC_ROWS * QC_COLS * 2 : 0);
    constexpr int OFF_BAR = OFF_PMAX + 4 * QC_COLS * 4;
    const float* in = reinterpret_cast<const float*>(base_ptr + OFF_IN);
    uint4* rnd = reinterpret_cast<uint4*>(base_ptr + OFF_RND);
    uint32_t* pmax = reinterpret_cast<uint32_t*>(base_ptr + OFF_PMAX);
    const uint32_t full_bar = base + OFF_BAR;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + OFF_BAR + 8 * QC_STAGES);

    const int tid = threadIdx.x, n = tid & (QC_COLS - 1), q = tid >> 6;
    if (tid == 0) {
        for (int s = 0; s < QC_STAGES; ++s) mbar_init(full_bar + 8 * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    const int first = blockIdx.x, step = gridDim.x;
    if (tid == 0) {
        if (p.at.place == BESIDE) asm volatile("fence.proxy.async.global;" ::: "memory");      // what was acquired is read by the copy engine
        for (int s = 0; s < QC_STAGES; ++s) {
            const int t = first + s * step;
            if (t < total_tiles) {
                mbar_expect_tx(full_bar + 8 * s, QC_IN_BYTES);
                tma_load_2d(base + OFF_IN + s * QC_IN_BYTES, &mapX, (t % tiles_n) * (QC_COLS * 4), (t / tiles_n) * QC_ROWS, full_bar + 8 * s);
            }
        }
    }
    uint32_t s = 0, ph = 0;
    bool stores_pending = false;
    for (int t = first; t < total_tiles; t += step) {
        const int nt = t % tiles_n, kt = t / tiles_n;
        const int64_t col = (int64_t)nt * QC_COLS + n;
        if (SR) {
            // one Philox call per eight consecutive source elements of a row (R % 8 == 0 here); the draws
            // do not depend on the data, so they are made while the tile may still be in flight (the
            // previous tile's readers of the table are past the barrier that precedes its store)
            for (int i = tid; i < QC_ROWS * (QC_COLS / 8); i += QC_THREADS) {
                const uint64_t L = (uint64_t)((int64_t)kt * QC_ROWS + (i >> 3)) * (uint64_t)R + (uint64_t)(nt * QC_COLS + (i & 7) * 8);
                rnd[i] = draws_of_group(p, L >> 3);
            }
        }
        // (uniform verdict: a wait that gave up in some threads only would split the CTA barriers below)
        if (!__syncthreads_and(mbar_wait(full_bar + 8 * s, ph, abort_flag, status, 601))) break;
        const float* tile = in + (size_t)s * (QC_IN_BYTES / 4);
        float v[32];
        uint32_t am = 0;
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
            v[j] = tile[(q * 32 + j) * QC_COLS + n];
            v[j + 1] = tile[(q * 32 + j + 1) * QC_COLS + n];
            am = max3_abs_bits(am, v[j], v[j + 1]);
        }
        // Blocks of 32 need no exchange of maxima; they are stored all the same, because a thread may reach the barrier only when its
        // loads of the tile have returned. Without a value that depends on them before it, a warp's loads could still wait in the load
        // unit's queue while the copy engine, which that queue does not order, filled the stage again: about one product in a
        // hundred at 1024 x 4096 x 4096 had 32 columns of mantissas from the next tile.
        pmax[q * QC_COLS + n] = am;
        // the packed tile of the previous iteration must have left shared memory before it is rewritten
        if (tid == 0 && stores_pending) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncthreads();
        // every thread holds its values in registers now: refill this stage with the tile after next
        if (tid == 0) {
            const int t2 = t + QC_STAGES * step;
            if (t2 < total_tiles) {
                mbar_expect_tx(full_bar + 8 * s, QC_IN_BYTES);
                tma_load_2d(base + OFF_IN + s * QC_IN_BYTES, &mapX, (t2 % tiles_n) * (QC_COLS * 4), (t2 / tiles_n) * QC_ROWS, full_bar + 8 * s);
            }
        }
        if (LB == 0) am = max(max(pmax[n], pmax[QC_COLS + n]), max(pmax[2 * QC_COLS + n], pmax[3 * QC_COLS + n]));
        if (LB == 1) am = max(pmax[(q & 2) * QC_COLS + n], pmax[((q & 2) + 1) * QC_COLS + n]);
        const int sexp = given ? (col < R ? (int)given[col] : -63) : block_exponent(am, p.m, p.exp_mode);
        const int64_t kb = ((int64_t)kt << LB) + (q >> (2 - LB));
        if constexpr (is_form(PLANES)) {
            check_exponent<PLANES>(sexp, FormArgs{status});
            if ((q & ((4 >> LB) - 1)) == 0 && kb < nkb && col < R) store_exponent<PLANES>(exps, kb * rs + col, sexp);
        } else if (!given && (q & ((4 >> LB) - 1)) == 0 && kb < nkb && col < rs) {
            exps[kb * rs + col] = col < R ? (int8_t)sexp : (int8_t)0;   // padding lines: zero
        }

        uint32_t hi[8], lo[8];
        uint32_t fo[is_form(PLANES) ? 2 : 1][16];
        const uint16_t* rnd16 = reinterpret_cast<const uint16_t*>(rnd);
        const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
        const float sc = pow2f(SR ? 16 - sexp : -sexp);
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            uint32_t h[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int j = 4 * w + 2 * k;
                if (SR) {
                    // the draws of two vertical neighbours belong to different rows: two table entries
                    h[k] = round_sr_pair2(v[j], v[j + 1], sc, rnd16[(q * 32 + j) * QC_COLS + n], rnd16[(q * 32 + j + 1) * QC_COLS + n], qm, nqm);
                } else {
                    h[k] = round_rne_pair(v[j], v[j + 1], sc, qm, nqm);
                }
            }
            if constexpr (is_form(PLANES)) {
                form_pair<PLANES>(h[0], pow2f(sexp), fo[0][2 * w], fo[1][2 * w]);
                form_pair<PLANES>(h[1], pow2f(sexp), fo[0][2 * w + 1], fo[1][2 * w + 1]);
            } else {
                pack4<PLANES>(h[0], h[1], hi[w], lo[w]);
            }
        }
        if constexpr (is_form(PLANES)) {
            if (col < R) {
#pragma unroll
                for (int pl = 0; pl < (PLANES == FORM_WIDE_B ? 2 : 1); ++pl) {
                    int8_t* dst = form_out + 2 * (pl * plane_stride + col * kst + (int64_t)kt * QC_ROWS + 32 * q);
                    store_sector(dst, &fo[pl][0]);
                    store_sector(dst + 32, &fo[pl][8]);
                }
            }
            if (SR) __syncthreads();                             // the table of draws is rewritten by the next tile
            if (++s == QC_STAGES) { s = 0; ph ^= 1u; }
            continue;
        }
        // 128B swizzle of the store tile: 16-byte chunk c of row n sits at chunk position c ^ (n % 8)
        unsigned char* orow = base_ptr + (n >> 3) * 1024 + (n & 7) * 128;
        const int c0 = ((2 * q) ^ (n & 7)) << 4, c1 = ((2 * q + 1) ^ (n & 7)) << 4;
        *reinterpret_cast<uint4*>(orow + c0) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(orow + c1) = make_uint4(hi[4], hi[5], hi[6], hi[7]);
        if (PLANES == 2) {
            *reinterpret_cast<uint4*>(orow + QC_OUT_BYTES + c0) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            *reinterpret_cast<uint4*>(orow + QC_OUT_BYTES + c1) = make_uint4(lo[4], lo[5], lo[6], lo[7]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            tma_store_2d(&mapM0, kt * QC_ROWS, nt * QC_COLS, base);
            if (PLANES == 2) tma_store_2d(&mapM1, kt * QC_ROWS, nt * QC_COLS, base + QC_OUT_BYTES);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        stores_pending = true;
        if (++s == QC_STAGES) { s = 0; ph ^= 1u; }
    }
    // the stores must be complete when the CTA leaves (a load still in flight after an abandoned
    // wait has had the whole wait budget, seconds, to land)
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Whole-axis blocks down the columns (one exponent per column of the stored matrix): pass 1 of 2. Each CTA takes
// 256 columns and a band of rows, reads rows coalesced and folds its band's maxima into one word per column. Bands of 128 rows
// where that makes four CTAs per SM, otherwise of 32: a thread's loads leave eight at a time. Every band adds an atomic per column,
// and thousands of them on the words of few columns take longer than the loads: 65536 x 64 14.9 us with bands of 128, 19.3 of 32;
// 65536 x 200 26.9 / 35.3, 16384 x 512 16.7 / 18.6, but 12000 x 300 20.4 / 18.4, 16384 x 1000 26.8 / 24.8, 8192 x 64 12.4 / 10.4.
constexpr int CMAX_ROWS = 128, CMAX_ROWS_SHORT = 32;
__global__ void __launch_bounds__(256)
col_amax_kernel(const float* __restrict__ x, int64_t K, int64_t R, int64_t ld, int band, uint32_t* __restrict__ amax) {
    chain_start();
    const int64_t col = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (col >= R) return;
    const int64_t k0 = (int64_t)blockIdx.y * band, k1 = min(K, k0 + band);
    uint32_t am = 0;
#pragma unroll 8
    for (int64_t k = k0; k < k1; ++k) am = max(am, abs_bits(__ldg(x + k * ld + col)));
    atomicMax(amax + col, am);
}
__global__ void col_exps_kernel(const uint32_t* __restrict__ amax, int64_t R, QParams p, int8_t* __restrict__ exps) {
    chain_start();
    const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (col < R) exps[col] = (int8_t)block_exponent(amax[col], p.m, p.exp_mode);
}

template <int PLANES, int LB, bool SR>
int launch_col_tma(const float* x, int64_t K, int64_t rows, int64_t ld, const QParams& p, const Layout& L,
                   int8_t* mant, int8_t* exps, cudaStream_t st, const int8_t* given = nullptr) {
    CUtensorMap mX, mM0, mM1;
    int rc = make_map(&mX, x, (uint64_t)rows * 4, (uint64_t)K, (uint64_t)ld * 4, QC_COLS * 4, QC_ROWS, false);
    if (rc) return rc;
    mM0 = mX;
    if (!is_form(PLANES)) {
        rc = make_map(&mM0, mant, (uint64_t)L.kst, (uint64_t)rows, (uint64_t)L.kst, QC_ROWS, QC_COLS, true);
        if (rc) return rc;
    }
    mM1 = mM0;
    if (PLANES == 2) {
        rc = make_map(&mM1, mant + L.plane_stride, (uint64_t)L.kst, (uint64_t)rows, (uint64_t)L.kst, QC_ROWS, QC_COLS, true);
        if (rc) return rc;
    }
    constexpr int smem = 1024 + (is_form(PLANES) ? 0 : PLANES * QC_OUT_BYTES) + QC_STAGES * QC_IN_BYTES + (SR ? QC_ROWS * QC_COLS * 2 : 0) +
                         4 * QC_COLS * 4 + 64;
    // attribute and occupancy belong to the device: cached per device ordinal
    static int ctas_per_sm_dev[MAX_DEVICES] = {};
    const int dev = current_device();
    if (dev < 0) return HBFP_ERR_CUDA;
    if (!ctas_per_sm_dev[dev]) {
        HBFP_CUDA_OK(cudaFuncSetAttribute(quant_col_tma<PLANES, LB, SR>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        int nb = 0;
        HBFP_CUDA_OK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, quant_col_tma<PLANES, LB, SR>, QC_THREADS, smem));
        ctas_per_sm_dev[dev] = nb > 0 ? nb : 1;
    }
    const int ctas_per_sm = ctas_per_sm_dev[dev];
    int32_t* status = device_status_word();
    if (!status) return HBFP_ERR_CUDA;
    const int64_t tiles_n = (rows + QC_COLS - 1) / QC_COLS, tiles_k = L.kst / QC_ROWS;
    const int64_t total = tiles_n * tiles_k;
    const int64_t cap = (int64_t)sm_count() * ctas_per_sm;
    const int grid = (int)(total < cap ? total : cap);
    launch_placed(p.at, 0, quant_col_tma<PLANES, LB, SR>, grid, QC_THREADS, smem, st, mX, mM0, mM1, p, exps, L.rs, L.nkb, K, rows, (int)tiles_n,
                                                              (int)total, status, given, mant, L.kst, L.plane_stride);
    return launch_status();
}

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int LPB>
int launch_row_fast(const float* x, int64_t rows, int64_t K, int64_t ld, const QParams& p, const Layout& L,
                    int8_t* mant, int8_t* exps, cudaStream_t st) {
    dim3 grid((unsigned)((L.kst + 511) / 512), (unsigned)((rows + 31) / 32));
    // the last column tile must also cover the exponent rows of blocks that start before K
    if (p.rounding == 1) {
        if (L.planes == 1) launch_placed(p.at, 4 * rows * K, quant_row_fast<LPB, true, 1>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, nullptr, FormArgs{});
        else launch_placed(p.at, 4 * rows * K, quant_row_fast<LPB, true, 2>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, nullptr, FormArgs{});
    } else {
        if (L.planes == 1) launch_placed(p.at, 4 * rows * K, quant_row_fast<LPB, false, 1>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, nullptr, FormArgs{});
        else launch_placed(p.at, 4 * rows * K, quant_row_fast<LPB, false, 2>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, nullptr, FormArgs{});
    }
    return launch_status();
}

}  // namespace

// Launch of the full-tile kernel for tiles of 32 and 64 (defined in part 2 of this file). The parameter blocks are
// passed as opaque bytes: their types live in this file's unnamed namespace, which every part compiles alike.
int launch_tile_full_small(int mode, int planes, int t, bool general, unsigned gx, unsigned gy, const float* src, int64_t ld, int64_t d0,
                           int64_t d1, const void* qparams, int16_t* wide, int8_t* grid, int64_t grid_ld,
                           const void* tileviews, cudaStream_t st);

#if HBFP_QUANT_PART == 2

int launch_tile_full_small(int mode, int planes, int t, bool general, unsigned gx, unsigned gy, const float* src, int64_t ld, int64_t d0,
                           int64_t d1, const void* qparams, int16_t* wide, int8_t* grid, int64_t grid_ld,
                           const void* tileviews, cudaStream_t st) {
    QParams p;
    TileViews tv;
    memcpy(&p, qparams, sizeof(p));
    memcpy(&tv, tileviews, sizeof(tv));
    const dim3 grid_dim(gx, gy);
#define HBFP_TILE_FULL_SMALL(MODE, PLANES, TP)                                                                                              \
    do {                                                                                                                                    \
        if (general) launch_streamed(tile_bytes<MODE>(d0, d1), tile_kernel_full<MODE, PLANES, TP, true>, grid_dim, 256, 0, st, src, ld, d0, d1, p, wide, grid, grid_ld, tv); \
        else launch_streamed(tile_bytes<MODE>(d0, d1), tile_kernel_full<MODE, PLANES, TP, false>, grid_dim, 256, 0, st, src, ld, d0, d1, p, wide, grid, grid_ld, tv);      \
    } while (0)
#define HBFP_TILE_FULL_MODE(MODE)                                                                     \
    do {                                                                                              \
        if (planes == 1) { if (t == 32) HBFP_TILE_FULL_SMALL(MODE, 1, 32); else HBFP_TILE_FULL_SMALL(MODE, 1, 64); } \
        else { if (t == 32) HBFP_TILE_FULL_SMALL(MODE, 2, 32); else HBFP_TILE_FULL_SMALL(MODE, 2, 64); }             \
    } while (0)
    if (t != 32 && t != 64) return HBFP_ERR_INVALID_ARG;
    if (mode == 0) HBFP_TILE_FULL_MODE(0);
    else if (mode == 1) HBFP_TILE_FULL_MODE(1);
    else if (mode == 2) HBFP_TILE_FULL_MODE(2);
    else if (mode == 3) HBFP_TILE_FULL_MODE(3);
    else if (mode == 4) HBFP_TILE_FULL_MODE(4);
    else return HBFP_ERR_INVALID_ARG;
#undef HBFP_TILE_FULL_MODE
#undef HBFP_TILE_FULL_SMALL
    return launch_status();
}

#else   // part 1: everything else

// ------------------------------------------------------------------------------ launchers

int launch_quantize(const float* x, int64_t d0, int64_t d1, int64_t ld, int axis, const hbfp_format* f,
                    int8_t* mant, int8_t* exps, cudaStream_t st, const Placing& at) {
    const int64_t K = axis == 1 ? d1 : d0, rows = axis == 1 ? d0 : d1;
    Layout L;
    int rc = make_layout(rows, K, f, &L);
    if (rc) return rc;
    if (rows == 0) return HBFP_OK;
    const QParams p = make_params(f);
    QParams one = p, last = p;         // the only launch of a conversion, the last of several
    one.at = at;
    if (at.place == LEAD) last.at = at;
    if (K == 0) {
        HBFP_CUDA_OK(cudaMemsetAsync(mant, 0, (size_t)L.mant_bytes, st));
        HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L.exp_bytes, st));
        return HBFP_OK;
    }
    const bool aligned = ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && (ld % 4 == 0);
    if (rows * L.kst >= (int64_t)1 << 40) return HBFP_ERR_UNSUPPORTED;

    // row lengths that the 512-column tiles of quant_row_fast would leave ragged
    if (f->tile == 0 && axis == 1 && aligned && L.b == L.bp && L.b <= 128 && K % L.b == 0 && L.kst % 512 != 0 &&
        rows * (L.kst / 8) < (1ll << 32) - 4096) {
        switch (L.b) {
            case 32: return launch_row_flat<4>(x, rows, K, ld, one, L, mant, exps, st);
            case 64: return launch_row_flat<8>(x, rows, K, ld, one, L, mant, exps, st);
            case 128: return launch_row_flat<16>(x, rows, K, ld, one, L, mant, exps, st);
            default: break;
        }
    }
    // one block per row over the whole axis, longer than the fast kernel's tile: row maxima first (one warp per row),
    // then the fast kernel with the exponents given
    if (f->tile == 0 && axis == 1 && aligned && d1 % 8 == 0 && L.nkb == 1 && L.b == K && K > 256) {
        if (L.rs != rows) HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L.exp_bytes, st));
        // rows of 2048, 4096, 8192 or 16384 elements stay in a CTA's registers: one pass
        if ((K == 2048 || K == 4096 || K == 8192 || K == 16384) && L.kst == K && rows < (1ll << 31)) {
#define HBFP_QROW_WHOLE2(GV, SRV, PL) launch_placed(last.at, 4 * rows * K, quant_row_whole<GV, SRV, PL>, (unsigned)rows, 256, 0, st, x, ld, d1, p, mant, L.kst, L.plane_stride, exps)
#define HBFP_QROW_WHOLE(GV)                                                                          \
    do {                                                                                             \
        if (p.rounding == 1) { if (L.planes == 1) HBFP_QROW_WHOLE2(GV, true, 1); else HBFP_QROW_WHOLE2(GV, true, 2); }   \
        else { if (L.planes == 1) HBFP_QROW_WHOLE2(GV, false, 1); else HBFP_QROW_WHOLE2(GV, false, 2); }                 \
    } while (0)
            if (K == 2048) HBFP_QROW_WHOLE(1); else if (K == 4096) HBFP_QROW_WHOLE(2); else if (K == 8192) HBFP_QROW_WHOLE(4); else HBFP_QROW_WHOLE(8);
#undef HBFP_QROW_WHOLE
#undef HBFP_QROW_WHOLE2
            return launch_status();
        }
        const int64_t want = (rows * 32 + 255) / 256;
        launch_chained(exps_axis1, (unsigned)(want < 148 * 16 ? want : 148 * 16), 256, 0, st, x, rows, K, ld, L.b, L.nkb, p, exps, L.rs);
        if (launch_status()) return HBFP_ERR_CUDA;
        dim3 grid((unsigned)((L.kst + 511) / 512), (unsigned)((rows + 31) / 32));
#define HBFP_QROW_GIVEN(SRV, PL) launch_placed(last.at, 4 * rows * K, quant_row_fast<16, SRV, PL>, grid, 256, 0, st, x, rows, K, ld, p, mant, L.kst, L.plane_stride, exps, L.rs, L.nkb, exps, FormArgs{})
        if (p.rounding == 1) { if (L.planes == 1) HBFP_QROW_GIVEN(true, 1); else HBFP_QROW_GIVEN(true, 2); }
        else { if (L.planes == 1) HBFP_QROW_GIVEN(false, 1); else HBFP_QROW_GIVEN(false, 2); }
#undef HBFP_QROW_GIVEN
        return launch_status();
    }
    if (f->tile == 0 && axis == 1 && aligned && d1 % 8 == 0 && L.b == L.bp && L.b <= 256 &&
        rows <= 32ll * 65535) {
        switch (L.b) {
            case 32: return launch_row_fast<4>(x, rows, K, ld, one, L, mant, exps, st);
            case 64: return launch_row_fast<8>(x, rows, K, ld, one, L, mant, exps, st);
            case 128: return launch_row_fast<16>(x, rows, K, ld, one, L, mant, exps, st);
            case 256: return launch_row_fast<32>(x, rows, K, ld, one, L, mant, exps, st);
            default: break;
        }
    }
    // one block per column over the whole axis: column maxima first (scratch: the head of the mantissa buffer, which
    // the second pass overwrites), then a tile kernel with the exponents given: the streaming one for whole tiles, the ragged one
    // (pieces of 128) for every other length, pitch and alignment - 3432 x 597 170 us through the generic path (a thread per
    // column, an index division per element), now 20.4; 8000 x 8000 1386, now 121; 777 x 333 stochastic 45.5, now 14.8
    if (f->tile == 0 && axis == 0 && L.nkb == 1 && L.b == K && K > 128 && K < (1ll << 31) && rows < (1ll << 29) &&
        (K + CMAX_ROWS - 1) / CMAX_ROWS <= 65535 && ((rows + COLT - 1) / COLT) * (L.kst / 128) < (1ll << 31)) {
        const bool stream = aligned && K % QC_ROWS == 0 && L.kst == K && (p.rounding == 0 || rows % 8 == 0) &&
                            (reinterpret_cast<uintptr_t>(mant) & 127) == 0;
        if (L.rs != rows) HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L.exp_bytes, st));
        uint32_t* amax = reinterpret_cast<uint32_t*>(mant);
        HBFP_CUDA_OK(cudaMemsetAsync(amax, 0, (size_t)rows * 4, st));
        const int64_t wide = (rows + 255) / 256;
        const bool idle = wide * ((K + CMAX_ROWS - 1) / CMAX_ROWS) < 4 * 148;
        const int band = idle && (K <= 12288 || (K <= 20480 && wide >= 3)) ? CMAX_ROWS_SHORT : CMAX_ROWS;
        launch_streamed(4 * rows * K, col_amax_kernel, dim3((unsigned)wide, (unsigned)((K + band - 1) / band)), 256, 0, st, x, K, rows, ld, band, amax);
        launch_chained(col_exps_kernel, (unsigned)wide, 256, 0, st, amax, rows, p, exps);
        if (launch_status()) return HBFP_ERR_CUDA;
        if (stream) {
#define HBFP_QCOL_GIVEN(PL) (p.rounding ? launch_col_tma<PL, 0, true>(x, K, rows, ld, last, L, mant, exps, st, exps) \
                                        : launch_col_tma<PL, 0, false>(x, K, rows, ld, last, L, mant, exps, st, exps))
            return L.planes == 1 ? HBFP_QCOL_GIVEN(1) : HBFP_QCOL_GIVEN(2);
#undef HBFP_QCOL_GIVEN
        }
        const int64_t pieces = L.kst / 128;
        return L.planes == 1 ? launch_col_block<1>(x, K, rows, ld, 128, 128, pieces, last, L, mant, exps, st, FormArgs{}, exps)
                             : launch_col_block<2>(x, K, rows, ld, 128, 128, pieces, last, L, mant, exps, st, FormArgs{}, exps);
    }
    if (f->tile == 0 && axis == 0 && aligned && L.b == L.bp && L.b <= 128 && (p.rounding == 0 || rows % 8 == 0) &&
        (reinterpret_cast<uintptr_t>(mant) & 127) == 0 && rows < (1ll << 29) && K < (1ll << 31) &&
        ((rows + QC_COLS - 1) / QC_COLS) * (L.kst / QC_ROWS) < (1ll << 31)) {
#define HBFP_QCOL_TMA(PL, LBV) (p.rounding ? launch_col_tma<PL, LBV, true>(x, K, rows, ld, one, L, mant, exps, st) \
                                           : launch_col_tma<PL, LBV, false>(x, K, rows, ld, one, L, mant, exps, st))
        const int lb = L.b == 128 ? 0 : L.b == 64 ? 1 : 2;
        if (L.planes == 1) return lb == 0 ? HBFP_QCOL_TMA(1, 0) : lb == 1 ? HBFP_QCOL_TMA(1, 1) : HBFP_QCOL_TMA(1, 2);
        return lb == 0 ? HBFP_QCOL_TMA(2, 0) : lb == 1 ? HBFP_QCOL_TMA(2, 1) : HBFP_QCOL_TMA(2, 2);
#undef HBFP_QCOL_TMA
    }
    // every other block length up to 128, any pitch and alignment
    if (f->tile == 0 && axis == 0 && L.b <= 128 && ((rows + COLT - 1) / COLT) * L.nkb < (1ll << 31)) {
        return L.planes == 1 ? launch_col_block<1>(x, K, rows, ld, (int)L.b, L.bp, L.nkb, one, L, mant, exps, st, FormArgs{}, nullptr)
                             : launch_col_block<2>(x, K, rows, ld, (int)L.b, L.bp, L.nkb, one, L, mant, exps, st, FormArgs{}, nullptr);
    }
    if (f->tile == 0 && axis == 1 && L.b <= 128 && K < (1ll << 30) && rows * (L.kst / 8) < (1ll << 39)) {
        const bool vec = aligned && L.b % 4 == 0;          // every piece starts on a 16-byte boundary
        return L.planes == 1 ? launch_row_ragged<1>(vec, x, rows, K, ld, one, L, mant, exps, st) : launch_row_ragged<2>(vec, x, rows, K, ld, one, L, mant, exps, st);
    }
    if (f->tile > 0 && f->tile <= 128) {
        // single view of a tiled weight: the fused tile kernel with the other view switched off
        return axis == 0 ? launch_quantize_tiles(x, d0, d1, ld, f, mant, exps, nullptr, nullptr, nullptr, st)
                         : launch_quantize_tiles(x, d0, d1, ld, f, nullptr, nullptr, mant, exps, nullptr, st);
    }

    // generic two-pass path
    HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L.exp_bytes, st));
    if (f->tile == 0) {
        if (axis == 1) {
            int64_t items = rows * L.nkb;
            int64_t want = (items + 7) / 8;
            unsigned blocks = (unsigned)(want < 148 * 32 ? want : 148 * 32);
            launch_chained(exps_axis1, blocks, 256, 0, st, x, rows, K, ld, L.b, L.nkb, p, exps, L.rs);
        } else {
            launch_chained(exps_axis0, blocks_for(rows * L.nkb, 256), 256, 0, st, x, rows, K, ld, L.b, L.nkb, p, exps, L.rs);
        }
    } else {
        const int64_t t = f->tile, nu = (d0 + t - 1) / t, nv = (d1 + t - 1) / t;
        launch_chained(exps_tiles, blocks_for(nu * nv * 32, 256), 256, 0, st, x, d0, d1, ld, t, p, axis, exps, L.rs, nu, nv);
    }
    if (launch_status()) return HBFP_ERR_CUDA;
    if (L.planes == 1)
        launch_placed(last.at, 4 * rows * K, mant_generic<1>, blocks_for(rows * (L.kst / 4), 256), 256, 0, st, x, d1, rows, K, ld, axis, L.b, L.bp, L.nkb, p, exps, L.rs, mant, L.kst, L.plane_stride);
    else
        launch_placed(last.at, 4 * rows * K, mant_generic<2>, blocks_for(rows * (L.kst / 4), 256), 256, 0, st, x, d1, rows, K, ld, axis, L.b, L.bp, L.nkb, p, exps, L.rs, mant, L.kst, L.plane_stride);
    return launch_status();
}

namespace {

template <int FORM>
int quantize_form(const float* x, int64_t d1, int64_t ld, int axis, int64_t rows, int64_t K, const QParams& p, const Layout& L, int8_t* out, int8_t* scales,
                  const FormArgs& fa, cudaStream_t st) {
    const bool aligned = ((reinterpret_cast<uintptr_t>(x) & 15) == 0) && (ld % 4 == 0);
    if (axis == 1) {
        if (aligned && L.b == L.bp && K % L.b == 0 && L.kst % 512 != 0 && rows * (L.kst / 8) < (1ll << 32) - 4096)
            return L.b == 32 ? launch_row_flat<4, FORM>(x, rows, K, ld, p, L, out, scales, st, fa) : launch_row_flat<8, FORM>(x, rows, K, ld, p, L, out, scales, st, fa);
        if (aligned && d1 % 8 == 0 && L.b == L.bp && rows <= 32ll * 65535) {
            const dim3 grid((unsigned)((L.kst + 511) / 512), (unsigned)((rows + 31) / 32));
#define HBFP_QFAST(LPB, SRV) launch_placed(p.at, 4 * rows * K, quant_row_fast<LPB, SRV, FORM>, grid, 256, 0, st, x, rows, K, ld, p, out, L.kst, L.plane_stride, scales, L.rs, L.nkb, nullptr, fa)
            if (L.b == 32) { if (p.rounding) HBFP_QFAST(4, true); else HBFP_QFAST(4, false); }
            else { if (p.rounding) HBFP_QFAST(8, true); else HBFP_QFAST(8, false); }
#undef HBFP_QFAST
            return launch_status();
        }
        if (K >= (1ll << 30) || rows * (L.kst / 8) >= (1ll << 39)) return HBFP_ERR_UNSUPPORTED;
        return launch_row_ragged<FORM>(aligned && L.b % 4 == 0, x, rows, K, ld, p, L, out, scales, st, fa);
    }
    if (aligned && L.b == L.bp && (p.rounding == 0 || rows % 8 == 0) && rows < (1ll << 29) && K < (1ll << 31) &&
        ((rows + QC_COLS - 1) / QC_COLS) * (L.kst / QC_ROWS) < (1ll << 31)) {
        if (L.b == 64) return p.rounding ? launch_col_tma<FORM, 1, true>(x, K, rows, ld, p, L, out, scales, st) : launch_col_tma<FORM, 1, false>(x, K, rows, ld, p, L, out, scales, st);
        return p.rounding ? launch_col_tma<FORM, 2, true>(x, K, rows, ld, p, L, out, scales, st) : launch_col_tma<FORM, 2, false>(x, K, rows, ld, p, L, out, scales, st);
    }
    if (((rows + COLT - 1) / COLT) * L.nkb >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    return launch_col_block<FORM>(x, K, rows, ld, (int)L.b, L.bp, L.nkb, p, L, out, scales, st, fa, nullptr);
}

}  // namespace

// Converts an FP32 operand straight to a floating-point operand form: blocks of at most 64, no weight tiles, elements
// aligned to 32 bytes (HBFP_ERR_UNSUPPORTED otherwise; the caller converts to the packed layout and expands that).
int launch_quantize_form(const float* x, int64_t d0, int64_t d1, int64_t ld, int axis, const hbfp_format* f, int wide, bool is_b, const Placing& at,
                         const FpOperand& o, cudaStream_t st) {
    const int64_t K = axis == 1 ? d1 : d0, rows = axis == 1 ? d0 : d1;
    Layout L;
    int rc = make_layout(rows, K, f, &L);
    if (rc) return rc;
    if (f->tile != 0 || L.bp > 64 || rows == 0 || K == 0 || (L.planes == 2) != (wide != 0)) return HBFP_ERR_UNSUPPORTED;
    QParams p = make_params(f);
    p.at = at;
    const FormArgs fa{device_status_word()};
    if (!fa.status) return HBFP_ERR_CUDA;
    int8_t* out = static_cast<int8_t*>(o.p0);
    int8_t* scales = reinterpret_cast<int8_t*>(o.scales);
    if (is_b && wide) L.plane_stride = (static_cast<int8_t*>(o.p1) - out) / 2;        // in elements
    if (!wide) return quantize_form<FORM_SCALED>(x, d1, ld, axis, rows, K, p, L, out, scales, fa, st);
    return is_b ? quantize_form<FORM_WIDE_B>(x, d1, ld, axis, rows, K, p, L, out, scales, fa, st)
                : quantize_form<FORM_WIDE_A>(x, d1, ld, axis, rows, K, p, L, out, scales, fa, st);
}

namespace {

template <int MODE>
int launch_tiles(const float* src, int64_t ld, int64_t d0, int64_t d1, const hbfp_format* f, int16_t* wide,
                 int8_t* grid, int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1, float* value, int64_t ldv,
                 cudaStream_t st) {
    if (f->tile <= 0 || f->tile != f->block) return HBFP_ERR_INVALID_ARG;
    if (f->tile > 128) return HBFP_ERR_UNSUPPORTED;
    Layout L0, L1;
    int rc = make_layout(d1, d0, f, &L0);     // view c0: rows = d1, k = d0
    if (rc) return rc;
    rc = make_layout(d0, d1, f, &L1);         // view c1: rows = d0, k = d1
    if (rc) return rc;
    if (d0 == 0 || d1 == 0) return HBFP_OK;
    const QParams p = make_params(f);
    const int t = f->tile, tp = (int)L0.bp;
    const int64_t nu = L0.nkb, nv = L1.nkb;   // tiles along d0, along d1
    if (nu > 65535) return HBFP_ERR_UNSUPPORTED;
    const TileViews tv{mant_c0, L0.kst, L0.plane_stride, exps_c0, L0.rs, L0.nkb, mant_c1, L1.kst, L1.plane_stride, exps_c1, L1.rs, L1.nkb, value, ldv};
    const bool fast = (t % 8) == 0 && (d1 % 8) == 0 &&
                      (MODE == 2 || ((ld % 4) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0)) &&
                      (MODE == 3 || (reinterpret_cast<uintptr_t>(wide) & 15) == 0) &&
                      (!value || ((ldv % 4) == 0 && (reinterpret_cast<uintptr_t>(value) & 15) == 0));
    const dim3 grid_dim((unsigned)nv, (unsigned)nu);
    // tiles of 32 / 64 / 128, both views or none
    const bool full = fast && t == tp && ((mant_c0 != nullptr) == (mant_c1 != nullptr)) &&
                      (!mant_c0 || (exps_c0 && exps_c1));
    if (full) {
        // whole tiles, cut by 32-bit shifts
        const bool general = d0 % t != 0 || d1 % t != 0 || (MODE != 3 && 16 - p.m + (L0.planes == 2 ? 4 : 0) > 8);
#define HBFP_TILE_FULL(PLANES, RG) launch_streamed_long(tile_bytes<MODE>(d0, d1), tile_kernel_full<MODE, PLANES, 128, RG>, grid_dim, 256, 0, st, src, ld, d0, d1, p, wide, grid, nv, tv)
        if (t != 128)
            return launch_tile_full_small(MODE, (int)L0.planes, t, general, grid_dim.x, grid_dim.y, src, ld, d0, d1, &p, wide, grid, nv, &tv, st);
        if (L0.planes == 1) { if (general) HBFP_TILE_FULL(1, true); else HBFP_TILE_FULL(1, false); }
        else { if (general) HBFP_TILE_FULL(2, true); else HBFP_TILE_FULL(2, false); }
#undef HBFP_TILE_FULL
        return launch_status();
    }
    // A CTA per tile or strips of tiles (148 SMs; a wave of the one are 148 to 1184 CTAs, by the tile; us, the one / the other).
    //   Few small tiles: strips leave SMs idle, even cut down as below (100 x 100, t = 8, update 7.4 / 8.3, cut down, and 14.4 as they were;
    //   512 x 512, t = 24 8.7 / 9.7 and 11.5). What reads the wide words gains for longer (1000 x 1000, t = 24 12.8 / 14.5, from FP32 11.3 /
    //   11.3), without vectors for shorter.
    //   Aligned tiles above 32: sixteen bytes per access against four (4096 x 4096, t = 72, update 69 / 182, t = 120 58 / 100, t = 40 66 / 77).
    //   48 is the one length whose strips have no idle lane: many of those are faster in strips where no word is read (51 / 40).
    //   Others above 64: a strip is one tile, with 44 % of its lanes idle at t = 72 and one CTA per SM (2000 x 3001, t = 72, update 35 / 66, from
    //   FP32 27 / 44); the draws, made per element there and from a table here, take most of that back (86 / 100, t = 84 even; from FP32 even at 72).
    constexpr bool FROM_WORDS = MODE != 0 && MODE != 3, UPDATE = MODE == 1 || MODE == 4;
    const int64_t tiles = nu * nv;
    const bool draws = p.rounding && MODE != 2;
    bool per_tile;
    if (fast && t <= 32) per_tile = tiles <= (t == tp ? 592 : FROM_WORDS && t >= 16 ? 1776 : 1184);
    else if (fast && t == tp) per_tile = t == 64 && tiles <= 592;
    else if (fast) per_tile = FROM_WORDS || t != 48 || tiles <= 1184;
    else if (t <= 64) per_tile = t <= (FROM_WORDS ? 32 : 24) && tiles <= 592;
    else per_tile = draws ? UPDATE && t <= 76 && tiles > 592 : t <= (FROM_WORDS ? 96 : 88) && tiles > 148;
    if (per_tile) {
        const size_t smem = (size_t)t * (t + 4) * sizeof(float) + (size_t)tp * (tp + 2) * sizeof(int16_t);
#define HBFP_TILE(PLANES, FAST)                                                                                               \
    do {                                                                                                                      \
        rc = allow_shared<tile_kernel<MODE, PLANES, FAST>>(128 * 132 * sizeof(float) + 128 * 130 * sizeof(int16_t));          \
        if (rc) return rc;                                                                                                    \
        launch_streamed(tile_bytes<MODE>(d0, d1), tile_kernel<MODE, PLANES, FAST>, grid_dim, 256, smem, st, src, ld, d0, d1, t, tp, p, wide, grid, nv, tv); \
    } while (0)
        if (L0.planes == 1) { if (fast) HBFP_TILE(1, true); else HBFP_TILE(1, false); }
        else { if (fast) HBFP_TILE(2, true); else HBFP_TILE(2, false); }
#undef HBFP_TILE
        return launch_status();
    }
    // Strips of 64 or 96 columns (whichever the tiles fill better) and up to 64 rows, 128 x 128 for tiles above 64.
    StripShape sh{t, tp, tp == 32 ? 5 : tp == 64 ? 6 : 7, 1, t <= 8 ? 3 : t <= 16 ? 2 : t <= 32 ? 1 : 0, 0, (65536 + t - 1) / t, 0, (int)nu, (int)nv};
    const int warps = t > 64 ? 16 : 8;
    auto warp_rows = [&]() { return (t + (warps >> sh.lg_rv) - 1) / (warps >> sh.lg_rv); };
    if (t <= 64) {
        const int cv2 = std::min(64 / t, 160 / tp), cv3 = std::min(96 / t, 160 / tp);
        sh.cv = warp_rows() <= 6 && 2 * cv3 > 3 * cv2 ? cv3 : cv2;
        // smaller ones where these leave SMs idle
        auto strips = [&]() { return ((nu + (1 << sh.lg_rv) - 1) >> sh.lg_rv) * ((nv + sh.cv - 1) / sh.cv); };
        while (strips() < 148 && (sh.lg_rv > 0 || sh.cv > 1)) {
            if (sh.lg_rv > 0 && ((1 << sh.lg_rv) >= sh.cv || sh.cv == 1)) --sh.lg_rv;
            else sh.cv = (sh.cv + 1) / 2;
        }
    }
    sh.rpw = warp_rows();
    const int kc = t > 64 ? 4 : sh.cv * t > 64 ? 3 : 2;
    const int rv = 1 << sh.lg_rv, rows = kc == 3 ? 6 : 8, per = sh.cv * tp / 8;
    sh.recip_per = ((1 << 20) + per - 1) / per;
    if (nv >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    const dim3 strips((unsigned)((nv + sh.cv - 1) / sh.cv), (unsigned)((nu + rv - 1) / rv));
    const size_t smem = (size_t)rv * tp * (sh.cv * tp + 8) * 2 + (p.rounding && MODE != 2 ? (size_t)warps * rows * (4 * kc + 1) * 16 : 0);
#define HBFP_STRIP(PLANES, NW, RPW, KC, SRV)                                                                                                      \
    do {                                                                                                                                          \
        rc = allow_shared<tile_strip_kernel<MODE, PLANES, NW, RPW, KC, SRV>>(96 * 1024);       /* eight tile rows of five tiles of 8 with draws: 93 KB */     \
        if (rc) return rc;                                                                                                                        \
        launch_streamed_long(tile_bytes<MODE>(d0, d1), tile_strip_kernel<MODE, PLANES, NW, RPW, KC, SRV>, strips, 32 * NW, smem, st, src, ld, d0, d1, sh, p, wide, grid, nv, tv);  \
    } while (0)
#define HBFP_STRIP_SR(PLANES, NW, RPW, KC) do { if (p.rounding && MODE != 2) HBFP_STRIP(PLANES, NW, RPW, KC, MODE != 2); else HBFP_STRIP(PLANES, NW, RPW, KC, false); } while (0)
#define HBFP_STRIP_KC(PLANES) do { if (kc == 2) HBFP_STRIP_SR(PLANES, 8, 8, 2); else if (kc == 3) HBFP_STRIP_SR(PLANES, 8, 6, 3); else HBFP_STRIP_SR(PLANES, 16, 8, 4); } while (0)
    if (L0.planes == 1) HBFP_STRIP_KC(1); else HBFP_STRIP_KC(2);
#undef HBFP_STRIP_KC
#undef HBFP_STRIP_SR
#undef HBFP_STRIP
    return launch_status();
}

}  // namespace

int launch_quantize_tiles(const float* w, int64_t d0, int64_t d1, int64_t ld, const hbfp_format* f,
                          int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                          int8_t* tile_exps, cudaStream_t st) {
    return launch_tiles<3>(w, ld, d0, d1, f, nullptr, tile_exps, mant_c0, exps_c0, mant_c1, exps_c1, nullptr, 0, st);
}

// Convolution weights w [taps * c_in][c_out] with one exponent per (t input maps) x (t output maps) tile over
// all taps: view c0 (rows = c_out, k = taps * c_in) and / or view c1 (rows = taps * c_in, k = c_out).
int launch_quantize_conv_weights(const float* w, int64_t taps, int64_t c_in, int64_t c_out, int64_t ld,
                                 const hbfp_format* f, int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                                 int8_t* tile_exps, cudaStream_t st) {
    const int64_t t = f->tile;
    if (t <= 0 || f->block != t || taps <= 0 || c_in <= 0 || c_out <= 0) return HBFP_ERR_INVALID_ARG;
    if (c_in % t != 0) return HBFP_ERR_UNSUPPORTED;               // a K-block must not straddle two taps
    const int64_t d0 = taps * c_in, d1 = c_out, nu = c_in / t, nv = (c_out + t - 1) / t;
    const QParams p = make_params(f);
    if (nu * nv >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    Layout L[2];
    for (int axis = 0; axis < 2; ++axis) {
        int8_t* exps = axis == 0 ? exps_c0 : exps_c1;
        if (!(axis == 0 ? mant_c0 : mant_c1)) continue;
        int rc = make_layout(axis == 0 ? d1 : d0, axis == 0 ? d0 : d1, f, &L[axis]);
        if (rc) return rc;
        if (L[axis].rs != L[axis].rows) HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L[axis].exp_bytes, st));   // padding lines are zero
    }
    if (!mant_c0 && !mant_c1 && !tile_exps) return HBFP_OK;
    // few tiles: split each tile's rows over several CTAs, maxima merged in the head of a mantissa buffer (the
    // mantissa pass that follows overwrites it)
    int8_t* const scratch_buf = mant_c1 ? mant_c1 : mant_c0;
    const int64_t scratch_room = !scratch_buf ? 0 : (mant_c1 ? L[1].mant_bytes : L[0].mant_bytes);
    int64_t splits = (2 * 148 + nu * nv - 1) / (nu * nv);
    splits = std::min<int64_t>(splits, (taps * t + CONVW_THREADS / 32 - 1) / (CONVW_THREADS / 32));
    for (int pass = 0; pass < 2; ++pass) {
        uint32_t* amax = nullptr;
        if (splits > 1 && nu * nv * 4 <= scratch_room) amax = reinterpret_cast<uint32_t*>(scratch_buf);
        if (pass == 1 && !amax) break;
        if (pass == 0 && amax) HBFP_CUDA_OK(cudaMemsetAsync(amax, 0, (size_t)(nu * nv * 4), st));
        const dim3 grid((unsigned)(nu * nv), pass == 0 && amax ? (unsigned)splits : 1u);
        launch_chained(exps_conv_tiles, grid, CONVW_THREADS, 0, st, w, taps, c_in, c_out, ld, t, p, mant_c0 ? exps_c0 : nullptr,
                                                        mant_c0 ? L[0].rs : 0, mant_c1 ? exps_c1 : nullptr,
                                                        mant_c1 ? L[1].rs : 0, nu, nv, tile_exps, amax, pass == 1);
        if (launch_status()) return HBFP_ERR_CUDA;
    }
    for (int axis = 0; axis < 2; ++axis) {
        int8_t* mant = axis == 0 ? mant_c0 : mant_c1;
        const int8_t* exps = axis == 0 ? exps_c0 : exps_c1;
        if (!mant) continue;
        const Layout& A = L[axis];
        if (A.planes == 1)
            launch_chained(mant_generic<1>, blocks_for(A.rows * (A.kst / 4), 256), 256, 0, st, w, d1, A.rows, A.k, ld, axis, A.b, A.bp, A.nkb, p, exps, A.rs, mant, A.kst, A.plane_stride);
        else
            launch_chained(mant_generic<2>, blocks_for(A.rows * (A.kst / 4), 256), 256, 0, st, w, d1, A.rows, A.k, ld, axis, A.b, A.bp, A.nkb, p, exps, A.rs, mant, A.kst, A.plane_stride);
        if (launch_status()) return HBFP_ERR_CUDA;
    }
    return HBFP_OK;
}

int launch_wide(int mode, const float* src, int64_t ld, int64_t d0, int64_t d1, const hbfp_format* f,
                int16_t* wide, int8_t* wide_exps, int8_t* mant_c0, int8_t* exps_c0, int8_t* mant_c1, int8_t* exps_c1,
                float* value, int64_t ldv, cudaStream_t st) {
    if (mode == 0) return launch_tiles<0>(src, ld, d0, d1, f, wide, wide_exps, mant_c0, exps_c0, mant_c1, exps_c1, nullptr, 0, st);
    if (mode == 1 && value) return launch_tiles<4>(src, ld, d0, d1, f, wide, wide_exps, mant_c0, exps_c0, mant_c1, exps_c1, value, ldv, st);
    if (mode == 1) return launch_tiles<1>(src, ld, d0, d1, f, wide, wide_exps, mant_c0, exps_c0, mant_c1, exps_c1, nullptr, 0, st);
    return launch_tiles<2>(nullptr, d1, d0, d1, f, wide, wide_exps, mant_c0, exps_c0, mant_c1, exps_c1, nullptr, 0, st);
}

int launch_im2col_packed(const int8_t* xm, const int8_t* xe, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw,
                         int pad, const hbfp_format* f, int8_t* om, int8_t* oe, cudaStream_t st) {
    if (f->tile != 0 || f->block != c) return HBFP_ERR_INVALID_ARG;      // one block per pixel
    if (c > 128) return HBFP_ERR_UNSUPPORTED;
    const int64_t ho = h + 2 * pad - kh + 1, wo = w + 2 * pad - kw + 1;
    if (ho <= 0 || wo <= 0) return HBFP_ERR_INVALID_ARG;
    Layout Lx, Lo;
    int rc = make_layout(n * h * w, c, f, &Lx);
    if (rc) return rc;
    rc = make_layout(n * ho * wo, (int64_t)kh * kw * c, f, &Lo);
    if (rc) return rc;
    if (h > (1 << 20) || w > (1 << 20) || Lo.kst > (1ll << 30)) return HBFP_ERR_UNSUPPORTED;
    if (n == 0) return HBFP_OK;
    HBFP_CUDA_OK(cudaMemsetAsync(oe, 0, (size_t)Lo.exp_bytes, st));
    const int lg_bp = Lo.bp == 32 ? 5 : Lo.bp == 64 ? 6 : 7;
    if (kh * kw > IM2COL_MAX_TAPS || kh > 100 || kw > 100 || pad > 100) return HBFP_ERR_UNSUPPORTED;
    if (Lo.rows >= (1ll << 31) || Lx.rows >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    launch_chained(im2col_gather, blocks_for(Lo.rows, IM2COL_ROWS), 256, 0, st, xm, xe, (int)Lx.kst, Lx.plane_stride, (int)h, (int)w, (int)ho, (int)wo,
                                                                   kh, kw, pad, lg_bp, (int)Lo.planes, (uint32_t)Lo.rows, (int)Lo.kst,
                                                                   Lo.plane_stride, Lo.rs, om, oe);
    return launch_status();
}

int launch_im2col_cols(const float* x, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad,
                       const hbfp_format* f, int8_t* mant, int8_t* exps, cudaStream_t st) {
    if (f->tile != 0 || f->block <= 0) return HBFP_ERR_INVALID_ARG;
    const int64_t b = f->block;
    // Under stochastic rounding every entry takes the draw of the activation it is a copy of (its index in
    // x [n][h][w][c]): the matrix this operand is the conversion of never exists.
    // same-size output, blocks of whole image rows that do not straddle images
    if (2 * pad != kh - 1 || 2 * pad != kw - 1) return HBFP_ERR_UNSUPPORTED;
    if (!(b == 16 || b == 32 || b == 64 || b == 128) || b % w != 0 || w < 4 || (w & (w - 1)) != 0 || (h * w) % b != 0 ||
        c % 4 != 0 || (reinterpret_cast<uintptr_t>(x) & 15))
        return HBFP_ERR_UNSUPPORTED;
    Layout L;
    int rc = make_layout((int64_t)kh * kw * c, n * h * w, f, &L);
    if (rc) return rc;
    if (n == 0) return HBFP_OK;
    if (h > 32768 || c > 4096 || L.nkb >= (1ll << 31)) return HBFP_ERR_UNSUPPORTED;
    const size_t smem = (size_t)(b / w + kh - 1) * w * c * sizeof(float);
    constexpr int IM2COL_SMEM_MAX = 200 * 1024;
    if (smem > IM2COL_SMEM_MAX) return HBFP_ERR_UNSUPPORTED;
    const QParams p = make_params(f);
    if (L.rs != L.rows) HBFP_CUDA_OK(cudaMemsetAsync(exps, 0, (size_t)L.exp_bytes, st));
    if (L.kst != L.nkb * L.bp) HBFP_CUDA_OK(cudaMemsetAsync(mant, 0, (size_t)L.mant_bytes, st));     // row tails
    if (kw == 3 && b == 64 && w >= 8 && w <= 64 && (p.rounding == 0 || c % 8 == 0)) {
        const unsigned threads = (unsigned)std::min<int64_t>(192, round_up(kh * c, 32));
        const size_t table = p.rounding ? (size_t)(b / w + kh - 1) * w * c * 2 : 0;
#define HBFP_COLS3(PL, WV, SRV)                                                                                                      \
    do {                                                                                                                              \
        rc = allow_shared<im2col_cols3<PL, WV, SRV>>(IM2COL_SMEM_MAX / 2);          /* two bytes of draws for every four of values */    \
        if (rc) return rc;                                                                                                            \
        launch_streamed(4 * n * h * w * c, im2col_cols3<PL, WV, SRV>, (unsigned)L.nkb, threads, table, st, x, (int)h, (int)c, kh, pad, p, L.kst, L.plane_stride, L.rs, mant, exps); \
    } while (0)
#define HBFP_COLS3_SR(PL, WV) do { if (p.rounding) HBFP_COLS3(PL, WV, true); else HBFP_COLS3(PL, WV, false); } while (0)
#define HBFP_COLS3_W(PL) do { if (w == 8) HBFP_COLS3_SR(PL, 8); else if (w == 16) HBFP_COLS3_SR(PL, 16); else if (w == 32) HBFP_COLS3_SR(PL, 32); else HBFP_COLS3_SR(PL, 64); } while (0)
        if (L.planes == 1) HBFP_COLS3_W(1); else HBFP_COLS3_W(2);
#undef HBFP_COLS3_W
#undef HBFP_COLS3_SR
#undef HBFP_COLS3
        return launch_status();
    }
    int lg_w = 0;
    while ((1 << lg_w) < w) ++lg_w;
#define HBFP_COLS_LAUNCH2(PL, NPX, SRV)                                                                                       \
    do {                                                                                                                       \
        rc = allow_shared<im2col_cols<PL, NPX, SRV>>(IM2COL_SMEM_MAX);                                                          \
        if (rc) return rc;                                                                                                     \
        launch_streamed(4 * n * h * w * c, im2col_cols<PL, NPX, SRV>, (unsigned)L.nkb, 256, smem, st, x, (int)h, (int)w, lg_w, (int)c, kh, kw, pad, p, L.kst,     \
                                                                     L.plane_stride, L.rs, mant, exps);                        \
    } while (0)
#define HBFP_COLS_LAUNCH(PL, NPX)                                                 \
    do {                                                                          \
        if (p.rounding) HBFP_COLS_LAUNCH2(PL, NPX, true);                         \
        else HBFP_COLS_LAUNCH2(PL, NPX, false);                                   \
    } while (0)
    if (L.planes == 1) {
        if (b == 16) HBFP_COLS_LAUNCH(1, 4); else if (b == 32) HBFP_COLS_LAUNCH(1, 8); else if (b == 64) HBFP_COLS_LAUNCH(1, 16); else HBFP_COLS_LAUNCH(1, 32);
    } else {
        if (b == 16) HBFP_COLS_LAUNCH(2, 4); else if (b == 32) HBFP_COLS_LAUNCH(2, 8); else if (b == 64) HBFP_COLS_LAUNCH(2, 16); else HBFP_COLS_LAUNCH(2, 32);
    }
#undef HBFP_COLS_LAUNCH2
#undef HBFP_COLS_LAUNCH
    return launch_status();
}

int launch_conv_dgrad_filters(const Packed& c1, int taps, int64_t c_in, int64_t c_out, int t, int8_t* mant_out,
                              int8_t* exps_out, const Layout& Lo, cudaStream_t st) {
    if (c_in == 0) return HBFP_OK;
    if (Lo.rs != c_in) HBFP_CUDA_OK(cudaMemsetAsync(exps_out, 0, (size_t)Lo.exp_bytes, st));   // padding lines are zero
    const int64_t warps = c_in * taps;
    launch_chained(conv_dgrad_filters_kernel, blocks_for(warps * 32, 256), 256, 0, st, c1.mant, c1.exps, c1.L.kst, c1.L.plane_stride, c1.L.rs,
                                                                          taps, c_in, c_out, t, (int)c1.L.planes, mant_out, exps_out,
                                                                          Lo.kst, Lo.plane_stride, Lo.rs);
    return launch_status();
}

int launch_unpack(const Packed& p, int16_t* q, int8_t* s, cudaStream_t st) {
    const Layout& L = p.L;
    int64_t n = L.rows * (L.k > L.nkb ? L.k : L.nkb);
    if (n == 0) return HBFP_OK;
    launch_chained(unpack_kernel, blocks_for(n, 256), 256, 0, st, p.mant, p.exps, L.rows, L.k, L.b, L.bp, L.nkb, L.kst,
                                                     L.plane_stride, (int)L.planes, L.rs, q, s);
    return launch_status();
}

// Value of wide weight storage, Eq. 1: out[i][j] = q16[i][j] * 2^s16[i/t][j/t] (exact in binary32: 16-bit mantissas).
// Bound by its 6 bytes per weight. V = 4 weights of a row per access and four rows in flight per thread where the
// tile, the pitches and the bases are multiples of four (then the four share an exponent); one weight per access
// otherwise. A CTA covers 4 rows x (256 V) columns, so that no thread divides a linear index by the row length.
// One weight per thread with a 64-bit division each took 28.4 us for 1024 x 4096 weights (0.9 TB/s), this form 5.5 us; 437 and 63 us
// (6.4 TB/s) for 8192 x 8192.
template <int V>
__global__ void __launch_bounds__(256)
wide_dequant_kernel(const int16_t* __restrict__ wide, const int8_t* __restrict__ exps, int64_t d0, int64_t d1, int t,
                    int64_t tiles1, float* __restrict__ out, int64_t ldo) {
    chain_start();
    constexpr int ROWS = 4;
    const int64_t c = ((int64_t)blockIdx.x * 256 + threadIdx.x) * V;
    if (c >= d1) return;
    const int64_t tc = d1 < (1ll << 31) ? (int64_t)((uint32_t)c / (uint32_t)t) : c / t;
    for (int64_t r0 = (int64_t)blockIdx.y * ROWS; r0 < d0; r0 += (int64_t)gridDim.y * ROWS) {
        const int64_t tr = d0 < (1ll << 31) ? (int64_t)((uint32_t)r0 / (uint32_t)t) : r0 / t;
        const int r_in = (int)(r0 - tr * t);
        uint2 q[ROWS] = {};
        int e[ROWS] = {};
#pragma unroll
        for (int i = 0; i < ROWS; ++i)
            if (r0 + i < d0) {
                const int16_t* at = wide + (r0 + i) * d1 + c;
                if (V == 4) q[i] = *reinterpret_cast<const uint2*>(at);
                else q[i].x = (uint16_t)*at;
                // V = 4: tiles of whole groups of four rows, the four have one exponent
                e[i] = exps[(V == 4 ? tr : tr + (uint32_t)(r_in + i) / (uint32_t)t) * tiles1 + tc];
            }
#pragma unroll
        for (int i = 0; i < ROWS; ++i)
            if (r0 + i < d0) {
                const float sc = pow2f_stored(e[i]);
                float* to = out + (r0 + i) * ldo + c;
                const float2 a = wide_values(q[i].x, sc), b = wide_values(q[i].y, sc);
                if (V == 4) *reinterpret_cast<float4*>(to) = make_float4(a.x, a.y, b.x, b.y);
                else *to = a.x;
            }
    }
}

int launch_wide_dequantize(const int16_t* wide, const int8_t* exps, int64_t d0, int64_t d1, int tile, float* out,
                           int64_t ldo, cudaStream_t st) {
    if (d0 * d1 == 0) return HBFP_OK;
    const int64_t tiles1 = (d1 + tile - 1) / tile;
    const unsigned rows = (unsigned)std::min<int64_t>((d0 + 3) / 4, 65535);
    const bool vec = tile % 4 == 0 && d1 % 4 == 0 && ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(wide) & 7) == 0 &&
                     (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    if (vec) launch_streamed(2 * d0 * d1, wide_dequant_kernel<4>, dim3(blocks_for(d1, 1024), rows), 256, 0, st, wide, exps, d0, d1, tile, tiles1, out, ldo);
    else launch_streamed(2 * d0 * d1, wide_dequant_kernel<1>, dim3(blocks_for(d1, 256), rows), 256, 0, st, wide, exps, d0, d1, tile, tiles1, out, ldo);
    return launch_status();
}

int launch_dequantize(const Packed& p, float* out, int64_t ld, cudaStream_t st) {
    const Layout& L = p.L;
    if (L.rows * L.k == 0) return HBFP_OK;
    launch_streamed(L.planes * L.rows * L.k, dequant_kernel, blocks_for(L.rows * L.k, 256), 256, 0, st, p.mant, p.exps, L.rows, L.k, L.b, L.bp, L.kst,
                                                                 L.plane_stride, (int)L.planes, L.rs, out, ld);
    return launch_status();
}

#endif   // HBFP_QUANT_PART

}  // namespace hbfp
