// Arithmetic of the conversion (Sec. 4.1, Sec. 5.3) shared by the quantisers and by the GEMM kernels that convert an operand
// themselves: block exponent, rounding, draws, packing.
#pragma once

#include "common.cuh"
#include "tc_ptx.cuh"

namespace hbfp {
namespace {

// ------------------------------------------------------------------------------ arithmetic

struct QParams {
    int m;          // mantissa bits
    int qmax;       // 2^(m-1) - 1
    int exp_mode;
    int rounding;
    uint32_t key0, key1, stream_id;
    Placing at;     // of the launch
};

__device__ __forceinline__ uint32_t abs_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// Shared exponent (of the mantissa LSB) from the largest |x| of the block, given as its bit
// pattern: floor(log2 amax) + 1 is the biased exponent field minus 126.
__device__ __forceinline__ int block_exponent(uint32_t amax_bits, int m, int exp_mode) {
    int E = (int)(amax_bits >> 23);
    int e = E - 126;
    if (exp_mode == 1 && E != 0 && (amax_bits & 0x7fffffu) == 0u) e -= 1;
    int s = e - (m - 1);
    s = s < -63 ? -63 : s;
    return s > 127 ? 127 : s;
}

__device__ __forceinline__ float pow2f(int e) {   // 2^e for e in [-126, 127]
    return __uint_as_float((uint32_t)(e + 127) << 23);
}

__device__ __forceinline__ int clampq(int q, int qmax) { return max(-qmax, min(qmax, q)); }

// Bit pattern of max(m, |a|, |b|) for finite values, in one three-input instruction.
__device__ __forceinline__ uint32_t max3_abs_bits(uint32_t m, float a, float b) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(__uint_as_float(m)), "f"(fabsf(a)), "f"(fabsf(b)));
    return __float_as_uint(d);
}

// Stochastic rounding of two neighbours whose 16-bit draws are the halves of one word w: the
// floors of (Y + r) / 2^16 are the upper halfwords of the two sums, clamped as a signed pair.
// Returns the two mantissas as packed signed halfwords (element 0 in the low half).
__device__ __forceinline__ uint32_t round_sr_pair(float x0, float x1, float scale, uint32_t w, uint32_t qmax2, uint32_t nqmax2) {
    const int t0 = __float2int_rd(__fmul_rn(x0, scale)) + (int)(w & 0xFFFFu);
    const int t1 = __float2int_rd(__fmul_rn(x1, scale)) + (int)(w >> 16);
    const uint32_t h = __byte_perm((uint32_t)t0, (uint32_t)t1, 0x7632);
    return __vmaxs2(__vmins2(h, qmax2), nqmax2);
}

// The same for two values whose draws r0, r1 (16 bits each) come from different places.
__device__ __forceinline__ uint32_t round_sr_pair2(float x0, float x1, float scale, uint32_t r0, uint32_t r1, uint32_t qmax2, uint32_t nqmax2) {
    const int t0 = __float2int_rd(__fmul_rn(x0, scale)) + (int)r0;
    const int t1 = __float2int_rd(__fmul_rn(x1, scale)) + (int)r1;
    const uint32_t h = __byte_perm((uint32_t)t0, (uint32_t)t1, 0x7632);
    return __vmaxs2(__vmins2(h, qmax2), nqmax2);
}

// Nearest-even rounding of two values, clamped as a signed halfword pair (m <= 12: the unclamped
// value, at most 2^(m-1) in magnitude, fits a halfword). Adding 1.5 * 2^23 rounds the product (exact: a power of two) to the
// nearest even integer in the low bits of the sum: one FMA per value instead of a multiplication and a float-to-integer
// conversion, which runs at an eighth of the FMA rate.
__device__ __forceinline__ uint32_t round_rne_pair(float x0, float x1, float scale, uint32_t qmax2, uint32_t nqmax2) {
    const uint32_t q0 = __float_as_uint(__fmaf_rn(x0, scale, 12582912.0f)), q1 = __float_as_uint(__fmaf_rn(x1, scale, 12582912.0f));
    const uint32_t h = __byte_perm(q0, q1, 0x5410);
    return __vmaxs2(__vmins2(h, qmax2), nqmax2);
}

__device__ __forceinline__ uint32_t qmax_pair(int qmax) { return (uint32_t)qmax * 0x10001u; }
__device__ __forceinline__ uint32_t neg_qmax_pair(int qmax) { return ((uint32_t)(-qmax) & 0xFFFFu) * 0x10001u; }

// Bytes of the mantissa planes from two halfword pairs (four mantissas): the 8-bit plane, or for
// two planes (q = 16 hi + lo) bits 4..11 and bits 0..3 of every halfword.
template <int PLANES>
__device__ __forceinline__ void pack4(uint32_t h01, uint32_t h23, uint32_t& hi, uint32_t& lo) {
    if (PLANES == 1) {
        hi = __byte_perm(h01, h23, 0x6420);
        lo = 0;
    } else {
        hi = __byte_perm((h01 >> 4) & 0x00FF00FFu, (h23 >> 4) & 0x00FF00FFu, 0x6420);
        lo = __byte_perm(h01 & 0x000F000Fu, h23 & 0x000F000Fu, 0x6420);
    }
}

// Largest |x| of eight values, as a bit pattern.
__device__ __forceinline__ uint32_t amax8_bits(const float (&e8)[8]) {
    uint32_t am = 0;
#pragma unroll
    for (int j = 0; j < 8; j += 2) am = max3_abs_bits(am, e8[j], e8[j + 1]);
    return am;
}

// Rounds eight consecutive values that share the exponent s (w: their eight 16-bit draws in
// stochastic mode) and packs the plane(s), eight bytes each.
template <bool SR, int PLANES>
__device__ __forceinline__ void quantize_pack8(const float (&e8)[8], int s, const QParams& p, uint4 w, uint2& hi, uint2& lo) {
    const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
    const float sc = pow2f(SR ? 16 - s : -s);
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
    uint32_t h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        h[j] = SR ? round_sr_pair(e8[2 * j], e8[2 * j + 1], sc, ww[j], qm, nqm) : round_rne_pair(e8[2 * j], e8[2 * j + 1], sc, qm, nqm);
    pack4<PLANES>(h[0], h[1], hi.x, lo.x);
    pack4<PLANES>(h[2], h[3], hi.y, lo.y);
}

// ---- Output kinds. 1 and 2: the packed layout with one or two mantissa planes. The others are the operand forms of gemm_fp.cu,
// rows of kst two-byte elements: FORM_SCALED bfloat16 q * 2^s, FORM_WIDE_A binary16 q, FORM_WIDE_B binary16 h and l with
// q = 64 h + l (two planes plane_stride elements apart); the wide forms keep 2^s as floats in place of the exponents.
// Writing the form here instead of expanding packed operands saves a pass over both: 1024 x 4096 x 4096 backward-weight, b = 32,
// 94 -> 77 us; 4096 cube with 12 bits 354 -> 326 us; 1111 x 777 x 3001, b = 24, 65 -> 56 us.
constexpr int FORM_SCALED = 3, FORM_WIDE_A = 4, FORM_WIDE_B = 5;
__host__ __device__ constexpr bool is_form(int out) { return out >= FORM_SCALED; }
// what the row and column kernels need beside the packed case
struct FormArgs {
    int32_t* status;      // FORM_WIDE_A: exponents beyond the GEMM's exact range are reported here
};

// Two rounded values (packed signed halfwords) as the form's elements: a (and for FORM_WIDE_B b) hold two elements each.
template <int OUT>
__device__ __forceinline__ void form_pair(uint32_t h, float two_s, uint32_t& a, uint32_t& b) {
    // halfword + 2^15 in the low bits of 2^23: no integer-to-float conversion
    const uint32_t u = h ^ 0x80008000u;
    float f0 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7610)) - 8421376.0f;
    float f1 = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7632)) - 8421376.0f;
    if (OUT == FORM_SCALED) {
        a = __byte_perm(__float_as_uint(f0 * two_s), __float_as_uint(f1 * two_s), 0x7632);      // exact: the low halves are zero
        b = 0;
    } else {
        float l0 = 0.f, l1 = 0.f;
        if (OUT == FORM_WIDE_B) {
            const float h0 = __fmaf_rn(f0, 0.015625f, 12582912.0f) - 12582912.0f, h1 = __fmaf_rn(f1, 0.015625f, 12582912.0f) - 12582912.0f;
            l0 = __fmaf_rn(-64.0f, h0, f0);                                                       // in [-32, 32]
            l1 = __fmaf_rn(-64.0f, h1, f1);
            f0 = h0; f1 = h1;
        }
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(a) : "f"(f1), "f"(f0));
        if (OUT == FORM_WIDE_B) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(b) : "f"(l1), "f"(l0));
        else b = 0;
    }
}
// Eight consecutive values with the exponent s: sixteen bytes of the form (two planes for FORM_WIDE_B).
template <bool SR, int OUT>
__device__ __forceinline__ void quantize_form8(const float (&e8)[8], int s, const QParams& p, uint4 w, uint4& a, uint4& b) {
    const uint32_t qm = qmax_pair(p.qmax), nqm = neg_qmax_pair(p.qmax);
    const float sc = pow2f(SR ? 16 - s : -s), two_s = pow2f(s);
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
    uint32_t ra[4], rb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t h = SR ? round_sr_pair(e8[2 * j], e8[2 * j + 1], sc, ww[j], qm, nqm) : round_rne_pair(e8[2 * j], e8[2 * j + 1], sc, qm, nqm);
        form_pair<OUT>(h, two_s, ra[j], rb[j]);
    }
    a = make_uint4(ra[0], ra[1], ra[2], ra[3]);
    b = make_uint4(rb[0], rb[1], rb[2], rb[3]);
}
// The exponent (packed), nothing (FORM_SCALED) or the scale of a block.
template <int OUT>
__device__ __forceinline__ void store_exponent(int8_t* exps, int64_t at, int s) {
    if (!is_form(OUT)) exps[at] = (int8_t)s;
    else if (OUT != FORM_SCALED) reinterpret_cast<float*>(exps)[at] = pow2f(s);
}
// Eight consecutive elements at element offset `at` of the row-major result.
template <bool SR, int OUT>
__device__ __forceinline__ void round_and_store8(const float (&e8)[8], int s, const QParams& p, uint4 w, int8_t* mant, int64_t at, int64_t plane_stride, bool store) {
    if constexpr (is_form(OUT)) {
        uint4 a, b;
        quantize_form8<SR, OUT>(e8, s, p, w, a, b);
        if (store) {
            *reinterpret_cast<uint4*>(mant + 2 * at) = a;
            if (OUT == FORM_WIDE_B) *reinterpret_cast<uint4*>(mant + 2 * (at + plane_stride)) = b;
        }
    } else {
        uint2 hi, lo;
        quantize_pack8<SR, OUT>(e8, s, p, w, hi, lo);
        if (store) {
            *reinterpret_cast<uint2*>(mant + at) = hi;
            if (OUT == 2) *reinterpret_cast<uint2*>(mant + plane_stride + at) = lo;
        }
    }
}
// Eight zero elements there.
template <int OUT>
__device__ __forceinline__ void store_zero8(int8_t* mant, int64_t at, int64_t plane_stride) {
    if constexpr (is_form(OUT)) {
        *reinterpret_cast<uint4*>(mant + 2 * at) = make_uint4(0u, 0u, 0u, 0u);
        if (OUT == FORM_WIDE_B) *reinterpret_cast<uint4*>(mant + 2 * (at + plane_stride)) = make_uint4(0u, 0u, 0u, 0u);
    } else {
        *reinterpret_cast<uint2*>(mant + at) = make_uint2(0u, 0u);
        if (OUT == 2) *reinterpret_cast<uint2*>(mant + plane_stride + at) = make_uint2(0u, 0u);
    }
}
template <int OUT>
__device__ __forceinline__ void check_exponent(int s, const FormArgs& fa) {
    if (OUT == FORM_WIDE_A && s > 96) atomicCAS(fa.status, 0, STATUS_EXPONENT_RANGE);
}

// round-half-even( x * 2^-s ), saturated
__device__ __forceinline__ int round_rne(float x, int s, int qmax) {
    float y = __fmul_rn(x, pow2f(-s));           // s >= -63 and s <= 126 for finite input, m >= 3
    return clampq(__float2int_rn(y), qmax);
}

// stochastic: floor( (floor(fl32(x * 2^(16-s))) + r) / 2^16 ), saturated
__device__ __forceinline__ int round_sr(float x, int s, int qmax, uint32_t r) {
    float y = __fmul_rn(x, pow2f(16 - s));
    int Y = __float2int_rd(y);
    return clampq((Y + (int)r) >> 16, qmax);
}

// One whole 32-byte sector; p must be 32-byte aligned.
__device__ __forceinline__ void store_sector(int8_t* p, const uint32_t* w) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]),
                 "r"(w[6]), "r"(w[7]) : "memory");
}

// Philox4x32-10 (Salmon et al., SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint4 draws_of_group(const QParams& p, uint64_t g) {
    return philox4x32_10((uint32_t)g, (uint32_t)(g >> 32), p.stream_id, 0u, p.key0, p.key1);
}

// The draws of eight consecutive elements from index L on: they may straddle two Philox groups, the second call is made only then.
__device__ __forceinline__ uint4 draws_of_eight(const QParams& p, uint64_t L) {
    uint4 w = draws_of_group(p, L >> 3);
    const uint32_t sh = (uint32_t)(L & 7);
    if (sh) {
        // halfwords sh .. sh + 7 of the two groups
        const uint4 n4 = draws_of_group(p, (L >> 3) + 1);
        const uint32_t a[8] = {w.x, w.y, w.z, w.w, n4.x, n4.y, n4.z, n4.w};
        const uint32_t ws = sh >> 1;
        uint32_t t[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) t[j] = ws == 0 ? a[j] : ws == 1 ? a[(j + 1) & 7] : ws == 2 ? a[(j + 2) & 7] : a[(j + 3) & 7];
        if (sh & 1) w = make_uint4(__funnelshift_r(t[0], t[1], 16), __funnelshift_r(t[1], t[2], 16), __funnelshift_r(t[2], t[3], 16), __funnelshift_r(t[3], t[4], 16));
        else w = make_uint4(t[0], t[1], t[2], t[3]);
    }
    return w;
}

__device__ __forceinline__ uint32_t draw_from(uint4 w, uint32_t lane8) {   // lane8 = L & 7
    uint32_t word = (lane8 >> 1) == 0 ? w.x : (lane8 >> 1) == 1 ? w.y : (lane8 >> 1) == 2 ? w.z : w.w;
    return (word >> (16u * (lane8 & 1u))) & 0xFFFFu;
}

__device__ __forceinline__ uint32_t draw_of_element(const QParams& p, uint64_t L) {
    return draw_from(draws_of_group(p, L >> 3), (uint32_t)(L & 7));
}

__device__ __forceinline__ int quantize_one(float x, int s, const QParams& p, uint64_t L) {
    if (p.rounding == 0) return round_rne(x, s, p.qmax);
    return round_sr(x, s, p.qmax, draw_of_element(p, L));
}

// Exponent bytes of the lines beyond the matrix (rows .. rs of every block, at most fifteen) are documented as zero: written by all
// CTAs, sixteen threads per block. (By the first CTA alone a 57 x 52416 operand's 11 000 bytes took 4 us.)
__device__ __forceinline__ void zero_padding_lines(int8_t* exps, int64_t rows, int64_t rs, int64_t nkb) {
    if (rs == rows) return;
    const int64_t line = rows + (threadIdx.x & 15);
    if (line >= rs) return;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 4);
    for (int64_t kb = (int64_t)blockIdx.x * (blockDim.x >> 4) + (threadIdx.x >> 4); kb < nkb; kb += step) exps[kb * rs + line] = 0;
}

QParams make_params(const hbfp_format* f) {
    QParams p;
    p.m = f->mant_bits;
    p.qmax = (1 << (f->mant_bits - 1)) - 1;
    p.exp_mode = f->exp_mode;
    p.rounding = f->rounding;
    p.key0 = (uint32_t)f->seed;
    p.key1 = (uint32_t)(f->seed >> 32);
    p.stream_id = f->stream_id;
    p.at = Placing{};
    return p;
}

}  // namespace
}  // namespace hbfp
