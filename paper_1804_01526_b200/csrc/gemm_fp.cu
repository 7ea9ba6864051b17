// Tensor-core BFP GEMM on floating-point operand forms, for sm_100a: short blocks of 8-bit mantissas, and 9 to 12 bits.
//
// What bounds the integer kernels (gemm_tc.cu, gemm_tc2.cu) when blocks are short is not the MMA but the rescale: per
// K-block every output word needs an integer-to-float step, a row scale, a column scale and the tables that hold them,
// about 1000 cycles per 128 x 256 words whatever the block's length. Here the operands carry the scale instead:
//   form S (mantissas of at most 8 bits): every element is bfloat16 q * 2^s. q has 7 magnitude bits, so the value is
//     exact; every product of a block is a multiple of 2^(sA + sB) and their sum less than 2^24 multiples, so the MMAs
//     (kind::f16, FP32 accumulator) of ONE K-block leave exactly P * 2^(sA + sB) of Eq. 2 in tensor memory. What is left
//     of the rescale is one FP32 addition per word, the one rounding the definition allows: no tables, no conversion.
//   form W (9 to 12 bits): q fits binary16. The B operand is split q = 64 h + l (|h|, |l| <= 32) into two binary16
//     planes stacked along N, so that both partial sums of a block stay below 2^24 and are exact;
//     t = fma(H, 64 * 2^sA, L * 2^sA) is the one rounding of float(P), acc = fma(t, 2^sB, acc) the one of the sum.
//     Against three int8 parts (256 hi.hi + 16 mid + lo.lo): two tensor-memory words per output instead of three, three
//     packed operations instead of five, and nothing is written back.
// The blocks are added in ascending order, one rounding each: bit for bit the sequential definition when K is not split.
// bf16 MMAs run at half the int8 rate, so blocks of 128 at 8 bits stay with the integer kernels.
//
// One CTA per SM, persistent: warp 0 TMA producer, warp 1 MMA issuer and owner of tensor memory, warps 4-11 rescale (two
// per lane quarter, FP32 accumulators in registers). A K-block's MMAs overwrite one of two accumulator groups of 256
// columns (form W: 128 outputs, h and l); four groups of 128 columns were measured and are no faster. PAIR: two CTAs of a
// cluster compute a tile of 256 rows with cta_group::2 MMAs (plan_gemm_fp says when). Small outputs split K over the CTAs of a cluster: every CTA leaves its partial tile in shared memory and adds up a share of the rows over
// the cluster in ascending order - deterministic, no scratch, no second launch.
// Every wait is bounded (tc_ptx.cuh). No load is multicast.
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace hbfp {
namespace {

constexpr int FP_CONTROL_WARPS = 4, FP_PRODUCER_WARP = 0, FP_MMA_WARP = 1, FP_RW = 8;
constexpr int FP_THREADS = 32 * (FP_CONTROL_WARPS + FP_RW);
constexpr int FP_STAGE_ELEMS = 64;            // K elements per stage: one 128-byte swizzle row of 2-byte elements
constexpr int FORM_S = 0, FORM_W = 1;
// register split: totals stay inside 384 threads x 168 registers
constexpr int FP_REGS_RESCALE = 216, FP_REGS_CONTROL = 72;
static_assert(128 * FP_REGS_CONTROL + 32 * FP_RW * FP_REGS_RESCALE <= FP_THREADS * 168, "register split");

template <int FORM, int NCOL, int BP, bool PAIR>
struct FpCfg {
    static constexpr int NOUT = FORM == FORM_W ? NCOL / 2 : NCOL;      // output columns of a tile
    static constexpr int GROUPS = TMEM_COLS / NCOL > 4 ? 4 : TMEM_COLS / NCOL;   // accumulator groups
    static constexpr int NC = NOUT / 2;                                // output columns of a rescale warp
    static constexpr int CH = FORM == FORM_W ? 16 : (NC < 32 ? NC : 32);         // columns per tensor-memory read
    static constexpr int BPS = FP_STAGE_ELEMS / BP;                    // K-blocks per stage
    static constexpr int STEPS = BP / 16;                              // MMA steps per block
    static constexpr int A_BYTES = TILE_M * 128;
    static constexpr int B_ROWS = PAIR ? NCOL / 2 : NCOL;              // rows of B that a CTA stages
    static constexpr int STAGE = A_BYTES + B_ROWS * 128;
    // Form S leaves through one 32 x 32 FP32 box per rescale warp; form W stores from registers, its stages need the room.
    static constexpr int OUT_BYTES = FORM == FORM_S ? FP_RW * 4096 : 0;
    static constexpr int SC_SLOT = FORM == FORM_W ? 4 * BPS * (TILE_M + NOUT) : 0;   // scales of the blocks of a stage
    static constexpr int STAGES_RAW = (232448 - 2048 - OUT_BYTES - GROUPS * SC_SLOT) / (STAGE + SC_SLOT);
    static constexpr int STAGES = STAGES_RAW > 8 ? 8 : STAGES_RAW;
    // Scales arrive once per stage. A slot is overwritten SC_DEPTH stages later, when the MMAs of a block at least
    // SC_DEPTH - STAGES stages after the slot's have completed; those were issued only after every rescale warp had
    // handed back the group GROUPS blocks before, which it does after its last look at that block's scales.
    static constexpr int SC_DEPTH = FORM == FORM_W ? STAGES + GROUPS : 1;
    static constexpr int SMEM = 1024 + STAGES * STAGE + OUT_BYTES + (FORM == FORM_W ? SC_DEPTH * SC_SLOT : 0) + 1024;
    static_assert(STAGES >= 3 && SMEM <= 232448, "shared memory");
    static_assert(PAIR || STAGES * STAGE >= TILE_M * (NOUT + 4) * 4, "the partial tile of a split fits the stages");
};

struct FpProblem {
    int M, N, nkb;
    int tiles_m, tiles_n;
    int splits, kb_per_split;     // splits > 1: the CTAs of a cluster share a tile
    int tma_out;                  // C leaves through TMA stores (16-byte aligned, pitch of whole quads)
    const float* bias;            // may be null
    float* C;
    int64_t ldc;
    int32_t* status;
};

struct FpWork { int m0, n0; };

// Groups of tile rows (2048 matrix rows) sweep across N, so that their B panels are shared in L2.
template <int TM, int NOUT>
__device__ __forceinline__ FpWork fp_work(const FpProblem& p, int t) {
    constexpr int G = 2048 / TM;
    const int per_group = G * p.tiles_n;
    const int group = t / per_group, first_m = group * G;
    const int gsize = min(G, p.tiles_m - first_m), within = t - group * per_group;
    const int nt = within / gsize;
    return {(first_m + (within - nt * gsize)) * TM, nt * NOUT};
}

// ------------------------------------------------------------------------------ PTX

__device__ __forceinline__ uint32_t fp_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t fp_clusterid() { uint32_t r; asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t fp_map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void fp_cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Bounded wait of a single thread: prompt tries first.
__device__ __forceinline__ bool fp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status, int code) {
    for (int i = 0; i < 256; ++i)
        if (mbar_try(bar, parity)) return true;
    return mbar_wait(bar, parity, abort_flag, status, code);
}
__device__ __forceinline__ uint32_t fp_nclusters() { uint32_t r; asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r)); return r; }
// Tile copy of one CTA of a pair whose completion bytes are counted on a barrier of either CTA (a cluster address).
__device__ __forceinline__ void fp_tma_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar, uint64_t hint) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "l"(hint) : "memory");
}
constexpr uint64_t FP_L2_NORMAL = 0x1000000000000000ull;
// Arrives, once the MMAs issued so far have completed, on the barrier at this offset (PAIR: of the CTAs in the mask).
template <bool PAIR>
__device__ __forceinline__ void fp_commit(uint32_t bar, uint16_t mask = 3) {
    if (PAIR) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(mask) : "memory");
    else tc_commit(bar);
}
template <bool PAIR>
__device__ __forceinline__ void fp_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    if (PAIR)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// FP32 accumulator, K-major operands: bfloat16 (form S) or binary16 (form W).
template <int FORM, int NCOL, bool PAIR>
__device__ __forceinline__ constexpr uint32_t fp_idesc() {
    return (1u << 4) | (FORM == FORM_S ? ((1u << 7) | (1u << 10)) : 0u) | ((uint32_t)(NCOL >> 3) << 17) | ((uint32_t)((PAIR ? 2 * TILE_M : TILE_M) >> 4) << 24);
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
template <int N>
__device__ __forceinline__ void fp_next(uint32_t& i, uint32_t& ph) {
    if (++i == N) { i = 0; ph ^= 1u; }
}

// ------------------------------------------------------------------------------ rescale

struct FpRescale {
    uint32_t tfull_bar, tempty_bar, sfull_bar, tmem_base;     // tempty_bar: a cluster address, the leader's, with PAIR
    const float* scales;          // scale ring (form W): per slot [BPS][128 row scales], then [BPS][NOUT column scales]
    volatile int* abort_flag;
};
struct FpRing { uint32_t g, gph, sc, scph; };

// The K-blocks of one work item into acc2 (output columns [col0, col0 + NC) of this warp's rows). Ring positions are
// carried across items. Returns false when a wait was abandoned.
template <bool PAIR>
__device__ __forceinline__ void fp_hand_back(uint32_t bar) {
    if (PAIR) mbar_arrive_cluster_elect(bar); else mbar_arrive_elect(bar);
}
template <int FORM, int NCOL, int BP, bool PAIR>
__device__ __forceinline__ bool fp_blocks(uint64_t (&acc2)[FpCfg<FORM, NCOL, BP, PAIR>::NC / 2], const FpProblem& p, const FpRescale& a, int nblk, int col0, FpRing& r) {
    using C = FpCfg<FORM, NCOL, BP, PAIR>;
    constexpr int CH = C::CH, NCHK = C::NC / CH;
    const int lane = threadIdx.x & 31, quarter = (threadIdx.x >> 5) & 3;
    const uint32_t lane_addr = a.tmem_base + ((uint32_t)(quarter * 32) << 16) + col0;
    for (int kb = 0; kb < nblk; ++kb) {
        const uint32_t taddr = lane_addr + r.g * NCOL;
        const int jb = C::BPS > 1 ? kb % C::BPS : 0;
        if (!mbar_wait_warp_fast(a.tfull_bar + 8 * r.g, r.gph, a.abort_flag, p.status, 342)) return false;
        tc_fence_after();
        if constexpr (FORM == FORM_S) {
            uint32_t v[2][CH];
            tc_ldn(taddr, v[0]);
#pragma unroll
            for (int ch = 0; ch < NCHK; ++ch) {
                tc_wait_ld();
                if (ch + 1 < NCHK) {
                    tc_ldn(taddr + (ch + 1) * CH, v[(ch + 1) & 1]);
                } else {
                    tc_fence_before();
                    fp_hand_back<PAIR>(a.tempty_bar + 8 * r.g);
                }
                const uint32_t(&x)[CH] = v[ch & 1];
#pragma unroll
                for (int q = 0; q < CH; q += 2) acc2[(ch * CH + q) / 2] = fadd2(acc2[(ch * CH + q) / 2], pack2(x[q], x[q + 1]));
            }
        } else {
            uint32_t vh[2][CH], vl[2][CH];
            tc_ldn(taddr, vh[0]);
            tc_ldn(taddr + C::NOUT, vl[0]);
            if (jb == 0 && !mbar_wait_warp_fast(a.sfull_bar + 8 * r.sc, r.scph, a.abort_flag, p.status, 343)) return false;
            const float* slot = a.scales + r.sc * (C::SC_SLOT / 4);
            const float sa = slot[jb * TILE_M + quarter * 32 + lane], sa64 = 64.0f * sa;
            const uint64_t sa2 = pack2(__float_as_uint(sa), __float_as_uint(sa)), sh2 = pack2(__float_as_uint(sa64), __float_as_uint(sa64));
            const uint32_t tab = smem_u32(slot + C::BPS * TILE_M + jb * C::NOUT + col0);
#pragma unroll
            for (int ch = 0; ch < NCHK; ++ch) {
                uint64_t sb[CH / 2];
#pragma unroll
                for (int q = 0; q < CH; q += 2)
                    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(sb[q / 2]) : "r"(tab + 4u * (uint32_t)(ch * CH + q)));
                tc_wait_ld();
                if (ch + 1 < NCHK) {
                    tc_ldn(taddr + (ch + 1) * CH, vh[(ch + 1) & 1]);
                    tc_ldn(taddr + C::NOUT + (ch + 1) * CH, vl[(ch + 1) & 1]);
                } else {
                    tc_fence_before();
                    fp_hand_back<PAIR>(a.tempty_bar + 8 * r.g);
                }
                const uint32_t(&h)[CH] = vh[ch & 1];
                const uint32_t(&l)[CH] = vl[ch & 1];
#pragma unroll
                for (int q = 0; q < CH; q += 2) {
                    const uint64_t t = ffma2(pack2(h[q], h[q + 1]), sh2, fmul2(pack2(l[q], l[q + 1]), sa2));
                    acc2[(ch * CH + q) / 2] = ffma2(t, sb[q / 2], acc2[(ch * CH + q) / 2]);
                }
            }
        }
        fp_next<C::GROUPS>(r.g, r.gph);
        if (FORM == FORM_W && (jb == C::BPS - 1 || kb == nblk - 1)) fp_next<C::SC_DEPTH>(r.sc, r.scph);
    }
    return true;
}

// Form S carries the scale in the operands, so that where sA + sB is above 107 single products or part sums can leave binary32
// although the block's sum, after cancellation, would not. An infinity stays one (or becomes a NaN) through every later addition:
// one look at the finished accumulators finds it (0 * x + 0 is 0 for finite x only).
template <int NC>
__device__ __forceinline__ bool fp_all_finite(const uint64_t (&acc2)[NC / 2]) {
    uint64_t t[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int c = 0; c < NC / 2; ++c) t[c & 3] = ffma2(acc2[c], 0ull, t[c & 3]);
    float lo, hi;
    unpack2(fadd2(fadd2(t[0], t[1]), fadd2(t[2], t[3])), lo, hi);
    return lo == 0.f && hi == 0.f;
}

// Stores the columns [gj0, gj0 + NC) of row gi: whole 32-byte sectors per lane where the pitch allows it.
template <int NC>
__device__ __forceinline__ void fp_store_rows(const uint64_t (&acc2)[NC / 2], const FpProblem& p, int gi, int gj0) {
    if (gi >= p.M) return;
    float* rowp = p.C + (int64_t)gi * p.ldc + gj0;
    const bool wide = (p.ldc & 7) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 31) == 0;
    const bool quad = (p.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
#pragma unroll
    for (int c = 0; c < NC; c += 8) {
        if (wide && gj0 + c + 7 < p.N) {
            st_global_256(rowp + c, acc2[c / 2], acc2[c / 2 + 1], acc2[c / 2 + 2], acc2[c / 2 + 3]);
        } else {
#pragma unroll
            for (int h = c; h < c + 8; h += 4) {
                if (quad && gj0 + h + 3 < p.N) {
                    *reinterpret_cast<ulonglong2*>(rowp + h) = make_ulonglong2(acc2[h / 2], acc2[h / 2 + 1]);
                } else {
                    float e4[4];
                    unpack2(acc2[h / 2], e4[0], e4[1]);
                    unpack2(acc2[h / 2 + 1], e4[2], e4[3]);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (gj0 + h + e < p.N) rowp[h + e] = e4[e];
                }
            }
        }
    }
}

// The bias of the columns [gj0, gj0 + NC): one more addition per output, after the last block. One load per 32 columns and
// shuffles: a load per column held up the end of every tile by 2400 cycles.
template <int NC>
__device__ __forceinline__ void fp_add_bias(uint64_t (&acc2)[NC / 2], const FpProblem& p, int gj0) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < NC; h += 32) {
        const int gj = gj0 + h + lane;
        const float mine = gj < p.N ? __ldg(p.bias + gj) : 0.f;
#pragma unroll
        for (int c = 0; c < 32; c += 2)
            acc2[(h + c) / 2] = fadd2(acc2[(h + c) / 2], pack2(__float_as_uint(__shfl_sync(0xffffffffu, mine, c)), __float_as_uint(__shfl_sync(0xffffffffu, mine, c + 1))));
    }
}

// Split-K parts of a tile, one per CTA of the cluster: every part goes to its CTA's shared memory (rows padded so that
// eight lanes' 16-byte stores hit all banks), then each CTA adds up a share of the rows over the cluster in ascending
// order of K. Runs in the rescale warps; called whether or not their waits succeeded, so that every barrier is met.
template <int NOUT, int NC, bool BIAS>
__device__ __forceinline__ void fp_split_sum(const uint64_t (&acc2)[NC / 2], const FpProblem& p, uint32_t base, unsigned char* base_ptr,
                                             const FpWork& w, int rank, int row, int col0) {
    constexpr int NT = 32 * FP_RW;
    // the stages were last written by the copy engine and read by MMAs that every warp has seen complete
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
    float* mine = reinterpret_cast<float*>(base_ptr) + row * (NOUT + 4) + col0;
#pragma unroll
    for (int c = 0; c < NC; c += 4) *reinterpret_cast<ulonglong2*>(mine + c) = make_ulonglong2(acc2[c / 2], acc2[c / 2 + 1]);
    __syncwarp();
    fp_cluster_barrier();
    constexpr int QPR = NOUT / 4, QUADS = TILE_M * QPR;
    const int tid = (int)threadIdx.x - 32 * FP_CONTROL_WARPS;
    const bool quad = (p.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
    for (int i = rank * NT + tid; i < QUADS; i += p.splits * NT) {
        const int r = i / QPR, q4 = (i - r * QPR) * 4;
        const int gi = w.m0 + r, gj = w.n0 + q4;
        if (gi >= p.M || gj >= p.N) continue;
        const uint32_t at = base + 4u * (uint32_t)(r * (NOUT + 4) + q4);
        float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int sp = 0; sp < p.splits; ++sp) {
            float y[4];
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(y[0]), "=f"(y[1]), "=f"(y[2]), "=f"(y[3]) : "r"(fp_map_rank(at, (uint32_t)sp)) : "memory");
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = sp == 0 ? y[e] : __fadd_rn(x[e], y[e]);
        }
        if constexpr (BIAS)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (gj + e < p.N) x[e] = __fadd_rn(x[e], __ldg(p.bias + gj + e));
        float* dst = p.C + (int64_t)gi * p.ldc + gj;
        if (quad && gj + 3 < p.N) *reinterpret_cast<float4*>(dst) = make_float4(x[0], x[1], x[2], x[3]);
        else
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (gj + e < p.N) dst[e] = x[e];
    }
}

// ------------------------------------------------------------------------------ kernel

// BIAS is a parameter of the kernel and not a run-time branch: the branch alone cost the 12-bit kernel 4 % (222 -> 232 us, 4096 cube).
template <int FORM, int NCOL, int BP, bool PAIR, bool BIAS>
__global__ void __launch_bounds__(FP_THREADS, 1)
gemm_fp_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapB1,
               const __grid_constant__ CUtensorMap mapSA, const __grid_constant__ CUtensorMap mapSB,
               const __grid_constant__ CUtensorMap mapC, const FpProblem p) {
    using C = FpCfg<FORM, NCOL, BP, PAIR>;
    constexpr int STAGES = C::STAGES, GROUPS = C::GROUPS;
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
    constexpr uint32_t out_off = STAGES * C::STAGE;
    constexpr uint32_t sc_off = out_off + C::OUT_BYTES;
    constexpr uint32_t bar_off = sc_off + (FORM == FORM_W ? C::SC_DEPTH * C::SC_SLOT : 0);
    const uint32_t full_bar = base + bar_off;                 // operand tiles landed
    const uint32_t empty_bar = full_bar + 8 * STAGES;         // stage consumed
    const uint32_t tfull_bar = empty_bar + 8 * STAGES;        // block sums complete (MMA commit)
    const uint32_t tempty_bar = tfull_bar + 8 * GROUPS;       // group read by every rescale warp
    const uint32_t done_bar = tempty_bar + 8 * GROUPS;
    const uint32_t sfull_bar = done_bar + 8;                  // scales landed (form W)
    constexpr int BAR_BYTES = 16 * STAGES + 16 * GROUPS + 8 + 8 * C::SC_DEPTH;
    static_assert(BAR_BYTES + 8 <= 1024, "barrier area");
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + bar_off + BAR_BYTES);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int TM = PAIR ? 2 * TILE_M : TILE_M;
    const bool split = !PAIR && p.splits > 1;
    const int rank = PAIR || split ? (int)fp_ctarank() : 0;                       // PAIR: 0 is the leader
    const int first = PAIR || split ? (int)fp_clusterid() : (int)blockIdx.x;
    const int tiles = p.tiles_m * p.tiles_n, step = PAIR ? (int)fp_nclusters() : split ? tiles : (int)gridDim.x;     // split: a cluster has one tile
    const int kb0 = PAIR ? 0 : rank * p.kb_per_split;
    const int nblk = min(p.nkb - kb0, p.kb_per_split);        // at least one: the host sizes the splits
    const int nst = (nblk + C::BPS - 1) / C::BPS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar + 8 * s, 1);
            mbar_init(empty_bar + 8 * s, 1);
        }
        for (int g = 0; g < GROUPS; ++g) {
            mbar_init(tfull_bar + 8 * g, 1);
            mbar_init(tempty_bar + 8 * g, (PAIR ? 2 : 1) * FP_RW);
        }
        mbar_init(done_bar, 1);
        for (int i = 0; i < C::SC_DEPTH; ++i) mbar_init(sfull_bar + 8 * i, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == FP_MMA_WARP) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) fp_cluster_barrier();            // both CTAs' barriers and tensor memory exist before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_start();

    if (warp < FP_CONTROL_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FP_REGS_CONTROL));
        if (warp == FP_PRODUCER_WARP) {
            // -------------------------------------------------------------- TMA producer
            if (elect_one()) {
                const uint32_t full_addr = PAIR ? fp_map_rank(full_bar, 0) : full_bar;
                uint32_t s = 0, ph = 0, sc = 0, scph = 0, it = 0, nsc = 0;
                bool ok = true;
                for (int t = first; ok && t < tiles; t += step) {
                    const FpWork w = fp_work<TM, C::NOUT>(p, t);
                    const int my_m = w.m0 + (PAIR ? rank * TILE_M : 0);
                    int kbyte = kb0 * BP * 2, kb = kb0;
                    for (int si = 0; si < nst; ++si, kbyte += 128, ++it) {
                        if (!fp_wait(empty_bar + 8 * s, ph ^ 1, abort_flag, p.status, 141)) { ok = false; break; }
                        const uint32_t ms = base + s * C::STAGE;
                        if (PAIR) {
                            // both CTAs' tiles are counted on the leader's barrier; form S: each CTA stages half of the rows
                            // of B, form W: the leader the h plane and the other the l plane
                            if (rank == 0) mbar_expect_tx(full_bar + 8 * s, 2u * C::STAGE);
                            fp_tma_pair(ms, &mapA, kbyte, my_m, full_addr + 8 * s, L2_EVICT_LAST);
                            if (FORM == FORM_S) fp_tma_pair(ms + C::A_BYTES, &mapB, kbyte, w.n0 + rank * C::B_ROWS, full_addr + 8 * s, FP_L2_NORMAL);
                            else fp_tma_pair(ms + C::A_BYTES, rank == 0 ? &mapB : &mapB1, kbyte, w.n0, full_addr + 8 * s, FP_L2_NORMAL);
                        } else {
                            mbar_expect_tx(full_bar + 8 * s, (uint32_t)C::STAGE);
                            tma_load_2d_hint(ms, &mapA, kbyte, my_m, full_bar + 8 * s, L2_EVICT_LAST);
                            tma_load_2d(ms + C::A_BYTES, &mapB, kbyte, w.n0, full_bar + 8 * s);
                            if (FORM == FORM_W) tma_load_2d(ms + C::A_BYTES + C::NOUT * 128, &mapB1, kbyte, w.n0, full_bar + 8 * s);
                        }
                        if (FORM == FORM_W) {
                            mbar_expect_tx(sfull_bar + 8 * sc, (uint32_t)C::SC_SLOT);
                            const uint32_t sa = base + sc_off + sc * C::SC_SLOT;
                            tma_load_2d(sa, &mapSA, my_m, kb, sfull_bar + 8 * sc);
                            tma_load_2d(sa + 4 * C::BPS * TILE_M, &mapSB, w.n0, kb, sfull_bar + 8 * sc);
                            kb += C::BPS;
                            ++nsc;
                            fp_next<C::SC_DEPTH>(sc, scph);
                        }
                        fp_next<STAGES>(s, ph);
                    }
                }
                // every issued copy must have landed before the CTA may leave (in a normal run they have)
                const uint32_t back = it < (uint32_t)STAGES ? it : (uint32_t)STAGES;
                for (uint32_t k = 0; k < back; ++k) {
                    if (s == 0) { s = STAGES - 1; ph ^= 1u; } else { --s; }
                    if (!PAIR || rank == 0) mbar_wait(full_bar + 8 * s, ph, abort_flag, p.status, 142, false);
                }
                const uint32_t sback = nsc < (uint32_t)C::SC_DEPTH ? nsc : (uint32_t)C::SC_DEPTH;
                for (uint32_t k = 0; k < sback; ++k) {
                    if (sc == 0) { sc = C::SC_DEPTH - 1; scph ^= 1u; } else { --sc; }
                    mbar_wait(sfull_bar + 8 * sc, scph, abort_flag, p.status, 143, false);
                }
            }
        } else if (warp == FP_MMA_WARP) {
            // -------------------------------------------------------------- MMA issuer (PAIR: the leader's)
            if ((!PAIR || rank == 0) && elect_one()) {
                constexpr uint32_t idesc = fp_idesc<FORM, NCOL, PAIR>();
                uint32_t s = 0, ph = 0, g = 0, gph = 0;
                bool ok = true;
                for (int t = first; ok && t < tiles; t += step) {
                    int left = nblk;
                    for (int si = 0; ok && si < nst; ++si) {
                        if (!fp_wait(full_bar + 8 * s, ph, abort_flag, p.status, 241)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t ms = base + s * C::STAGE;
                        const uint64_t a_desc = smem_desc_sw128(ms), b_desc = smem_desc_sw128(ms + C::A_BYTES);
                        const int nb = C::BPS == 1 ? 1 : min(C::BPS, left);
#pragma unroll
                        for (int jb = 0; jb < C::BPS; ++jb) {
                            if (jb < nb) {
                                if (!fp_wait(tempty_bar + 8 * g, gph, abort_flag, p.status, 242)) { ok = false; break; }
                                tc_fence_after();
                                const uint32_t d = tmem_base + g * NCOL;
#pragma unroll
                                for (int q = 0; q < C::STEPS; ++q) {
                                    const uint64_t ko = (uint64_t)(2 * (jb * C::STEPS + q));     // 32 bytes per step, in 16-byte units
                                    fp_mma<PAIR>(d, a_desc + ko, b_desc + ko, idesc, q != 0);
                                }
                                fp_commit<PAIR>(tfull_bar + 8 * g);
                                fp_next<GROUPS>(g, gph);
                            }
                        }
                        left -= nb;
                        fp_commit<PAIR>(empty_bar + 8 * s);          // the stage is free once these MMAs have read it
                        fp_next<STAGES>(s, ph);
                    }
                }
                fp_commit<PAIR>(done_bar, 1);
                mbar_wait(done_bar, 0, abort_flag, p.status, 243, false);
            }
        }
        __syncwarp();
        if (split) fp_cluster_barrier();       // this warp's share of the barrier between writing and adding up the parts
    } else {
        // ------------------------------------------------------------------ rescale warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(FP_REGS_RESCALE));
        constexpr int NC = C::NC;
        const int rwarp = warp - FP_CONTROL_WARPS, quarter = warp & 3, col0 = (rwarp >> 2) * NC;
        const FpRescale ra{tfull_bar, PAIR ? fp_map_rank(tempty_bar, 0) : tempty_bar, sfull_bar, tmem_base, reinterpret_cast<const float*>(base_ptr + sc_off), abort_flag};
        for (int g = 0; g < GROUPS; ++g) fp_hand_back<PAIR>(ra.tempty_bar + 8 * g);      // every group starts out free
        uint64_t acc2[NC / 2];
        FpRing ring{0, 0, 0, 0};
        bool sent = false;
        for (int t = first; t < tiles; t += step) {
            const FpWork w = fp_work<TM, C::NOUT>(p, t);
#pragma unroll
            for (int c = 0; c < NC / 2; ++c) acc2[c] = 0ull;
            const bool ok = fp_blocks<FORM, NCOL, BP, PAIR>(acc2, p, ra, nblk, col0, ring);
            if (FORM == FORM_S && ok && !fp_all_finite<NC>(acc2)) atomicCAS(p.status, 0, STATUS_EXPONENT_RANGE);
            if constexpr (!PAIR) if (split) {
                __syncwarp();
                fp_split_sum<C::NOUT, NC, BIAS>(acc2, p, base, base_ptr, w, rank, quarter * 32 + lane, col0);
                break;
            }
            if (!ok) break;
            if constexpr (BIAS) fp_add_bias<NC>(acc2, p, w.n0 + col0);
            const int gi0 = w.m0 + (PAIR ? rank * TILE_M : 0) + quarter * 32;
            if constexpr (FORM == FORM_W) { fp_store_rows<NC>(acc2, p, gi0 + lane, w.n0 + col0); continue; }
#pragma unroll
            for (int cb = 0; cb < NC / 32; ++cb) {
                // 32 rows x 32 columns through shared memory (16-byte piece j of row r at piece j ^ (r & 7)): whole lines leave
                const uint32_t buf = base + out_off + (uint32_t)rwarp * 4096u;
                if (p.tma_out && sent) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t at = buf + (uint32_t)lane * 128u + (uint32_t)((j ^ (lane & 7)) << 4);
                    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(at), "l"(acc2[cb * 16 + 2 * j]), "l"(acc2[cb * 16 + 2 * j + 1]) : "memory");
                }
                const int gj0 = w.n0 + col0 + 32 * cb;
                if (p.tma_out) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                                     ::"l"(reinterpret_cast<uint64_t>(&mapC)), "r"(buf), "r"(gj0), "r"(gi0) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        sent = true;
                    }
                } else {
                    __syncwarp();
                    const float* box = reinterpret_cast<const float*>(base_ptr + out_off + rwarp * 4096);
                    float* dst = p.C + (int64_t)gi0 * p.ldc + gj0 + lane;
                    const bool in_n = gj0 + lane < p.N;
                    const int rows = min(32, p.M - gi0);
                    for (int r = 0; r < rows; ++r) {
                        const float x = box[r * 32 + (((lane >> 2) ^ (r & 7)) << 2) + (lane & 3)];
                        if (in_n) dst[(int64_t)r * p.ldc] = x;
                    }
                }
            }
        }
        if (sent) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }

    // ------------------------------------------------------------------ teardown
    tc_fence_before();
    __syncthreads();
    if (PAIR || split) fp_cluster_barrier();   // nobody leaves while its memory may be read or its barriers signalled
    if (warp == FP_MMA_WARP) {
        tc_fence_after();
        if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    }
}

// ------------------------------------------------------------------------------ operand forms from packed operands

// Eight packed mantissa bytes as exact floats: byte + 128 in the low mantissa bits of 2^23, minus the constant.
__device__ __forceinline__ void bytes_to_floats(uint2 b, float (&f)[8]) {
    const uint32_t w[2] = {b.x ^ 0x80808080u, b.y ^ 0x80808080u};
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = __uint_as_float(__byte_perm(w[i >> 2], 0x4B000000u, 0x7440 + (i & 3))) - 8388736.0f;
}
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {       // exact: the low halves of both words are zero
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
__device__ __forceinline__ uint32_t f16_pair(float a, float b) {        // exact for integers up to 2048
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

// Form S: rows x kst bytes of one-plane mantissas -> bfloat16 q * 2^s, 16 elements per thread.
__global__ void __launch_bounds__(256)
expand_s_kernel(const int8_t* __restrict__ q, const int8_t* __restrict__ exps, int64_t rows, int kst, int lg_bp, int nkb, int64_t rs,
                uint4* __restrict__ out, const Placing at) {
    const Chain chain(at);
    const int per = kst >> 4;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= rows * per) return;
    const int64_t r = i / per;
    const int o = (int)(i - r * per) << 4, kb = o >> lg_bp;
    const uint4 b = __ldcs(reinterpret_cast<const uint4*>(q + r * kst + o));
    const int s = kb < nkb ? (int)__ldca(reinterpret_cast<const signed char*>(exps) + (int64_t)kb * rs + r) : 0;
    const float sc = __uint_as_float((uint32_t)(s + 127) << 23);
    float f[8], h[8];
    bytes_to_floats(make_uint2(b.x, b.y), f);
    bytes_to_floats(make_uint2(b.z, b.w), h);
#pragma unroll
    for (int k = 0; k < 8; ++k) { f[k] *= sc; h[k] *= sc; }
    out[2 * i] = make_uint4(bf16_pair(f[0], f[1]), bf16_pair(f[2], f[3]), bf16_pair(f[4], f[5]), bf16_pair(f[6], f[7]));
    out[2 * i + 1] = make_uint4(bf16_pair(h[0], h[1]), bf16_pair(h[2], h[3]), bf16_pair(h[4], h[5]), bf16_pair(h[6], h[7]));
}

// Form W: two-plane mantissas q = 16 hi + lo -> binary16 q (A) or the split q = 64 h + l (B), and the block scales
// 2^s as floats [nkb][rs]. 8 elements per thread.
template <bool IS_B>
__global__ void __launch_bounds__(256)
expand_w_kernel(const int8_t* __restrict__ q, int64_t plane_stride, const int8_t* __restrict__ exps, int64_t rows, int kst, int lg_bp, int nkb,
                int64_t rs, uint4* __restrict__ out, uint4* __restrict__ out_l, float* __restrict__ scales, int32_t* status, const Placing at) {
    const Chain chain(at);
    const int per = kst >> 3;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= rows * per) return;
    const int64_t r = i / per;
    const int o = (int)(i - r * per) << 3, kb = o >> lg_bp;
    const uint2 bh = __ldcs(reinterpret_cast<const uint2*>(q + r * kst + o)), bl = __ldcs(reinterpret_cast<const uint2*>(q + plane_stride + r * kst + o));
    float fh[8], fl[8];
    bytes_to_floats(bh, fh);
    bytes_to_floats(bl, fl);
    if ((o & ((1 << lg_bp) - 1)) == 0 && kb < nkb) {
        const int s = __ldca(reinterpret_cast<const signed char*>(exps) + (int64_t)kb * rs + r);
        scales[(int64_t)kb * rs + r] = __uint_as_float((uint32_t)(s + 127) << 23);
        // the kernel forms P * 2^sA with |P| below 2^30: finite up to here, reported beyond
        if (!IS_B && s > 96) atomicCAS(status, 0, STATUS_EXPONENT_RANGE);
    }
    if (!IS_B) {
#pragma unroll
        for (int k = 0; k < 8; ++k) fh[k] = fmaf(16.0f, fh[k], fl[k]);
        out[i] = make_uint4(f16_pair(fh[0], fh[1]), f16_pair(fh[2], fh[3]), f16_pair(fh[4], fh[5]), f16_pair(fh[6], fh[7]));
    } else {
        // h = floor((q + 32) / 64), l = q - 64 h in [-32, 31]
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float v = fmaf(16.0f, fh[k], fl[k]);
            fh[k] = floorf((v + 32.0f) * 0.015625f);
            fl[k] = fmaf(-64.0f, fh[k], v);
        }
        out[i] = make_uint4(f16_pair(fh[0], fh[1]), f16_pair(fh[2], fh[3]), f16_pair(fh[4], fh[5]), f16_pair(fh[6], fh[7]));
        out_l[i] = make_uint4(f16_pair(fl[0], fl[1]), f16_pair(fl[2], fl[3]), f16_pair(fl[4], fl[5]), f16_pair(fl[6], fl[7]));
    }
}

// ------------------------------------------------------------------------------ host side

int make_map_f32(CUtensorMap* m, const void* ptr, uint64_t inner, uint64_t outer, uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer, bool swizzle128) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return HBFP_ERR_CUDA;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {pitch_elems * 4};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? HBFP_OK : HBFP_ERR_CUDA;
}

// Shared-memory attribute and, for pairs, the number of clusters the device holds: they belong to the device.
template <int FORM, int NCOL, int BP, bool PAIR, bool BIAS>
int fp_device_setup(int* clusters) {
    using C = FpCfg<FORM, NCOL, BP, PAIR>;
    static int ready[MAX_DEVICES] = {};        // 0: not yet, else 1 + clusters
    const int dev = current_device();
    if (dev < 0) return HBFP_ERR_CUDA;
    if (!ready[dev]) {
        HBFP_CUDA_OK(cudaFuncSetAttribute(gemm_fp_kernel<FORM, NCOL, BP, PAIR, BIAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
        int n = 0;
        if (PAIR) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(2 * sm_count(), 1, 1);
            cfg.blockDim = dim3(FP_THREADS, 1, 1);
            cfg.dynamicSmemBytes = C::SMEM;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, gemm_fp_kernel<FORM, NCOL, BP, PAIR, BIAS>, &cfg) != cudaSuccess || n < 1) {
                cudaGetLastError();
                return HBFP_ERR_CUDA;
            }
        }
        ready[dev] = 1 + n;
    }
    *clusters = ready[dev] - 1;
    return HBFP_OK;
}

template <int FORM, int NCOL, int BP, bool PAIR, bool BIAS>
int fp_launch(FpProblem p, const FpOperand& a, const FpOperand& b, cudaStream_t st) {
    using C = FpCfg<FORM, NCOL, BP, PAIR>;
    constexpr int TM = PAIR ? 2 * TILE_M : TILE_M;
    p.tiles_m = (p.M + TM - 1) / TM;
    p.tiles_n = (p.N + C::NOUT - 1) / C::NOUT;
    int clusters = 0;
    int rc = fp_device_setup<FORM, NCOL, BP, PAIR, BIAS>(&clusters);
    if (rc) return rc;
    CUtensorMap mA, mB, mB1, mSA, mSB, mC;
    rc = make_map(&mA, a.p0, 2 * a.kst, a.rows, 2 * a.kst, 128, TILE_M, true);
    if (rc) return rc;
    constexpr int B_BOX = FORM == FORM_W ? C::NOUT : C::B_ROWS;
    rc = make_map(&mB, b.p0, 2 * b.kst, b.rows, 2 * b.kst, 128, B_BOX, true);
    if (rc) return rc;
    mB1 = mSA = mSB = mC = mB;
    if (FORM == FORM_W) {
        rc = make_map(&mB1, b.p1, 2 * b.kst, b.rows, 2 * b.kst, 128, C::NOUT, true);
        if (rc) return rc;
        rc = make_map_f32(&mSA, a.scales, a.rs, p.nkb, a.rs, TILE_M, C::BPS, false);
        if (rc) return rc;
        rc = make_map_f32(&mSB, b.scales, b.rs, p.nkb, b.rs, C::NOUT, C::BPS, false);
        if (rc) return rc;
    }
    p.tma_out = FORM == FORM_S && p.splits == 1 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0 && (p.ldc & 3) == 0;
    if (p.tma_out) {
        rc = make_map_f32(&mC, p.C, p.N, p.M, p.ldc, 32, 32, true);
        if (rc) return rc;
    }
    const int tiles = p.tiles_m * p.tiles_n;
    const int grid = PAIR ? 2 * (tiles < clusters ? tiles : clusters) : p.splits > 1 ? tiles * p.splits : (tiles < sm_count() ? tiles : sm_count());
    // A long launch of the 12-bit form is not chained: its three operand planes are the heaviest traffic there is, and CTAs placed as SMs
    // fall free share panels in L2 less well than CTAs placed on an empty chip, which costs a long launch more than its start. Chained /
    // not, with conversions, in order of K-blocks x tiles of a CTA: 2048 cube, b = 64 (128) 59.3 / 61.5 us; 4096 x 4096 x 1024, b = 32 (224)
    // 144.3 / 144.6; 1024 x 4096 x 4096, b = 24 (342) 208.6 / 209.6; 3072 cube, b = 32 (384) 220.5 / 221.1; from there on 4096 cube, b = 64
    // (448) 301.9 / 301.7; 8192 x 8192 x 512, b = 32 (448) 295.0 / 289.0; 3072 cube, b = 24 (512) 285.0 / 284.5; 4096 cube, b = 32 (896)
    // 486.5 / 484.0; 4096 cube, b = 24 (1197) 640.2 / 633.5. The 8-bit form gains by it at every size: 2048 cube, b = 32 (128) 40.1 / 42.8,
    // 4096 cube, b = 64 (256) 149.9 / 153.0, b = 32 (512) 205.0 / 207.5, b = 24 (684) 325.7 / 328.3, 4096 x 4096 x 8192, b = 32 (1024) 484.4 /
    // 486.6.
    const int ctas = PAIR ? grid / 2 : grid;
    const bool chained = FORM == FORM_S || p.splits > 1 || (int64_t)((tiles + ctas - 1) / ctas) * p.nkb < 400;
    launch_chained_clusters(gemm_fp_kernel<FORM, NCOL, BP, PAIR, BIAS>, PAIR ? 2 : p.splits, grid, FP_THREADS, C::SMEM, st, chained, mA, mB, mB1, mSA, mSB, mC, p);
    note_product(st);
    return launch_status();
}

template <int FORM, int BP, bool BIAS>
int fp_launch_bp(const FpProblem& p, const FpPlan& plan, const FpOperand& a, const FpOperand& b, cudaStream_t st) {
    if (plan.pair) return fp_launch<FORM, 256, BP, true, BIAS>(p, a, b, st);
    if (plan.ncol == 256) return fp_launch<FORM, 256, BP, false, BIAS>(p, a, b, st);
    if (plan.ncol == 128) return fp_launch<FORM, 128, BP, false, BIAS>(p, a, b, st);
    if constexpr (FORM == FORM_S) return fp_launch<FORM, 64, BP, false, BIAS>(p, a, b, st);
    return HBFP_ERR_UNSUPPORTED;
}
template <int FORM, int BP>
int fp_launch_bias(const FpProblem& p, const FpPlan& plan, const FpOperand& a, const FpOperand& b, cudaStream_t st) {
    return p.bias ? fp_launch_bp<FORM, BP, true>(p, plan, a, b, st) : fp_launch_bp<FORM, BP, false>(p, plan, a, b, st);
}

inline int log2_of(int64_t v) { int l = 0; while ((1ll << l) < v) ++l; return l; }

}  // namespace

// (The times below are both sides' before launches were chained: what each launch adds has since become less on either side.)
FpPlan plan_gemm_fp(int64_t M, int64_t N, const Layout& la, const Layout& lb, int passes) {
    FpPlan f{};
    if (M <= 0 || N <= 0 || la.nkb <= 0 || la.planes != lb.planes || la.bp != lb.bp || la.nkb != lb.nkb || la.b != lb.b) return f;
    const bool w = la.planes == 2;
    // blocks of 128: the integer kernels are as fast (8 bits) or faster (12 bits, 4096 cube: 230 against 310 us)
    if (la.bp > 64) return f;
    // (within what launch_quantize_form covers, so that a conversion straight to the form is never refused)
    if (M > (1ll << 28) || N > (1ll << 28) || la.kst > (1ll << 29)) return f;
    const int64_t lines = M > N ? M : N;
    if (lines * (la.kst / 8) >= (1ll << 39) || ((lines + 31) / 32) * la.nkb >= (1ll << 31)) return f;
    // Packed operands cost a pass each to take the form. It pays where every element is used often enough and the product is
    // large (all with both passes): 2048 cube 34 against 51 us (8 bits, b = 32), 27 against 31 (b = 64), 48 against 58 (12 bits,
    // b = 64), 4096 cube 186 / 290, 123 / 159, 261 / 368; but 1024 x 1024 x 2048 20 / 20, 18 / 14 and 24 / 18 us.
    // FP32 operands are converted straight to the form, which pays at (nearly) every size: see below.
    if (passes > 0 && (M * N < 600 * (M + N) || (double)M * (double)N * (double)(la.nkb * la.b) < 8.0e9)) return f;
    f.form = w ? FORM_W : FORM_S;
    const int64_t SMS = 148;                       // planning constant: the target part
    const int64_t nst = (la.nkb * la.bp + FP_STAGE_ELEMS - 1) / FP_STAGE_ELEMS;
    f.splits = 1;
    // The time of a block grows with the tile's columns but not in proportion. K is split only where all clusters run at once:
    // a cluster's CTAs share a GPU processing cluster, so that of 148 SMs only this many clusters of one CTA per SM are resident
    // (cudaOccupancyMaxActiveClusters). 36 clusters of four took two rounds: 1111 x 777 x 3001 with b = 24 51.4 us with its
    // conversions, 63 clusters of two 41.2; 1500 x 600 x 3000, b = 64: 38.4 against 30.9; 128 x 4000 x 2000, b = 32: 37.7 against 27.0.
    static constexpr int resident[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    double best = 1e30;
    for (int ncol = 256; ncol >= (w ? 128 : 64); ncol /= 2) {
        const int64_t nout = w ? ncol / 2 : ncol, tiles = ((M + 127) / 128) * ((N + nout - 1) / nout);
        const double cost = ncol == 256 ? 1.0 : ncol == 128 ? 0.55 : 0.45;
        for (int64_t sp = 1; sp <= 8; ++sp) {
            if (sp > 1 && (tiles > resident[sp] || nst < 4 * sp)) continue;
            if ((nst + (nst + sp - 1) / sp - 1) / ((nst + sp - 1) / sp) != sp) continue;       // a split would be empty
            const double waves = (double)((tiles * sp + SMS - 1) / SMS);
            const double t = waves * ((double)((nst + sp - 1) / sp) * cost + 4.0 + (sp > 1 ? 3.0 : 0.0));
            if (t < best * 0.999) { best = t; f.ncol = ncol; f.splits = (int)sp; }
        }
    }
    // A few tiles with a long contraction want more splits than a cluster has CTAs: the integer kernels (split-K over the whole
    // chip, a second launch adds the parts) take them, 64 x 64 x 16384 19 against 25 us, 576 x 64 x 32768 39 against 58. Otherwise
    // from FP32 operands (b = 32): 128 x 10 x 1024 12 against 24 us, 512 x 512 x 1024 13 / 18, 1111 x 777 x 3001 41 / 47, 8192 x 256 x 256
    // 13 / 15, 4096 cube 197 / 329.
    {
        const int64_t nout = w ? f.ncol / 2 : f.ncol, ctas = ((M + 127) / 128) * ((N + nout - 1) / nout) * f.splits;
        const int64_t per = (nst + f.splits - 1) / f.splits;       // stages of a CTA
        if (ctas < 74 && nst / f.splits > 24) return FpPlan{};
        // The narrowest tiles in eight splits say the same of shorter contractions: 128 x 200 x 10865 (b = 64) 22 against 18 us,
        // 64 x 56 x 12416 (12 bits, b = 32) 27 against 20. With 104 CTAs and more the forms keep blocks of 32 (209 x 448 x 14464,
        // 12 bits, 38 against 43) and lose long ones of 64, whose MMAs wait for operands: 208 x 384 x 52072 71 against 54.
        if (f.ncol == (w ? 128 : 64) && f.splits == 8 && ((ctas < 104 && per >= 13) || (la.bp == 64 && per >= 28))) return FpPlan{};
        // the same without a split, where the tiles alone occupy the chip: 1944 x 576 x 10752, b = 64, 96 against 84
        if (f.ncol == (w ? 128 : 64) && la.bp == 64 && ctas < 148 && per >= 100) return FpPlan{};
    }
    // Blocks of 64 feed the tensor cores twice as fast as blocks of 32, and one SM's shared memory cannot deliver it: a stage
    // costs 48 KB written and 48 KB read (768 cycles) for 512 cycles of MMAs. A pair of SMs stages and reads a third less each
    // (4096 cube with conversions of the packed operands: 8 bits 136 -> 123 us, 12 bits 281 -> 261 us; blocks of 32 gain
    // nothing, 186 against 192).
    const int64_t pair_tiles = ((M + 255) / 256) * ((N + (w ? 127 : 255)) / (w ? 128 : 256));
    if (la.bp == 64 && f.splits == 1 && f.ncol == 256 && pair_tiles >= 74) f.pair = 1;
    const int64_t unit = FP_STAGE_ELEMS / la.bp;      // blocks per stage
    int64_t kbps = (la.nkb + f.splits - 1) / f.splits;
    kbps = (kbps + unit - 1) / unit * unit;
    if (f.splits > 1 && (la.nkb + kbps - 1) / kbps != f.splits) { f.splits = 1; kbps = la.nkb; }
    f.kb_per_split = (int)kbps;
    f.planes_b = w ? 2 : 1;
    f.use = 1;
    return f;
}

int launch_expand(const Packed& x, const FpPlan& plan, bool is_b, const Placing& at, const FpOperand& out, cudaStream_t st) {
    const Layout& L = x.L;
    const int lg = log2_of(L.bp);
    if (plan.form == FORM_S) {
        const int64_t n = L.rows * (L.kst / 16);
        launch_placed(at, L.rows * L.kst, expand_s_kernel, (unsigned)((n + 255) / 256), 256, 0, st, x.mant, x.exps, L.rows, (int)L.kst, lg, (int)L.nkb, L.rs, static_cast<uint4*>(out.p0), at);
        return launch_status();
    }
    int32_t* status = device_status_word();
    if (!status) return HBFP_ERR_CUDA;
    const int64_t n = L.rows * (L.kst / 8);
    const unsigned g = (unsigned)((n + 255) / 256);
    if (is_b) launch_placed(at, L.rows * L.kst * 2, expand_w_kernel<true>, g, 256, 0, st, x.mant, L.plane_stride, x.exps, L.rows, (int)L.kst, lg, (int)L.nkb, L.rs, static_cast<uint4*>(out.p0), static_cast<uint4*>(out.p1), out.scales, status, at);
    else launch_placed(at, L.rows * L.kst * 2, expand_w_kernel<false>, g, 256, 0, st, x.mant, L.plane_stride, x.exps, L.rows, (int)L.kst, lg, (int)L.nkb, L.rs, static_cast<uint4*>(out.p0), nullptr, out.scales, status, at);
    return launch_status();
}

int launch_gemm_fp(int64_t M, int64_t N, const Layout& la, const FpPlan& plan, const FpOperand& a, const FpOperand& b, const float* bias, float* Cout, int64_t ldc, cudaStream_t st) {
    FpProblem p{};
    p.M = (int)M;
    p.N = (int)N;
    p.nkb = (int)la.nkb;
    p.splits = plan.splits;
    p.kb_per_split = plan.kb_per_split;
    p.bias = bias;
    p.C = Cout;
    p.ldc = ldc;
    p.status = device_status_word();
    if (!p.status) return HBFP_ERR_CUDA;
    if (plan.form == FORM_S) return la.bp == 32 ? fp_launch_bias<FORM_S, 32>(p, plan, a, b, st) : fp_launch_bias<FORM_S, 64>(p, plan, a, b, st);
    return la.bp == 32 ? fp_launch_bias<FORM_W, 32>(p, plan, a, b, st) : fp_launch_bias<FORM_W, 64>(p, plan, a, b, st);
}

}  // namespace hbfp
