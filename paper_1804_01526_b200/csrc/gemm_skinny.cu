// BFP GEMM of a few rows of FP32 activations with weights that were packed ahead of time, conversion included, in one launch.
//
// Bound: reading the weights. 16 x 4096 x 4096 is 17 MB of mantissas (2.6 us at the copy bandwidth) and little arithmetic, but
// the general path spends three launches on it: the conversion, a GEMM whose 128-row tiles of activations are seven eighths
// padding and the addition of split-K parts. Here the weights are the 128-row operand of the MMA and the activations the narrow
// one: a CTA takes 128 weight rows and a range of K, asks for all of its weights at once (128-byte columns by TMA, one barrier
// each), and converts the activations of that range into the swizzled shared-memory operand while they fly. Every K-block gets
// its own columns of tensor memory (int32, exact), so the MMAs of a CTA run without waiting for the rescale warps unless K is
// long; those read each block once, acc = fma(P * 2^sB, 2^sA, acc), ascending, one rounding per block. The CTAs that share an
// output tile form a cluster along K and add their parts through distributed shared memory in ascending order: deterministic,
// no scratch. (The same with warp-level binary16 MMAs, weights converted in registers: 14.8 us at 16 x 4096 x 4096 - the
// legacy MMA issues once per 8 cycles and SM, and the arithmetic around it costs as much again.)
#include <cuda.h>

#include "quant_math.cuh"

namespace hbfp {
namespace {

constexpr int SK_CONV_WARPS = 8, SK_THREADS = 32 * (SK_CONV_WARPS + 1), SK_SEG = STAGE_K;     // K bytes per TMA box
constexpr int SK_MAX_SEGS = 16, SK_NT = TILE_M, SK_MAX_GROUPS = 32;
constexpr int SK_SMEM_LIMIT = 232448 - 1024;

struct SkinnyProblem {
    const float* x;                 // [M][K], pitch ld
    int64_t ld;
    int M, N, K, b, nkb;
    const int8_t* w_exps;           // [nkb][rs]
    int64_t rs;
    int segs, segs_per_cta, splits; // 128-byte columns of the packed weights: all, of a CTA; CTAs of a cluster
    int tmem_cols;
    int off_x, off_xs, off_we, off_bar;   // shared memory
    int vec;                        // pieces of eight activations are 16-byte aligned
    const float* bias;              // may be null
    float* C;
    int64_t ldc;
    int32_t* status;
    QParams q;
};

__device__ __forceinline__ uint32_t sk_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t sk_map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void sk_cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint64_t sk_mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// ROWS: activation rows of a CTA (columns of an accumulator), BP: padded block length.
template <int ROWS, int BP, bool SR>
__global__ void __launch_bounds__(SK_THREADS, 2)
gemm_skinny_kernel(const __grid_constant__ CUtensorMap mapW, const SkinnyProblem p) {
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* sm = smem_dyn + (base - smem_u32(smem_dyn));
    float* xs = reinterpret_cast<float*>(sm + p.off_xs);          // [block][ROWS]: 2^s of the activations
    int8_t* we = reinterpret_cast<int8_t*>(sm + p.off_we);        // [block][SK_NT]: exponents of the weights
    const uint32_t full_bar = base + p.off_bar;                   // weights of a segment landed
    const uint32_t done_bar = full_bar + 8 * p.segs_per_cta;      // block sums of a segment complete
    const uint32_t free_bar = done_bar + 8 * p.segs_per_cta;      // accumulator columns read by every rescale warp
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + p.off_bar + 16 * p.segs_per_cta + 8 * (p.tmem_cols / ROWS));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = p.splits > 1 ? (int)sk_ctarank() : 0;
    const int n0 = blockIdx.y * SK_NT, m0 = blockIdx.z * ROWS;
    const int seg0 = rank * p.segs_per_cta, nseg = min(p.segs_per_cta, p.segs - seg0);      // at least one: the host sizes the splits
    constexpr int BPS = SK_SEG / BP;                              // blocks per segment
    const int kb0 = seg0 * BPS, groups = p.tmem_cols / ROWS;

    if (warp == SK_CONV_WARPS) {
        if (lane == 0) {
            for (int i = 0; i < nseg; ++i) { mbar_init(full_bar + 8 * i, 1); mbar_init(done_bar + 8 * i, 1); }
            for (int i = 0; i < groups; ++i) mbar_init(free_bar + 8 * i, SK_CONV_WARPS);
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            chain_wait();
            for (int i = 0; i < nseg; ++i) {
                mbar_expect_tx(full_bar + 8 * i, SK_NT * SK_SEG);
                tma_load_2d(base + i * (SK_NT * SK_SEG), &mapW, (seg0 + i) * SK_SEG, n0, full_bar + 8 * i);
            }
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        chain_wait();
        chain_next();
    } else {
        chain_wait();
        // exponents of the weight rows, sixteen at a time (blocks and rows beyond the matrix: 0, their mantissas are 0)
        for (int i = tid; i < nseg * BPS * (SK_NT / 16); i += 32 * SK_CONV_WARPS) {
            const int kb = kb0 + i / (SK_NT / 16), r = n0 + 16 * (i % (SK_NT / 16));
            const bool in = kb < p.nkb && r < p.rs;
            const int8_t* src = in ? p.w_exps + (int64_t)kb * p.rs + r : p.w_exps;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + p.off_we + 16 * i), "l"(src), "r"(in ? 16 : 0) : "memory");
        }
        // Activations in pieces of eight packed positions, LPB lanes per block: a thread keeps its position and walks down the
        // rows, rpp rows at a time (the threads left over only take part in the shuffles).
        constexpr int LPB = BP / 8, UNR = 4;
        const int gpr = nseg * (SK_SEG / 8), rpp = 32 * SK_CONV_WARPS / gpr;
        const int r0 = tid / gpr, pos = 8 * (tid - r0 * gpr);
        const int kb = kb0 + pos / BP, within = pos & (BP - 1), k = kb * p.b + within;
        const int n = r0 < rpp && kb < p.nkb ? min(p.b - within, p.K - k) : 0;       // elements of the piece
        const int off = pos & (SK_SEG - 1);
        unsigned char* xt = sm + p.off_x + (pos / SK_SEG) * (ROWS * SK_SEG) + (off & 8);
        float* xst = xs + (pos / BP) * ROWS;
        for (int rb = 0; rb < ROWS; rb += UNR * rpp) {
            float e8[UNR][8];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int r = rb + u * rpp + r0;
                const float* src = p.x + (int64_t)(m0 + r) * p.ld + k;
                const int nr = r < ROWS && m0 + r < p.M ? n : 0;
                if (nr >= 8 && p.vec) {
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
                if (rb + u * rpp >= ROWS) break;                          // all threads alike
                const int r = rb + u * rpp + r0;
                uint32_t am = amax8_bits(e8[u]);
#pragma unroll
                for (int o = 1; o < LPB; o <<= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, o));
                const int s = block_exponent(am, p.q.m, p.q.exp_mode);
                const uint4 w = SR ? draws_of_eight(p.q, (uint64_t)((int64_t)(m0 + r) * p.K + k)) : make_uint4(0u, 0u, 0u, 0u);
                uint2 h, unused;
                quantize_pack8<SR, 1>(e8[u], s, p.q, w, h, unused);
                if (r < ROWS && r0 < rpp) {
                    *reinterpret_cast<uint2*>(xt + r * SK_SEG + (((off >> 4) ^ (r & 7)) << 4)) = h;
                    if (within == 0) xst[r] = pow2f(s);
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // the MMAs read what was written here
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == SK_CONV_WARPS) {
        // the whole warp waits and one lane issues: a look at a barrier costs a warp 119 cycles, a lane that polls in a loop 317
        constexpr uint32_t idesc = idesc_i8<ROWS>();
        int g = 0, ph = 1, issued = 0;
        bool ok = true, again = false;                  // again: the accumulator columns are in use for the second time and more
        for (int i = 0; ok && i < nseg; ++i) {
            ok = mbar_wait_warp_fast(full_bar + 8 * i, 0, abort_flag, p.status, 161);
            if (!ok) break;
            tc_fence_after();
            const uint64_t a_desc = smem_desc_sw128(base + i * (SK_NT * SK_SEG)), b_desc = smem_desc_sw128(base + p.off_x + i * (ROWS * SK_SEG));
#pragma unroll
            for (int jb = 0; jb < BPS; ++jb) {
                if (again) {
                    ok = ok && mbar_wait_warp_fast(free_bar + 8 * g, (uint32_t)ph, abort_flag, p.status, 162);
                    if (!ok) break;
                    tc_fence_after();
                }
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BP / 32; ++k) {
                        const uint64_t ko = (uint64_t)(2 * (jb * (BP / 32) + k));      // 32 bytes per step, in 16-byte units
                        tc_mma_i8(tmem_base + g * ROWS, a_desc + ko, b_desc + ko, idesc, k != 0);
                    }
                    if (jb == BPS - 1) tc_commit(done_bar + 8 * i);
                }
                if (++g == groups) { g = 0; ph ^= 1; again = true; }
            }
            if (ok) issued = i + 1;
        }
        // nothing of this CTA is in flight when it leaves (in a normal run all has completed). MMAs of a segment that was given up
        // half way write tensor memory, which goes back below: they too are committed and waited for, abort flag or not.
        if (!ok) {
            if (elect_one()) tc_commit(done_bar + 8 * issued);
            ++issued;
            for (int i = 0; i < nseg; ++i) mbar_wait(full_bar + 8 * i, 0, abort_flag, p.status, 163, false);
        }
        for (int i = 0; i < issued; ++i)
            if (!mbar_wait_warp_fast(done_bar + 8 * i, 0, abort_flag, p.status, 164)) mbar_wait(done_bar + 8 * i, 0, abort_flag, p.status, 164, false);
        __syncwarp();
    } else {
        constexpr int NC = ROWS / 2;                              // accumulator columns of a warp
        const int quarter = warp & 3, col0 = (warp >> 2) * NC, nrow = quarter * 32 + lane;
        uint64_t acc[NC / 2];
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) acc[c] = 0ull;
        int g = 0;
        for (int i = 0; i < nseg; ++i) {
            if (!mbar_wait_warp_fast(done_bar + 8 * i, 0, abort_flag, p.status, 165)) break;
            tc_fence_after();
            // as many of the segment's blocks at a time as registers hold
            constexpr int AT_ONCE = BPS * NC <= 64 ? BPS : (64 / NC < 1 ? 1 : 64 / NC);
#pragma unroll
            for (int j0 = 0; j0 < BPS; j0 += AT_ONCE) {
                uint32_t v[AT_ONCE][NC];
                const int gfirst = g;
#pragma unroll
                for (int jb = 0; jb < AT_ONCE; ++jb) {
                    tc_ldn(tmem_base + ((uint32_t)(quarter * 32) << 16) + g * ROWS + col0, v[jb]);
                    if (++g == groups) g = 0;
                }
                float fb[AT_ONCE];
#pragma unroll
                for (int jb = 0; jb < AT_ONCE; ++jb) {
                    const int sb = we[(i * BPS + j0 + jb) * SK_NT + nrow];
                    fb[jb] = pow2f(sb);
                    if (sb > 104) atomicCAS(p.status, 0, STATUS_EXPONENT_RANGE);        // |P| < 2^22: P * 2^sB is finite up to here
                }
                tc_wait_ld();
                tc_fence_before();
#pragma unroll
                for (int jb = 0, q = gfirst; jb < AT_ONCE; ++jb) {
                    mbar_arrive_elect(free_bar + 8 * q);
                    if (++q == groups) q = 0;
                }
#pragma unroll
                for (int jb = 0; jb < AT_ONCE; ++jb) {
                    const uint64_t fb2 = pack2(__float_as_uint(fb[jb]), __float_as_uint(fb[jb]));
                    const uint64_t nbias = pack2(0xCB400000u, 0xCB400000u);             // -1.5 * 2^23
                    const ulonglong2* fa = reinterpret_cast<const ulonglong2*>(xs + (i * BPS + j0 + jb) * ROWS + col0);
#pragma unroll
                    for (int c = 0; c < NC / 2; c += 2) {
                        const ulonglong2 f = fa[c / 2];
                        // P + 1.5 * 2^23 as the bits of a float, then minus the constant: exact for |P| < 2^22
                        const uint64_t t0 = fadd2(pack2(v[jb][2 * c] + BIAS_BITS, v[jb][2 * c + 1] + BIAS_BITS), nbias);
                        const uint64_t t1 = fadd2(pack2(v[jb][2 * c + 2] + BIAS_BITS, v[jb][2 * c + 3] + BIAS_BITS), nbias);
                        acc[c] = ffma2(sk_mul2(t0, fb2), f.x, acc[c]);
                        acc[c + 1] = ffma2(sk_mul2(t1, fb2), f.y, acc[c + 1]);
                    }
                }
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * SK_CONV_WARPS) : "memory");     // the MMAs are through with the weights: their place holds the part
        float* part = reinterpret_cast<float*>(sm) + nrow;                          // [ROWS][SK_NT]
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) {
            float lo, hi;
            unpack2(acc[c], lo, hi);
            part[(col0 + 2 * c) * SK_NT] = lo;
            part[(col0 + 2 * c + 1) * SK_NT] = hi;
        }
    }
    tc_fence_before();
    __syncthreads();
    // Tensor memory goes back before the CTA waits for its cluster, on every way through the kernel: a CTA that holds columns
    // depends on nobody but itself, so one that blocks in tcgen05.alloc waits for work that always ends - whatever launches, of this
    // or of other plans, on this or on other streams, share the SMs. (Held across the barriers, two clusters that each hold columns
    // on one SM and ask for them on the other would wait for one another for good.) The library's other tensor-core kernels take an
    // SM's registers whole and are nobody's neighbours.
    if (warp == SK_CONV_WARPS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
    }
    if (p.splits > 1) sk_cluster_barrier();
    // each CTA adds up a share of the outputs, parts in ascending order of K
    constexpr int QPR = SK_NT / 4;
    const bool quad = (p.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
    if (tid < 32 * SK_CONV_WARPS)
        for (int i = rank * 32 * SK_CONV_WARPS + tid; i < ROWS * QPR; i += p.splits * 32 * SK_CONV_WARPS) {
            const int r = i / QPR, c = 4 * (i - r * QPR);
            const int gi = m0 + r, gj = n0 + c;
            if (gi >= p.M || gj >= p.N) continue;
            const uint32_t from = base + 16u * (uint32_t)i;
            float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
            for (int sp = 0; sp < p.splits; ++sp) {
                float v[4];
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                             : "r"(p.splits > 1 ? sk_map_rank(from, (uint32_t)sp) : from) : "memory");
#pragma unroll
                for (int e = 0; e < 4; ++e) y[e] = sp == 0 ? v[e] : __fadd_rn(y[e], v[e]);
            }
            if (p.bias)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gj + e < p.N) y[e] = __fadd_rn(y[e], __ldg(p.bias + gj + e));
            float* dst = p.C + (int64_t)gi * p.ldc + gj;
            if (quad && gj + 3 < p.N) *reinterpret_cast<float4*>(dst) = make_float4(y[0], y[1], y[2], y[3]);
            else
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gj + e < p.N) dst[e] = y[e];
        }
    __syncwarp();
    // no neighbour still reads this CTA's part (what it read has arrived in registers, so the arrival orders nothing more)
    if (p.splits > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// ------------------------------------------------------------------------------ host side

struct SkinnyPlan { int rows, splits, segs_per_cta, tmem_cols; size_t smem; };

inline size_t sk_smem(int rows, int bp, int nseg, int cols, SkinnyProblem* p) {
    const int blocks = nseg * (SK_SEG / bp);
    size_t at = (size_t)nseg * SK_NT * SK_SEG;
    const size_t part = (size_t)rows * SK_NT * 4;
    if (part > at) at = part;
    if (p) p->off_x = (int)at;
    at += (size_t)nseg * rows * SK_SEG;
    if (p) p->off_xs = (int)at;
    at += (size_t)blocks * rows * 4;
    if (p) p->off_we = (int)at;
    at += (size_t)blocks * SK_NT;
    if (p) p->off_bar = (int)at;
    return at + 16 * nseg + 8 * (cols / rows) + 8 + 1024;
}

// Splits of K by the estimated time (in SM cycles) of the slowest SM. A CTA is a chain of latencies (start, activations, first
// weights, barrier of the cluster, store: 3000 cycles) and per 128 bytes of K a look at a barrier, four MMAs and a rescale; the
// CTAs of an SM share its intake. Measured at 16 x 4096 x 4096: 8 splits 8.8 us, 6 10.9, 5 (two rounds) 16.6, 4 9.2, 3 12.1. Several
// CTAs share an SM where shared memory allows it; the clusters that are resident at once are those of one GPU processing
// cluster (see plan_gemm_fp).
bool sk_plan(int64_t M, int64_t N, const Layout& lb, SkinnyPlan* out) {
    static constexpr int resident[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    const int bp = (int)lb.bp, segs = (int)(round_up(lb.nkb * lb.bp, SK_SEG) / SK_SEG);
    const int rows = M <= 16 ? 16 : M <= 32 ? 32 : 64;
    const int64_t tiles = (N + SK_NT - 1) / SK_NT * ((M + rows - 1) / rows);
    double best = 1e30;
    for (int sp = 8; sp >= 1; --sp) {
        const int per = (segs + sp - 1) / sp, blocks = per * (SK_SEG / bp);
        if ((segs + per - 1) / per != sp || per > SK_MAX_SEGS) continue;
        // Every resident CTA asks for tensor memory when it starts, and one that finds too little of it waits until a neighbour is
        // through with its MMAs: what the CTAs of a launch that fit an SM ask for together is kept within its 512 columns, by shared
        // memory. That is a matter of time only; the kernel gives its columns back before it waits for anyone.
        int cols = 32;
        while (cols < blocks * rows && cols < 512) cols *= 2;
        if (cols / rows > SK_MAX_GROUPS) cols = SK_MAX_GROUPS * rows;
        size_t smem = sk_smem(rows, bp, per, cols, nullptr);
        if (smem > SK_SMEM_LIMIT) continue;
        int room = (int)(233472 / (smem + 1024));
        if (cols == 512 && room > 1) cols = 256;
        if (room > 512 / cols) { room = 512 / cols; smem = 233472 / (room + 1); }       // (room + 1) x (smem + 1024) no longer fits
        const double share = (double)tiles / resident[sp];                              // clusters per slot
        const double rounds = share <= room ? 1.0 : (double)(int64_t)(share / room + 0.999);
        const double together = share >= room ? room : (double)(int64_t)(share + 0.999);
        const double alone = per * (500.0 + 6.0 * rows), intake = together * per * (300.0 + 4.0 * rows);
        const double t = rounds * (3000.0 + (alone > intake ? alone : intake));
        if (t < best * 0.98) { best = t; *out = SkinnyPlan{rows, sp, per, cols, smem}; }
    }
    return best < 1e30;
}

template <int ROWS, int BP, bool SR>
int sk_launch(const SkinnyProblem& p, const CUtensorMap& mW, size_t smem, dim3 grid, cudaStream_t st) {
    static bool ready[MAX_DEVICES] = {};               // the attribute belongs to the device (same value from any thread)
    const int dev = current_device();
    if (dev < 0) return HBFP_ERR_CUDA;
    if (!ready[dev]) {
        HBFP_CUDA_OK(cudaFuncSetAttribute(gemm_skinny_kernel<ROWS, BP, SR>, cudaFuncAttributeMaxDynamicSharedMemorySize, SK_SMEM_LIMIT));
        ready[dev] = true;
    }
    launch_chained_clusters(gemm_skinny_kernel<ROWS, BP, SR>, p.splits, grid, SK_THREADS, smem, st, true, mW, p);
    note_product(st);
    return launch_status();
}
template <int ROWS, bool SR>
int sk_launch_bp(int bp, const SkinnyProblem& p, const CUtensorMap& mW, size_t smem, dim3 grid, cudaStream_t st) {
    if (bp == 32) return sk_launch<ROWS, 32, SR>(p, mW, smem, grid, st);
    if (bp == 64) return sk_launch<ROWS, 64, SR>(p, mW, smem, grid, st);
    return sk_launch<ROWS, 128, SR>(p, mW, smem, grid, st);
}
template <bool SR>
int sk_launch_rows(int rows, int bp, const SkinnyProblem& p, const CUtensorMap& mW, size_t smem, dim3 grid, cudaStream_t st) {
    if (rows == 16) return sk_launch_bp<16, SR>(bp, p, mW, smem, grid, st);
    if (rows == 32) return sk_launch_bp<32, SR>(bp, p, mW, smem, grid, st);
    return sk_launch_bp<64, SR>(bp, p, mW, smem, grid, st);
}

}  // namespace

bool skinny_gemm_eligible(int64_t M, int64_t N, const Layout& la, const Layout& lb, int bits_a, int bits_b) {
    if (la.planes != 1 || lb.planes != 1 || lb.bp > 128 || lb.nkb <= 0 || la.b != lb.b) return false;
    const int64_t qa = (1ll << (bits_a - 1)) - 1, qb = (1ll << (bits_b - 1)) - 1;
    if (qa * qb * lb.b >= (1ll << 22)) return false;              // block sums exact through the biased conversion
    if (M < 1 || N > (1 << 20) || lb.kst > (1 << 20)) return false;
    // The activations are converted once per CTA along N and rows beyond 64 read the weights again, so the bytes of weights up to
    // which one launch beats conversion, GEMM and split-K sum fall with the rows. Device time, here / there: 16 rows 4096 x 4096
    // 9.7 / 17.4 us, 8192 x 8192 (b = 24) 80 / 91; 32 rows 4096 x 4096 11.5 / 18.6; 64 rows 4096 x 4096 20.9 / 19.8, 33 rows
    // 8192 x 1024 11.5 / 16.6, 64 rows 8192 x 2000 19.0 / 14.1; 128 rows 1024 x 1024 8.9 / 11.7 (b = 24: 12.9 / 13.1), 4096 x 4096 40 / 22.
    const int64_t bytes = N * lb.kst;
    if (M > (bytes <= (3 << 19) ? 128 : bytes <= (1 << 23) ? 64 : bytes <= (1 << 25) ? 32 : 16)) return false;
    SkinnyPlan plan;
    return sk_plan(M, N, lb, &plan);
}

int launch_gemm_skinny(int64_t M, int64_t N, int64_t K, const float* x, int64_t ld, const hbfp_format* fx, const Packed& w, const float* bias, float* C,
                       int64_t ldc, cudaStream_t st) {
    SkinnyPlan plan;
    if (!sk_plan(M, N, w.L, &plan)) return HBFP_ERR_UNSUPPORTED;
    const int bp = (int)w.L.bp;
    SkinnyProblem p{};
    p.x = x;
    p.ld = ld;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.b = (int)w.L.b;
    p.nkb = (int)w.L.nkb;
    p.w_exps = w.exps;
    p.rs = w.L.rs;
    p.segs = (int)(round_up(w.L.nkb * w.L.bp, SK_SEG) / SK_SEG);
    p.segs_per_cta = plan.segs_per_cta;
    p.splits = plan.splits;
    p.tmem_cols = plan.tmem_cols;
    sk_smem(plan.rows, bp, plan.segs_per_cta, plan.tmem_cols, &p);
    p.vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0 && (ld & 3) == 0 && (p.b & 3) == 0;
    p.bias = bias;
    p.C = C;
    p.ldc = ldc;
    p.status = device_status_word();
    if (!p.status) return HBFP_ERR_CUDA;
    p.q = make_params(fx);
    CUtensorMap mW;
    const int rc = make_map(&mW, w.mant, w.L.kst, w.L.rows, w.L.kst, SK_SEG, SK_NT, true);
    if (rc) return rc;
    const dim3 grid(plan.splits, (unsigned)((N + SK_NT - 1) / SK_NT), (unsigned)((M + plan.rows - 1) / plan.rows));
    return fx->rounding == 1 ? sk_launch_rows<true>(plan.rows, bp, p, mW, plan.smem, grid, st)
                             : sk_launch_rows<false>(plan.rows, bp, p, mW, plan.smem, grid, st);
}

}  // namespace hbfp
