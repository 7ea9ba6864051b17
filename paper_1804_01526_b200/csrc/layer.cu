// The FP32 parts of a dense layer around its products (Sec. 5.1: everything but the dot products stays FP32). Both are bound by
// reading (and for the bias writing) one matrix once.
#include "common.cuh"

namespace hbfp {
namespace {

// C += bias on every row, for products whose kernel does not add it in its own store. V = 4: rows of whole 16-byte quads.
template <int V>
__global__ void __launch_bounds__(256)
add_bias_kernel(float* __restrict__ C, uint32_t N, int64_t ldc, const float* __restrict__ bias, int64_t total) {
    chain_start();
    const uint32_t per = N / V;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (int64_t)gridDim.x * 256) {
        const int64_t r = i / per;
        const uint32_t c = (uint32_t)(i - r * per) * V;
        float* at = C + r * ldc + c;
        if (V == 4) {
            const float4 x = *reinterpret_cast<const float4*>(at), b = __ldg(reinterpret_cast<const float4*>(bias + c));
            *reinterpret_cast<float4*>(at) = make_float4(__fadd_rn(x.x, b.x), __fadd_rn(x.y, b.y), __fadd_rn(x.z, b.z), __fadd_rn(x.w, b.w));
        } else {
            *at = __fadd_rn(*at, __ldg(bias + c));
        }
    }
}

// Column sums of x [rows][cols]. A CTA takes 32 * V columns and a share of the rows: lane = V neighbouring columns, eight
// warps (and UNR independent chains in each) along the rows; the CTAs of a cluster split the rows further and the first adds up
// their parts from their shared memory. Deterministic, one launch, nothing to clear.
constexpr int CS_WARPS = 8, CS_UNR = 8;
template <int V>
__global__ void __launch_bounds__(32 * CS_WARPS)
column_sums_kernel(const float* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, int splits, float* __restrict__ out) {
    chain_start();
    __shared__ __align__(16) float part[CS_WARPS][32 * V];
    __shared__ __align__(16) float total[32 * V];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t col = (int64_t)blockIdx.y * (32 * V) + lane * V;
    const int64_t share = (rows + splits - 1) / splits, r_end = min(rows, (int64_t)(blockIdx.x + 1) * share);
    float acc[CS_UNR][V];
#pragma unroll
    for (int u = 0; u < CS_UNR; ++u)
#pragma unroll
        for (int e = 0; e < V; ++e) acc[u][e] = 0.f;
    if (col < cols) {
        auto add = [&](int u, const float* src) {
            if (V == 4) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(src));
                acc[u][0] += v.x; acc[u][1] += v.y; acc[u][2] += v.z; acc[u][3] += v.w;
            } else {
                acc[u][0] += __ldg(src);
            }
        };
        int64_t r0 = blockIdx.x * share + warp;
        const int64_t step = CS_WARPS * ld;
        const float* src = x + r0 * ld + col;
        // whole rounds without a condition, so that their loads leave together
        for (; r0 + (CS_UNR - 1) * CS_WARPS < r_end; r0 += CS_WARPS * CS_UNR, src += CS_UNR * step)
#pragma unroll
            for (int u = 0; u < CS_UNR; ++u) add(u, src + u * step);
        for (int u = 0; r0 < r_end; r0 += CS_WARPS, src += step, ++u) {
#pragma unroll
            for (int k = 0; k < CS_UNR; ++k)
                if (k == u) add(k, src);
        }
    }
#pragma unroll
    for (int step = CS_UNR / 2; step >= 1; step /= 2)
#pragma unroll
        for (int u = 0; u < step; ++u)
#pragma unroll
            for (int e = 0; e < V; ++e) acc[u][e] += acc[u + step][e];
#pragma unroll
    for (int e = 0; e < V; ++e) part[warp][lane * V + e] = acc[0][e];
    __syncthreads();
    for (int c = threadIdx.x; c < 32 * V; c += 32 * CS_WARPS) {
        float t = part[0][c];
#pragma unroll
        for (int w = 1; w < CS_WARPS; ++w) t += part[w][c];
        total[c] = t;
    }
    __syncwarp();
    if (splits > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
    if (blockIdx.x == 0)
        for (int c = threadIdx.x; c < 32 * V; c += 32 * CS_WARPS) {
            float t = total[c];
            for (int s = 1; s < splits; ++s) {
                uint32_t at;
                float v;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(total + c)), "r"(s));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
                t += v;
            }
            const int64_t gc = (int64_t)blockIdx.y * (32 * V) + c;
            if (gc < cols) out[gc] = t;
        }
    __syncwarp();
    if (splits > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// The scatter of the gradient of an im2col matrix cols [n h w][kh kw c] (stride 1, output as large as the input) back onto the pixels:
// out[n][y][x] = sum over the taps (i, j), ascending, of cols[n][y - i + pad][x - j + pad][i][j], from +0, taps outside the image left
// out. V channels and one pixel per thread, tap after tap; bound by reading the matrix once and by the latency of its taps (131072 pixels
// x 9 x 32: 168 MB in 38.9 us, 4.3 TB/s; x 9 x 96 5.2). As a padded tensor, nine shifted additions and a copy it moved five times as much.
template <int V>
__global__ void __launch_bounds__(256)
fold_taps_kernel(const float* __restrict__ cols, uint32_t h, uint32_t w, uint32_t x0, uint32_t part, uint32_t cv, int kh, int kw, int pad, float* __restrict__ out) {
    chain_start();
    const uint32_t i = blockIdx.y * blockDim.x + threadIdx.x;              // within `part` pixels from x0 on of the image row blockIdx.x
    if (i >= part * cv) return;
    const int x = (int)(x0 + i / cv), y = (int)(blockIdx.x % h);
    const uint32_t ch = (i % cv) * V;
    const int64_t px = (int64_t)blockIdx.x * w + x, c = (int64_t)cv * V, pitch = (int64_t)kh * kw * c;
    float acc[V];
#pragma unroll
    for (int e = 0; e < V; ++e) acc[e] = 0.f;
    for (int di = 0; di < kh; ++di) {
        const int sy = y - di + pad;
        if (sy < 0 || sy >= (int)h) continue;
#pragma unroll 3
        for (int dj = 0; dj < kw; ++dj) {
            const int sx = x - dj + pad;
            if (sx < 0 || sx >= (int)w) continue;
            const float* src = cols + (px + (int64_t)(pad - di) * w + (pad - dj)) * pitch + (di * kw + dj) * c + ch;
            if (V == 4) {
                const float4 v = __ldcs(reinterpret_cast<const float4*>(src));
                acc[0] = __fadd_rn(acc[0], v.x); acc[1 % V] = __fadd_rn(acc[1 % V], v.y);
                acc[2 % V] = __fadd_rn(acc[2 % V], v.z); acc[3 % V] = __fadd_rn(acc[3 % V], v.w);
            } else {
                acc[0] = __fadd_rn(acc[0], __ldcs(src));
            }
        }
    }
    float* dst = out + px * c + ch;
    if (V == 4) *reinterpret_cast<float4*>(dst) = make_float4(acc[0], acc[1 % V], acc[2 % V], acc[3 % V]);
    else *dst = acc[0];
}

template <int V>
int column_sums(const float* x, int64_t rows, int64_t cols, int64_t ld, float* out, cudaStream_t st) {
    constexpr int64_t MOST = 65535ll * 32 * V;                    // columns a grid can have
    // a share of at least one round of loads, more CTAs than that only add to the exchange
    int splits = 1;
    while (splits < 8 && rows >= 2 * splits * CS_WARPS * CS_UNR) splits *= 2;
    for (int64_t c0 = 0; c0 < cols; c0 += MOST) {
        const int64_t n = cols - c0 < MOST ? cols - c0 : MOST;
        launch_chained_clusters(column_sums_kernel<V>, splits, dim3(splits, (unsigned)((n + 32 * V - 1) / (32 * V))), 32 * CS_WARPS, 0, st, chain_streamed(4 * rows * n, st), x + c0, rows, n, ld,
                                splits, out + c0);
        if (launch_status()) return HBFP_ERR_CUDA;
    }
    return HBFP_OK;
}

}  // namespace

int launch_add_bias(float* C, int64_t M, int64_t N, int64_t ldc, const float* bias, cudaStream_t st) {
    const bool quad = ((reinterpret_cast<uintptr_t>(C) | reinterpret_cast<uintptr_t>(bias)) & 15) == 0 && (ldc & 3) == 0 && (N & 3) == 0;
    const int64_t total = quad ? M * (N / 4) : M * N;
    const int64_t blocks = (total + 255) / 256, cap = 148 * 32;
    const unsigned grid = (unsigned)(blocks < cap ? blocks : cap);
    if (quad) launch_streamed(4 * M * N, add_bias_kernel<4>, grid, 256, 0, st, C, (uint32_t)N, ldc, bias, total);
    else launch_streamed(4 * M * N, add_bias_kernel<1>, grid, 256, 0, st, C, (uint32_t)N, ldc, bias, total);
    return launch_status();
}

int launch_fold_taps(const float* cols, int64_t n, int64_t h, int64_t w, int64_t c, int kh, int kw, int pad, float* out, cudaStream_t st) {
    if (n == 0) return HBFP_OK;
    const bool quad = c % 4 == 0 && ((reinterpret_cast<uintptr_t>(cols) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int64_t cv = quad ? c / 4 : c;
    const int threads = w * cv < 256 ? (int)round_up(w * cv, 32) : 256;
    // a grid has 65535 chunks of a row: wider rows in parts
    const int64_t most = 65535ll * threads / cv;
    if (n * h >= (1ll << 31) || w >= (1ll << 31) || most == 0) return HBFP_ERR_UNSUPPORTED;
    for (int64_t x0 = 0; x0 < w; x0 += most) {
        const uint32_t part = (uint32_t)(w - x0 < most ? w - x0 : most);
        const dim3 grid((unsigned)(n * h), (unsigned)((part * cv + threads - 1) / threads));
        if (quad) launch_streamed(4 * n * h * part * c * kh * kw, fold_taps_kernel<4>, grid, threads, 0, st, cols, (uint32_t)h, (uint32_t)w, (uint32_t)x0, part, (uint32_t)cv, kh, kw, pad, out);
        else launch_streamed(4 * n * h * part * c * kh * kw, fold_taps_kernel<1>, grid, threads, 0, st, cols, (uint32_t)h, (uint32_t)w, (uint32_t)x0, part, (uint32_t)cv, kh, kw, pad, out);
        if (launch_status()) return HBFP_ERR_CUDA;
    }
    return HBFP_OK;
}

int launch_column_sums(const float* x, int64_t rows, int64_t cols, int64_t ld, float* out, cudaStream_t st) {
    if (cols == 0) return HBFP_OK;
    // four columns per lane where that still leaves a CTA per SM
    const bool quad = (reinterpret_cast<uintptr_t>(x) & 15) == 0 && (ld & 3) == 0 && (cols & 3) == 0 && cols >= 2048;
    return quad ? column_sums<4>(x, rows, cols, ld, out, st) : column_sums<1>(x, rows, cols, ld, out, st);
}

}  // namespace hbfp
