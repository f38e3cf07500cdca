// Functional-connectivity kernels of the tvbx engine (arXiv 2311.13337,
// Sec. "Output": the FC is obtained from the covariance of the simulated
// series; Eq. 6: Pearson correlation; Table 2 "mean_FC").
//
// The E series is read through a SeriesLayout: the engine's set-blocked
// [P/4][T][N][4] or the sets-fastest [T][N][P]. For each set the kernels
// form block moments over the samples [t_begin, t_end):
//   G_b[k][j] = sum_{t in block b} (x_k(t) - m_k)(x_j(t) - m_j),
//   s_b[k]    = sum_{t in block b} (x_k(t) - m_k),
// with the shift m_k = the running mean kept by the simulation, or a given
// shift (any shift is exact; a close one avoids cancellation). The covariance over a union of
// blocks of length L is sum G_b - (sum s_b)(sum s_b)^T / L. Every producer's
// G_b is symmetric up to FP32 rounding, so the readers take the diagonal and
// the upper triangle (k < j) and write the FC symmetric.

#include <algorithm>

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"
#include "ptx_async.cuh"

namespace tvbx {

// ---------------------------------------------------------------------------
// Gram block moments in FP32. A CTA owns m groups of 4 sets (the 16-byte pieces
// of a sample), one moment block of samples and a range of 8 x 8 tiles of the
// upper triangle; a thread owns one tile of one set in registers. Chunks of Tt
// samples, copied a chunk ahead by cp.async into slots of their own threads, go
// minus the shift to one of two shared buffers [set][Tt][Npad] (regions fastest): a thread reads 16 values for 64
// multiply-adds, and the threads of a row of tiles share 8 of them. Column N of
// the buffer is 1, so the row sums are the Gram column N. Bound by the FP32
// pipe: 45 tiles per set at 68 regions, 81% of whose products are needed.
// Measured 4.16 ms on 4,096 x 68 x 5,000 (FMA pipe 51% busy; staging and shared
// memory take the rest); 4 x 4 tiles of 8 sets took 30 ms.
// ---------------------------------------------------------------------------
constexpr int FCR_MAXB = 12;      // most moment blocks the reductions take in registers
constexpr int FM_TILE = 8;
constexpr int FM_THREADS = 192;   // at most; two CTAs per SM (a third needs 96 registers, with spills)
constexpr int FM_LOADS = 6;       // 16-byte pieces a thread copies per chunk

struct FmPlan {
    int32_t npad;             // regions and the column of ones, rounded up to the tile
    int32_t tasks_per_set;    // tiles of the upper triangle
    int32_t m;                // groups of 4 sets per CTA
    int32_t chunks, per_chunk;// CTAs that share a group's tiles, tiles of each
    int32_t threads;
    int32_t Tt;               // samples per chunk
    int32_t merge;            // moment sub-blocks (of FcArgs::blk samples) added up in a stored block
    size_t smem;
};

static FmPlan fm_plan(int32_t N, int64_t P)
{
    FmPlan f;
    f.npad = (N + 1 + FM_TILE - 1) / FM_TILE * FM_TILE;
    const int nt = f.npad / FM_TILE;
    f.tasks_per_set = nt * (nt + 1) / 2;
    const int64_t groups = (P + 3) / 4;
    // few regions: several groups fill a CTA, as long as there are CTAs for every SM
    f.merge = 1;
    f.m = 1;
    while (f.m < 8 && 2 * f.m * 4 * f.tasks_per_set <= FM_THREADS && groups / (2 * f.m) >= 304) f.m *= 2;
    const int total = 4 * f.m * f.tasks_per_set;
    f.chunks = (total + FM_THREADS - 1) / FM_THREADS;
    f.per_chunk = (total + f.chunks - 1) / f.chunks;
    f.threads = (f.per_chunk + 31) / 32 * 32;
    if (f.threads < 64) f.threads = 64;
    f.Tt = FM_LOADS * f.threads / (N * f.m);
    f.Tt = f.Tt < 1 ? 1 : (f.Tt > 16 ? 16 : f.Tt);
    f.smem = sizeof(float) * (size_t)(4 * f.m) * (2 * (size_t)f.Tt * f.npad + N) +
             sizeof(float4) * (size_t)FM_LOADS * f.threads;
    return f;
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// two FP32 values in a register pair; fma.rn.f32x2 rounds each lane as fmaf
__device__ __forceinline__ uint64_t pair2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair2(uint64_t v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t x, uint64_t y)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(x), "l"(y));
}

// position of region k in a row of the buffer: 16-byte pieces 8 apart swap with
// their neighbour, so that the 32-byte strides of a warp's tiles meet every bank
__device__ __forceinline__ int fm_pos(int k)
{
    const int c = k >> 2;
    return ((c ^ ((c >> 3) & 1)) << 2) | (k & 3);
}

template <bool VEC>
__global__ void __launch_bounds__(FM_THREADS, 2)
fc_moments_kernel(const __grid_constant__ FcArgs a, const __grid_constant__ FmPlan f)
{
    extern __shared__ __align__(16) float fm_smem[];
    const int N = a.N, npad = f.npad, Tt = f.Tt, sets = 4 * f.m;
    const int tid = threadIdx.x, nthr = blockDim.x;
    float* xs = fm_smem;                                       // [2][sets][Tt][npad]
    const int buf = sets * Tt * npad;
    float4* sh = reinterpret_cast<float4*>(xs + 2 * buf);      // [m][N], the 4 sets of a group
    const int64_t b = blockIdx.x % a.n_blocks;
    const int64_t g0 = blockIdx.x / a.n_blocks * f.m;          // first group
    const int64_t Tn = a.t_end - a.t_begin;
    const int64_t blk = a.blk > 0 ? a.blk : Tn;
    int64_t t_lo = a.t_begin + b * blk;   // of the sub-block at hand

    for (int i = tid; i < 2 * buf; i += nthr) xs[i] = 0.0f;
    for (int i = tid; i < f.m * N; i += nthr) {
        const int g = i / N, k = i - g * N;
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int q = 0; q < 4; ++q) {
            const int64_t p = 4 * (g0 + g) + q;
            if (p >= a.P) continue;
            if (a.state) v[q] = a.state[(int64_t)SV_SUM_E * N * a.P + (int64_t)k * a.P + p] / (float)Tn;
            else if (a.shift) v[q] = a.shift[(int64_t)k * a.P + p];
        }
        sh[i] = make_float4(v[0], v[1], v[2], v[3]);
    }
    __syncthreads();
    for (int i = tid; i < 2 * sets * Tt; i += nthr) xs[i * npad + fm_pos(N)] = 1.0f;

    // this thread's tile
    const int task = blockIdx.y * f.per_chunk + tid;
    const bool works = tid < f.per_chunk && task < sets * f.tasks_per_set;
    int q = 0, kb = 0, jb = 0;
    if (works) {
        q = task / f.tasks_per_set;
        int r = task - q * f.tasks_per_set;
        const int nt = npad / FM_TILE;
        while (r >= nt - kb) { r -= nt - kb; ++kb; }
        jb = kb + r;
    }
    const int64_t p = 4 * g0 + q;
    const int ck0 = fm_pos(FM_TILE * kb), ck1 = fm_pos(FM_TILE * kb + 4);
    const int cj0 = fm_pos(FM_TILE * jb), cj1 = fm_pos(FM_TILE * jb + 4);
    uint64_t acc2[FM_TILE][FM_TILE / 2];   // two neighbouring columns each

    // 16-byte pieces (row = group and sample, region) of a chunk, dealt to the
    // threads in turn, a chunk ahead: VEC by cp.async into slots of their own
    // threads, else (rows that are not 16-byte aligned) in registers
    const int row_first = tid / N, k_first = tid - row_first * N, row_step = nthr / N, k_step = nthr - row_step * N;
    const int rows = f.m * Tt;
    float4* raw = reinterpret_cast<float4*>(sh + f.m * N) + tid;   // [FM_LOADS][threads]
    float4 v[VEC ? 1 : FM_LOADS];
    int64_t len = 0;
    auto fetch = [&](int64_t t0) {
        const int n = len - t0 < Tt ? (int)(len - t0) : Tt;
        const float* chunk = a.series + g0 * a.sl.sg + (t_lo + t0) * a.sl.st;
        int row = row_first, k = k_first;
#pragma unroll
        for (int u = 0; u < FM_LOADS; ++u) {
            const int g = f.m > 1 ? row / Tt : 0, t = f.m > 1 ? row - g * Tt : row;
            const int left = (int)(a.P - 4 * g0) - 4 * g;   // sets from this group on (a.P < 2^31)
            if (row < rows && t < n && left > 0) {
                const float* src = chunk + t * a.sl.st + k * a.sl.sk;
                if (f.m > 1) src += g * a.sl.sg;
                if constexpr (VEC) {
                    if (left >= 4) cp_async16(raw + u * nthr, src);
                    else
                        for (int c = 0; c < left; ++c) cp_async4(reinterpret_cast<float*>(raw + u * nthr) + c, src + c);
                } else {
                    v[u].x = src[0];
                    if (left > 1) v[u].y = src[1];
                    if (left > 2) v[u].z = src[2];
                    if (left > 3) v[u].w = src[3];
                }
            }
            row += row_step;
            k += k_step;
            if (k >= N) { k -= N; ++row; }
        }
        if constexpr (VEC) cp_async_commit();
    };
    auto put = [&](float* dst) {
        int row = row_first, k = k_first;
#pragma unroll
        for (int u = 0; u < FM_LOADS; ++u) {
            if (row < rows) {
                const int g = f.m > 1 ? row / Tt : 0;
                const float4 s4 = sh[g * N + k], x = VEC ? raw[u * nthr] : v[VEC ? 0 : u];
                float* at = dst + (3 * g * Tt + row) * npad + fm_pos(k);   // row 4 g Tt + t
                at[0] = x.x - s4.x;
                at[Tt * npad] = x.y - s4.y;
                at[2 * Tt * npad] = x.z - s4.z;
                at[3 * Tt * npad] = x.w - s4.w;
            }
            row += row_step;
            k += k_step;
            if (k >= N) { k -= N; ++row; }
        }
    };
    float* G = a.blocks + (p * a.n_blocks + b) * ((int64_t)N * N + N);
    const bool whole = kb < jb && FM_TILE * (jb + 1) <= N && N % 4 == 0;   // inside the triangle, rows 16-byte aligned
    float* cur = xs + buf;
    for (int sub = 0; sub < f.merge; ++sub, t_lo += blk) {
        len = (t_lo + blk < a.t_end ? t_lo + blk : a.t_end) - t_lo;
        if (len <= 0) break;
#pragma unroll
        for (int r = 0; r < FM_TILE; ++r)
#pragma unroll
            for (int c = 0; c < FM_TILE / 2; ++c) acc2[r][c] = 0;
        fetch(0);
        for (int64_t t0 = 0; t0 < len; t0 += Tt) {
            cur = cur == xs ? xs + buf : xs;
            if constexpr (VEC) cp_async_wait_all();
            put(cur);
            if (t0 + Tt < len) fetch(t0 + Tt);
            __syncthreads();   // chunk visible; every read of the other buffer's last chunk done
            if (!works) continue;
            const int n = len - t0 < Tt ? (int)(len - t0) : Tt;
            const float* row = cur + q * Tt * npad;
#pragma unroll 2
            for (int t = 0; t < n; ++t, row += npad) {
                const float4 x0 = *reinterpret_cast<const float4*>(row + ck0), x1 = *reinterpret_cast<const float4*>(row + ck1);
                const float4 y0 = *reinterpret_cast<const float4*>(row + cj0), y1 = *reinterpret_cast<const float4*>(row + cj1);
                const float x[FM_TILE] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
                const uint64_t y[FM_TILE / 2] = {pair2(y0.x, y0.y), pair2(y0.z, y0.w), pair2(y1.x, y1.y), pair2(y1.z, y1.w)};
#pragma unroll
                for (int r = 0; r < FM_TILE; ++r) {
                    const uint64_t xr = pair2(x[r], x[r]);
#pragma unroll
                    for (int c = 0; c < FM_TILE / 2; ++c) fma2(acc2[r][c], xr, y[c]);
                }
            }
        }
        if (!works || p >= a.P) continue;
        // the first sub-block's sums, or the sums so far and this one's
#pragma unroll
        for (int r = 0; r < FM_TILE; ++r) {
            const int k = FM_TILE * kb + r;
            if (k >= N) continue;
            float s[FM_TILE];
#pragma unroll
            for (int c = 0; c < FM_TILE / 2; ++c) unpair2(acc2[r][c], s[2 * c], s[2 * c + 1]);
            float* at = G + (int64_t)k * N + FM_TILE * jb;
            if (whole) {
                float4 lo = make_float4(s[0], s[1], s[2], s[3]), hi = make_float4(s[4], s[5], s[6], s[7]);
                if (sub > 0) {
                    const float4 l0 = reinterpret_cast<float4*>(at)[0], h0 = reinterpret_cast<float4*>(at)[1];
                    lo = make_float4(l0.x + lo.x, l0.y + lo.y, l0.z + lo.z, l0.w + lo.w);
                    hi = make_float4(h0.x + hi.x, h0.y + hi.y, h0.z + hi.z, h0.w + hi.w);
                }
                reinterpret_cast<float4*>(at)[0] = lo;
                reinterpret_cast<float4*>(at)[1] = hi;
            } else {
#pragma unroll
                for (int c = 0; c < FM_TILE; ++c) {
                    const int j = FM_TILE * jb + c;
                    float* to = j < N && j >= k ? at + c : (j == N ? G + (int64_t)N * N + k : nullptr);
                    if (to) *to = sub > 0 ? *to + s[c] : s[c];
                }
            }
        }
    }
}

// Per set: FC of each window (blocks [w, w + m)), upper-triangle vectors, and
// the Pearson correlation between every pair of window vectors.
__global__ void fcd_kernel(const float* __restrict__ blocks, int32_t N, int32_t n_blocks,
                           int32_t m, int32_t nw, int64_t Lw, float* __restrict__ vec,
                           float* __restrict__ fcd)
{
    extern __shared__ float sm[];   // diag [N] + mom [nw] + red
    const int p = blockIdx.x;
    const int M = N * (N - 1) / 2;
    const int64_t stride_b = (int64_t)N * N + N;
    const float* B = blocks + (int64_t)p * n_blocks * stride_b;
    float* V = vec + (int64_t)p * nw * M;
    float* dg = sm;
    float* mom = sm + N;         // [nw] means then inverse norms
    float* red = mom + 2 * nw;
    const float invL = 1.0f / (float)Lw;
    for (int w = 0; w < nw; ++w) {
        for (int k = threadIdx.x; k < N; k += blockDim.x) {
            float g = 0.0f, s = 0.0f;
            for (int b = w; b < w + m; ++b) {
                g += B[b * stride_b + (int64_t)k * N + k];
                s += B[b * stride_b + (int64_t)N * N + k];
            }
            const float v = g - s * s * invL;
            dg[k] = v > 0.0f ? sqrtf(v) : 0.0f;
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < M; idx += blockDim.x) {
            // idx -> (k, j), k < j, row by row
            int k = 0, r = idx;
            while (r >= N - 1 - k) { r -= N - 1 - k; ++k; }
            const int j = k + 1 + r;
            float g = 0.0f, sk = 0.0f, sj = 0.0f;
            for (int b = w; b < w + m; ++b) {
                g += B[b * stride_b + (int64_t)k * N + j];   // upper triangle (the matrices are symmetric)
                sk += B[b * stride_b + (int64_t)N * N + k];
                sj += B[b * stride_b + (int64_t)N * N + j];
            }
            const float c = g - sk * sj * invL;
            const float d = dg[k] * dg[j];
            V[(int64_t)w * M + idx] = d > 0.0f ? c / d : 0.0f;
        }
        __syncthreads();
    }
    // centre each window vector and normalise it
    for (int w = 0; w < nw; ++w) {
        float s = 0.0f;
        for (int i = threadIdx.x; i < M; i += blockDim.x) s += V[(int64_t)w * M + i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.0f;
            for (int q = 0; q < (int)(blockDim.x / 32); ++q) t += red[q];
            mom[w] = t / (float)M;
        }
        __syncthreads();
        const float mu = mom[w];
        float ss = 0.0f;
        for (int i = threadIdx.x; i < M; i += blockDim.x) {
            const float v = V[(int64_t)w * M + i] - mu;
            V[(int64_t)w * M + i] = v;
            ss += v * v;
        }
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        __syncthreads();
        if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.0f;
            for (int q = 0; q < (int)(blockDim.x / 32); ++q) t += red[q];
            mom[nw + w] = t > 0.0f ? rsqrtf(t) : 0.0f;
        }
        __syncthreads();
    }
    for (int pair = 0; pair < nw * nw; ++pair) {
        const int u = pair / nw, v = pair - u * nw;
        if (v < u) continue;
        float s = 0.0f;
        for (int i = threadIdx.x; i < M; i += blockDim.x) s += V[(int64_t)u * M + i] * V[(int64_t)v * M + i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.0f;
            for (int q = 0; q < (int)(blockDim.x / 32); ++q) t += red[q];
            float r = t * mom[nw + u] * mom[nw + v];
            if (u == v) r = 1.0f;
            fcd[((int64_t)p * nw + u) * nw + v] = r;
            fcd[((int64_t)p * nw + v) * nw + u] = r;
        }
        __syncthreads();
    }
}

__global__ void summary_kernel(const float* __restrict__ state, int32_t N, int32_t P, int64_t n_samples,
                               float* __restrict__ mean_e_hz, float* __restrict__ mean_i_hz)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= P) return;
    float se = 0.0f, si = 0.0f;
    for (int k = 0; k < N; ++k) {
        se += state[(int64_t)SV_SUM_E * N * P + (int64_t)k * P + p];
        si += state[(int64_t)SV_SUM_I * N * P + (int64_t)k * P + p];
    }
    const float scale = n_samples > 0 ? 1000.0f / ((float)N * (float)n_samples) : 0.0f;
    mean_e_hz[p] = se * scale;
    mean_i_hz[p] = si * scale;
}

cudaError_t launch_fc_moments(const FcArgs& a, cudaStream_t s)
{
    if (a.N > 384) return cudaErrorInvalidValue;
    FmPlan f = fm_plan(a.N, a.P);
    f.merge = a.merge > 0 ? a.merge : 1;
    const bool vec = a.sl.sk % 4 == 0 && a.sl.st % 4 == 0 && a.sl.sg % 4 == 0 &&
                     (reinterpret_cast<uintptr_t>(a.series) & 15) == 0;
    auto kern = vec ? fc_moments_kernel<true> : fc_moments_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem);
    if (e != cudaSuccess) return e;
    const int64_t groups = ((a.P + 3) / 4 + f.m - 1) / f.m;
    note_launch();
    kern<<<dim3((unsigned)(groups * a.n_blocks), f.chunks), f.threads, f.smem, s>>>(a, f);
    return cudaGetLastError();
}

// Moment sub-blocks of an FC without windows, of at least 256 samples and at
// most 12: a function of the samples alone, so that a set's sums do not depend
// on how many sets there are. Few sets store them as blocks that CTAs of their
// own form (*merge 1, and the reduction adds them in order); otherwise one CTA
// adds them up in the same order (*merge: their number).
int32_t fc_moment_blocks(int32_t N, int64_t P, int64_t Tn, int32_t* blk, int32_t* merge)
{
    int64_t n = Tn / 256 < 1 ? 1 : (Tn / 256 > FCR_MAXB ? FCR_MAXB : Tn / 256);
    *blk = 0;
    *merge = 1;
    if (N > 384 || n == 1) return 1;
    *blk = (int32_t)((Tn + n - 1) / n);
    n = (Tn + *blk - 1) / *blk;
    const FmPlan f = fm_plan(N, P);
    if (((P + 3) / 4 + f.m - 1) / f.m * f.chunks < 4 * 304) return (int32_t)n;   // 304 CTAs are resident
    *merge = (int32_t)n;
    return 1;
}

// Shift of each (region, set): mean of up to 64 evenly spaced samples of
// [t_begin, t_end). Any shift gives the same moments in exact arithmetic; one
// within a few standard deviations of the mean keeps the low-precision
// operands of the tensor-core path small relative to the fluctuations.
// Consecutive threads take consecutive elements of a sample: sets fastest in
// the [T][N][P] layout, (region, set within the group of 4) in the
// set-blocked one.
__global__ void fc_shift_kernel(const float* __restrict__ series, const SeriesLayout sl, int32_t N, int64_t P,
                                int64_t t_begin, int64_t t_end, float* __restrict__ shift)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t k, p;
    if (sl.sk == 4) {   // i = (group, region, set within the group)
        const int64_t g = i / (4 * (int64_t)N), q = i - g * 4 * (int64_t)N;
        k = q >> 2;
        p = 4 * g + (q & 3);
        if (p >= P) return;
    } else {            // i = (region, set)
        if (i >= (int64_t)N * P) return;
        k = i / P;
        p = i - k * P;
    }
    const int64_t o = k * P + p;   // shift[k][p]
    const int64_t Tn = t_end - t_begin;
    const int64_t n = Tn < 64 ? Tn : 64;
    float s = 0.0f;
    if (Tn <= (int64_t)(UINT32_MAX / 64)) {   // the same sample indices in 32-bit arithmetic
        const uint32_t tn = (uint32_t)Tn, nn = (uint32_t)n;
#pragma unroll 8
        for (uint32_t q = 0; q < nn; ++q) s += series[series_index(sl, t_begin + (q * tn) / nn, k, p)];
    } else {
        for (int64_t q = 0; q < n; ++q) s += series[series_index(sl, t_begin + (q * Tn) / n, k, p)];
    }
    shift[o] = n > 0 ? s / (float)n : 0.0f;
}

// acc += add over n floats: the block moments of one chunk of a streamed
// series folded into the moments of the run (the blocks of all chunks share
// one shift, so their sums add).
__global__ void fc_accumulate_kernel(const float* __restrict__ add, float* __restrict__ acc, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc[i] += add[i];
}

cudaError_t launch_fc_accumulate(const float* add, float* acc, int64_t n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    note_launch();
    fc_accumulate_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, s>>>(add, acc, n);
    return cudaGetLastError();
}

cudaError_t launch_fc_shift(const float* series, const SeriesLayout& sl, int32_t N, int64_t P, int64_t t_begin,
                            int64_t t_end, float* shift, cudaStream_t s)
{
    // threads: N P, or N x (P rounded up to 4) in the set-blocked layout
    const int64_t n = (int64_t)N * (sl.sk == 4 ? (P + 3) / 4 * 4 : P);
    note_launch();
    fc_shift_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(series, sl, N, P, t_begin, t_end, shift);
    return cudaGetLastError();
}

// Per set, from the block moments: Pearson FC over all samples, chi, mean
// off-diagonal FC and the FCD over nw > 0 windows of m blocks (Lw samples
// each) in one pass. One CTA per set; one warp per FC row; the
// window FC vectors (upper triangles) stay in shared memory. MW > 0: m == MW
// and n_blocks <= FCR_MAXB, block values in registers with compile-time
// indices; MW == 0: any m and n_blocks, block values re-read.
//
// Every producer writes a Gram matrix that is symmetric up to FP32 rounding
// (the SIMT kernel exactly, the tensor-core forms as H H^T or
// H H^T + H L^T + L H^T), so only the upper triangle is read: row r from
// column r + 1 on, along the row (coalesced).
constexpr int RED_THREADS = 512;
constexpr int RED_WARPS = RED_THREADS / 32;

// Work items of the row pass: (row r, first column of a 32-column chunk right
// of the diagonal), row by row; their number is sum over L = 1 .. N-1 of
// ceil(L / 32).
static __host__ __device__ inline int fc_reduce_items(int N)
{
    const int Q = (N - 1) / 32, R = (N - 1) % 32;
    return N > 1 ? 16 * Q * (Q + 1) + R * (Q + 1) : 0;
}

static __device__ __forceinline__ float warp_sum(float x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// The same without windows. The upper triangle is read along the rows, and both
// triangles of the FC are written along theirs: through the whole matrix in
// shared memory (WHOLE, up to FIN_WHOLE regions), else through the transposes
// of 32 x 32 tiles (column writes measured 1.62 ms on 32,768 x 68 and 2.79 ms
// on 4,096 x 360; tiles throughout 0.94 and 1.96).
constexpr int FIN_WHOLE = 112;   // 50 KB: four CTAs per SM
constexpr int FIN_THREADS = 256;
constexpr int FIN_WARPS = FIN_THREADS / 32;

template <bool WHOLE>
__global__ void __launch_bounds__(FIN_THREADS, 3)
fc_finish_kernel(const __grid_constant__ FcArgs a)
{
    extern __shared__ float sm[];
    const int N = a.N, nb = a.n_blocks;
    const int64_t p = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t stride_b = (int64_t)N * N + N;
    const float* B = a.blocks + p * nb * stride_b;
    const int64_t Tn = a.t_end - a.t_begin;
    float* sS = sm;                        // [N] row sums
    float* isd = sS + N;                   // [N] 1 / sd (0 if sd = 0)
    __shared__ float red[3][FIN_WARPS];
    const float invT = Tn > 0 ? 1.0f / (float)Tn : 0.0f;
    float* fc = a.fc ? a.fc + p * N * N : nullptr;

    float s_all = 0.0f, s_diag = 0.0f, s_fc = 0.0f;
    bool zero = false;
    for (int k = tid; k < N; k += FIN_THREADS) {
        float g = 0.0f, sk = 0.0f;
        for (int b = 0; b < nb; ++b) {
            g += B[b * stride_b + (int64_t)k * N + k];
            sk += B[b * stride_b + (int64_t)N * N + k];
        }
        const float v = g - sk * sk * invT;
        sS[k] = sk;
        isd[k] = v > 0.0f ? rsqrtf(v) : 0.0f;
        s_all += v;
        s_diag += v;
        if (!(isd[k] > 0.0f)) zero = true;   // no variance, or one that overflowed
    }
    if (zero) atomicOr(a.status + p, TVBX_SET_ZERO_VAR);
    __syncthreads();
    if constexpr (WHOLE) {
        // the whole FC in shared memory, pitch N | 1 (columns meet every bank)
        const int pitch = N | 1;
        float* F = isd + N;
        for (int r = warp; r < N; r += FIN_WARPS) {
            const float* Br = B + (int64_t)r * N;
            const float sr = sS[r], ir = isd[r];
            if (lane == 0) F[r * pitch + r] = 1.0f;
#pragma unroll 3
            for (int j = r + 1 + lane; j < N; j += 32) {
                float g = 0.0f;
                for (int b = 0; b < nb; ++b) g += Br[b * stride_b + j];
                const float c = g - sr * sS[j] * invT;
                const float x = c * ir * isd[j];
                s_all += 2.0f * c;
                s_fc += 2.0f * x;
                F[r * pitch + j] = x;
                F[j * pitch + r] = x;
            }
        }
        __syncthreads();
        if (fc)
            for (int i = tid; i < N * N; i += FIN_THREADS) fc[i] = F[i / N * pitch + i % N];
    } else {
        const int nt = (N + 31) / 32;
        float (*tr)[32][33] = reinterpret_cast<float (*)[32][33]>(isd + N);   // [2] tiles
        int parity = 0;
        for (int ti = 0; ti < nt; ++ti)
            for (int tj = ti; tj < nt; ++tj, parity ^= 1) {
                const int j = 32 * tj + lane;
                const float sj = j < N ? sS[j] : 0.0f, ij = j < N ? isd[j] : 0.0f;
                float g[32 / FIN_WARPS];
#pragma unroll
                for (int u = 0; u < 32 / FIN_WARPS; ++u) g[u] = 0.0f;
                for (int b = 0; b < nb; ++b)
#pragma unroll
                    for (int u = 0; u < 32 / FIN_WARPS; ++u) {
                        const int r = 32 * ti + warp + u * FIN_WARPS;
                        if (r < N && j < N && j > r) g[u] += B[b * stride_b + (int64_t)r * N + j];
                    }
#pragma unroll
                for (int u = 0; u < 32 / FIN_WARPS; ++u) {
                    const int rr = warp + u * FIN_WARPS, r = 32 * ti + rr;
                    if (r >= N || j >= N || j < r) continue;
                    if (j == r) {
                        if (fc) fc[(int64_t)r * N + r] = 1.0f;
                        continue;
                    }
                    const float c = g[u] - sS[r] * sj * invT;
                    const float x = c * isd[r] * ij;
                    s_all += 2.0f * c;
                    s_fc += 2.0f * x;
                    if (fc) fc[(int64_t)r * N + j] = x;
                    tr[parity][rr][lane] = x;
                }
                if (!fc) continue;
                __syncthreads();   // the tile is whole; the other buffer's readers are done with the tile before
                const int c0 = 32 * ti + lane;
#pragma unroll
                for (int u = 0; u < 32 / FIN_WARPS; ++u) {
                    const int rr = warp + u * FIN_WARPS, r = 32 * tj + rr;
                    if (r < N && c0 < r) fc[(int64_t)r * N + c0] = tr[parity][lane][rr];
                }
            }
    }
    s_all = warp_sum(s_all);
    s_diag = warp_sum(s_diag);
    s_fc = warp_sum(s_fc);
    if (lane == 0) { red[0][warp] = s_all; red[1][warp] = s_diag; red[2][warp] = s_fc; }
    __syncthreads();
    if (tid == 0) {
        float A = 0.0f, D = 0.0f, F = 0.0f;
        for (int w = 0; w < FIN_WARPS; ++w) { A += red[0][w]; D += red[1][w]; F += red[2][w]; }
        const float num = A / ((float)N * (float)N), den = D / (float)N;
        a.chi[p] = den > 0.0f ? sqrtf(fmaxf(num / den, 0.0f)) : 0.0f;
        a.mean_fc[p] = N > 1 ? F / ((float)N * (float)(N - 1)) : 0.0f;
    }
}

template <int MW>
__global__ void __launch_bounds__(RED_THREADS)
fc_reduce_kernel(const __grid_constant__ FcArgs a, int32_t m, int32_t nw, int64_t Lw, float* __restrict__ fcd)
{
    extern __shared__ float sm[];
    const int N = a.N, nb = a.n_blocks;
    const int64_t p = blockIdx.x;
    const int M = N * (N - 1) / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int64_t stride_b = (int64_t)N * N + N;
    const float* B = a.blocks + p * nb * stride_b;
    const int64_t Tn = a.t_end - a.t_begin;
    float* sSf = sm;                        // [N] row sums over all blocks
    float* isd = sSf + N;                   // [N] 1 / sd over all samples (0 if sd = 0)
    float* cdg = isd + N;                   // [N] variance over all samples
    float* sSw = cdg + N;                   // [nw][N] window row sums
    float* isdw = sSw + nw * N;             // [nw][N] window 1 / sd
    float* V = isdw + nw * N;               // [nw][M] window FC upper triangles
    float* red = V + (size_t)nw * M;        // [48] sums, [nw] inverse norms
    int* items = reinterpret_cast<int*>(red + 48 + nw);   // row-pass items
    const int n_items = fc_reduce_items(N);
    const float invT = Tn > 0 ? 1.0f / (float)Tn : 0.0f;
    const float invL = Lw > 0 ? 1.0f / (float)Lw : 0.0f;

    if (tid == RED_THREADS - 1) {
        int q = 0;
        for (int r = 0; r + 1 < N; ++r)
            for (int c = r + 1; c < N; c += 32) items[q++] = (r << 16) | c;
    }
    for (int k = tid; k < N; k += blockDim.x) {
        const float* sk_b = B + (int64_t)N * N + k;
        const float* dk_b = B + (int64_t)k * N + k;
        float g = 0.0f, sk = 0.0f;
        for (int b = 0; b < nb; ++b) { g += dk_b[b * stride_b]; sk += sk_b[b * stride_b]; }
        const float v = g - sk * sk * invT;
        sSf[k] = sk;
        cdg[k] = v;
        isd[k] = v > 0.0f ? rsqrtf(v) : 0.0f;
        for (int w = 0; w < nw; ++w) {
            float gw = 0.0f, sw = 0.0f;
            for (int b = w; b < w + m; ++b) { gw += dk_b[b * stride_b]; sw += sk_b[b * stride_b]; }
            const float vw = gw - sw * sw * invL;
            sSw[w * N + k] = sw;
            isdw[w * N + k] = vw > 0.0f ? rsqrtf(vw) : 0.0f;
        }
    }
    __syncthreads();

    float s_all = 0.0f, s_diag = 0.0f, s_fc = 0.0f;
    bool zero = false;
    float* fc = a.fc ? a.fc + p * N * N : nullptr;
    for (int k = tid; k < N; k += blockDim.x) {
        s_all += cdg[k];
        s_diag += cdg[k];
        if (!(isd[k] > 0.0f)) zero = true;
        if (fc) fc[(int64_t)k * N + k] = 1.0f;
    }
    // the row pass: items (row, 32-column chunk) dealt to the warps in turn,
    // so every warp gets the same number of chunks up to one
    for (int it = warp; it < n_items; it += RED_WARPS) {
        const int r = items[it] >> 16, jj = (items[it] & 0xffff) + lane;
        const float sr = sSf[r], ir = isd[r];
        const int e0 = r * N - r * (r + 1) / 2 - r - 1;   // triangle index of (r, jj) is e0 + jj
        const float* Br = B + (int64_t)r * N;              // row r of block 0
        if (jj < N) {
            // the block matrices at (r, jj)
            float g = 0.0f;
            float pre[FCR_MAXB + 1];
            if constexpr (MW > 0) {
                pre[0] = 0.0f;
#pragma unroll
                for (int b = 0; b < FCR_MAXB; ++b) {
                    const float gb = b < nb ? Br[b * stride_b + jj] : 0.0f;
                    pre[b + 1] = pre[b] + gb;
                }
                g = pre[FCR_MAXB];
            } else {
                for (int b = 0; b < nb; ++b) g += Br[b * stride_b + jj];
            }
            const float c = g - sr * sSf[jj] * invT;
            const float f = c * ir * isd[jj];
            s_all += 2.0f * c;
            s_fc += 2.0f * f;
            if (fc) {
                fc[(int64_t)r * N + jj] = f;
                fc[(int64_t)jj * N + r] = f;
            }
            if constexpr (MW > 0) {
#pragma unroll
                for (int w = 0; w + MW <= FCR_MAXB; ++w) {
                    if (w < nw) {
                        const float gw = pre[w + MW] - pre[w];
                        const float cw = gw - sSw[w * N + r] * sSw[w * N + jj] * invL;
                        V[(size_t)w * M + e0 + jj] = cw * isdw[w * N + r] * isdw[w * N + jj];
                    }
                }
            } else {
                for (int w = 0; w < nw; ++w) {
                    float gw = 0.0f;
                    for (int b = w; b < w + m; ++b)
                        gw += Br[b * stride_b + jj];
                    const float cw = gw - sSw[w * N + r] * sSw[w * N + jj] * invL;
                    V[(size_t)w * M + e0 + jj] = cw * isdw[w * N + r] * isdw[w * N + jj];
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        s_all += __shfl_xor_sync(0xffffffffu, s_all, o);
        s_diag += __shfl_xor_sync(0xffffffffu, s_diag, o);
        s_fc += __shfl_xor_sync(0xffffffffu, s_fc, o);
    }
    if (lane == 0) { red[warp] = s_all; red[16 + warp] = s_diag; red[32 + warp] = s_fc; }
    if (zero) atomicOr(a.status + p, TVBX_SET_ZERO_VAR);
    __syncthreads();
    if (tid == 0) {
        float A = 0.0f, D = 0.0f, F = 0.0f;
        for (int w = 0; w < nwarps; ++w) { A += red[w]; D += red[16 + w]; F += red[32 + w]; }
        const float num = A / ((float)N * (float)N), den = D / (float)N;
        a.chi[p] = den > 0.0f ? sqrtf(fmaxf(num / den, 0.0f)) : 0.0f;
        a.mean_fc[p] = N > 1 ? F / ((float)N * (float)(N - 1)) : 0.0f;
    }

    // FCD: centre and normalise each window vector (a warp per window), then
    // the products of window u with up to four windows v > u per warp item
    // (window u read once for all four)
    float* mom = red + 48;   // [nw] inverse norms
    for (int w = warp; w < nw; w += RED_WARPS) {
        float* v = V + (size_t)w * M;
        float sum = 0.0f;
        for (int i = lane; i < M; i += 32) sum += v[i];
        const float mean = warp_sum(sum) / (float)M;
        float ss = 0.0f;
        for (int i = lane; i < M; i += 32) {
            const float x = v[i] - mean;
            v[i] = x;
            ss += x * x;
        }
        ss = warp_sum(ss);
        if (lane == 0) {
            mom[w] = ss > 0.0f ? rsqrtf(ss) : 0.0f;
            fcd[(p * nw + w) * nw + w] = 1.0f;
        }
    }
    __syncthreads();
    int n_pitems = 0;   // items (u, first v) with v = u + 1, u + 5, ...
    for (int u = 0; u < nw; ++u) n_pitems += (nw - 1 - u + 3) / 4;
    for (int it = warp; it < n_pitems; it += RED_WARPS) {
        int u = 0, rem = it;
        while (rem >= (nw - 1 - u + 3) / 4) { rem -= (nw - 1 - u + 3) / 4; ++u; }
        const int v0 = u + 1 + 4 * rem, nv = nw - v0 < 4 ? nw - v0 : 4;
        const float* x = V + (size_t)u * M;
        const float* y0 = V + (size_t)v0 * M;
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int i = lane; i < M; i += 32) {
            const float xi = x[i];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < nv) acc[c] += xi * y0[(size_t)c * M + i];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c < nv) {
                const float dot = warp_sum(acc[c]);
                if (lane == 0) {
                    const int v2 = v0 + c;
                    const float r = dot * mom[u] * mom[v2];
                    fcd[(p * nw + u) * nw + v2] = r;
                    fcd[(p * nw + v2) * nw + u] = r;
                }
            }
        }
    }
}

static size_t fc_reduce_smem(int N, int nb, int nw)
{
    (void)nb;
    const size_t M = (size_t)N * (N - 1) / 2;
    return sizeof(float) * (3 * (size_t)N + 2 * (size_t)nw * N + (size_t)nw * M + 48 + (size_t)nw) +
           sizeof(int) * (size_t)fc_reduce_items(N);
}

template <int MW>
static cudaError_t launch_reduce_mw(const FcArgs& a, int32_t m, int32_t nw, int64_t Lw, float* fcd, size_t smem,
                                    cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(fc_reduce_kernel<MW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    note_launch();
    fc_reduce_kernel<MW><<<a.P, RED_THREADS, smem, s>>>(a, m, nw, Lw, fcd);
    return cudaGetLastError();
}

cudaError_t launch_fc_reduce(const FcArgs& a, int32_t m, int32_t nw, int64_t Lw, float* vec_scratch, float* fcd,
                             cudaStream_t s)
{
    if (nw == 0) return launch_fc_finalize(a, s);
    const size_t smem = fc_reduce_smem(a.N, a.n_blocks, nw);
    if (smem > 200 * 1024) {
        // window vectors too large for shared memory: the FC pass without
        // windows, then the FCD with the vectors in global scratch
        cudaError_t e = launch_fc_finalize(a, s);
        if (e != cudaSuccess) return e;
        return launch_fcd(a.blocks, a.P, a.N, a.n_blocks, m, nw, Lw, vec_scratch, fcd, s);
    }
    if (a.n_blocks <= FCR_MAXB) {
        switch (m) {
        case 1: return launch_reduce_mw<1>(a, m, nw, Lw, fcd, smem, s);
        case 2: return launch_reduce_mw<2>(a, m, nw, Lw, fcd, smem, s);
        case 3: return launch_reduce_mw<3>(a, m, nw, Lw, fcd, smem, s);
        case 4: return launch_reduce_mw<4>(a, m, nw, Lw, fcd, smem, s);
        default: break;
        }
    }
    return launch_reduce_mw<0>(a, m, nw, Lw, fcd, smem, s);
}

cudaError_t launch_fc_finalize(const FcArgs& a, cudaStream_t s)
{
    const bool whole = a.N <= FIN_WHOLE;
    const size_t smem = sizeof(float) * (2 * (size_t)a.N + (whole ? (size_t)a.N * (a.N | 1) : 2 * 32 * 33));
    auto kern = whole ? fc_finish_kernel<true> : fc_finish_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    note_launch();
    kern<<<a.P, FIN_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

size_t fc_reduce_needs_vec_scratch(int N, int nb, int nw) { return fc_reduce_smem(N, nb, nw) > 200 * 1024; }

cudaError_t launch_fcd(const float* blocks, int32_t P, int32_t N, int32_t n_blocks,
                       int32_t blocks_per_window, int32_t n_windows, int64_t window_samples,
                       float* vec_scratch, float* fcd, cudaStream_t s)
{
    const size_t smem = sizeof(float) * ((size_t)N + 2 * n_windows + 64);
    note_launch();
    fcd_kernel<<<P, 256, smem, s>>>(blocks, N, n_blocks, blocks_per_window, n_windows, window_samples,
                                    vec_scratch, fcd);
    return cudaGetLastError();
}

cudaError_t launch_summary(const float* state, int32_t N, int32_t P, int64_t n_samples,
                           float* mean_e_hz, float* mean_i_hz, cudaStream_t s)
{
    note_launch();
    summary_kernel<<<(P + 255) / 256, 256, 0, s>>>(state, N, P, n_samples, mean_e_hz, mean_i_hz);
    return cudaGetLastError();
}

}  // namespace tvbx
