// Table 2 analysis metrics of the excitatory rate series (arXiv 2311.13337,
// Sec. "Analysis metrics", Table 2: mean_PLI, mean_UD_duration,
// psd_fmax_ampmax, fit_psd_slope; Sec. "Vast parameter space exploration and
// analysis" names the PLI the mean phase lag index).
//
// Input: series [P][N][T] (set-major, time fastest; the layout of
// tvbx_series_range). Each series contributes its last T' samples, T' the
// largest number <= T whose prime factors are 2, 3 and 5, so every discrete
// Fourier transform below has length T'.
//
// Sets are processed in batches of B (scratch: the analytic signals of B
// sets, B * N * T' complex floats):
//  * an_series_kernel, one CTA per (set, region): the mean of the row to FP64;
//    UP / DOWN runs against that mean (rounded to FP32); the forward DFT of
//    the mean-removed row (in place in one shared-memory buffer: the row is
//    stored digit-reversed and transformed by decimation-in-time stages of
//    radix 2, 3, 4, 5; twiddles from a host FP64 table); the periodogram on
//    the PSD band; the analytic signal (real part: the row; imaginary part: the
//    inverse transform of -i times the positive-frequency spectrum, decimation
//    in frequency, in place, read back through the digit reversal), written to
//    scratch; for even T' both transforms are complex ones of length T'/2 of
//    the sample pairs;
//  * an_pli_kernel, one CTA per (time slice, set): time tiles of the N analytic signals in
//    shared memory; a thread owns a 4 x 4 block of region pairs and counts
//    sign(Im(z_k conj(z_j))) from the differences of the two rounded products,
//    so identical signals give exactly 0;
//  * an_finalize_kernel, one CTA per set: region-mean PSD, its peak on the
//    band, the least-squares fit of log10 PSD on log10 f (FP64), the pooled
//    UP / DOWN durations.

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"
#include "ptx_async.cuh"
#include "tvbx.h"

namespace tvbx {
namespace {

constexpr int AN_MAX_T = 8192;
constexpr int AN_MAX_STAGES = 16;
constexpr int AN_THREADS = 256;
// samples per time tile of the PLI kernel: TT (64; 32 or 8 when the two buffers of
// many regions would not fit); padded row stride of a tile plane TT + 4 floats
constexpr int PLI_TT_MAX = 64;
constexpr int PLI_TT_MIN = 8;
constexpr int PLI_THREADS = 160;   // 153 blocks of pairs at 68 regions

struct FftPlan {
    int n;
    int n_stages;
    int radix[AN_MAX_STAGES];
    // stage s (radix[s], DIT or DIF) has L1 = radix[0] ... radix[s-1]:
    // magic[s] = ceil(2^32 / L1) (0 for L1 = 1), so idx / L1 = umulhi(idx, magic)
    uint32_t magic[AN_MAX_STAGES];
    // twiddles of stage s in the plan's table: w_L^{j q} (L = L1 radix[s]) at
    // tw_off[s] + (q - 1) L1 + j, so that neighbouring butterflies read
    // neighbouring entries
    int tw_off[AN_MAX_STAGES];
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

__device__ __forceinline__ float2 twiddle(const float2* __restrict__ tw, int e, bool inv)
{
    float2 w = __ldg(tw + e);
    if (inv) w.y = -w.y;
    return w;
}

// R-point DFT v_k = sum_q w_R^{k q} u_q with w_R = exp(sg 2 pi i / R), in the
// symmetric forms (cos and sin of 2 pi / 3 and 2 pi k / 5).
template <int R>
__device__ __forceinline__ void butterfly(const float2 (&u)[R], float2 (&v)[R], float sg)
{
    if constexpr (R == 2) {
        v[0] = cadd(u[0], u[1]);
        v[1] = csub(u[0], u[1]);
    } else if constexpr (R == 4) {
        const float2 s02 = cadd(u[0], u[2]), d02 = csub(u[0], u[2]);
        const float2 s13 = cadd(u[1], u[3]), d13 = csub(u[1], u[3]);
        const float2 jd13 = make_float2(-sg * d13.y, sg * d13.x);   // (sg i) d13
        v[0] = cadd(s02, s13);
        v[1] = cadd(d02, jd13);
        v[2] = csub(s02, s13);
        v[3] = csub(d02, jd13);
    } else if constexpr (R == 3) {
        constexpr float S3 = 0.86602540378443865f;   // sin(2 pi / 3); cos(2 pi / 3) = -1/2
        const float2 t1 = cadd(u[1], u[2]), t2 = csub(u[1], u[2]);
        const float2 a0 = make_float2(fmaf(-0.5f, t1.x, u[0].x), fmaf(-0.5f, t1.y, u[0].y));
        const float bx = sg * S3 * t2.x, by = sg * S3 * t2.y;   // (sg S3) t2, times i below
        v[0] = cadd(u[0], t1);
        v[1] = make_float2(a0.x - by, a0.y + bx);
        v[2] = make_float2(a0.x + by, a0.y - bx);
    } else {
        constexpr float C1 = 0.30901699437494742f, C2 = -0.80901699437494742f;
        constexpr float S1 = 0.95105651629515357f, S2 = 0.58778525229247313f;
        const float2 t1 = cadd(u[1], u[4]), t2 = cadd(u[2], u[3]);
        const float2 t3 = csub(u[1], u[4]), t4 = csub(u[2], u[3]);
        const float2 a1 = make_float2(fmaf(C1, t1.x, fmaf(C2, t2.x, u[0].x)), fmaf(C1, t1.y, fmaf(C2, t2.y, u[0].y)));
        const float2 a2 = make_float2(fmaf(C2, t1.x, fmaf(C1, t2.x, u[0].x)), fmaf(C2, t1.y, fmaf(C1, t2.y, u[0].y)));
        // b1 = sg (S1 t3 + S2 t4), b2 = sg (S2 t3 - S1 t4)
        const float b1x = sg * fmaf(S1, t3.x, S2 * t4.x), b1y = sg * fmaf(S1, t3.y, S2 * t4.y);
        const float b2x = sg * fmaf(S2, t3.x, -S1 * t4.x), b2y = sg * fmaf(S2, t3.y, -S1 * t4.y);
        v[0] = make_float2(u[0].x + t1.x + t2.x, u[0].y + t1.y + t2.y);
        v[1] = make_float2(a1.x - b1y, a1.y + b1x);   // a1 + i b1
        v[4] = make_float2(a1.x + b1y, a1.y - b1x);   // a1 - i b1
        v[2] = make_float2(a2.x - b2y, a2.y + b2x);   // a2 + i b2
        v[3] = make_float2(a2.x + b2y, a2.y - b2x);   // a2 - i b2
    }
}

// In-place decimation-in-time stage of radix R on a (length n, input in
// digit-reversed order): butterfly j of a block of span L = L1 R combines
// a[blk L + j + q L1], twiddled by w_L^{j q} before the R-point DFT. tw: the
// stage's twiddles.
template <int R>
__device__ void dit_stage(float2* a, int n, int L1, uint32_t magic, const float2* __restrict__ tw, bool inv)
{
    const int L = L1 * R, m = n / R;
    const float sg = inv ? 1.0f : -1.0f;
    for (int idx = threadIdx.x; idx < m; idx += blockDim.x) {
        const int blk = magic ? (int)__umulhi((uint32_t)idx, magic) : idx;   // idx / L1
        const int j = idx - blk * L1;
        float2* p = a + blk * L + j;
        float2 u[R], v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const float2 y = p[q * L1];
            u[q] = (q == 0 || j == 0) ? y : cmul(y, twiddle(tw, (q - 1) * L1 + j, inv));
        }
        butterfly<R>(u, v, sg);
#pragma unroll
        for (int k = 0; k < R; ++k) p[k * L1] = v[k];
    }
}

// In-place decimation-in-frequency stage of radix R (natural-order input,
// span L = L1 R): the R-point DFT of a[blk L + j + q L1], each output k then
// twiddled by w_L^{j k}; after all stages the result is digit-reversed.
template <int R>
__device__ void dif_stage(float2* a, int n, int L1, uint32_t magic, const float2* __restrict__ tw, bool inv)
{
    const int L = L1 * R, m = n / R;
    const float sg = inv ? 1.0f : -1.0f;
    for (int idx = threadIdx.x; idx < m; idx += blockDim.x) {
        const int blk = magic ? (int)__umulhi((uint32_t)idx, magic) : idx;   // idx / L1
        const int j = idx - blk * L1;
        float2* p = a + blk * L + j;
        float2 u[R], v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) u[q] = p[q * L1];
        butterfly<R>(u, v, sg);
#pragma unroll
        for (int k = 0; k < R; ++k)
            p[k * L1] = (k == 0 || j == 0) ? v[k] : cmul(v[k], twiddle(tw, (k - 1) * L1 + j, inv));
    }
}

// Forward transform in place: a holds the input in digit-reversed order
// (a[perm[t]] = x[t]) and ends in natural order. tw: the plan's table. total:
// points of all the series that lie one after the other in a.
__device__ void fft_dit(float2* a, const FftPlan& plan, const float2* __restrict__ tw, bool inv, int total)
{
    int L1 = 1;
    for (int s = 0; s < plan.n_stages; ++s) {
        const int r = plan.radix[s];
        const uint32_t mg = plan.magic[s];
        const float2* ts = tw + plan.tw_off[s];
        switch (r) {
        case 2: dit_stage<2>(a, total, L1, mg, ts, inv); break;
        case 3: dit_stage<3>(a, total, L1, mg, ts, inv); break;
        case 4: dit_stage<4>(a, total, L1, mg, ts, inv); break;
        default: dit_stage<5>(a, total, L1, mg, ts, inv); break;
        }
        __syncthreads();
        L1 *= r;
    }
}

// Transform in place from natural order to digit-reversed order (result t at
// a[perm[t]]): the stages in reverse radix order.
__device__ void fft_dif(float2* a, const FftPlan& plan, const float2* __restrict__ tw, bool inv, int total)
{
    int L = plan.n;
    for (int s = plan.n_stages - 1; s >= 0; --s) {
        const int r = plan.radix[s];
        const int L1 = L / r;
        const uint32_t mg = plan.magic[s];
        const float2* ts = tw + plan.tw_off[s];
        switch (r) {
        case 2: dif_stage<2>(a, total, L1, mg, ts, inv); break;
        case 3: dif_stage<3>(a, total, L1, mg, ts, inv); break;
        case 4: dif_stage<4>(a, total, L1, mg, ts, inv); break;
        default: dif_stage<5>(a, total, L1, mg, ts, inv); break;
        }
        __syncthreads();
        L = L1;
    }
}

template <class T>
__device__ __forceinline__ T block_sum(T v, T* red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    T s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    return s;
}

// a + b rounded, and what the rounding left off.
__device__ __forceinline__ float two_sum(float a, float b, float& rest)
{
    const float sum = __fadd_rn(a, b), bb = __fsub_rn(sum, a);
    rest = __fadd_rn(__fsub_rn(a, __fsub_rn(sum, bb)), __fsub_rn(b, bb));
    return sum;
}

// One CTA per (set in batch, region). The row is held once in shared memory
// in digit-reversed order (a[perm[t]] = x_t), transformed in place forward
// (DIT, natural-order spectrum) and back (DIF, digit-reversed analytic
// signal).
//
// HALF (n even): the real row goes through a complex transform of length
// M = n / 2, z_m = x_2m + i x_2m+1 stored digit-reversed for the half plan
// (a[perm[m]] = z_m); with E, O the transforms of the even and odd samples,
// E_k = (Z_k + conj Z_{M-k}) / 2, O_k = -i (Z_k - conj Z_{M-k}) / 2, and
// X_k = E_k + w^k O_k, X_{M-k} = conj(E_k - w^k O_k), X_M = E_0 - O_0
// (w = exp(-2 pi i / n)). The analytic signal's real part is the mean-removed
// row itself, so only its imaginary part y, a real row with the spectrum
// -i X_k (0 < k < M; 0 at k = 0, M), is transformed back, again at half the
// length: with e = E_k and t = w^k O_k, the packed spectrum of y is
// -i t + e w^-k at k and i conj(t) - conj(e) w^k at M - k. Both untanglings
// are one pass over the pairs (k, M - k), in place.
//
// z_out: per (set, region) the real and then the imaginary part of the
// analytic signal, ns floats each (n rounded up to 4, zeros at the end).
// UP / DOWN: with the transitions t_1 < ... < t_m (samples whose state differs
// from the one before), the complete runs are [t_i, t_{i+1}). Their number in
// a state is the number of transitions into it, without the last one, and
// their samples are all samples of that state in [t_1, t_m); so sums, a
// minimum and a maximum over the samples give them, with no run followed.
//
// Bound by the L1 / shared-memory data path (the FFT passes and their
// twiddles): full-length inverse transforms, twiddles gathered from one
// natural-order table and a pass that followed the runs measured 6.0 ms on
// 1,024 x 68 x 5,000.
template <bool HALF>
__global__ void __launch_bounds__(AN_THREADS)
an_series_kernel(const float* __restrict__ series, int N, int64_t T, FftPlan plan, FftPlan plan_h,
                 const float2* __restrict__ tw, const float2* __restrict__ tws, const int* __restrict__ perm,
                 int band_lo, int band_n, float psd_scale, int64_t p0, float* __restrict__ psd_out,
                 int* __restrict__ ud_out, float* __restrict__ z_out, int ns)
{
    extern __shared__ float2 an_smem[];
    __shared__ double red_d[AN_THREADS / 32];
    __shared__ int red_i[5][AN_THREADS / 32];
    const int n = plan.n, M = n / 2;
    float2* a = an_smem;
    const int b = blockIdx.x / N, k = blockIdx.x - b * N;
    const float* row = series + ((p0 + b) * (int64_t)N + k) * T + (T - n);
    // mean: a thread's samples in three floats by error-free additions, no fewer
    // bits than FP64 keeps (1,024 x 68 x 5,000: 5.64 ms a call, 5.79 with FP64
    // additions), the threads in FP64
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        float rest;
        hi = two_sum(hi, row[t], rest);
        mid = two_sum(mid, rest, rest);
        lo = __fadd_rn(lo, rest);
    }
    double total = block_sum((double)hi + ((double)mid + (double)lo), red_d);
    if (!isfinite(total)) {   // infinities, or a sum beyond FP32: in FP64 throughout
        double s = 0.0;
        for (int t = threadIdx.x; t < n; t += blockDim.x) s += (double)row[t];
        total = block_sum(s, red_d);
    }
    const float theta = (float)(total / (double)n);
    // the mean-removed row in digit-reversed order, and the UP / DOWN counts
    int ups = 0, into_up = 0, into_dn = 0, first = n, last = -1;
    auto count = [&](int t, bool up, float before) {
        ups += up;
        if (t == 0 || up == (before > theta)) return;
        into_up += up;
        into_dn += !up;
        first = min(first, t);
        last = max(last, t);
    };
    if constexpr (HALF) {
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            const float x0 = row[2 * m], x1 = row[2 * m + 1];
            a[__ldg(perm + m)] = make_float2(x0 - theta, x1 - theta);
            count(2 * m, x0 > theta, m > 0 ? row[2 * m - 1] : 0.0f);
            count(2 * m + 1, x1 > theta, x0);
        }
    } else {
        for (int t = threadIdx.x; t < n; t += blockDim.x) {
            const float x = row[t];
            a[__ldg(perm + t)] = make_float2(x - theta, 0.0f);
            count(t, x > theta, t > 0 ? row[t - 1] : 0.0f);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ups = __reduce_add_sync(0xffffffffu, ups);
    into_up = __reduce_add_sync(0xffffffffu, into_up);
    into_dn = __reduce_add_sync(0xffffffffu, into_dn);
    first = __reduce_min_sync(0xffffffffu, first);
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0) {
        red_i[0][warp] = ups;
        red_i[1][warp] = into_up;
        red_i[2][warp] = into_dn;
        red_i[3][warp] = first;
        red_i[4][warp] = last;
    }
    __syncthreads();   // also: the row is whole
    if (threadIdx.x == 0) {
        for (int w = 1; w < AN_THREADS / 32; ++w) {
            ups += red_i[0][w];
            into_up += red_i[1][w];
            into_dn += red_i[2][w];
            first = min(first, red_i[3][w]);
            last = max(last, red_i[4][w]);
        }
        int nu = 0, su = 0, nd = 0, sd = 0;
        if (last > first) {   // at least two transitions
            const bool up_first = row[first] > theta, up_last = row[last] > theta;
            nu = into_up - up_last;
            nd = into_dn - !up_last;
            su = ups - (up_first ? 0 : first) - (up_last ? n - last : 0);
            sd = last - first - su;
        }
        int* u = ud_out + ((int64_t)b * N + k) * 4;
        u[0] = nu; u[1] = su; u[2] = nd; u[3] = sd;
    }
    float* pr = psd_out + ((int64_t)b * N + k) * band_n;
    if constexpr (HALF) {
        fft_dit(a, plan_h, tws, false, M);
        for (int i = threadIdx.x; i <= M / 2; i += blockDim.x) {
            if (i == 0) {
                a[0] = make_float2(0.0f, 0.0f);
                continue;
            }
            const float2 zk = a[i], zm = a[M - i], w = __ldg(tw + i);
            const float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));   // (Z_i + conj Z_{M-i}) / 2
            const float2 o = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));  // -i (Z_i - conj Z_{M-i}) / 2
            const float2 t = cmul(w, o);
            const float2 xk = cadd(e, t), xm = csub(e, t);                               // X_i, conj X_{M-i}
            if (i >= band_lo && i < band_lo + band_n) pr[i - band_lo] = psd_scale * fmaf(xk.x, xk.x, xk.y * xk.y);
            if (M - i != i && M - i >= band_lo && M - i < band_lo + band_n)
                pr[M - i - band_lo] = psd_scale * fmaf(xm.x, xm.x, xm.y * xm.y);
            const float2 c = cmul(e, make_float2(w.x, -w.y));                            // e w^-i
            a[i] = make_float2(c.x + t.y, c.y - t.x);
            if (M - i != i) a[M - i] = make_float2(t.y - c.x, t.x + c.y);                // i conj(t) - conj(c)
        }
        __syncthreads();
        fft_dif(a, plan_h, tws, true, M);
        const float inv_m = 1.0f / (float)M;
        float* xr = z_out + ((int64_t)b * N + k) * 2 * ns;
        float2* yr = reinterpret_cast<float2*>(xr + ns);
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            const float2 v = a[__ldg(perm + m)];
            yr[m] = make_float2(v.x * inv_m, v.y * inv_m);
        }
        for (int t = threadIdx.x; t < n; t += blockDim.x) xr[t] = row[t] - theta;
        for (int t = n + threadIdx.x; t < ns; t += blockDim.x) xr[t] = xr[ns + t] = 0.0f;
        return;
    } else {
        fft_dit(a, plan, tws, false, n);
        for (int i = threadIdx.x; i < band_n; i += blockDim.x) {
            const float2 v = a[band_lo + i];
            pr[i] = psd_scale * fmaf(v.x, v.x, v.y * v.y);
        }
        __syncthreads();   // the band is read before the spectrum is overwritten
        // analytic signal: spectrum times h (h_0 = 1, h_i = 2 below n/2, h_{n/2} = 1, 0 above)
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            float h = 0.0f;
            if (i == 0 || 2 * i == n) h = 1.0f;
            else if (2 * i < n) h = 2.0f;
            const float2 v = a[i];
            a[i] = make_float2(h * v.x, h * v.y);
        }
        __syncthreads();
    }
    fft_dif(a, plan, tws, true, n);
    const float inv_n = 1.0f / (float)n;
    float* xr = z_out + ((int64_t)b * N + k) * 2 * ns;
    for (int t = threadIdx.x; t < ns; t += blockDim.x) {
        const float2 v = t < n ? a[__ldg(perm + t)] : make_float2(0.0f, 0.0f);
        xr[t] = v.x * inv_n;
        xr[ns + t] = v.y * inv_n;
    }
}

// Packed products with a zero addend: a product that is zero is +0, and -0 is
// left only where a negative one underflows. So of two products without a sign
// the difference below is +0, but for -0 less +0 (which signless_sums counts).
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(0ull));
    return d;
}
// c - a b in each lane. With b = 1 it is the rounded difference of two already
// rounded products; a packed subtraction of two packed products may be
// contracted into a fused multiply-add (observed), which leaves the rounding
// error of one product instead of an exact 0 for identical signals.
__device__ __forceinline__ uint64_t diff_f32x2(uint64_t c, uint64_t a)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(0xbf800000bf800000ull), "l"(c));
    return d;
}
// The signs of both lanes as two halves: -1 (negative) or 0 in bits 0-15 and 16-31.
__device__ __forceinline__ uint32_t sign_halves(uint64_t d)
{
    uint32_t t;
    asm("prmt.b32 %0, %1, %2, 0xffbb;" : "=r"(t) : "r"((uint32_t)d), "r"((uint32_t)(d >> 32)));
    return t;
}
// min(m, |d|) over both lanes; NaN once a lane is NaN
__device__ __forceinline__ float min_abs(float m, uint64_t d)
{
    float r;
    asm("{\n .reg .f32 x, y;\n abs.f32 x, %1;\n abs.f32 y, %2;\n min.NaN.f32 %0, x, y, %3;\n}"
        : "=f"(r) : "f"(__uint_as_float((uint32_t)d)), "f"(__uint_as_float((uint32_t)(d >> 32))), "f"(m));
    return r;
}
// Negatives among the samples whose sign_halves were summed into s (fewer than
// 65,536 per half): with l negatives in the low half and h in the high one,
// -s = 65536 (h - l) + l.
__device__ __forceinline__ int negatives(uint32_t s)
{
    const uint32_t l = -s & 0xffffu, h = (((-s - l) >> 16) + l) & 0xffffu;
    return (int)(l + h);
}
// Adds to none[u][v] what the n samples of the pairs of rows xk + u row and
// xj + v row (imaginary parts a plane further) that have no sign (a difference
// that is zero or NaN) count for as positive or negative ones: 1, or -1 for -0.
__device__ __noinline__ void signless_sums(const float* xk, const float* xj, int row, int plane, int n, int (&none)[4][4])
{
    int c[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) c[u][v] = none[u][v];
#pragma unroll 1
    for (int t = 0; t < n; t += 4) {
        ulonglong2 ak[4], bk[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            ak[u] = *reinterpret_cast<const ulonglong2*>(xk + u * row + t);
            bk[u] = *reinterpret_cast<const ulonglong2*>(xk + plane + u * row + t);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const ulonglong2 aj = *reinterpret_cast<const ulonglong2*>(xj + v * row + t);
            const ulonglong2 bj = *reinterpret_cast<const ulonglong2*>(xj + plane + v * row + t);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t d[2] = {diff_f32x2(mul_f32x2(bk[u].x, aj.x), mul_f32x2(ak[u].x, bj.x)),
                                       diff_f32x2(mul_f32x2(bk[u].y, aj.y), mul_f32x2(ak[u].y, bj.y))};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int x = (int)(uint32_t)(d[i >> 1] >> (i & 1) * 32);
                    if (!(fabsf(__int_as_float(x)) > 0.0f)) c[u][v] += 1 | (x >> 31);
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) none[u][v] = c[u][v];
}

// One CTA per (time slice, set): cnt[k][j] += sum_t sign(Im(z_k conj(z_j))) for
// k < j over the slice (slices of a set balance the CTAs over the SMs: one CTA
// per set left a third of the last wave). Time tiles of the planes of real and
// imaginary parts come by cp.async into one of two buffers while the other is
// used. A thread owns a 4 x 4 block of region pairs: per pair and two samples
// two packed products p, q and the packed difference p - q, whose signs are
// summed as halves, two differences to an add, and whose smallest magnitude is
// kept; only where that is 0 or NaN does a thread go over the tile again for its
// samples without a sign (equal rows, silent regions, products that underflow, the
// zeros after a row's end), the others being positive or negative: 1,024 x 68 x
// 5,000 of silent regions take 14.5 ms with the transforms (16.9 with a count, and
// an atomic, per pair). Bound by the FMA and ALU pipes, about 3 issue
// slots per pair and sample, 2.5 ms per 1,024 x 68 x 5,000 (sign bits of p - q and of
// q - p shifted into words took 4 and 3.2 ms, comparisons and adds with
// predicates 17 and 4.98 ms).
template <int PLI_TT>
__global__ void __maxnreg__(128)   // 16 warps per SM: three CTAs of five
an_pli_kernel(const float* __restrict__ z_all, int N, int ns, int slice, int slices, int* __restrict__ cnt_all)
{
    constexpr int PLI_TS = PLI_TT + 4;
    // buffers [2][plane][(r mod 4) * NB + r / 4][PLI_TS]: the rows the lanes of a
    // quarter-warp read together (4 apart in r) are adjacent, and the stride
    // (4 mod 32 words) puts their 16-byte pieces in distinct banks
    extern __shared__ __align__(16) float tile[];
    const int b = blockIdx.x / slices;
    const int t_lo = (blockIdx.x - b * slices) * slice, t_hi = min(ns, t_lo + slice);   // multiples of 4
    const float* z = z_all + (int64_t)b * N * 2 * ns;
    const int NB = (N + 3) / 4, NR = NB * 4;
    const int plane = NR * PLI_TS, buf = 2 * plane;
    const int nbp = NB * (NB + 1) / 2;
    for (int r = N; r < NR; ++r)   // padded rows stay 0
        for (int i = threadIdx.x; i < 4 * PLI_TS; i += blockDim.x)
            tile[i / PLI_TS * plane + ((r & 3) * NB + (r >> 2)) * PLI_TS + i % PLI_TS] = 0.0f;
    auto fetch = [&](int t0, float* dst) {
        constexpr int C = PLI_TT / 4;   // 16-byte pieces per row
        for (int i = threadIdx.x; i < 2 * N * C; i += blockDim.x) {
            const int rp = i / C, c = i - rp * C, r = rp >> 1, pl = rp & 1;
            if (t0 + 4 * c < t_hi)
                cp_async16(dst + pl * plane + ((r & 3) * NB + (r >> 2)) * PLI_TS + 4 * c,
                           z + (int64_t)rp * ns + t0 + 4 * c);
        }
        cp_async_commit();
    };
    for (int base = 0; base < nbp; base += blockDim.x) {
        const int bp = base + threadIdx.x;
        int bk = 0, bj = 0;
        if (bp < nbp) {   // block pair (bk <= bj), row by row
            int rem = bp;
            while (rem >= NB - bk) { rem -= NB - bk; ++bk; }
            bj = bk + rem;
        }
        uint32_t sg[4][4];
        float least[4][4];   // smallest |p - q| of a tile
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) sg[u][v] = 0u;
        int none[4][4] = {};   // in local memory
        __syncthreads();   // the buffers are free
        fetch(t_lo, tile);
        float* cur = tile;
        for (int t0 = t_lo; t0 < t_hi; t0 += PLI_TT) {
            cp_async_wait_all();
            __syncthreads();   // this tile is whole, the other buffer's last reads are done
            float* next = cur == tile ? tile + buf : tile;
            if (t0 + PLI_TT < t_hi) fetch(t0 + PLI_TT, next);
            const int tl = min(PLI_TT, t_hi - t0);
            if (bp < nbp) {
                const float* xk0 = cur + bk * PLI_TS;
                const float* xj0 = cur + bj * PLI_TS;
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) least[u][v] = 1.0f;   // any positive number
                for (int t = 0; t < tl; t += 4) {
                    ulonglong2 xk[4], yk[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        xk[u] = *reinterpret_cast<const ulonglong2*>(xk0 + u * NB * PLI_TS + t);
                        yk[u] = *reinterpret_cast<const ulonglong2*>(xk0 + plane + u * NB * PLI_TS + t);
                    }
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const ulonglong2 xj = *reinterpret_cast<const ulonglong2*>(xj0 + v * NB * PLI_TS + t);
                        const ulonglong2 yj = *reinterpret_cast<const ulonglong2*>(xj0 + plane + v * NB * PLI_TS + t);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            // Im(z_k conj(z_j)) = y_k x_j - x_k y_j, each product rounded
                            const uint64_t d0 = diff_f32x2(mul_f32x2(yk[u].x, xj.x), mul_f32x2(xk[u].x, yj.x));
                            const uint64_t d1 = diff_f32x2(mul_f32x2(yk[u].y, xj.y), mul_f32x2(xk[u].y, yj.y));
                            sg[u][v] += sign_halves(d0) + sign_halves(d1);
                            least[u][v] = min_abs(min_abs(least[u][v], d0), d1);
                        }
                    }
                }
                bool any = false;   // pairs with a sample without a sign
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int kk = bk * 4 + u, jj = bj * 4 + v;
                        any = any || (!(least[u][v] > 0.0f) && kk < jj && jj < N);
                    }
                if (any) signless_sums(xk0, xj0, NB * PLI_TS, plane, tl, none);
            }
            cur = next;
        }
        if (bp < nbp) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int kk = bk * 4 + u, jj = bj * 4 + v;
                    if (kk < jj && jj < N)
                        atomicAdd(cnt_all + ((int64_t)b * N + kk) * N + jj,
                                  t_hi - t_lo - 2 * negatives(sg[u][v]) - none[u][v]);
                }
        }
    }
}

// One CTA per set: mean phase lag index (the mean over k < j of |cnt| / n), PSD
// mean over regions, peak, fit; UP / DOWN means.
__global__ void __launch_bounds__(AN_THREADS)
an_finalize_kernel(const float* __restrict__ psd, const int* __restrict__ ud, const int* __restrict__ cnt, int N, int n,
                   int band_lo, int band_n, double df, double dt_ms, int64_t p0, float* __restrict__ out)
{
    extern __shared__ float an_psd[];   // [band_n]
    __shared__ double red_d[4][AN_THREADS / 32];
    __shared__ float s_best[AN_THREADS];
    __shared__ int s_besti[AN_THREADS];
    __shared__ int s_pos;
    __shared__ float red_f[AN_THREADS / 32];
    const int b = blockIdx.x;
    float lag = 0.0f;
    const int* cb = cnt + (int64_t)b * N * N;
    for (int k = threadIdx.x >> 5; k < N; k += AN_THREADS / 32)
        for (int j = k + 1 + (threadIdx.x & 31); j < N; j += 32) lag += (float)abs(cb[k * N + j]) / (float)n;
    lag = block_sum(lag, red_f);
    const float* pb = psd + (int64_t)b * N * band_n;
    for (int i = threadIdx.x; i < band_n; i += blockDim.x) {
        float s = 0.0f;
        for (int k = 0; k < N; ++k) s += pb[(int64_t)k * band_n + i];
        an_psd[i] = s / (float)N;
    }
    if (threadIdx.x == 0) s_pos = 1;
    __syncthreads();
    // peak: largest value, ties to the lower frequency
    float best = -INFINITY;
    int bi = -1;
    for (int i = threadIdx.x; i < band_n; i += blockDim.x)
        if (an_psd[i] > best) { best = an_psd[i]; bi = i; }
    s_best[threadIdx.x] = best;
    s_besti[threadIdx.x] = bi;
    // least squares of log10 PSD on log10 f (FP64)
    double su = 0.0, sv = 0.0, suu = 0.0, suv = 0.0;
    for (int i = threadIdx.x; i < band_n; i += blockDim.x) {
        const float pv = an_psd[i];
        if (!(pv > 0.0f)) { s_pos = 0; continue; }
        const double u = log10((double)(band_lo + i) * df), v = log10((double)pv);
        su += u; sv += v; suu += u * u; suv += u * v;
    }
    su = block_sum(su, red_d[0]);
    sv = block_sum(sv, red_d[1]);
    suu = block_sum(suu, red_d[2]);
    suv = block_sum(suv, red_d[3]);
    if (threadIdx.x == 0) {
        float bv = -INFINITY;
        int bix = -1;
        for (int t = 0; t < (int)blockDim.x; ++t)
            if (s_besti[t] >= 0 && (s_best[t] > bv || (s_best[t] == bv && s_besti[t] < bix))) {
                bv = s_best[t];
                bix = s_besti[t];
            }
        int64_t nu = 0, suL = 0, nd = 0, sdL = 0;
        for (int k = 0; k < N; ++k) {
            const int* u = ud + ((int64_t)b * N + k) * 4;
            nu += u[0]; suL += u[1]; nd += u[2]; sdL += u[3];
        }
        const float nan = __int_as_float(0x7fc00000);
        float* o = out + (p0 + b) * (int64_t)TVBX_AN_COUNT;
        o[TVBX_AN_MEAN_PLI] = N > 1 ? lag / (float)(N * (N - 1) / 2) : nan;
        o[TVBX_AN_PSD_FMAX] = bix >= 0 ? (float)((double)(band_lo + bix) * df) : nan;
        o[TVBX_AN_PSD_AMPMAX] = bix >= 0 ? bv : nan;
        const double nb = (double)band_n;
        const double den = nb * suu - su * su;
        if (band_n >= 2 && s_pos && den != 0.0) {
            const double slope = (nb * suv - su * sv) / den;
            o[TVBX_AN_PSD_A] = (float)(-slope);
            o[TVBX_AN_PSD_B] = (float)pow(10.0, (sv - slope * su) / nb);
        } else {
            o[TVBX_AN_PSD_A] = nan;
            o[TVBX_AN_PSD_B] = nan;
        }
        o[TVBX_AN_UP_MS] = nu ? (float)((double)suL * dt_ms / (double)nu) : nan;
        o[TVBX_AN_DOWN_MS] = nd ? (float)((double)sdL * dt_ms / (double)nd) : nan;
        o[TVBX_AN_N_UP] = (float)nu;
        o[TVBX_AN_UP_SAMPLES] = (float)suL;
        o[TVBX_AN_N_DOWN] = (float)nd;
        o[TVBX_AN_DOWN_SAMPLES] = (float)sdL;
    }
}

// ---------------------------------------------------------------------------
// phFCD (Sec. "Output": the phase functional connectivity dynamics of the
// BOLD series; Deco et al. 2017): phases of the band-limited analytic
// signals, phase-coherence matrices dFC_kj(t) = cos(theta_k - theta_j), and
// the cosine similarity of their upper triangles for every t1 < t2. With unit
// phasors u_k(t), the dot product of two triangles is
//   ((|sum_k u_k(t1) u_k(t2)|^2 - N) + (|sum_k u_k(t1) conj u_k(t2)|^2 - N)) / 4,
// so a pair of times costs two complex sums over the regions.
// ---------------------------------------------------------------------------
constexpr int PF_TILE = 64;
constexpr int PF_THREADS = 256;

// Unit phasors of the band-limited analytic signals, U[b][k][t] for the T' kept
// samples. A CTA takes S adjacent sets of a region (S a power of two, S n <=
// AN_MAX_T): a short BOLD series alone leaves most threads of a stage idle, and
// the sets of a sample are neighbours in memory (one series per CTA and
// 8-byte writes at stride N: 441 us on 512 x 68 x 300).
__global__ void __launch_bounds__(AN_THREADS)
an_phase_kernel(const float* __restrict__ bold, int N, int64_t P, int64_t Tb, FftPlan plan,
                const float2* __restrict__ tw, const int* __restrict__ perm, int band_lo, int band_hi, int discard,
                int64_t p0, int nb, int S, float2* __restrict__ U)
{
    extern __shared__ float2 an_smem[];
    __shared__ double part[AN_THREADS];
    __shared__ float mean[AN_THREADS];
    const int n = plan.n, Tp = n - 2 * discard;
    float2* a = an_smem;   // [S][n], each series in digit-reversed order, transformed in place
    const int b0 = blockIdx.x / N * S, k = blockIdx.x % N;
    const int64_t NP = (int64_t)N * P;
    const float* col = bold + (Tb - n) * NP + (int64_t)k * P + p0 + b0;
    const int q = threadIdx.x % S;   // this thread's series, times threadIdx.x / S, + AN_THREADS / S, ...
    double s = 0.0;
    for (int t = threadIdx.x / S; t < n; t += AN_THREADS / S) {
        const float x = b0 + q < nb ? col[(int64_t)t * NP + q] : 0.0f;
        a[q * n + __ldg(perm + t)] = make_float2(x, 0.0f);
        s += (double)x;
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int h = AN_THREADS / 2; h >= S; h >>= 1) {
        if (threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x < S) mean[threadIdx.x] = (float)(part[threadIdx.x] / (double)n);
    __syncthreads();
    const float mu = mean[q];
    for (int t = threadIdx.x / S; t < n; t += AN_THREADS / S) a[q * n + t].x -= mu;
    __syncthreads();
    fft_dit(a, plan, tw, false, S * n);
    for (int i = threadIdx.x / S; i < n; i += AN_THREADS / S) {
        const float h = (i >= band_lo && i <= band_hi) ? 2.0f : 0.0f;
        a[q * n + i] = make_float2(h * a[q * n + i].x, h * a[q * n + i].y);
    }
    __syncthreads();
    fft_dif(a, plan, tw, true, S * n);
    for (int i = threadIdx.x; i < S * Tp; i += AN_THREADS) {
        const int r = i / Tp, t = i - r * Tp;
        if (b0 + r >= nb) break;
        const float2 v = a[r * n + __ldg(perm + t + discard)];
        const float len = hypotf(v.x, v.y);
        U[((int64_t)(b0 + r) * N + k) * Tp + t] = len > 0.0f ? make_float2(v.x / len, v.y / len) : make_float2(1.0f, 0.0f);
    }
}

// (x, x) (c, d) + acc in both lanes
__device__ __forceinline__ void fma_f32x2(uint64_t& acc, float x, uint64_t cd)
{
    uint64_t xx;
    asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(xx), "l"(cd));
}

// One CTA per (tile pair ta <= tc of 64 x 64 times, set in batch). Tiles are
// stored region-major in shared memory; thread (m, q) owns times
// ta*64 + q + 16 i and tc*64 + m + 16 j (i, j < 4), so a half-warp reads 16
// consecutive 8-byte phasors. With the four real sums xx, xy, yx, yy over the
// regions, |sum u u'|^2 + |sum u conj u'|^2 = 2 (xx^2 + xy^2 + yx^2 + yy^2):
// two packed multiply-adds per pair and region where the two complex sums took
// eight scalar ones (832 us on 512 x 68 x 300).
__global__ void __launch_bounds__(PF_THREADS)
an_phfcd_kernel(const float2* __restrict__ U, int N, int Tp, int64_t p0, int64_t M2, float* __restrict__ out)
{
    extern __shared__ float2 pf_smem[];
    float2* Ua = pf_smem;                       // [N][64]
    float2* Uc = pf_smem + (size_t)N * PF_TILE;  // [N][64]
    __shared__ float nrm_a[PF_TILE], nrm_c[PF_TILE];
    const int nt = (Tp + PF_TILE - 1) / PF_TILE;
    int ta = 0, rem = blockIdx.x;
    while (rem >= nt - ta) { rem -= nt - ta; ++ta; }
    const int tc = ta + rem;
    const int b = blockIdx.y;
    const float2* Ub = U + (int64_t)b * N * Tp;
    for (int i = threadIdx.x; i < PF_TILE * N; i += blockDim.x) {
        const int k = i / PF_TILE, r = i % PF_TILE;
        const int t1 = ta * PF_TILE + r, t2 = tc * PF_TILE + r;
        Ua[i] = t1 < Tp ? Ub[(int64_t)k * Tp + t1] : make_float2(0.0f, 0.0f);
        Uc[i] = t2 < Tp ? Ub[(int64_t)k * Tp + t2] : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    // |V(t)| from S = sum_k u_k^2: |V|^2 = ((|S|^2 - N) + N^2 - N) / 4
    if (threadIdx.x < 2 * PF_TILE) {
        const int r = threadIdx.x & (PF_TILE - 1);
        const float2* T = threadIdx.x < PF_TILE ? Ua : Uc;
        float sx = 0.0f, sy = 0.0f;
        for (int k = 0; k < N; ++k) {
            const float2 u = T[k * PF_TILE + r];
            sx += u.x * u.x - u.y * u.y;
            sy += 2.0f * u.x * u.y;
        }
        const float fN = (float)N;
        const float v2 = 0.25f * (fmaf(sx, sx, sy * sy) - fN + fN * fN - fN);
        (threadIdx.x < PF_TILE ? nrm_a : nrm_c)[r] = sqrtf(fmaxf(v2, 0.0f));
    }
    __syncthreads();
    const int q = threadIdx.x >> 4, m = threadIdx.x & 15;
    uint64_t xv[4][4], yv[4][4];   // (xx, xy), (yx, yy)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) xv[i][j] = yv[i][j] = 0;
#pragma unroll 2
    for (int k = 0; k < N; ++k) {
        float2 ua[4];
        uint64_t uc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ua[i] = Ua[k * PF_TILE + q + 16 * i];
            uc[i] = *reinterpret_cast<const uint64_t*>(Uc + k * PF_TILE + m + 16 * i);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                fma_f32x2(xv[i][j], ua[i].x, uc[j]);
                fma_f32x2(yv[i][j], ua[i].y, uc[j]);
            }
    }
    const float fN = (float)N;
    float* o = out + (p0 + b) * M2;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ra = q + 16 * i, rc = m + 16 * j;
            const int t1 = ta * PF_TILE + ra, t2 = tc * PF_TILE + rc;
            if (t1 < t2 && t2 < Tp) {
                const float xx = __uint_as_float((uint32_t)xv[i][j]), xy = __uint_as_float((uint32_t)(xv[i][j] >> 32));
                const float yx = __uint_as_float((uint32_t)yv[i][j]), yy = __uint_as_float((uint32_t)(yv[i][j] >> 32));
                const float dot = 0.5f * (fmaf(xx, xx, yy * yy) + fmaf(xy, xy, yx * yx) - fN);
                const int64_t e = (int64_t)t1 * Tp - (int64_t)t1 * (t1 + 1) / 2 + (t2 - t1 - 1);
                o[e] = dot / (nrm_a[ra] * nrm_c[rc]);
            }
        }
}

int smooth_length(int64_t n)
{
    for (int64_t m = std::min<int64_t>(n, AN_MAX_T); m > 0; --m) {
        int64_t r = m;
        for (int f : {2, 3, 5})
            while (r % f == 0) r /= f;
        if (r == 1) return (int)m;
    }
    return 0;
}

bool make_plan(int n, FftPlan& p)
{
    p.n = n;
    p.n_stages = 0;
    int r = n;
    // radix 5s, then 3s, then 4s, then a final 2
    for (int f : {5, 3, 4, 2}) {
        while (r % f == 0) {
            if (p.n_stages == AN_MAX_STAGES) return false;
            p.radix[p.n_stages++] = f;
            r /= f;
        }
    }
    if (r != 1) return false;
    uint64_t L1 = 1;
    int off = 0;
    for (int s = 0; s < p.n_stages; ++s) {
        p.tw_off[s] = off;
        off += (p.radix[s] - 1) * (int)L1;
        // idx < 2^13 and L1 < 2^13: floor(idx * ceil(2^32 / L1) / 2^32) = floor(idx / L1)
        p.magic[s] = L1 == 1 ? 0u : (uint32_t)((((uint64_t)1 << 32) + L1 - 1) / L1);
        L1 *= (uint64_t)p.radix[s];
    }
    return true;
}

// exp(-2 pi i e / n) for 0 <= e < n, from FP64.
std::vector<float2> roots(int n)
{
    std::vector<float2> w(n);
    for (int e = 0; e < n; ++e) {
        const double ang = -2.0 * 3.14159265358979323846 * (double)e / (double)n;
        w[e] = make_float2((float)std::cos(ang), (float)std::sin(ang));
    }
    return w;
}

// The plan's twiddle table (FftPlan::tw_off) from the roots of a multiple of its length.
std::vector<float2> stage_twiddles(const FftPlan& p, const std::vector<float2>& w)
{
    std::vector<float2> t;
    int L1 = 1;
    for (int s = 0; s < p.n_stages; ++s) {
        const int step = (int)w.size() / (L1 * p.radix[s]);
        for (int q = 1; q < p.radix[s]; ++q)
            for (int j = 0; j < L1; ++j) t.push_back(w[(size_t)step * j * q]);
        L1 *= p.radix[s];
    }
    return t;
}

// Digit reversal of the plan: the decimation-in-time stages (radix[0] first)
// take x_t at position perm[t], and the decimation-in-frequency stages leave
// output t at perm[t]. With t = sum_k d_k W_k in the number system whose
// least significant digit has radix radix[m-1] (W_0 = 1, W_{k+1} = W_k
// radix[m-1-k]), perm[t] = sum_k d_{m-1-k} V_k with V_0 = 1,
// V_{k+1} = V_k radix[k].
std::vector<int> digit_reversal(const FftPlan& p)
{
    const int m = p.n_stages;
    std::vector<int> perm(p.n);
    for (int t = 0; t < p.n; ++t) {
        int d[AN_MAX_STAGES];
        int rem = t;
        for (int k = 0; k < m; ++k) {
            const int r = p.radix[m - 1 - k];
            d[k] = rem % r;
            rem /= r;
        }
        int v = 0, w = 1;
        for (int k = 0; k < m; ++k) {
            v += d[m - 1 - k] * w;
            w *= p.radix[k];
        }
        perm[t] = v;
    }
    return perm;
}

#define ACK(call, what)                                                                              \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ == cudaErrorMemoryAllocation) return report_error(TVBX_E_OOM, "%s: out of memory", what); \
        if (e_ != cudaSuccess) return report_error(TVBX_E_CUDA, "%s: %s", what, cudaGetErrorString(e_)); \
    } while (0)

struct AnScratch {
    std::vector<void*> ptrs;
    cudaStream_t s;
    explicit AnScratch(cudaStream_t st) : s(st) {}
    template <class T> cudaError_t get(T** p, size_t n)
    {
        void* q = nullptr;
        cudaError_t e = cudaMallocAsync(&q, sizeof(T) * (n ? n : 1), s);
        if (e == cudaSuccess) {
            ptrs.push_back(q);
            *p = static_cast<T*>(q);
        }
        return e;
    }
    ~AnScratch()
    {
        for (void* q : ptrs) cudaFreeAsync(q, s);
    }
};

// Copy stream and events of a host-input analysis (released when the call
// returns; work still queued completes first). Before the release, the
// compute stream s waits for everything queued on the copy stream, so the
// staging buffers, freed on s afterwards, outlive every copy into them even
// when the call returns early on an error.
struct HostPipe {
    cudaStream_t s = nullptr;
    cudaStream_t cs = nullptr;
    cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // start, ready[2], free[2]
    ~HostPipe()
    {
        if (cs) {
            cudaEvent_t done = nullptr;
            if (cudaEventCreateWithFlags(&done, cudaEventDisableTiming) == cudaSuccess) {
                if (cudaEventRecord(done, cs) == cudaSuccess) cudaStreamWaitEvent(s, done, 0);
                cudaEventDestroy(done);
            } else {
                cudaStreamSynchronize(cs);
            }
        }
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        if (cs) cudaStreamDestroy(cs);
    }
};

// Whether p is ordinary host memory (pageable or pinned) rather than memory
// a kernel can read.
bool is_host_pointer(const void* p)
{
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return true;
    }
    return pa.type == cudaMemoryTypeHost || pa.type == cudaMemoryTypeUnregistered;
}

}  // namespace
}  // namespace tvbx

using namespace tvbx;

extern "C" tvbx_status tvbx_series_analysis(const float* series, int32_t n_regions, int64_t n_sets, int64_t n_samples,
                                            double dt_ms, float* out, int32_t* n_used, void* cuda_stream)
{
    const int N = n_regions;
    const int64_t P = n_sets, T = n_samples;
    if (!series || !out) return report_error(TVBX_E_INVALID_ARG, "NULL series or out");
    if (N < 1 || N > 752 || P < 1 || T < 2)
        return report_error(TVBX_E_INVALID_ARG, "need 1 <= n_regions <= 752, n_sets >= 1, n_samples >= 2");
    if (!(dt_ms > 0.0) || !std::isfinite(dt_ms)) return report_error(TVBX_E_INVALID_ARG, "dt_ms must be > 0");
    const int n = smooth_length(T);
    FftPlan plan;
    if (n < 2 || !make_plan(n, plan)) return report_error(TVBX_E_INVALID_ARG, "no transform length for %lld samples", (long long)T);
    // PSD band [1, 100] Hz: bins 1 <= i < n/2 with f_i = i / (n dt) in the band
    const double dt_s = dt_ms * 1e-3;
    int band_lo = -1, band_hi = -1;
    for (int i = 1; 2 * i < n; ++i) {
        const double f = (double)i / ((double)n * dt_s);
        if (f >= 1.0 && f <= 100.0) {
            if (band_lo < 0) band_lo = i;
            band_hi = i;
        }
    }
    const int band_n = band_lo < 0 ? 0 : band_hi - band_lo + 1;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // batch of sets: analytic signals and pair counts of B sets in at most ~2 GiB
    const int ns = (n + 3) / 4 * 4;
    const int64_t per_set = (int64_t)N * ns * 8 + (int64_t)N * N * 4;
    int64_t B = std::max<int64_t>(1, std::min<int64_t>(P, ((int64_t)1 << 31) / std::max<int64_t>(per_set, 1)));
    const size_t pli_row = sizeof(float) * 4 * (size_t)((N + 3) / 4 * 4);   // two buffers of two planes
    const int tt = pli_row * (PLI_TT_MAX + 4) <= 110 * 1024 ? PLI_TT_MAX : (pli_row * 36 <= 200 * 1024 ? 32 : PLI_TT_MIN);
    const size_t smem_pli = pli_row * (size_t)(tt + 4);
    if (smem_pli > 200 * 1024) return report_error(TVBX_E_INVALID_ARG, "too many regions for the PLI tile");
    auto pli_kernel = tt == PLI_TT_MAX ? an_pli_kernel<PLI_TT_MAX>
                                       : (tt == 32 ? an_pli_kernel<32> : an_pli_kernel<PLI_TT_MIN>);
    ACK(cudaFuncSetAttribute(pli_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_pli),
        "analysis shared memory");
    // time slices of about 640 samples, whole tiles
    const int slice = std::min((ns + PLI_TT_MAX - 1) / PLI_TT_MAX * PLI_TT_MAX, 10 * PLI_TT_MAX);
    const int slices = (ns + slice - 1) / slice;
    const std::vector<float2> htw = roots(n);
    AnScratch scr(s);
    float2* tw;
    float *z, *psd;
    int *ud, *cnt;
    // even lengths: complex transforms of half the length
    FftPlan plan_h = plan;
    const bool half = n % 2 == 0 && n >= 4 && make_plan(n / 2, plan_h);
    const FftPlan& used = half ? plan_h : plan;
    const std::vector<float2> htws = stage_twiddles(used, htw);
    const std::vector<int> hperm = digit_reversal(used);
    float2* tws;
    int* perm;
    ACK(scr.get(&tw, n), "analysis twiddles");
    ACK(scr.get(&tws, htws.size()), "analysis twiddles");
    ACK(scr.get(&perm, used.n), "analysis digit reversal");
    ACK(cudaMemcpyAsync(perm, hperm.data(), sizeof(int) * used.n, cudaMemcpyHostToDevice, s), "analysis digit reversal");
    ACK(cudaMemcpyAsync(tws, htws.data(), sizeof(float2) * htws.size(), cudaMemcpyHostToDevice, s), "analysis twiddles");
    ACK(scr.get(&z, (size_t)B * N * 2 * ns), "analysis signals");
    ACK(scr.get(&psd, (size_t)B * N * std::max(band_n, 1)), "analysis PSD");
    ACK(scr.get(&cnt, (size_t)B * N * N), "analysis PLI");
    ACK(scr.get(&ud, (size_t)B * N * 4), "analysis UP/DOWN");
    ACK(cudaMemcpyAsync(tw, htw.data(), sizeof(float2) * n, cudaMemcpyHostToDevice, s), "analysis twiddles");
    const size_t smem_series = sizeof(float2) * (size_t)(half ? n / 2 : n);
    auto series_kernel = half ? an_series_kernel<true> : an_series_kernel<false>;
    ACK(cudaFuncSetAttribute(series_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_series),
        "analysis shared memory");
    const size_t smem_fin = sizeof(float) * (size_t)std::max(band_n, 1);
    ACK(cudaFuncSetAttribute(an_finalize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_fin),
        "analysis shared memory");
    const float psd_scale = (float)(2.0 * dt_s / (double)n * 1e6);   // kHz^2 -> Hz^2, one-sided
    const double df = 1.0 / ((double)n * dt_s);
    // host input: batch b + 1 is copied on a second stream into one of two
    // staging buffers while batch b is analysed on s
    const bool host_in = is_host_pointer(series);
    HostPipe hp;
    hp.s = s;
    float* stage[2] = {nullptr, nullptr};
    if (host_in) {
        ACK(scr.get(&stage[0], (size_t)B * N * T), "analysis staging");
        ACK(scr.get(&stage[1], (size_t)B * N * T), "analysis staging");
        ACK(cudaStreamCreateWithFlags(&hp.cs, cudaStreamNonBlocking), "analysis copy stream");
        for (cudaEvent_t& e : hp.ev) ACK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "analysis events");
        ACK(cudaEventRecord(hp.ev[0], s), "analysis events");   // the staging buffers exist
        ACK(cudaStreamWaitEvent(hp.cs, hp.ev[0], 0), "analysis events");
    }
    int64_t batch = 0;
    for (int64_t p0 = 0; p0 < P; p0 += B, ++batch) {
        const int64_t nb = std::min<int64_t>(B, P - p0);
        const float* in = series;
        int64_t in_p0 = p0;
        const int slot = (int)(batch & 1);
        if (host_in) {
            if (batch >= 2) ACK(cudaStreamWaitEvent(hp.cs, hp.ev[3 + slot], 0), "analysis events");
            ACK(cudaMemcpyAsync(stage[slot], series + p0 * N * T, sizeof(float) * (size_t)(nb * N * T),
                                cudaMemcpyHostToDevice, hp.cs),
                "analysis series upload");
            ACK(cudaEventRecord(hp.ev[1 + slot], hp.cs), "analysis events");
            ACK(cudaStreamWaitEvent(s, hp.ev[1 + slot], 0), "analysis events");
            in = stage[slot];
            in_p0 = 0;
        }
        note_launch(3);
        series_kernel<<<(unsigned)(nb * N), AN_THREADS, smem_series, s>>>(in, N, T, plan, plan_h, tw, tws, perm,
                                                                        band_lo, band_n, psd_scale, in_p0, psd,
                                                                        ud, z, ns);
        ACK(cudaGetLastError(), "analysis series");
        if (host_in) ACK(cudaEventRecord(hp.ev[3 + slot], s), "analysis events");   // the slot was read
        ACK(cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)nb * N * N, s), "analysis PLI");
        pli_kernel<<<(unsigned)(nb * slices), PLI_THREADS, smem_pli, s>>>(z, N, ns, slice, slices, cnt);
        ACK(cudaGetLastError(), "analysis PLI");
        an_finalize_kernel<<<(unsigned)nb, AN_THREADS, smem_fin, s>>>(psd, ud, cnt, N, n, band_lo, band_n, df, dt_ms,
                                                                       p0, out);
        ACK(cudaGetLastError(), "analysis finalize");
    }
    if (n_used) *n_used = n;
    return TVBX_OK;
}

extern "C" tvbx_status tvbx_phfcd(const float* bold, int32_t n_regions, int64_t n_sets, int64_t n_tr, double tr_s,
                                  double f_lo_hz, double f_hi_hz, int32_t discard, float* out, int32_t* n_used,
                                  void* cuda_stream)
{
    const int N = n_regions;
    const int64_t P = n_sets;
    if (!bold || !out) return report_error(TVBX_E_INVALID_ARG, "NULL bold or out");
    if (N < 2 || N > 200 || P < 1 || n_tr < 2 || discard < 0)
        return report_error(TVBX_E_INVALID_ARG, "need 2 <= n_regions <= 200, n_sets >= 1, n_tr >= 2, discard >= 0");
    if (!(tr_s > 0.0) || !std::isfinite(tr_s) || !(f_lo_hz <= f_hi_hz))
        return report_error(TVBX_E_INVALID_ARG, "need tr_s > 0 and f_lo_hz <= f_hi_hz");
    const int n = smooth_length(n_tr);
    FftPlan plan;
    if (n < 2 || !make_plan(n, plan)) return report_error(TVBX_E_INVALID_ARG, "no transform length for %lld samples", (long long)n_tr);
    const int Tp = n - 2 * discard;
    if (Tp < 2) return report_error(TVBX_E_INVALID_ARG, "fewer than 2 samples left after discarding %d at each end", discard);
    int band_lo = n, band_hi = -1;   // empty unless a bin 0 < i < n/2 has its frequency in the band
    for (int i = 1; 2 * i < n; ++i) {
        const double f = (double)i / ((double)n * tr_s);
        if (f >= f_lo_hz && f <= f_hi_hz) {
            band_lo = std::min(band_lo, i);
            band_hi = std::max(band_hi, i);
        }
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int64_t per_set = (int64_t)Tp * N * 8;
    const int64_t B = std::max<int64_t>(1, std::min<int64_t>(P, ((int64_t)1 << 30) / std::max<int64_t>(per_set, 1)));
    const std::vector<float2> htw = stage_twiddles(plan, roots(n));
    AnScratch scr(s);
    float2 *tw, *U;
    ACK(scr.get(&tw, htw.size()), "phFCD twiddles");
    int* perm;
    ACK(scr.get(&perm, n), "phFCD digit reversal");
    const std::vector<int> hperm = digit_reversal(plan);
    ACK(cudaMemcpyAsync(perm, hperm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s), "phFCD digit reversal");
    ACK(scr.get(&U, (size_t)B * Tp * N), "phFCD phasors");
    ACK(cudaMemcpyAsync(tw, htw.data(), sizeof(float2) * htw.size(), cudaMemcpyHostToDevice, s), "phFCD twiddles");
    int S = 1;   // sets per CTA of the phase kernel
    while (S < 8 && 2 * S * n <= AN_MAX_T / 2) S *= 2;
    const size_t smem_phase = sizeof(float2) * (size_t)n * S;
    ACK(cudaFuncSetAttribute(an_phase_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_phase),
        "phFCD shared memory");
    const size_t smem_pf = sizeof(float2) * 2 * (size_t)N * PF_TILE;
    if (smem_pf > 200 * 1024) return report_error(TVBX_E_INVALID_ARG, "too many regions for the phFCD tiles");
    ACK(cudaFuncSetAttribute(an_phfcd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_pf),
        "phFCD shared memory");
    const int nt = (Tp + PF_TILE - 1) / PF_TILE;
    const int64_t M2 = (int64_t)Tp * (Tp - 1) / 2;
    for (int64_t p0 = 0; p0 < P; p0 += B) {
        const int64_t nb = std::min<int64_t>(B, P - p0);
        note_launch(2);
        an_phase_kernel<<<(unsigned)((nb + S - 1) / S * N), AN_THREADS, smem_phase, s>>>(
            bold, N, P, n_tr, plan, tw, perm, band_lo, band_hi, discard, p0, (int)nb, S, U);
        ACK(cudaGetLastError(), "phFCD phases");
        an_phfcd_kernel<<<dim3((unsigned)(nt * (nt + 1) / 2), (unsigned)nb), PF_THREADS, smem_pf, s>>>(U, N, Tp, p0,
                                                                                                       M2, out);
        ACK(cudaGetLastError(), "phFCD");
    }
    if (n_used) *n_used = Tp;
    return TVBX_OK;
}
