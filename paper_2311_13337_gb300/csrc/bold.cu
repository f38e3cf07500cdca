// Balloon-Windkessel BOLD signal of the simulated excitatory rates
// (arXiv 2311.13337, Sec. "Output": a Balloon-Windkessel kernel, Stephan et
// al. 2007, turns the simulated activity into BOLD series for comparison with
// fMRI).
//
// Model (Friston et al. 2000; Stephan et al. 2007), drive z = E rate in kHz,
// time in seconds:
//   ds/dt = z - kappa s - gamma (f - 1),  df/dt = s,
//   tau dv/dt = f - v^(1/alpha),
//   tau dq/dt = f E(f) / E0 - v^(1/alpha) q / v,  E(f) = 1 - (1 - E0)^(1/f),
//   y = V0 (k1 (1 - q) + k2 (1 - q/v) + k3 (1 - v)).
// One thread per (region, set) integrates forward Euler with the step of the
// rate samples. The state is kept as deviations from rest (f - 1, v - 1,
// q - 1) and the powers are written as functions of those deviations
// (series for small arguments, log1p / expm1 beyond), so FP32 resolves the
// small excursions a drive of a few Hz causes (about 1e-3 of the resting
// values) instead of rounding them against 1, and a zero drive keeps the
// resting state exactly.
//
// Layouts: series [T][N][P] (consecutive threads read consecutive sets), BOLD
// [T / decim][N][P], state [4][N][P] = s, f - 1, v - 1, q - 1.

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "internal.h"
#include "tvbx.h"

namespace tvbx {
namespace {

constexpr int BOLD_AHEAD = 8;     // samples fetched ahead
constexpr int BOLD_THREADS = 128;

struct BoldDev {
    float kappa, gamma, inv_tau, inv_alpha, r_E0, lnE, V0, k1, k2, k3, dt;   // r_E0 = (1 - E0) / E0
    float ca[8];   // binomial coefficients C(1/alpha, k), k = 1 .. 8
    float v_series;   // |v - 1| up to which the binomial series is used (0: never)
    float v_small, f_small;   // |v - 1| and |f - 1| up to which both series end at degree 4
};

// (1 + v)^a - 1 for |v| <= v_series: the binomial series sum_k C(a, k) v^k to
// degree 8 (Horner); v_series is chosen on the host so that the rest of the
// series stays below 1e-8 of the first term (exact for integer a <= 8).
// Beyond it, expm1(a log1p(v)).
static __device__ __forceinline__ float pow1p_m1(float v, const BoldDev& c)
{
    if (fabsf(v) <= c.v_series) {
        float h = c.ca[7];
#pragma unroll
        for (int k = 6; k >= 0; --k) h = fmaf(h, v, c.ca[k]);
        return h * v;
    }
    if (v != v) return v;
    return expm1f(log1pf(v) * c.inv_alpha);
}

// e^x - 1 for |x| <= 1/4 by its Taylor series to degree 8 (the rest is below
// 4.4e-11 of the first term: about x^8 / 9!), else expm1f
static __device__ __forceinline__ float expm1_small(float x)
{
    if (fabsf(x) <= 0.25f) {
        float h = 1.0f / 40320.0f;                 // 1/8!
        h = fmaf(h, x, 1.0f / 5040.0f);            // 1/7!
        h = fmaf(h, x, 1.0f / 720.0f);             // 1/6!
        h = fmaf(h, x, 1.0f / 120.0f);             // 1/5!
        h = fmaf(h, x, 1.0f / 24.0f);              // 1/4!
        h = fmaf(h, x, 1.0f / 6.0f);               // 1/3!
        h = fmaf(h, x, 0.5f);                      // 1/2!
        h = fmaf(h, x, 1.0f);
        return h * x;
    }
    if (x != x) return x;
    return expm1f(x);
}

// 1 / x by the SM's approximate reciprocal (about 1 ulp; x is the blood
// volume 1 + (v - 1), near 1, so no denormals arise)
static __device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The signal: 1 - q = -qt, 1 - q / v = (vt - qt) / (1 + vt), 1 - v = -vt.
static __device__ __forceinline__ float bold_of(const BoldDev& c, float vt, float qt)
{
    return c.V0 * fmaf(c.k3, -vt, fmaf(c.k1, -qt, c.k2 * (vt - qt) / (1.0f + vt)));
}

// One element per thread, for counts and addresses that bold_kernel2 does not
// take: the same operations, so the same numbers.
__global__ void bold_kernel(const float* __restrict__ series, int64_t NP, int64_t T, int decim, BoldDev c,
                            float* __restrict__ state, int reset, float* __restrict__ out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= NP) return;
    float s = 0.0f, ft = 0.0f, vt = 0.0f, qt = 0.0f;
    if (state && !reset) {
        s = state[i];
        ft = state[NP + i];
        vt = state[2 * NP + i];
        qt = state[3 * NP + i];
    }
    int phase = 0;
    int64_t o = 0;
    auto step = [&](float z) {
        const float f = 1.0f + ft;
        const float x = -c.lnE * ft * rcp_approx(f);
        float vpa_m1, em1;   // v^(1/alpha) - 1, e^x - 1
        if (fabsf(vt) <= c.v_small && fabsf(ft) <= c.f_small) {
            vpa_m1 = fmaf(fmaf(fmaf(c.ca[3], vt, c.ca[2]), vt, c.ca[1]), vt, c.ca[0]) * vt;
            em1 = fmaf(fmaf(fmaf(1.0f / 24.0f, x, 1.0f / 6.0f), x, 0.5f), x, 1.0f) * x;
        } else {
            vpa_m1 = pow1p_m1(vt, c);
            em1 = expm1_small(x);
        }
        // f E(f) / E0 - 1 = ft - (1 + ft) r_E0 expm1(-ln(1 - E0) ft / f), since
        // (1 - E0)^(1/f) = (1 - E0) exp(-ln(1 - E0) ft / f): exactly 0 at rest
        const float fE_m1 = fmaf(f * -c.r_E0, em1, ft);
        // v^(1/alpha - 1) q - 1, with v^(1/alpha - 1) - 1 = (v^(1/alpha) - v) / v
        // = (vpa_m1 - vt) / (1 + vt) (no cancellation: vpa_m1 is about vt / alpha)
        const float vq_m1 = fmaf((vpa_m1 - vt) * rcp_approx(1.0f + vt), 1.0f + qt, qt);
        const float ds = fmaf(-c.gamma, ft, fmaf(-c.kappa, s, z));
        const float nft = fmaf(c.dt, s, ft);
        const float nvt = fmaf(c.dt * c.inv_tau, ft - vpa_m1, vt);
        const float nqt = fmaf(c.dt * c.inv_tau, fE_m1 - vq_m1, qt);
        s = fmaf(c.dt, ds, s);
        ft = nft;
        vt = nvt;
        qt = nqt;
        if (++phase == decim) {
            phase = 0;
            out[o * NP + i] = bold_of(c, vt, qt);
            ++o;
        }
    };
    const float* at = series + i;
    auto fetch = [&](float (&z)[BOLD_AHEAD]) {
#pragma unroll
        for (int u = 0; u < BOLD_AHEAD; ++u, at += NP) z[u] = __ldg(at);
    };
    float za[BOLD_AHEAD], zb[BOLD_AHEAD];
    int64_t t = 0;
    if (T >= BOLD_AHEAD) fetch(za);
    for (; t + BOLD_AHEAD <= T; t += BOLD_AHEAD) {
        const bool more = t + 2 * BOLD_AHEAD <= T;
        if (more) fetch(zb);
#pragma unroll 1
        for (int u = 0; u < BOLD_AHEAD; ++u) {
            step(za[0]);
#pragma unroll
            for (int k = 0; k + 1 < BOLD_AHEAD; ++k) za[k] = za[k + 1];
        }
        if (more) {
#pragma unroll
            for (int u = 0; u < BOLD_AHEAD; ++u) za[u] = zb[u];
        }
    }
    for (; t < T; ++t, at += NP) step(__ldg(at));
    if (state) {
        state[i] = s;
        state[NP + i] = ft;
        state[2 * NP + i] = vt;
        state[3 * NP + i] = qt;
    }
}

// Two FP32 values in a 64-bit register pair and the packed f32x2 operations
// of sm_100-class SMs (each lane rounds like the scalar instruction).
static __device__ __forceinline__ uint64_t p2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
static __device__ __forceinline__ float2 u2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
static __device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
static __device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
static __device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
static __device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// v^(1/alpha) - 1 and e^x - 1 of two elements beyond the range of the short
// series: packed to degree 8 where both lanes are in range, else lane by lane.
// A lane that is NaN takes the other's way and stays NaN. Inlined: as a call it
// cost 16% of the whole (2,048 x 68 x 10,000 1.82 ms, now 1.54) for what it kept
// on the stack, and rates that are not finite were slower than without it.
static __device__ __forceinline__ void powers(const BoldDev& c, uint64_t vt, uint64_t x, uint64_t& vpa_m1, uint64_t& em1)
{
    const float2 v0 = u2(vt), x0 = u2(x);
    const float2 v = make_float2(v0.x == v0.x ? v0.x : 0.0f, v0.y == v0.y ? v0.y : 0.0f);
    const float2 xf = make_float2(x0.x == x0.x ? x0.x : 0.0f, x0.y == x0.y ? x0.y : 0.0f);
    float2 r, e;
    if (fabsf(v.x) <= c.v_series && fabsf(v.y) <= c.v_series) {
        const uint64_t vp = p2(v.x, v.y);
        uint64_t h = p2(c.ca[7], c.ca[7]);
#pragma unroll
        for (int k = 6; k >= 0; --k) h = fma2(h, vp, p2(c.ca[k], c.ca[k]));
        r = u2(mul2(h, vp));
    } else {
        r = make_float2(pow1p_m1(v.x, c), pow1p_m1(v.y, c));
    }
    if (fabsf(xf.x) <= 0.25f && fabsf(xf.y) <= 0.25f) {
        const uint64_t xp = p2(xf.x, xf.y);
        uint64_t h = p2(1.0f / 40320.0f, 1.0f / 40320.0f);
        h = fma2(h, xp, p2(1.0f / 5040.0f, 1.0f / 5040.0f));
        h = fma2(h, xp, p2(1.0f / 720.0f, 1.0f / 720.0f));
        h = fma2(h, xp, p2(1.0f / 120.0f, 1.0f / 120.0f));
        h = fma2(h, xp, p2(1.0f / 24.0f, 1.0f / 24.0f));
        h = fma2(h, xp, p2(1.0f / 6.0f, 1.0f / 6.0f));
        h = fma2(h, xp, p2(0.5f, 0.5f));
        h = fma2(h, xp, p2(1.0f, 1.0f));
        e = u2(mul2(h, xp));
    } else {
        e = make_float2(expm1_small(xf.x), expm1_small(xf.y));
    }
    vpa_m1 = p2(v0.x == v0.x ? r.x : v0.x, v0.y == v0.y ? r.y : v0.y);
    em1 = p2(x0.x == x0.x ? e.x : x0.x, x0.y == x0.y ? e.y : x0.y);
}

// The same integration for two neighbouring (region, set) elements per
// thread, i and i + 1 (i even; NP even, so every sample row starts 8-byte
// aligned), in packed f32x2 arithmetic; reciprocals, the general forms of the
// powers and the output are lane by lane. While v - 1 and f - 1 of a lane
// are within v_small and f_small (rates up to about 25 Hz), both series end at
// degree 4, which leaves the same 1e-8 of their first term as the longer ones
// do at their bounds; each lane by its own values, so that an element does not
// depend on its neighbour. The rates come BOLD_AHEAD samples ahead: one load per
// step, waited for, bound the kernel by memory latency below a full chip
// (2,048 x 68 x 10,000: 4.58 ms; now 1.54).
__global__ void __launch_bounds__(BOLD_THREADS)
bold_kernel2(const float* __restrict__ series, int64_t NP, int64_t T, int decim, BoldDev c,
                             float* __restrict__ state, int reset, float* __restrict__ out)
{
    const int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
    if (i >= NP) return;
    float2 s0 = make_float2(0.0f, 0.0f), f0 = s0, v0 = s0, q0 = s0;
    if (state && !reset) {
        s0 = *reinterpret_cast<const float2*>(state + i);
        f0 = *reinterpret_cast<const float2*>(state + NP + i);
        v0 = *reinterpret_cast<const float2*>(state + 2 * NP + i);
        q0 = *reinterpret_cast<const float2*>(state + 3 * NP + i);
    }
    uint64_t s = p2(s0.x, s0.y), ft = p2(f0.x, f0.y), vt = p2(v0.x, v0.y), qt = p2(q0.x, q0.y);
    const uint64_t one = p2(1.0f, 1.0f), m_kappa = p2(-c.kappa, -c.kappa), m_gamma = p2(-c.gamma, -c.gamma);
    const uint64_t dt = p2(c.dt, c.dt), dtt = p2(c.dt * c.inv_tau, c.dt * c.inv_tau);
    const uint64_t m_rE0 = p2(-c.r_E0, -c.r_E0);
    uint64_t ca[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) ca[k] = p2(c.ca[k], c.ca[k]);
    const uint64_t m_lnE = p2(-c.lnE, -c.lnE);
    const uint64_t e2 = p2(0.5f, 0.5f), e3 = p2(1.0f / 6.0f, 1.0f / 6.0f), e4 = p2(1.0f / 24.0f, 1.0f / 24.0f);
    int phase = 0;
    int64_t o = 0;
    auto step = [&](float2 zf) {
        const uint64_t z = p2(zf.x, zf.y);
        const uint64_t f = add2(one, ft), w = add2(one, vt);
        const float2 vtf = u2(vt), ftf = u2(ft), ff = u2(f), wf = u2(w);
        uint64_t vpa_m1;   // v^(1/alpha) - 1
        uint64_t em1;      // e^x - 1 of the oxygen extraction, x = -ln(1 - E0) ft / f
        const uint64_t rv = p2(rcp_approx(wf.x), rcp_approx(wf.y));
        const uint64_t x = mul2(mul2(m_lnE, ft), p2(rcp_approx(ff.x), rcp_approx(ff.y)));
        if (fabsf(vtf.x) <= c.v_small && fabsf(vtf.y) <= c.v_small && fabsf(ftf.x) <= c.f_small &&
            fabsf(ftf.y) <= c.f_small) {
            vpa_m1 = mul2(fma2(fma2(fma2(ca[3], vt, ca[2]), vt, ca[1]), vt, ca[0]), vt);
            em1 = mul2(fma2(fma2(fma2(e4, x, e3), x, e2), x, one), x);
        } else {
            powers(c, vt, x, vpa_m1, em1);
            // an element's series do not depend on its neighbour
            const bool near0 = fabsf(vtf.x) <= c.v_small && fabsf(ftf.x) <= c.f_small;
            const bool near1 = fabsf(vtf.y) <= c.v_small && fabsf(ftf.y) <= c.f_small;
            if (near0 || near1) {
                const float2 vf = u2(vpa_m1), ef = u2(em1);
                const float2 vn = u2(mul2(fma2(fma2(fma2(ca[3], vt, ca[2]), vt, ca[1]), vt, ca[0]), vt));
                const float2 en = u2(mul2(fma2(fma2(fma2(e4, x, e3), x, e2), x, one), x));
                vpa_m1 = p2(near0 ? vn.x : vf.x, near1 ? vn.y : vf.y);
                em1 = p2(near0 ? en.x : ef.x, near1 ? en.y : ef.y);
            }
        }
        const uint64_t fE_m1 = fma2(mul2(f, m_rE0), em1, ft);
        const uint64_t vq_m1 = fma2(mul2(sub2(vpa_m1, vt), rv), add2(one, qt), qt);
        const uint64_t ds = fma2(m_gamma, ft, fma2(m_kappa, s, z));
        const uint64_t nft = fma2(dt, s, ft);
        const uint64_t nvt = fma2(dtt, sub2(ft, vpa_m1), vt);
        const uint64_t nqt = fma2(dtt, sub2(fE_m1, vq_m1), qt);
        s = fma2(dt, ds, s);
        ft = nft;
        vt = nvt;
        qt = nqt;
        if (++phase == decim) {
            phase = 0;
            const float2 a = u2(vt), b = u2(qt);
            *reinterpret_cast<float2*>(out + o * NP + i) = make_float2(bold_of(c, a.x, b.x), bold_of(c, a.y, b.y));
            ++o;
        }
    };
    // rates of BOLD_AHEAD samples at a time, the next ones on the way
    const float* at = series + i;
    auto fetch = [&](float2 (&z)[BOLD_AHEAD]) {
#pragma unroll
        for (int u = 0; u < BOLD_AHEAD; ++u, at += NP) z[u] = __ldg(reinterpret_cast<const float2*>(at));
    };
    float2 za[BOLD_AHEAD], zb[BOLD_AHEAD];
    int64_t t = 0;
    if (T >= BOLD_AHEAD) fetch(za);
    for (; t + BOLD_AHEAD <= T; t += BOLD_AHEAD) {
        const bool more = t + 2 * BOLD_AHEAD <= T;
        if (more) fetch(zb);
#pragma unroll
        for (int u = 0; u < BOLD_AHEAD; ++u) step(za[u]);
        if (more) {
#pragma unroll
            for (int u = 0; u < BOLD_AHEAD; ++u) za[u] = zb[u];
        }
    }
    for (; t < T; ++t, at += NP) step(__ldg(reinterpret_cast<const float2*>(at)));
    if (state) {
        *reinterpret_cast<float2*>(state + i) = u2(s);
        *reinterpret_cast<float2*>(state + NP + i) = u2(ft);
        *reinterpret_cast<float2*>(state + 2 * NP + i) = u2(vt);
        *reinterpret_cast<float2*>(state + 3 * NP + i) = u2(qt);
    }
}

}  // namespace
}  // namespace tvbx

using namespace tvbx;

extern "C" tvbx_status tvbx_bold_defaults(tvbx_bold_params* out)
{
    if (!out) return report_error(TVBX_E_INVALID_ARG, "NULL out");
    out->kappa = 0.65;
    out->gamma = 0.41;
    out->tau = 0.98;
    out->alpha = 0.32;
    out->E0 = 0.34;
    out->V0 = 0.02;
    out->theta0 = 40.3;
    out->r0 = 25.0;
    out->TE = 0.04;
    out->eps = 1.0;
    return TVBX_OK;
}

extern "C" tvbx_status tvbx_bold(const float* series, int32_t n_regions, int64_t n_sets, int64_t n_samples,
                                 double dt_ms, int32_t decim, const tvbx_bold_params* params, float* state,
                                 int32_t reset_state, float* bold_out, void* cuda_stream)
{
    if (!series || !bold_out) return report_error(TVBX_E_INVALID_ARG, "NULL series or bold_out");
    if (n_regions < 1 || n_sets < 1 || n_samples < 0 || decim < 1)
        return report_error(TVBX_E_INVALID_ARG, "need n_regions >= 1, n_sets >= 1, n_samples >= 0, decim >= 1");
    if (!(dt_ms > 0.0) || !std::isfinite(dt_ms)) return report_error(TVBX_E_INVALID_ARG, "dt_ms must be > 0");
    tvbx_bold_params p;
    if (params) p = *params;
    else tvbx_bold_defaults(&p);
    if (!(p.tau > 0.0) || !(p.alpha > 0.0) || !(p.E0 > 0.0 && p.E0 < 1.0))
        return report_error(TVBX_E_INVALID_ARG, "need tau > 0, alpha > 0, 0 < E0 < 1");
    BoldDev c;
    c.kappa = (float)p.kappa;
    c.gamma = (float)p.gamma;
    c.inv_tau = (float)(1.0 / p.tau);
    c.inv_alpha = (float)(1.0 / p.alpha);
    c.r_E0 = (float)((1.0 - p.E0) / p.E0);
    c.lnE = (float)std::log1p(-p.E0);
    c.V0 = (float)p.V0;
    c.k1 = (float)(4.3 * p.theta0 * p.E0 * p.TE);
    c.k2 = (float)(p.eps * p.r0 * p.E0 * p.TE);
    c.k3 = (float)(1.0 - p.eps);
    c.dt = (float)(dt_ms * 1e-3);
    // binomial coefficients of (1 + v)^a, a = 1 / alpha, and the largest
    // |v| (a power of 2 from 1/4 down) at which the series beyond degree 8
    // stays below 1e-8 of its first term a |v|
    {
        const double a = 1.0 / p.alpha;
        double C[41];
        C[0] = 1.0;
        for (int k = 1; k <= 40; ++k) C[k] = C[k - 1] * (a - (k - 1)) / k;
        for (int k = 0; k < 8; ++k) c.ca[k] = (float)C[k + 1];
        c.v_series = 0.0f;
        for (double vm = 0.25; vm >= 1.0 / 1024.0; vm *= 0.5) {
            double tail = 0.0, pw = std::pow(vm, 9);
            for (int k = 9; k <= 40; ++k, pw *= vm) tail += std::fabs(C[k]) * pw;
            if (tail <= 1e-8 * std::fabs(a) * vm) {
                c.v_series = (float)vm;
                break;
            }
        }
        // the same below degree 5, and for e^x - 1 (|x| <= 1/32, where x^4 / 120 < 1e-8),
        // x = -ln(1 - E0) (f - 1) / f
        c.v_small = 0.0f;
        for (double vm = std::min(0.0625, (double)c.v_series); vm >= 1.0 / 4096.0; vm *= 0.5) {
            double tail = 0.0, pw = std::pow(vm, 5);
            for (int k = 5; k <= 40; ++k, pw *= vm) tail += std::fabs(C[k]) * pw;
            if (tail <= 1e-8 * std::fabs(a) * vm) {
                c.v_small = (float)vm;
                break;
            }
        }
        c.f_small = (float)((1.0 / 32.0) / (1.0 / 32.0 - std::log1p(-p.E0)));
    }
    const int64_t NP = (int64_t)n_regions * n_sets;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    note_launch();
    // two elements per thread when every row of series, BOLD and state starts
    // 8-byte aligned (NP even, 8-byte aligned buffers), else one
    const bool pair = NP % 2 == 0 && (uintptr_t)series % 8 == 0 && (uintptr_t)bold_out % 8 == 0 &&
                      (!state || (uintptr_t)state % 8 == 0);
    if (pair)
        bold_kernel2<<<(unsigned)((NP / 2 + BOLD_THREADS - 1) / BOLD_THREADS), BOLD_THREADS, 0, s>>>(series, NP, n_samples, decim, c, state,
                                                                      reset_state, bold_out);
    else
        bold_kernel<<<(unsigned)((NP + BOLD_THREADS - 1) / BOLD_THREADS), BOLD_THREADS, 0, s>>>(series, NP, n_samples, decim, c, state, reset_state,
                                                                bold_out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return report_error(TVBX_E_CUDA, "BOLD: %s", cudaGetErrorString(e));
    return TVBX_OK;
}
