// Windowed simulation kernels of the tvbx engine (arXiv 2311.13337, the
// lock-step integration of Eq. 1-5 with forward Euler).
//
// Step n + b reads values of steps up to n + b - d_min, d_min the connectome's
// shortest delay, and step n's are known: over a window of B <= d_min + 1 steps
// every (set, region) pair is independent of the others, and the coupling sums
// of all B steps can be formed from the ring before the first of them is taken. One launch advances every
// pair by one window; launch order is the only synchronisation, so nothing
// waits at a barrier, any number of regions or sets fills the chip evenly, and
// each row entry is read once per window instead of once per step.
//
// A thread owns one region of one set (float) or of two adjacent sets (float2,
// packed FP32x2); in sweeps too small to fill the chip two threads share one.
// It
//  1. forms the coupling sums of the window, up to 8 steps at a time, in CSR
//     order (the sums of the other kernels, bit for bit): independent loads
//     that do not wait for the sums;
//  2. loads its state, takes the B steps in registers, and writes E of each
//     step to the ring; then stores the state.
//
// Ring layout: [tile][N][H + WIN_FAR][pb], a tile of pb sets holding the H last
// steps of a region contiguously, with the first WIN_FAR slots repeated after
// slot H - 1: the rows an entry reads are one run that never wraps.
// H = d_max + 1 + B, so that the window's own writes never meet a row that
// another thread of the same launch may still read.
//
// Short delays (B < 8, large connectomes at high speeds): a window alone would
// read each row entry for a few steps only. sim_far_kernel then sums the entries
// with d >= WIN_FAR, which come first in each CSR row, for WIN_FAR steps at once
// into a buffer [tile][WIN_FAR][N][pb]; the windows start from those sums and add
// the few nearer entries. Zero delays read the step before the window's only one.

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "internal.h"
#include "launch_next.cuh"
#include "model_device.cuh"

namespace tvbx {

namespace {

// 128 threads and 128 registers: four CTAs per SM. Five or six (102, 85
// registers, more spills) and three measured slower (32,768 x 68 sweep, 500
// steps: 23.5 ms against 27.3, 31.5 and 25.4).
constexpr int WIN_THREADS = 128;

template <class V> struct VSets;
template <> struct VSets<float> { static constexpr int n = 1; };
template <> struct VSets<float2> { static constexpr int n = 2; };

__device__ __forceinline__ void load_v(float& x, const float* p, bool, bool) { x = *p; }
__device__ __forceinline__ void load_v(float2& x, const float* p, bool, bool act1)
{
    x.x = p[0];
    x.y = act1 ? p[1] : 0.0f;
}
__device__ __forceinline__ void store_v(float* p, float x, bool) { *p = x; }
__device__ __forceinline__ void store_v(float* p, float2 x, bool act1)
{
    p[0] = x.x;
    if (act1) p[1] = x.y;
}

__device__ __noinline__ float next_ou(const DevModel& m, uint64_t seed, uint32_t n, uint32_t k, uint32_t p, float OU)
{
    const float xi = std_normal(seed, n, k, p);
    return fmaf(m.ou_a, m.ou_mu - OU, fmaf(m.ou_b, xi, OU));
}

// Coupling sums of G steps from row `at` on: row entries [e0, e1) added to acc.
// ring: row (j, slot) at (j HR + slot) pb. Four entries' loads are in flight
// together (one: 27.1 ms, two: 23.5 ms, four: 21.9 ms on the sweep above).
template <int G, class V>
__device__ __forceinline__ void gather(V (&acc)[G], const GroupDev& grp, const float* ring, int e0, int e1, int at,
                                       int H, int HR, int pb)
{
    const uint32_t* __restrict__ cd_p = grp.col_dly;
    const float* __restrict__ w_p = grp.w;
#pragma unroll 4
    for (int e = e0; e < e1; ++e) {
        const uint32_t cd = __ldg(cd_p + e);
        const V w = vbc<V>(__ldg(w_p + e));
        int sl = at - (int)(cd >> 16);
        sl += sl < 0 ? H : 0;
        const float* row = ring + (uint32_t)(((cd & 0xffffu) * (uint32_t)HR + (uint32_t)sl) * (uint32_t)pb);
#pragma unroll
        for (int b = 0; b < G; ++b) acc[b] = vfma(w, *reinterpret_cast<const V*>(row + b * pb), acc[b]);
    }
}

// The pair of the calling thread: region k of sets tile.q0 + q (and + 1).
struct WinSlot {
    int k, q;
    bool act1;
};
template <int S>
__device__ __forceinline__ WinSlot win_slot(const TileDev& tile, int i)   // i: the pair within the tile
{
    const int width = (tile.nq + S - 1) / S;   // pairs per region
    WinSlot w;
    w.k = i / width;
    w.q = (i - w.k * width) * S;
    w.act1 = w.q + 1 < tile.nq;
    return w;
}

// Sums of a pair's entries with d >= WIN_FAR over the WIN_FAR steps from n0 on,
// to the tile's far buffer.
template <class V, int PB>
__device__ __forceinline__ void far_pair(const SimArgs& a, const TileDev& tile, const GroupDev& grp, const WinSlot ws,
                                         int pb, uint32_t n0, float* far)
{
    const int N = a.N, H = grp.H, HR = H + WIN_FAR;
    V acc[WIN_FAR];
#pragma unroll
    for (int b = 0; b < WIN_FAR; ++b) acc[b] = vbc<V>(0.0f);
    gather<WIN_FAR>(acc, grp, grp.ring + (int64_t)tile.q0 * N * HR + ws.q, grp.row_ptr[ws.k], grp.row_near[ws.k],
                    (int)(n0 % (uint32_t)H), H, HR, pb);
    float* out = far + (int64_t)ws.k * pb + ws.q;
#pragma unroll
    for (int b = 0; b < WIN_FAR; ++b) *reinterpret_cast<V*>(out + (int64_t)b * N * pb) = acc[b];
}

// The far sums of every pair from step a.n0 on. Bound by the L2 reads of the
// rows (4 B per weight and step; 72% of the L2 rate on 1,024 x 360); a launch
// covers WIN_FAR steps so that the rows that different regions read are mostly
// the same ones (85% L2 hits).
template <class V, int PB>
__global__ void __launch_bounds__(WIN_THREADS, 4)
sim_far_kernel(const __grid_constant__ SimArgs a, int32_t pb_rt, int32_t blocks_per_tile, float* __restrict__ far)
{
    const int pb = PB > 0 ? PB : pb_rt;
    const int32_t ti = blockIdx.x / blocks_per_tile;
    const TileDev tile = a.tiles[ti];
    const WinSlot ws = win_slot<VSets<V>::n>(tile, (blockIdx.x % blocks_per_tile) * blockDim.x + threadIdx.x);
    after_last_launch();
    if (ws.k >= a.N) return;
    far_pair<V, PB>(a, tile, a.groups[tile.group], ws, pb, (uint32_t)a.n0, far + (int64_t)ti * WIN_FAR * a.N * pb);
}

// One window of `steps` steps of one thread's pair (region ws.k of sets
// tile.q0 + ws.q, + 1) from step n0. NEAR: the sums start from far (the
// tile's row of the window's first step) and add the nearer entries. m: the
// model, in constant memory. stash: this thread's coupling sums, a step every
// WIN_THREADS.
template <class V, int PB, bool NEAR>
__device__ __forceinline__ void window_pair(const SimArgs& a, const DevModel& m, const TileDev& tile,
                                            const GroupDev& grp, const WinSlot ws, int pb, uint32_t n0, int steps,
                                            int64_t table_step, const float* far, V* stash)
{
    constexpr int S = VSets<V>::n;
    const int N = a.N, k = ws.k, q = ws.q;
    const bool act1 = ws.act1;
    const int H = grp.H, HR = H + WIN_FAR;
    const int slot0 = (int)(n0 % (uint32_t)H);
    float* ring = grp.ring + (int64_t)tile.q0 * N * HR + q;
    const int ts = a.ts;
    const bool own_noise = a.noise_per_set != 0;

    // 1. coupling sums of the window
    {
        const int e0 = NEAR ? grp.row_near[k] : grp.row_ptr[k], e1 = grp.row_end[k];
        const float* far_k = NEAR ? far + (int64_t)k * pb + q : nullptr;
        int b0 = 0;
        auto pass = [&](auto g_c) {
            constexpr int G = decltype(g_c)::value;
            for (; b0 + G <= steps; b0 += G) {
                V acc[G];
#pragma unroll
                for (int b = 0; b < G; ++b)
                    acc[b] = NEAR ? *reinterpret_cast<const V*>(far_k + (int64_t)(b0 + b) * N * pb) : vbc<V>(0.0f);
                int at = slot0 + b0;
                at -= at >= H ? H : 0;
                gather<G>(acc, grp, ring, e0, e1, at, H, HR, pb);
#pragma unroll
                for (int b = 0; b < G; ++b) stash[(b0 + b) * WIN_THREADS] = acc[b];
            }
        };
        pass(std::integral_constant<int, 8>{});
        pass(std::integral_constant<int, 4>{});
        pass(std::integral_constant<int, 2>{});
        pass(std::integral_constant<int, 1>{});
    }

    // 2. the window's steps
    const int64_t NP = (int64_t)N * a.P;
    const int64_t p = grp.p_base + tile.q0 + q;
    float* st = a.state + (int64_t)k * a.P + p;
    ParamsV<V> sp;
    {
        const float* prm = a.prm + p;
        load_v(sp.g, prm + (int64_t)TVBX_AXIS_G * a.P, true, act1);
        load_v(sp.b_e, prm + (int64_t)TVBX_AXIS_B_E * a.P, true, act1);
        load_v(sp.inv_tw, prm + (int64_t)TVBX_AXIS_TAU_W_E * a.P, true, act1);
        sp.inv_tw = vmap(sp.inv_tw, [](float u) { return 1.0f / u; });
        load_v(sp.ELe, prm + (int64_t)TVBX_AXIS_E_L_E * a.P, true, act1);
        load_v(sp.ELi, prm + (int64_t)TVBX_AXIS_E_L_I * a.P, true, act1);
        load_v(sp.a_e, prm + (int64_t)TVBX_AXIS_A_E * a.P, true, act1);
        load_v(sp.wn, prm + (int64_t)TVBX_AXIS_W_NOISE * a.P, true, act1);
        load_v(sp.cFee, prm + (int64_t)TVBX_AXIS_CF_EE * a.P, true, act1);
        load_v(sp.cFei, prm + (int64_t)TVBX_AXIS_CF_EI * a.P, true, act1);
        load_v(sp.cFie, prm + (int64_t)TVBX_AXIS_CF_IE * a.P, true, act1);
        load_v(sp.cFii, prm + (int64_t)TVBX_AXIS_CF_II * a.P, true, act1);
    }
    PairV<V> x;
    V accE, accI, ou;
    load_v(x.E, st + SV_E * NP, true, act1);
    load_v(x.I, st + SV_I * NP, true, act1);
    load_v(x.Cee, st + SV_CEE * NP, true, act1);
    load_v(x.Cei, st + SV_CEI * NP, true, act1);
    load_v(x.Cii, st + SV_CII * NP, true, act1);
    load_v(x.We, st + SV_WE * NP, true, act1);
    load_v(x.Wi, st + SV_WI * NP, true, act1);
    load_v(x.cWe, st + SV_CWE * NP, true, act1);
    load_v(x.cWi, st + SV_CWI * NP, true, act1);
    load_v(accE, st + SV_ACC_E * NP, true, act1);
    load_v(accI, st + SV_ACC_I * NP, true, act1);
    uint32_t pn[2] = {0u, 0u};
    if (own_noise) {
        load_v(ou, st + SV_OU * NP, true, act1);
        pn[0] = (uint32_t)(a.p_offset + a.ext_index[p]);
        if (S > 1 && act1) pn[1] = (uint32_t)(a.p_offset + a.ext_index[p + 1]);
    } else {
        ou = vbc<V>(0.0f);
    }
    Track<V> trk = track_init<V>();
    const float inv_ts = 1.0f / (float)ts;
    // samples are the means of ts post-step states: steps left to the next one, and its index
    int left = ts - (int)(n0 % (uint32_t)ts);
    int64_t t = n0 / (uint32_t)ts;
    int slot_w = slot0;
    float* const ring_k = ring + (uint32_t)(k * HR) * (uint32_t)pb;
    const float* ou_p = a.ou_table + (own_noise ? 0 : table_step * N + k);
    for (int b = 0; b < steps; ++b) {
        const V OU = own_noise ? ou : vbc<V>(__ldg(ou_p));
        ou_p += own_noise ? 0 : N;
        pair_step(m, sp, x, stash[b * WIN_THREADS], OU, trk);
        if (own_noise) {
#pragma unroll
            for (int l = 0; l < S; ++l)
                set_lane(ou, l, next_ou(m, a.seed, n0 + (uint32_t)b, (uint32_t)k, pn[l], lane(OU, l)));
        }
        ++slot_w;
        slot_w -= slot_w == H ? H : 0;
        float* dst = ring_k + slot_w * pb;
        store_v(dst, x.E, act1);
        if (slot_w < WIN_FAR) store_v(dst + H * pb, x.E, act1);
        accE = vadd(accE, x.E);
        accI = vadd(accI, x.I);
        if (--left == 0) {
            if (t < a.T) {
                const V xE = vmul(accE, vbc<V>(inv_ts)), xI = vmul(accI, vbc<V>(inv_ts));
#pragma unroll
                for (int l = 0; l < S; ++l) {
                    if (l && !act1) continue;
                    const int64_t so = series_index(a.sl, t, k, p + l);
                    a.series[so] = lane(xE, l);
                    if (a.series_i) a.series_i[so] = lane(xI, l);
                    if (t >= a.transient) {
                        float sE = st[SV_SUM_E * NP + l], cE = st[SV_CMP_E * NP + l];
                        float sI = st[SV_SUM_I * NP + l], cI = st[SV_CMP_I * NP + l];
                        kahan_add(sE, cE, lane(xE, l));
                        kahan_add(sI, cI, lane(xI, l));
                        st[SV_SUM_E * NP + l] = sE;
                        st[SV_CMP_E * NP + l] = cE;
                        st[SV_SUM_I * NP + l] = sI;
                        st[SV_CMP_I * NP + l] = cI;
                    }
                }
            }
            left = ts;
            ++t;
            accE = vbc<V>(0.0f);
            accI = vbc<V>(0.0f);
        }
    }
    store_v(st + SV_E * NP, x.E, act1);
    store_v(st + SV_I * NP, x.I, act1);
    store_v(st + SV_CEE * NP, x.Cee, act1);
    store_v(st + SV_CEI * NP, x.Cei, act1);
    store_v(st + SV_CII * NP, x.Cii, act1);
    store_v(st + SV_WE * NP, x.We, act1);
    store_v(st + SV_WI * NP, x.Wi, act1);
    store_v(st + SV_CWE * NP, x.cWe, act1);
    store_v(st + SV_CWI * NP, x.cWi, act1);
    store_v(st + SV_ACC_E * NP, accE, act1);
    store_v(st + SV_ACC_I * NP, accI, act1);
    if (own_noise) store_v(st + SV_OU * NP, ou, act1);
#pragma unroll
    for (int l = 0; l < S; ++l) {
        const uint32_t f = track_flags(m, trk, l);
        if (f && (l == 0 || act1)) atomicOr(a.status + p + l, f);
    }
}

// One window of a.n_chunk steps from step a.n0. PB: sets per tile (0: the
// runtime width pb_rt).
template <class V, int PB, bool NEAR>
__global__ void __launch_bounds__(WIN_THREADS, 4)
sim_window_kernel(const __grid_constant__ SimArgs a, int32_t pb_rt, int32_t blocks_per_tile, int64_t table_step,
                  const float* __restrict__ far)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    const int pb = PB > 0 ? PB : pb_rt;
    const int32_t ti = blockIdx.x / blocks_per_tile;
    const TileDev tile = a.tiles[ti];
    const WinSlot ws = win_slot<VSets<V>::n>(tile, (blockIdx.x % blocks_per_tile) * blockDim.x + threadIdx.x);
    after_last_launch();
    if (ws.k >= a.N) return;
    window_pair<V, PB, NEAR>(a, a.m, tile, a.groups[tile.group], ws, pb, (uint32_t)a.n0, a.n_chunk, table_step,
                             NEAR ? far + (int64_t)ti * WIN_FAR * a.N * pb : nullptr,
                             reinterpret_cast<V*>(win_smem) + threadIdx.x);
}

// The window of a sweep too small to fill the chip, where the chain of one step
// bounds it: two lanes per pair, one per population (pair_step_split), each
// forming the coupling sums of half the steps. The next step's noise and
// coupling are read during a step: 16 x 68 took 0.85 ms per 1,000 steps with
// that and 0.99 without. (In sim_window_kernel, whose warps hide those reads
// from one another, the extra registers cost more: 32,768 x 68 went from 21.8
// to 22.4 ms.) Needs the reduced transfer function (tau_e == tau_i).
template <bool NEAR>
__global__ void __launch_bounds__(WIN_THREADS, 2)
sim_window_split_kernel(const __grid_constant__ SimArgs a, int32_t pb, int32_t blocks_per_tile, int64_t table_step,
                        const float* __restrict__ far)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    constexpr int PAIRS = WIN_THREADS / 2;
    const int32_t ti = blockIdx.x / blocks_per_tile;
    const TileDev tile = a.tiles[ti];
    const GroupDev& grp = a.groups[tile.group];
    const DevModel& m = a.m;
    const int N = a.N, pop = threadIdx.x & 1;
    const WinSlot ws = win_slot<1>(tile, ((blockIdx.x % blocks_per_tile) * blockDim.x + threadIdx.x) >> 1);
    const uint32_t lanes = __ballot_sync(0xffffffffu, ws.k < N);
    after_last_launch();
    if (ws.k >= N) return;
    const int k = ws.k, q = ws.q, H = grp.H, HR = H + WIN_FAR, steps = a.n_chunk, ts = a.ts;
    const bool own_noise = a.noise_per_set != 0;
    const uint32_t n0 = (uint32_t)a.n0;
    const int slot0 = (int)(n0 % (uint32_t)H);
    float* ring = grp.ring + (int64_t)tile.q0 * N * HR + q;
    float* stash = reinterpret_cast<float*>(win_smem) + (threadIdx.x >> 1);   // step b at stash[b * PAIRS]

    // 1. coupling sums: of every 2 G steps a lane takes G
    {
        const int e0 = NEAR ? grp.row_near[k] : grp.row_ptr[k], e1 = grp.row_end[k];
        const float* far_k = NEAR ? far + ((int64_t)ti * WIN_FAR * N + k) * pb + q : nullptr;
        int b0 = 0;
        auto pass = [&](auto g_c) {
            constexpr int G = decltype(g_c)::value;
            for (; b0 + 2 * G <= steps || (G == 1 && b0 < steps); b0 += 2 * G) {
                const int c0 = b0 + pop * G;
                if (c0 >= steps) continue;   // an odd last step
                float acc[G];
#pragma unroll
                for (int b = 0; b < G; ++b) acc[b] = NEAR ? far_k[(int64_t)(c0 + b) * N * pb] : 0.0f;
                int at = slot0 + c0;
                at -= at >= H ? H : 0;
                gather<G>(acc, grp, ring, e0, e1, at, H, HR, pb);
#pragma unroll
                for (int b = 0; b < G; ++b) stash[(c0 + b) * PAIRS] = acc[b];
            }
        };
        pass(std::integral_constant<int, 8>{});
        pass(std::integral_constant<int, 4>{});
        pass(std::integral_constant<int, 2>{});
        pass(std::integral_constant<int, 1>{});
    }
    __syncwarp(lanes);

    // 2. the window's steps; the even lane writes
    const int64_t NP = (int64_t)N * a.P;
    const int64_t p = grp.p_base + tile.q0 + q;
    float* st = a.state + (int64_t)k * a.P + p;
    const SetParams sp = load_set_params(a.prm, a.P, p);
    const float EL = pop ? sp.ELi : sp.ELe, cFe = pop ? sp.cFie : sp.cFee, cFi = pop ? sp.cFii : sp.cFei;
    float cp[10];
#pragma unroll
    for (int c = 0; c < 10; ++c) cp[c] = pop ? m.cp_i[c] : m.cp_e[c];
    const auto poly = [&cp](int c) { return cp[c]; };
    PairState x{st[SV_E * NP],  st[SV_I * NP],  st[SV_CEE * NP], st[SV_CEI * NP], st[SV_CII * NP],
                st[SV_WE * NP], st[SV_WI * NP], st[SV_CWE * NP], st[SV_CWI * NP]};
    float accE = st[SV_ACC_E * NP], accI = st[SV_ACC_I * NP], ou = own_noise ? st[SV_OU * NP] : 0.0f;
    const uint32_t pn = own_noise ? (uint32_t)(a.p_offset + a.ext_index[p]) : 0u;
    Track<float> trk = track_init<float>();
    const float inv_ts = 1.0f / (float)ts;
    int left = ts - (int)(n0 % (uint32_t)ts);
    int64_t t = n0 / (uint32_t)ts;
    int slot_w = slot0;
    float* const ring_k = ring + (uint32_t)(k * HR) * (uint32_t)pb;
    const float* ou_p = a.ou_table + (own_noise ? 0 : table_step * N + k);
    float ou_next = own_noise ? 0.0f : __ldg(ou_p), c_next = stash[0];   // the next step's, on the way
    for (int b = 0; b < steps; ++b) {
        const float OU = own_noise ? ou : ou_next, c = c_next;
        if (b + 1 < steps) {
            if (!own_noise) ou_next = __ldg(ou_p += N);
            c_next = stash[(b + 1) * PAIRS];
        }
        pair_step_split(m, poly, pop, EL, cFe, cFi, sp, x, c, OU, trk, lanes);
        if (own_noise) ou = next_ou(m, a.seed, n0 + (uint32_t)b, (uint32_t)k, pn, OU);
        ++slot_w;
        slot_w -= slot_w == H ? H : 0;
        accE = vadd(accE, x.E);
        accI = vadd(accI, x.I);
        if (pop == 0) {
            float* dst = ring_k + slot_w * pb;
            *dst = x.E;
            if (slot_w < WIN_FAR) dst[H * pb] = x.E;
        }
        if (--left == 0) {
            if (t < a.T && pop == 0) {
                const float xE = vmul(accE, inv_ts), xI = vmul(accI, inv_ts);
                const int64_t so = series_index(a.sl, t, k, p);
                a.series[so] = xE;
                if (a.series_i) a.series_i[so] = xI;
                if (t >= a.transient) {
                    float sE = st[SV_SUM_E * NP], cE = st[SV_CMP_E * NP];
                    float sI = st[SV_SUM_I * NP], cI = st[SV_CMP_I * NP];
                    kahan_add(sE, cE, xE);
                    kahan_add(sI, cI, xI);
                    st[SV_SUM_E * NP] = sE;
                    st[SV_CMP_E * NP] = cE;
                    st[SV_SUM_I * NP] = sI;
                    st[SV_CMP_I * NP] = cI;
                }
            }
            left = ts;
            ++t;
            accE = 0.0f;
            accI = 0.0f;
        }
    }
    if (pop) return;
    const float v[11] = {x.E, x.I, x.Cee, x.Cei, x.Cii, x.We, x.Wi, x.cWe, x.cWi, accE, accI};
    constexpr int at[11] = {SV_E, SV_I, SV_CEE, SV_CEI, SV_CII, SV_WE, SV_WI, SV_CWE, SV_CWI, SV_ACC_E, SV_ACC_I};
#pragma unroll
    for (int c = 0; c < 11; ++c) st[at[c] * NP] = v[c];
    if (own_noise) st[SV_OU * NP] = ou;
    const uint32_t f = track_flags(m, trk, 0);
    if (f) atomicOr(a.status + p, f);
}

// Window `turn` of a job: its first step within the round, its length (0: the
// round is over) and its first row of the far sums. A window stays within the
// WIN_FAR steps whose far sums are at hand.
struct WinTurn {
    int w0, len, row;
};
__host__ __device__ __forceinline__ WinTurn win_turn(int turn, int steps, bool far, int n_chunk)
{
    WinTurn t;
    t.row = 0;
    if (far) {
        const int per = (WIN_FAR + steps - 1) / steps;   // windows per far block
        t.row = turn % per * steps;
        t.w0 = turn / per * WIN_FAR + t.row;
        t.len = WIN_FAR - t.row < steps ? WIN_FAR - t.row : steps;
    } else {
        t.w0 = turn * steps;
        t.len = steps;
    }
    if (t.len > n_chunk - t.w0) t.len = n_chunk - t.w0 > 0 ? n_chunk - t.w0 : 0;
    return t;
}

// A batch of sweeps that all have windows and share the model m: one launch
// takes every job through its window `turn` (FAR: forms the far sums of the
// jobs that start a far block with it). blocks[i] names block i's job and its
// index among the job's blocks. The register-tile body, whose CTAs keep a tile
// of 4 to 28 sets through a whole round, took 19.4 ms of an eight-job batch of
// 64 to 1,024 sets; a windowed body over such tiles reads rows of 16 bytes and
// took 34 ms.
template <class V, bool FAR>
__global__ void __launch_bounds__(WIN_THREADS, 4)
sim_batch_window_kernel(const __grid_constant__ DevModel m, const BatchJob* __restrict__ jobs,
                        const BatchItem* __restrict__ blocks, int32_t turn)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    __shared__ BatchJob s_job;
    constexpr int S = VSets<V>::n;
    const BatchItem bi = blocks[blockIdx.x];
    const uint32_t* src = reinterpret_cast<const uint32_t*>(jobs + bi.job);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&s_job);
    for (int w = threadIdx.x; w < (int)(sizeof(BatchJob) / 4); w += WIN_THREADS) dst[w] = src[w];
    __syncthreads();
    after_last_launch();
    const SimArgs& a = s_job.a;
    const WinTurn t = win_turn(turn, s_job.win_steps, s_job.far != nullptr, a.n_chunk);
    if (t.len == 0 || (FAR && (!s_job.far || t.row != 0))) return;
    const int N = a.N, bpt = (N * (WIN_BATCH_PB / S) + WIN_THREADS - 1) / WIN_THREADS;
    const int ti = bi.tile / bpt;
    const TileDev tile = a.tiles[ti];
    const GroupDev grp = a.groups[tile.group];
    const WinSlot ws = win_slot<S>(tile, (bi.tile - ti * bpt) * WIN_THREADS + threadIdx.x);
    if (ws.k >= N) return;
    const uint32_t n0 = (uint32_t)a.n0 + (uint32_t)t.w0;
    float* far = s_job.far ? s_job.far + (int64_t)ti * WIN_FAR * N * WIN_BATCH_PB : nullptr;
    V* stash = reinterpret_cast<V*>(win_smem) + threadIdx.x;
    if constexpr (FAR) {
        far_pair<V, WIN_BATCH_PB>(a, tile, grp, ws, WIN_BATCH_PB, n0, far);
    } else if (far) {
        window_pair<V, WIN_BATCH_PB, true>(a, m, tile, grp, ws, WIN_BATCH_PB, n0, t.len, t.w0,
                                           far + (int64_t)t.row * N * WIN_BATCH_PB, stash);
    } else {
        window_pair<V, WIN_BATCH_PB, false>(a, m, tile, grp, ws, WIN_BATCH_PB, n0, t.len, t.w0, nullptr, stash);
    }
}

// [tile][N][H + WIN_FAR][pb] <-> slots [f0, f0 + nf) of [H0][N][stride], whose slot f
// holds the latest step t <= n with t = f mod H0. Blocks along the sets of one region
// and slot (blockIdx.y, .z): the divisions are a block's, not an element's (0.2 ms per
// 64 MB with the latter).
template <bool OUT>
__global__ void ring_convert_kernel(float* __restrict__ ring, int32_t H, int32_t pb, int32_t N, int32_t P_g,
                                    int32_t stride, int32_t H0, int64_t n, int32_t f0, float E0,
                                    float* __restrict__ rows)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, f = f0 + (int)blockIdx.z;
    if (c >= stride) return;
    float* row = rows + ((int64_t)blockIdx.z * N + j) * stride + c;
    if (c >= P_g) {
        if (OUT) *row = E0;
        return;
    }
    int64_t back = (n - f) % H0;
    back += back < 0 ? H0 : 0;
    int64_t slot = (n - back) % H;
    slot += slot < 0 ? H : 0;
    const int tile = c / pb;
    float* at = ring + (((int64_t)tile * N + j) * (H + WIN_FAR) + slot) * pb + (c - tile * pb);
    if (OUT) {
        *row = *at;
    } else {
        *at = *row;
        if (slot < WIN_FAR) at[(int64_t)H * pb] = *row;
    }
}

// A window takes 5 to 400 us: launches that start under the end of the last one
// (launch_next) took 16 x 68 from 0.85 to 0.77 ms per 1,000 steps, 1,001 x 68 at
// six speeds from 1.47 to 1.39, an eight-job batch from 8.9 to 8.4.
//
// far sums (when due) and the window of every pair; S sets per thread, or (SPLIT) two threads per set
template <class V, int PB, bool SPLIT = false>
cudaError_t launch_v(const SimArgs& a, const WindowPlan& w, int32_t n_tiles, int64_t table_step, float* far,
                     int32_t far_row, cudaStream_t s)
{
    constexpr int S = VSets<V>::n;
    const int64_t per_tile = (int64_t)a.N * ((w.pb + S - 1) / S);
    const int32_t bpt = (int32_t)((per_tile + w.threads - 1) / w.threads);
    const int32_t bpt_w = SPLIT ? (int32_t)((2 * per_tile + w.threads - 1) / w.threads) : bpt;
    const unsigned grid = (unsigned)((int64_t)n_tiles * bpt_w);
    const size_t smem = sizeof(V) * (size_t)WIN_THREADS * a.n_chunk / (SPLIT ? 2 : 1);
    float* row = nullptr;
    if (w.far) {
        if (far_row == 0) {
            const cudaError_t e = launch_next(sim_far_kernel<V, PB>, (unsigned)((int64_t)n_tiles * bpt), w.threads, 0, s,
                                              a, w.pb, bpt, far);
            if (e != cudaSuccess) return e;
        }
        row = far + (int64_t)far_row * a.N * w.pb;
    }
    if constexpr (SPLIT)
        return launch_next(w.far ? sim_window_split_kernel<true> : sim_window_split_kernel<false>, grid, w.threads, smem,
                           s, a, w.pb, bpt_w, table_step, row);
    else
        return launch_next(w.far ? sim_window_kernel<V, PB, true> : sim_window_kernel<V, PB, false>, grid, w.threads,
                           smem, s, a, w.pb, bpt_w, table_step, row);
}

}  // namespace

void sim_window_plan(int32_t d_min, int32_t N, int64_t P, int64_t P_group, bool reduced, int sms, WindowPlan& w)
{
    // d_min + 1 steps, less those that would need a gather pass of their own: 24 of
    // 28 steps (32,768 x 68: 20.97 ms against 21.03, 21.70 at 27), 16 of 17 (1,001 x
    // 68: 1.38 against 1.48), 8 of 13 (500 x 192: 1.67 against 1.84, 1.68 at 12), 4
    // of 5 (16,384 x 68: 5.45 against 5.65); 6, 4, 3 and 2 beat 5, 3, 2 and 1
    w.steps = d_min < WIN_MAX_STEPS - 1 ? d_min + 1 : WIN_MAX_STEPS;
    if (w.steps >= 8) w.steps -= w.steps % 8;
    else if (w.steps >= 5) w.steps -= w.steps % 2;
    w.far = w.steps < WIN_NEAR_BELOW;
    // packed pairs of sets (fewer instructions per step, half the threads) from
    // four warps per scheduler of single ones on: 1,001 x 68 (448 pairs per SM)
    // took 1.50 ms packed and 1.45 single, 1,500 x 68 the same either way. Two
    // lanes per pair while the chain of a step bounds the sweep: 16 x 68 took
    // 0.85 ms per 1,000 steps against 1.39 (0.66 with windows of 24 that start
    // under the last one's end), 400 x 68 (179 pairs per SM) 0.50 against 0.62, 600
    // x 68 (268) 0.95 against 0.74.
    const int64_t pairs = (int64_t)N * P;
    w.packed = reduced && pairs >= (int64_t)sms * 512;
    w.split = reduced && pairs <= (int64_t)sms * 192;
    w.pb = 64;
    while (w.pb > 2 && w.pb / 2 >= P_group) w.pb /= 2;
    const int64_t threads = w.packed ? (pairs + 1) / 2 : (w.split ? 2 * pairs : pairs);
    // smaller CTAs spread a sweep that cannot fill the chip over more SMs
    w.threads = threads >= (int64_t)sms * WIN_THREADS ? WIN_THREADS : (threads >= (int64_t)sms * 64 ? 64 : 32);
}

cudaError_t launch_sim_window(const SimArgs& a, const WindowPlan& w, int32_t n_tiles, int64_t table_step, float* far,
                              int32_t far_row, cudaStream_t s)
{
    if (n_tiles <= 0 || a.n_chunk <= 0) return cudaSuccess;
    if (w.packed) return w.pb == 64 ? launch_v<float2, 64>(a, w, n_tiles, table_step, far, far_row, s)
                                    : launch_v<float2, 0>(a, w, n_tiles, table_step, far, far_row, s);
    return w.split ? launch_v<float, 0, true>(a, w, n_tiles, table_step, far, far_row, s)
                   : launch_v<float, 0>(a, w, n_tiles, table_step, far, far_row, s);
}

int32_t sim_batch_window_blocks(int32_t N, bool packed)
{
    return (N * (packed ? WIN_BATCH_PB / 2 : WIN_BATCH_PB) + WIN_THREADS - 1) / WIN_THREADS;
}

int32_t sim_batch_window_turns(int32_t steps, bool far, int32_t n_chunk)
{
    if (n_chunk <= 0) return 0;
    if (!far) return (n_chunk + steps - 1) / steps;
    const int32_t per = (WIN_FAR + steps - 1) / steps, rest = n_chunk % WIN_FAR;
    return n_chunk / WIN_FAR * per + (rest + steps - 1) / steps;
}

cudaError_t launch_sim_batch_window(const DevModel& m, bool packed, bool far, const BatchJob* jobs,
                                    const BatchItem* blocks, int32_t n_blocks, int32_t turn, int32_t steps,
                                    cudaStream_t s)
{
    if (n_blocks <= 0) return cudaSuccess;
    auto kern = packed ? (far ? sim_batch_window_kernel<float2, true> : sim_batch_window_kernel<float2, false>)
                       : (far ? sim_batch_window_kernel<float, true> : sim_batch_window_kernel<float, false>);
    return launch_next(kern, n_blocks, WIN_THREADS, far ? 0 : (packed ? 8 : 4) * (size_t)WIN_THREADS * steps, s, m, jobs,
                       blocks, turn);
}

cudaError_t launch_ring_convert(bool out, float* ring, const WindowPlan& w, int32_t H, int32_t N, int32_t P_g,
                                int32_t stride, int32_t H0, int64_t n, int32_t f0, int32_t nf, float E0, float* rows,
                                cudaStream_t s)
{
    note_launch();
    auto kern = out ? ring_convert_kernel<true> : ring_convert_kernel<false>;
    if (nf < 1) return cudaSuccess;
    const unsigned threads = stride < 256 ? (unsigned)stride : 256;   // whole warps: the stride is a multiple of 32
    kern<<<dim3((stride + threads - 1) / threads, N, nf), threads, 0, s>>>(ring, H, w.pb, N, P_g, stride, H0, n, f0, E0,
                                                                         rows);
    return cudaGetLastError();
}

}  // namespace tvbx
