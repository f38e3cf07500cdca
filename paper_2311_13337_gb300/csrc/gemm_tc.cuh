// Tensor-core (tcgen05) matrix product of the surrogate network, with the
// operands of gemm_simt.cuh:
//   C(m, n) = sum_k A(m, k) B(n, k),  A(m, k) = A[m sam + k sak],
//   B(n, k) = B[n sbn + k sbk],  blockIdx.z = ensemble member,
// and the same epilogues (bias, bias + ReLU, mask).
//
// Split precision. An FP32 operand X is split into BF16 parts X = H + L
// (H = bf16(X), L = bf16(X - H)); a BF16 operand (the network's weights) is
// its own H with L = 0. The product takes H_A H_B + L_A H_B (+ H_A L_B when
// both operands are FP32) on the tensor cores in kind::f16 (BF16 x BF16) with
// FP32 accumulation in tensor memory: the error of the split is about 2^-16
// of each operand, far below the FP32 reference product's own rounding over
// these K.
//
// Layout. A CTA of 128 threads owns a 128 x 128 tile of C. Per chunk of 64
// K (one 128-byte row of BF16) the threads read their shares of the A and B
// tiles (lanes along K where K is contiguous, else along the rows: the backward
// products read transposed operands) into registers, split, and write the
// parts to shared memory in the 128-byte swizzled K-major layout; one thread
// then issues the MMAs of the four 16-wide K slices and commits them to an
// mbarrier; the next chunk is read under them, and every thread waits (bounded)
// before it overwrites the operands. The accumulator (128 lanes x up to 128
// FP32 columns) is read back by the four warps, each its 32 lanes (rows), and
// stored with the epilogue along the rows. Rows and columns beyond M, N and K
// are staged as zeros. The products are small (1,024 x 256 x 256 per member)
// and bound by latency: a row per thread, read and written 4 bytes at a time,
// measured 113, 53 and 31 us for the masked, forward and weight products.
//
// Split K. A product with few output tiles and a long K (the weight
// gradients: K = the mini-batch rows) would occupy a handful of SMs, so its
// K chunks are divided among `splits` CTAs per tile; each writes its partial
// tile to a scratch array and a second kernel adds the partials in split
// order (deterministic), for the plain-store epilogue only.
#pragma once

#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_simt.cuh"
#include "internal.h"
#include "launch_next.cuh"
#include "ptx_async.cuh"

namespace tvbx {

constexpr int TCG_M = 128;       // rows of C per CTA (the MMA's M)
constexpr int TCG_N = 128;       // columns of C per CTA (MMA N <= 128, a multiple of 16)
constexpr int TCG_K = 64;        // K per staged chunk: 64 BF16 = one 128-byte row
constexpr int TCG_THREADS = 128;
constexpr int TCG_TILE_BYTES = TCG_M * TCG_K * 2;   // one operand part, 16 KB
constexpr size_t TCG_SMEM = 4 * (size_t)TCG_TILE_BYTES + 1024;   // A hi/lo, B hi/lo, slack for alignment

// Byte offset of element (r, k) (k < 64) of a 128-byte swizzled K-major tile.
static __device__ __forceinline__ uint32_t tcg_sw_off(int r, int k)
{
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((((k >> 3) ^ (r & 7)) & 7) << 4) + ((k & 7) << 1));
}

static __device__ __forceinline__ uint32_t tcg_pack2(__nv_bfloat16 a, __nv_bfloat16 b)
{
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// Registers of one thread's share of an operand chunk (128 rows x 64 K).
template <typename T> struct TcgRegs {
    uint32_t v[16 * sizeof(T)];   // FP32: 64 values; BF16: 64 values in pairs
};

// Load the chunk [0, 128) x [k0, k0 + 64) of an operand of R valid rows and K
// columns; zeros beyond. X points at row 0. K-contiguous operands (s_k == 1):
// lanes along the row, 16 bytes each (vec: rows start 16-byte aligned), else
// lanes along the rows, which are then neighbours (s_row == 1).
static __device__ __forceinline__ void tcg_load(TcgRegs<float>& f, const float* X, int64_t s_row, int64_t s_k, bool vec,
                                                int R, int k0, int K)
{
    const int t = threadIdx.x;
    if (s_k == 1) {
#pragma unroll
        for (int p = 0; p < 16; ++p) {
            const int r = 8 * p + (t >> 4), k = k0 + 4 * (t & 15);
            float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r < R) {
                const float* at = X + r * s_row + k;
                if (vec && k + 4 <= K) {
                    x = *reinterpret_cast<const float4*>(at);
                } else {
                    if (k < K) x.x = at[0];
                    if (k + 1 < K) x.y = at[1];
                    if (k + 2 < K) x.z = at[2];
                    if (k + 3 < K) x.w = at[3];
                }
            }
            f.v[4 * p] = __float_as_uint(x.x);
            f.v[4 * p + 1] = __float_as_uint(x.y);
            f.v[4 * p + 2] = __float_as_uint(x.z);
            f.v[4 * p + 3] = __float_as_uint(x.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < TCG_K; ++k)
            f.v[k] = t < R && k0 + k < K ? __float_as_uint(X[t * s_row + (k0 + k) * s_k]) : 0u;
    }
}
static __device__ __forceinline__ void tcg_load(TcgRegs<__nv_bfloat16>& f, const __nv_bfloat16* X, int64_t s_row,
                                                int64_t s_k, bool vec, int R, int k0, int K)
{
    const int t = threadIdx.x;
    const uint16_t* U = reinterpret_cast<const uint16_t*>(X);
    if (s_k == 1) {
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const int r = 16 * p + (t >> 3), k = k0 + 8 * (t & 7);
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (r < R) {
                const uint16_t* at = U + r * s_row + k;
                if (vec && k + 8 <= K) {
                    x = *reinterpret_cast<const uint4*>(at);
                } else {
                    uint32_t w[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        w[q] = (k + 2 * q < K ? at[2 * q] : 0u) | (k + 2 * q + 1 < K ? (uint32_t)at[2 * q + 1] << 16 : 0u);
                    x = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            f.v[4 * p] = x.x;
            f.v[4 * p + 1] = x.y;
            f.v[4 * p + 2] = x.z;
            f.v[4 * p + 3] = x.w;
        }
    } else {
        // lanes along K, two K of eight neighbouring rows each: 4 pairs (k, k + 1)
        // of row group (t >> 5) + 4 p, in f.v[8 p + row]
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const int r = 8 * ((t >> 5) + 4 * p), k = k0 + 2 * (t & 31);
            uint32_t w[2][4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint16_t* at = U + r + (k + h) * s_k;
                if (k + h >= K) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) w[h][q] = 0u;
                } else if (vec && r + 8 <= R) {
                    const uint4 x = *reinterpret_cast<const uint4*>(at);
                    w[h][0] = x.x; w[h][1] = x.y; w[h][2] = x.z; w[h][3] = x.w;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        w[h][q] = (r + 2 * q < R ? at[2 * q] : 0u) | (r + 2 * q + 1 < R ? (uint32_t)at[2 * q + 1] << 16 : 0u);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                f.v[8 * p + 2 * q] = __byte_perm(w[0][q], w[1][q], 0x5410);
                f.v[8 * p + 2 * q + 1] = __byte_perm(w[0][q], w[1][q], 0x7632);
            }
        }
    }
}

// Split the loaded values into BF16 parts and write them to the swizzled tiles
// at sh (high) and sl (low; a BF16 operand has none).
static __device__ __forceinline__ void tcg_split2(float x, float y, uint32_t& h, uint32_t& l)
{
    const __nv_bfloat16 hx = __float2bfloat16_rn(x), hy = __float2bfloat16_rn(y);
    h = tcg_pack2(hx, hy);
    l = tcg_pack2(__float2bfloat16_rn(x - __bfloat162float(hx)), __float2bfloat16_rn(y - __bfloat162float(hy)));
}
static __device__ __forceinline__ void tcg_store4(uint32_t at, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(at), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
static __device__ __forceinline__ void tcg_put(const TcgRegs<float>& f, int64_t s_k, uint32_t sh, uint32_t sl)
{
    const int t = threadIdx.x;
    if (s_k == 1) {
#pragma unroll
        for (int p = 0; p < 16; ++p) {
            uint32_t h[2], l[2];
            tcg_split2(__uint_as_float(f.v[4 * p]), __uint_as_float(f.v[4 * p + 1]), h[0], l[0]);
            tcg_split2(__uint_as_float(f.v[4 * p + 2]), __uint_as_float(f.v[4 * p + 3]), h[1], l[1]);
            const uint32_t off = tcg_sw_off(8 * p + (t >> 4), 4 * (t & 15));
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};\n" ::"r"(sh + off), "r"(h[0]), "r"(h[1]) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};\n" ::"r"(sl + off), "r"(l[0]), "r"(l[1]) : "memory");
        }
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                tcg_split2(__uint_as_float(f.v[8 * c + 2 * q]), __uint_as_float(f.v[8 * c + 2 * q + 1]), h[q], l[q]);
            const uint32_t off = tcg_sw_off(t, 8 * c);
            tcg_store4(sh + off, h[0], h[1], h[2], h[3]);
            tcg_store4(sl + off, l[0], l[1], l[2], l[3]);
        }
    }
}
static __device__ __forceinline__ void tcg_put(const TcgRegs<__nv_bfloat16>& f, int64_t s_k, uint32_t sh, uint32_t)
{
    const int t = threadIdx.x;
    if (s_k == 1) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            tcg_store4(sh + tcg_sw_off(16 * c + (t >> 3), 8 * (t & 7)), f.v[4 * c], f.v[4 * c + 1], f.v[4 * c + 2],
                       f.v[4 * c + 3]);
    } else {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(sh + tcg_sw_off(8 * ((t >> 5) + 4 * p) + i, 2 * (t & 31))),
                             "r"(f.v[8 * p + i])
                             : "memory");
    }
}

template <typename TA, typename TB, int EPI>
__global__ void __launch_bounds__(TCG_THREADS) mlp_gemm_tc_kernel(const GemmArgs g, uint32_t* __restrict__ error,
                                                                  uint32_t wait_limit, int splits, int chunks_per_split,
                                                                  float* __restrict__ part)
{
    extern __shared__ __align__(1024) uint8_t tcg_smem_raw[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    // 1024-byte aligned operand tiles (the swizzle pattern is tied to address bits)
    const uint32_t raw = smem_u32(tcg_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t sAh = base, sAl = base + TCG_TILE_BYTES, sBh = base + 2 * TCG_TILE_BYTES,
                   sBl = base + 3 * TCG_TILE_BYTES;
    constexpr bool B_SPLIT = !std::is_same<TB, __nv_bfloat16>::value;
    constexpr bool A_SPLIT = !std::is_same<TA, __nv_bfloat16>::value;

    const int64_t mem = blockIdx.z / splits;
    const int split = (int)(blockIdx.z % splits);
    const TA* A = static_cast<const TA*>(g.A) + mem * g.a_mem;
    const TB* B = static_cast<const TB*>(g.B) + mem * g.b_mem;
    const int m0 = blockIdx.y * TCG_M, n0 = blockIdx.x * TCG_N;
    const int nvalid = min(TCG_N, g.N - n0);
    const uint32_t nmma = (uint32_t)((nvalid + 15) / 16 * 16);   // MMA N: a multiple of 16
    const uint32_t idesc = tc_idesc(1u, (uint32_t)TCG_M, nmma);
    const int t = threadIdx.x;

    if (t == 0) {
        mbar_init(&mbar, 1);
        abort_flag = 0;
        fence_mbarrier_init();
    }
    if (t < 32) tmem_alloc(&tmem_slot, (uint32_t)TCG_N);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    after_last_launch();

    const TA* Am = A + (int64_t)m0 * g.sam;
    const TB* Bn = B + (int64_t)n0 * g.sbn;
    // 16-byte pieces along the contiguous direction
    const bool a_vec = (reinterpret_cast<uintptr_t>(Am) & 15) == 0 && (g.sak == 1 ? g.sam : g.sak) * sizeof(TA) % 16 == 0;
    const bool b_vec = (reinterpret_cast<uintptr_t>(Bn) & 15) == 0 && (g.sbk == 1 ? g.sbn : g.sbk) * sizeof(TB) % 16 == 0;
    TcgRegs<TA> ra;
    TcgRegs<TB> rb;

    uint32_t parity = 0;
    const int n_chunks = (g.K + TCG_K - 1) / TCG_K;
    const int ch0 = split * chunks_per_split, ch1 = min(n_chunks, ch0 + chunks_per_split);   // ch0 < ch1 (host)
    tcg_load(ra, Am, g.sam, g.sak, a_vec, g.M - m0, ch0 * TCG_K, g.K);
    tcg_load(rb, Bn, g.sbn, g.sbk, b_vec, g.N - n0, ch0 * TCG_K, g.K);
    for (int ch = ch0; ch < ch1; ++ch) {
        tcg_put(ra, g.sak, sAh, sAl);
        tcg_put(rb, g.sbk, sBh, sBl);
        fence_proxy_async_shared();   // the operand writes, visible to the tensor cores
        __syncthreads();
        if (t == 0 && !abort_flag) {
            tc_fence_after();
#pragma unroll
            for (int sl = 0; sl < TCG_K / 16; ++sl) {
                const uint32_t koff = (uint32_t)(sl * 32);   // 16 BF16 = 32 bytes into each row
                const uint64_t ah = sw128_desc(sAh + koff), bh = sw128_desc(sBh + koff);
                tc_mma<0>(tmem, ah, bh, idesc, (ch > ch0 || sl > 0) ? 1u : 0u);
                if (A_SPLIT) tc_mma<0>(tmem, sw128_desc(sAl + koff), bh, idesc, 1u);
                if (B_SPLIT) tc_mma<0>(tmem, ah, sw128_desc(sBl + koff), idesc, 1u);
            }
            tc_commit(&mbar);
        }
        if (ch + 1 < ch1) {   // the next chunk, under the MMAs
            tcg_load(ra, Am, g.sam, g.sak, a_vec, g.M - m0, (ch + 1) * TCG_K, g.K);
            tcg_load(rb, Bn, g.sbn, g.sbk, b_vec, g.N - n0, (ch + 1) * TCG_K, g.K);
        }
        // every thread: wait (bounded) until the MMAs have read the operands
        if (!abort_flag && !mbar_wait_bounded(&mbar, parity, wait_limit)) {
            atomicOr(error, TVBX_DEVERR_TIMEOUT);
            abort_flag = 1;
        }
        parity ^= 1u;
        tc_fence_after();
        __syncthreads();
    }

    // epilogue: warp w drains accumulator lanes 32 w .. 32 w + 31 (rows of C)
    // to the operands' shared memory, 16-byte pieces swizzled by the row, and
    // writes its rows from there, lanes along the columns
    const int warp = t >> 5, lane = t & 31;
    float* C = g.C + mem * g.c_mem;
    int64_t ldc = g.ldc;
    if (part) {   // split K: this split's partial tile, [split][member][M][N]
        const int64_t E = gridDim.z / splits;
        C = part + ((int64_t)split * E + mem) * (int64_t)g.M * g.N;
        ldc = g.N;
    }
    if (!abort_flag) {
        auto piece = [&](int row, int c) { return base + (uint32_t)(row * 4 * TCG_N + ((c ^ (row & 31)) << 4)); };
        for (int cb = 0; cb * 16 < nvalid; ++cb) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(cb * 16), v);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                tcg_store4(piece(t, 4 * cb + q), __float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                           __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
        }
        __syncwarp();
        const int n = n0 + 4 * lane;
        const int left = g.N - n;
        const float* mask = EPI == EPI_MASK ? g.mask + mem * g.mask_mem + n : nullptr;
        const bool vec = left >= 4 && ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C + n) & 15) == 0 &&
                         (EPI != EPI_MASK || (g.ldm % 4 == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0));
        float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < left) bias[i] = g.bias[mem * g.bias_mem + n + i];
        const int rows = min(32, g.M - m0 - 32 * warp);
        if (left > 0) {
#pragma unroll 4
            for (int r = 0; r < rows; ++r) {
                const int row = 32 * warp + r;
                float x[4];
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                             : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
                             : "r"(piece(row, lane)));
                float* out = C + (int64_t)(m0 + row) * ldc + n;
                float mk[4] = {1.0f, 1.0f, 1.0f, 1.0f};
                if (EPI == EPI_MASK) {
                    const float* at = mask + (int64_t)(m0 + row) * g.ldm;
                    if (vec) {
                        const float4 q = *reinterpret_cast<const float4*>(at);
                        mk[0] = q.x; mk[1] = q.y; mk[2] = q.z; mk[3] = q.w;
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < left) mk[i] = at[i];
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU) x[i] += bias[i];
                    if (EPI == EPI_BIAS_RELU) x[i] = fmaxf(x[i], 0.0f);
                    if (EPI == EPI_MASK && !(mk[i] > 0.0f)) x[i] = 0.0f;
                }
                if (vec) {
                    *reinterpret_cast<float4*>(out) = make_float4(x[0], x[1], x[2], x[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < left) out[i] = x[i];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (t < 32) tmem_dealloc(tmem, (uint32_t)TCG_N);
}

// Column sums of X [E][rows][n] to out, a member every out_mem (a layer's bias
// gradient): 8 row-interleaved sums per column.
struct ColumnSums {
    const float* X = nullptr;
    float* out = nullptr;
    int rows = 0, n = 0;
    int64_t out_mem = 0;
};
__device__ __forceinline__ void column_sums(const ColumnSums& c, int mem, int block)
{
    const int o = block * 32 + (threadIdx.x & 31);
    const int q = threadIdx.x >> 5;
    float s = 0.0f;
    if (o < c.n)
#pragma unroll 16
        for (int r = q; r < c.rows; r += 8) s += c.X[((int64_t)mem * c.rows + r) * c.n + o];
    __shared__ float red[8][33];
    red[q][threadIdx.x & 31] = s;
    __syncthreads();
    if (q == 0 && o < c.n) {
        float t = 0.0f;
        for (int i = 0; i < 8; ++i) t += red[i][threadIdx.x & 31];
        c.out[mem * c.out_mem + o] = t;
    }
}

// The first `sums` blocks: column sums. The others: C(member) = sum over splits
// of the partial tiles, in split order. Both wait on memory with few loads in
// flight, so they share a launch; 256 threads.
__global__ void __launch_bounds__(256)
mlp_reduce_kernel(const ColumnSums c, int sums, const float* __restrict__ part, int splits, int E, int M, int N,
                  float* __restrict__ C, int64_t ldc, int64_t c_mem)
{
    after_last_launch();
    if ((int)blockIdx.x < sums) {
        const int per = sums / E;
        column_sums(c, blockIdx.x / per, blockIdx.x % per);
        return;
    }
    const int64_t MN = (int64_t)M * N, total = (int64_t)E * MN, step = (int64_t)(gridDim.x - sums) * blockDim.x;
    for (int64_t i = (int64_t)(blockIdx.x - sums) * blockDim.x + threadIdx.x; i < total; i += step) {
        const int64_t mem = i / MN, r = i % MN;
        float acc = 0.0f;
#pragma unroll 8
        for (int sp = 0; sp < splits; ++sp) acc += part[((int64_t)sp * E + mem) * MN + r];
        C[mem * c_mem + (r / N) * ldc + r % N] = acc;
    }
}

// Launch on E members; error: device word that receives TVBX_DEVERR_TIMEOUT
// when a bounded wait expires (the outputs are then invalid). part / part_cap
// (floats): scratch for split K (plain-store epilogue only; nullptr: none).
// sums: column sums to form beside the product (X nullptr: none).
template <typename TA, typename TB, int EPI>
static inline cudaError_t gemm_tc(const GemmArgs& g, int E, uint32_t* error, uint32_t wait_limit, cudaStream_t s,
                                  float* part = nullptr, size_t part_cap = 0,
                                  const ColumnSums& sums = {})
{
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return cudaSuccess;
    auto kern = mlp_gemm_tc_kernel<TA, TB, EPI>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TCG_SMEM);
    if (e != cudaSuccess) return e;
    const int tiles = ((g.N + TCG_N - 1) / TCG_N) * ((g.M + TCG_M - 1) / TCG_M) * E;
    const int n_chunks = (g.K + TCG_K - 1) / TCG_K;
    int splits = 1;
    if (EPI == EPI_STORE && part) {
        // about two CTAs per SM of the 152, as far as the chunks and the scratch allow
        splits = std::min(n_chunks, std::max(1, 304 / tiles));
        const size_t per_split = (size_t)E * g.M * g.N;
        splits = (int)std::min<size_t>((size_t)splits, part_cap / per_split);
        splits = std::max(splits, 1);
    }
    const int cps = (n_chunks + splits - 1) / splits;
    splits = (n_chunks + cps - 1) / cps;   // every split owns at least one chunk
    dim3 grid((g.N + TCG_N - 1) / TCG_N, (g.M + TCG_M - 1) / TCG_M, E * splits);
    e = launch_next(kern, grid, TCG_THREADS, TCG_SMEM, s, g, error, wait_limit, splits, cps, splits > 1 ? part : nullptr);
    const int sum_blocks = sums.X ? (sums.n + 31) / 32 * E : 0;
    if (e != cudaSuccess || (splits == 1 && sum_blocks == 0)) return e;
    const int64_t total = (int64_t)E * g.M * g.N;
    const int blocks = splits > 1 ? (int)std::min<int64_t>((total + 255) / 256, 4 * 152) : 0;
    return launch_next(mlp_reduce_kernel, dim3(sum_blocks + blocks), 256, 0, s, sums, sum_blocks, part, splits, E, g.M, g.N,
                       g.C, g.ldc, g.c_mem);
}

}  // namespace tvbx
