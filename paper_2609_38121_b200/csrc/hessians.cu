// Attention-aware Hessians on the GPU (Appendix C, "Aggregation for WUSH-A"): for one calibration sequence and
// every key/value head h, the key and value Hessians summed over the perturbed position s,
//   H_K(h) = (2 / tau^2) sum_t sum_{g,g'} A_{gg'}(t) q_{g,t} q_{g',t}^T,
//   A_{gg'}(t) = sum_{s<=t} p_{g,t,s} p_{g',t,s} (v_s - o_{g,t})^T Gamma_{gg'} (v_s - o_{g',t}),
//   H_V(h) = 2 sum_{g,g'} (sum_t sum_{s<=t} p_{g,t,s} p_{g',t,s}) Gamma_{gg'},     Gamma_{gg'} = W_O(h,g) W_O(h,g')^T,
// which is the appendix's key / value Hessian with the sums over s and t exchanged.  Expanding the bilinear form,
//   A_{gg'}(t) = W2 - W1 . (Gamma_{gg'} o_{g',t}) - W1 . (Gamma_{g'g} o_{g,t}) + W0 o_{g,t} . (Gamma_{gg'} o_{g',t}),
//   W0 = sum_s w_s,  W1 = sum_s w_s v_s,  W2 = sum_s w_s (v_s^T Gamma_{gg'} v_s),  w_s = p_{g,t,s} p_{g',t,s},
// and, with the sum over s kept together (no cancellation between the terms of the expansion),
//   A_{gg'}(t) = sum_s w_s (alpha_{gg'}(s) - v_s . U_{gg'}(t) + kappa_{gg'}(t)),   alpha = v_s . Gamma_{gg'} v_s,
//   U = Gamma_{gg'} o_{g',t} + Gamma_{g'g} o_{g,t},   kappa = o_{g,t} . Gamma_{gg'} o_{g',t},   A_{gg'} = A_{g'g}.
//
// Every step is a contraction over 128 channels or over positions.  Where one operand is bf16 already and the other fp32 (or
// both fp32), the fp32 one is split into three bf16 terms, 24 bits, and the products run on the tensor cores (mma.sync: the
// long sums have to be added up outside the tensor core, which cuts them towards zero, so every 16 products come back to registers).
// 1024 tokens of 32 / 8 heads: 1343 us as register-blocked fp32 products out of shared memory, bound by fp32 issue and shared-memory
// reads alike (pairs_kernel 626, rows_kernel 366, project_kernel 215); now 610 us (243, 96, 136).  Error of H_K against 64 bits, 2-norm, mean of five seeds:
// 3.6e-7 -> 1.6e-7; of H_V 4.9e-8 -> 3.3e-8:
//   gamma_kernel      Gamma_{gg'}, 128 x 128 x d_model, fp32 products, float64 across groups of 16
//   rows_kernel       causal softmax statistics (max, 1 / sum) and head outputs o_{g,t}: 64 x 64 tiles
//   project_kernel    U, kappa and alpha: 128 x 128 tiles
//   pairs_kernel      logits of all query heads and v_s . U of up to 10 pairs over tiles of 128 keys; A, W0
//   key_kernel        H_K: sum over (t, g) of q_{g,t} (sum_g' A_{gg'}(t) q_{g',t})^T, float64 across positions
//   finish_kernel     H_V = 2 sum_{gg'} (sum_t W0) Gamma_{gg'}; the slices of H_K added up in order
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <limits>
#include <type_traits>

#include "host_common.h"
#include "layout.cuh"

namespace wushkv {
namespace {

constexpr int HS_PITCH = D + 4;            // floats per staged row

struct HessParams {
    int S, n_kv, n_q, G, d_model, n_pairs;
    float inv_tau, scale2;       // 1 / tau; log2(e) / tau
    const unsigned short* Q;     // [S][n_q][D] bf16
    const unsigned short* K;     // [S][n_kv][D]
    const unsigned short* V;     // [S][n_kv][D]
    const float* W_O;            // [n_q][D][d_model]
    float* gamma;                // [n_kv][G][G][D][D]
    float* row_m;                // [S][n_q] maximum of the logits times log2(e)
    float* row_linv;             // [S][n_q] 1 / sum of the exponentials
    float* Oh;                   // [S][n_q][D]
    float* U;                    // [S][n_kv][n_pairs][D]
    float* kappa;                // [S][n_kv][n_pairs], where A goes: pairs_kernel reads a position's before it writes its A
    float* alpha;                // [S][n_kv][n_pairs]
    float* A;                    // [S][n_kv][n_pairs]   pairs g <= g' in row-major order
    float* W0;                   // [S][n_kv][n_pairs]
    double* key_part;            // [n_slices][n_kv][36][16][16] sums of key_kernel over a slice of positions, over Oh and U
    int n_slices, slice_len;
    double* H_K;                 // [n_kv][D][D]
    double* H_V;
};
__device__ __forceinline__ void pair_heads(int k, int G, int& g, int& gp) {
    g = 0;
    while (k >= G - g) { k -= G - g; ++g; }
    gp = g + k;
}
// Products on the tensor cores at fp32's precision: bf16 operands as they are, fp32 operands as three bf16 terms (24 bits), fp32 sums.
__device__ __forceinline__ unsigned hs_smem_addr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void hs_ldsm(unsigned addr, unsigned (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void hs_ldsm_t(unsigned addr, unsigned (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void hs_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// The tensor core cuts the sum it adds to towards zero, and over a chain of products of one sign pattern that adds up (with every sum kept
// there H_K's error is 5.7e-7 and H_V's 2.7e-7, 2-norm, where fp32 products have 3.6e-7 and 4.9e-8; 558 us): long sums are added up in fp32, the tensor core
// sums 16 products, or terms that are 2^-8 of the result or less.
__device__ __forceinline__ void hs_mma_add(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    float d[4];
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] += d[e];
}
__device__ __forceinline__ unsigned hs_pack(float lo, float hi) {
    unsigned r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// (x, y) as three pairs of bf16 whose sum is the fp32 values up to 2^-24 of each.  The first term stops at bf16's largest number, which
// fp32's range exceeds (the second makes up for it).
__device__ __forceinline__ void hs_split(float x, float y, unsigned& hi, unsigned& mid, unsigned& lo) {
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(y), "f"(x));
    const float x1 = x - __uint_as_float(hi << 16), y1 = y - __uint_as_float(hi & 0xffff0000u);
    mid = hs_pack(x1, y1);
    lo = hs_pack(x1 - __uint_as_float(mid << 16), y1 - __uint_as_float(mid & 0xffff0000u));
}
__device__ __forceinline__ float hs_ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// rows of 128 bf16 in shared memory, 16-byte pieces exchanged by the row's low bits: eight rows' pieces lie in different banks
__device__ __forceinline__ unsigned hs_piece(int row, int piece) { return 256u * row + (static_cast<unsigned>(piece ^ (row & 7)) << 4); }
// rows [s0, s0 + N) of a [S][heads][D] bf16 tensor's head h to shared memory, zeros beyond S
template <int N, int THREADS>
__device__ __forceinline__ void hs_request(unsigned dst, const unsigned short* X, int s0, int S, int heads, int h) {
#pragma unroll
    for (int n = 0; n < N * 16 / THREADS; ++n) {
        const int item = threadIdx.x + n * THREADS, row = item >> 4, piece = item & 15;
        const bool in = s0 + row < S;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + hs_piece(row, piece)),
                     "l"(X + (static_cast<long long>(in ? s0 + row : 0) * heads + h) * D + 8 * piece), "r"(in ? 16u : 0u) : "memory");
    }
}
__device__ __forceinline__ void hs_requested() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void hs_landed() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }

// C[i][j] += sum_k a[k][i] b[k][j] for one staged group of 16 k; thread: rows 4 (tid >> 4) .., columns outer_column(tid, e).
constexpr int OUTER_K = 16;
__device__ __forceinline__ int outer_column(int tid, int e) { return 4 * (tid & 15) + (e < 4 ? e : 60 + e); }
__device__ __forceinline__ void outer_group(const float (*a)[HS_PITCH], const float (*b)[HS_PITCH], double (&acc)[4][8]) {
    const int i0 = 4 * (threadIdx.x >> 4), j0 = 4 * (threadIdx.x & 15);
    float part[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int e = 0; e < 8; ++e) part[r][e] = 0.f;
#pragma unroll 4
    for (int k = 0; k < OUTER_K; ++k) {
        const float4 av = *reinterpret_cast<const float4*>(&a[k][i0]);
        const float4 b0 = *reinterpret_cast<const float4*>(&b[k][j0]), b1 = *reinterpret_cast<const float4*>(&b[k][64 + j0]);
        const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            part[0][e] = fmaf(av.x, bv[e], part[0][e]); part[1][e] = fmaf(av.y, bv[e], part[1][e]);
            part[2][e] = fmaf(av.z, bv[e], part[2][e]); part[3][e] = fmaf(av.w, bv[e], part[3][e]);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[r][e] += static_cast<double>(part[r][e]);
}

// Gamma_{gg'}[i][j] = sum_m W_g[i][m] W_g'[j][m] and its transpose Gamma_{g'g}; grid (pairs, n_kv, 4 blocks of 32 rows i), 128
// threads: with few pairs the time is that of one CTA's groups of 16 m, whose loads are in flight while the group before
// is multiplied (a CTA per pair with its loads waited for: 58 us for one pair and d_model 320).
__global__ void __launch_bounds__(128, 3) gamma_kernel(HessParams P) {
    __shared__ __align__(16) float a_s[OUTER_K][HS_PITCH], b_s[OUTER_K][HS_PITCH];
    int g, gp;
    pair_heads(blockIdx.x, P.G, g, gp);
    const int h = blockIdx.y, tid = threadIdx.x, r0 = 32 * blockIdx.z;
    const float* Wa = P.W_O + (static_cast<long long>(h * P.G + g) * D + r0) * P.d_model;
    const float* Wb = P.W_O + static_cast<long long>(h * P.G + gp) * D * P.d_model;
    double acc[4][8] = {};
    float ta[4], tb[16];
    auto fetch = [&](int m0) {
        const int m = m0 + (tid & 15);
        const bool in = m < P.d_model;
#pragma unroll
        for (int n = 0; n < 16; ++n) {
            const long long off = static_cast<long long>((tid >> 4) + 8 * n) * P.d_model + m;
            tb[n] = in ? Wb[off] : 0.f;
            if (n < 4) ta[n] = in ? Wa[off] : 0.f;
        }
    };
    fetch(0);
    for (int m0 = 0; m0 < P.d_model; m0 += OUTER_K) {
        __syncthreads();
#pragma unroll
        for (int n = 0; n < 16; ++n) {
            b_s[tid & 15][(tid >> 4) + 8 * n] = tb[n];
            if (n < 4) a_s[tid & 15][(tid >> 4) + 8 * n] = ta[n];
        }
        __syncthreads();
        fetch(m0 + OUTER_K);
        outer_group(a_s, b_s, acc);
    }
    float* out = P.gamma + (static_cast<long long>(h * P.G + g) * P.G + gp) * D * D;
    float* outT = P.gamma + (static_cast<long long>(h * P.G + gp) * P.G + g) * D * D;
    const int i0 = r0 + 4 * (tid >> 4);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = outer_column(tid, e);
            const float v = static_cast<float>(acc[r][e]);
            out[(i0 + r) * D + j] = v;
            if (g != gp) outT[j * D + i0 + r] = v;
        }
}

// Causal softmax statistics and o = sum_s p_s v_s of 64 positions of one query head, over tiles of 64 keys: a warp per 16 positions,
// logits as exact bf16 products, probabilities as three bf16 terms against V; the next key and value tiles arrive during the products.
// grid (position tiles, n_q), the longest first, 128 threads, two CTAs per SM.  Bound by the tensor pipe (256 MMAs of 16 x 8 x 16 per
// warp and tile, 35 us of it for 1024 tokens of 32 heads) and the exponentials between them.  (Register-blocked fp32 products out
// of shared memory took 366 us there, this 96.)
constexpr int RT = 64;
constexpr int ROWS_SMEM = 5 * RT * 256;                 // queries, two stages of keys and values
__global__ void __launch_bounds__(128, 2) rows_kernel(HessParams P) {
    extern __shared__ __align__(128) unsigned char hs_smem[];
    const int t0 = (gridDim.x - 1 - blockIdx.x) * RT, j = blockIdx.y, h = j / P.G, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned sq = hs_smem_addr(hs_smem), skv = sq + RT * 256;
    const int s_end = min(t0 + RT, P.S);
    hs_request<RT, 128>(sq, P.Q, t0, P.S, P.n_q, j);
    hs_request<RT, 128>(skv, P.K, 0, P.S, P.n_kv, h);
    hs_request<RT, 128>(skv + RT * 256, P.V, 0, P.S, P.n_kv, h);
    hs_requested();
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, o[16][4];
#pragma unroll
    for (int n = 0; n < 16; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    unsigned q[8][4];
    const int t_row = t0 + 16 * warp + (lane >> 2);     // this thread's positions: t_row, t_row + 8
    for (int s0 = 0, st = 0; s0 < s_end; s0 += RT, st ^= 1) {
        const unsigned sk = skv + 2 * RT * 256 * st, sv = sk + RT * 256;
        hs_landed<0>();
        __syncthreads();
        if (s0 + RT < s_end) {
            hs_request<RT, 128>(skv + 2 * RT * 256 * (st ^ 1), P.K, s0 + RT, P.S, P.n_kv, h);
            hs_request<RT, 128>(skv + 2 * RT * 256 * (st ^ 1) + RT * 256, P.V, s0 + RT, P.S, P.n_kv, h);
            hs_requested();
        }
        if (s0 == 0) {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) hs_ldsm(sq + hs_piece(16 * warp + (lane & 15), 2 * ks + (lane >> 4)), q[ks]);
        }
        float z[8][4];
#pragma unroll
        for (int n = 0; n < 8; ++n) z[n][0] = z[n][1] = z[n][2] = z[n][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
#pragma unroll
            for (int n = 0; n < 8; n += 2) {
                unsigned b[4];
                hs_ldsm(sk + hs_piece(8 * n + (lane & 7) + ((lane >> 4) << 3), 2 * ks + ((lane >> 3) & 1)), b);
                hs_mma_add(z[n], q[ks], b[0], b[1]);
                hs_mma_add(z[n + 1], q[ks], b[2], b[3]);
            }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float mx = -INFINITY;
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int e = 2 * r; e < 2 * r + 2; ++e) {
                    if (s0 + 8 * n + 2 * (lane & 3) + (e & 1) > t_row + 8 * r) z[n][e] = -INFINITY;
                    mx = fmaxf(mx, z[n][e]);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float mn = fmaxf(m[r], mx * P.scale2), sc = hs_ex2(m[r] - mn);      // every position sees a key of the first tile: mn is finite
            float sum = 0.f;
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int e = 2 * r; e < 2 * r + 2; ++e) { z[n][e] = hs_ex2(fmaf(z[n][e], P.scale2, -mn)); sum += z[n][e]; }
            l[r] = l[r] * sc + sum;                                             // of this thread's keys
            m[r] = mn;
#pragma unroll
            for (int n = 0; n < 16; ++n) { o[n][2 * r] *= sc; o[n][2 * r + 1] *= sc; }
        }
        unsigned p0[4][4], p1[4][4], p2[4][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                hs_split(z[2 * ks + (i >> 1)][2 * (i & 1)], z[2 * ks + (i >> 1)][2 * (i & 1) + 1], p0[ks][i], p1[ks][i], p2[ks][i]);
#pragma unroll
        for (int n = 0; n < 16; n += 2) {
            float small[2][4] = {};
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                unsigned b[4];
                hs_ldsm_t(sv + hs_piece(16 * ks + (lane & 15), n + (lane >> 4)), b);
                hs_mma(small[0], p2[ks], b[0], b[1]); hs_mma(small[1], p2[ks], b[2], b[3]);
                hs_mma(small[0], p1[ks], b[0], b[1]); hs_mma(small[1], p1[ks], b[2], b[3]);
                hs_mma_add(o[n], p0[ks], b[0], b[1]); hs_mma_add(o[n + 1], p0[ks], b[2], b[3]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) { o[n][e] += small[0][e]; o[n + 1][e] += small[1][e]; }
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
        const int t = t_row + 8 * r;
        if (t >= P.S) continue;
        const float linv = 1.f / l[r];
        if ((lane & 3) == 0) { P.row_m[static_cast<long long>(t) * P.n_q + j] = m[r]; P.row_linv[static_cast<long long>(t) * P.n_q + j] = linv; }
        float* dst = P.Oh + (static_cast<long long>(t) * P.n_q + j) * D + 2 * (lane & 3);
#pragma unroll
        for (int n = 0; n < 16; ++n) *reinterpret_cast<float2*>(dst + 8 * n) = make_float2(o[n][2 * r] * linv, o[n][2 * r + 1] * linv);
    }
}

// U, kappa and alpha of 128 positions and one pair: y = Gamma x, a warp per 16 positions, Gamma as three bf16 terms in shared memory and x
// as three terms in registers; of the nine products the three below 2^-26 of the result are left out.  alpha uses the first Gamma
// that is staged (v . Gamma_{gg'} v = v . Gamma_{g'g} v); for g = g' both halves of U are the same product.  grid (position tiles, pairs,
// n_kv), 256 threads.  Bound by the tensor pipe.  1024 tokens of 32 / 8 heads: 215 us as register-blocked fp32 products, now 136.
constexpr int PROJECT_T = 128, PROJECT_SMEM = 3 * D * 256;
__global__ void __launch_bounds__(256, 1) project_kernel(HessParams P) {
    extern __shared__ __align__(128) unsigned char hs_smem[];
    const unsigned base = hs_smem_addr(hs_smem);
    int g, gp;
    pair_heads(blockIdx.y, P.G, g, gp);
    const int h = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t_row = blockIdx.x * PROJECT_T + 16 * warp + (lane >> 2);      // this thread's positions: t_row, t_row + 8
    const bool active = blockIdx.x * PROJECT_T + 16 * warp < P.S;
    const long long t_in[2] = {min(t_row, P.S - 1), min(t_row + 8, P.S - 1)};
    float y[16][4];
    unsigned x[3][8][4];
    auto clear = [&] {
#pragma unroll
        for (int n = 0; n < 16; ++n) y[n][0] = y[n][1] = y[n][2] = y[n][3] = 0.f;
    };
    auto stage_gamma = [&](int ga, int gb) {
        const float* src = P.gamma + (static_cast<long long>(h * P.G + ga) * P.G + gb) * D * D;
#pragma unroll 4
        for (int item = tid; item < D * 16; item += 256) {
            const float4 u = reinterpret_cast<const float4*>(src)[2 * item], v = reinterpret_cast<const float4*>(src)[2 * item + 1];
            uint4 w[3];
            hs_split(u.x, u.y, w[0].x, w[1].x, w[2].x);
            hs_split(u.z, u.w, w[0].y, w[1].y, w[2].y);
            hs_split(v.x, v.y, w[0].z, w[1].z, w[2].z);
            hs_split(v.z, v.w, w[0].w, w[1].w, w[2].w);
#pragma unroll
            for (int i = 0; i < 3; ++i) *reinterpret_cast<uint4*>(hs_smem + i * D * 256 + hs_piece(item >> 4, item & 15)) = w[i];
        }
    };
    auto output_of = [&](int gx, int r, int col) -> float2 {                 // two channels of a head's output at position t_row + 8 r
        return *reinterpret_cast<const float2*>(P.Oh + (t_in[r] * P.n_q + h * P.G + gx) * D + col + 2 * (lane & 3));
    };
    auto load_o = [&](int gx) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 v = output_of(gx, i & 1, 16 * ks + 8 * (i >> 1));
                hs_split(v.x, v.y, x[0][ks][i], x[1][ks][i], x[2][ks][i]);
            }
    };
    auto product = [&](auto terms_tag) {                                     // y += Gamma x with x in one or three terms
        constexpr int TERMS = decltype(terms_tag)::value;
#pragma unroll
        for (int n = 0; n < 16; n += 4) {
            float small[4][4] = {};
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                unsigned b[3][2][4];
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        hs_ldsm(base + i * D * 256 + hs_piece(8 * n + 16 * q + (lane & 7) + ((lane >> 4) << 3), 2 * ks + ((lane >> 3) & 1)), b[i][q]);
#pragma unroll
                for (int sum = 2; sum >= 0; --sum)                           // the small products first
#pragma unroll
                    for (int i = 0; i <= sum; ++i) {
                        if (sum - i >= TERMS) continue;
#pragma unroll
                        for (int q = 0; q < 2; ++q)
#pragma unroll
                            for (int w = 0; w < 2; ++w) {
                                if (sum > 0) hs_mma(small[2 * q + w], x[sum - i][ks], b[i][q][2 * w], b[i][q][2 * w + 1]);
                                else hs_mma_add(y[n + 2 * q + w], x[0][ks], b[0][q][2 * w], b[0][q][2 * w + 1]);
                            }
                    }
            }
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
                for (int e = 0; e < 4; ++e) y[n + w][e] += small[w][e];
        }
    };
    auto row_sums = [&](const float (&d)[2], float* out) {                   // over the four lanes of a row
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float v = d[r];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if ((lane & 3) == 0 && t_row + 8 * r < P.S) out[(t_in[r] * P.n_kv + h) * P.n_pairs + blockIdx.y] = v;
        }
    };
    stage_gamma(g, gp);
    __syncthreads();
    if (active) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x[0][ks][i] = *reinterpret_cast<const unsigned*>(P.V + (t_in[i & 1] * P.n_kv + h) * D + 16 * ks + 8 * (i >> 1) + 2 * (lane & 3));
        clear();
        product(std::integral_constant<int, 1>{});
        float d[2] = {0.f, 0.f};
#pragma unroll
        for (int n = 0; n < 16; ++n)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const unsigned v = x[0][n >> 1][2 * (n & 1) + r];
                d[r] = fmaf(__uint_as_float(v << 16), y[n][2 * r], d[r]);
                d[r] = fmaf(__uint_as_float(v & 0xffff0000u), y[n][2 * r + 1], d[r]);
            }
        row_sums(d, P.alpha);
        load_o(gp);
        clear();
        product(std::integral_constant<int, 3>{});
        d[0] = d[1] = 0.f;
#pragma unroll
        for (int n = 0; n < 16; ++n)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float2 v = output_of(g, r, 8 * n);
                d[r] = fmaf(v.x, y[n][2 * r], d[r]);
                d[r] = fmaf(v.y, y[n][2 * r + 1], d[r]);
            }
        row_sums(d, P.kappa);
    }
    if (g != gp) {
        __syncthreads();
        stage_gamma(gp, g);
        __syncthreads();
        if (active) {
            load_o(g);
            product(std::integral_constant<int, 3>{});
        }
    } else {
#pragma unroll
        for (int n = 0; n < 16; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) y[n][e] += y[n][e];
    }
    if (!active) return;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (t_row + 8 * r >= P.S) continue;
        float* dst = P.U + ((t_in[r] * P.n_kv + h) * P.n_pairs + blockIdx.y) * D + 2 * (lane & 3);
#pragma unroll
        for (int n = 0; n < 16; ++n) *reinterpret_cast<float2*>(dst + 8 * n) = make_float2(y[n][2 * r], y[n][2 * r + 1]);
    }
}

// A and W0 of T positions and up to NC pairs of query heads, over tiles of 128 keys: a warp takes 16 positions x NT tiles of 8 keys and
// holds the probabilities of all heads, then v . U of one pair after the other, in the same places of its accumulators, so that
// nothing but the sums over the keys crosses threads.  U is split into three bf16 terms while it is staged; a tile's values are held as operands
// in registers, so the next tile arrives while the pairs are multiplied.  grid (position tiles, pair chunks, n_kv), 256 threads.
// Up to 4 heads two position tiles of 16 and chunks of up to 5 pairs, beyond that one and up to 10: what fits in shared memory beside
// the heads' queries.  1024 tokens of 32 / 8 heads: 626 us as register-blocked fp32 products (fp32 and shared-memory pipes half
// busy each), now 243.
constexpr int KT = 128;                                 // keys per tile
constexpr int pairs_m_tiles(int G) { return G <= 4 ? 2 : 1; }
constexpr int pair_chunks(int G) { return (G * (G + 1) / 2 + (G <= 4 ? 4 : 9)) / (G <= 4 ? 5 : 10); }
constexpr int pairs_per_chunk(int G) { return (G * (G + 1) / 2 + pair_chunks(G) - 1) / pair_chunks(G); }
template <int G>
struct PairsShape {
    static constexpr int MT = pairs_m_tiles(G), T = 16 * MT, NC = pairs_per_chunk(G), KW = 8 / MT, NT = KT / KW / 8, CHUNKS = pair_chunks(G);
    static constexpr int OFF_U = G * T * 256, OFF_K = OFF_U + 3 * NC * T * 256, OFF_V = OFF_K + KT * 256, OFF_AL = OFF_V + KT * 256,
                         OFF_STAT = OFF_AL + NC * KT * 4, OFF_KAPPA = OFF_STAT + G * T * 8, SMEM = OFF_KAPPA + NC * T * 4;
    static_assert(SMEM <= 232448 && KW * T * NC * 2 * 4 <= KT * 256, "shared memory; the warps' sums over the keys' place");
};
template <int G>
__global__ void __launch_bounds__(256, 1) pairs_kernel(HessParams P) {
    using Sh = PairsShape<G>;
    constexpr int MT = Sh::MT, T = Sh::T, NC = Sh::NC, KW = Sh::KW, NT = Sh::NT;
    extern __shared__ __align__(128) unsigned char hs_smem[];
    const unsigned base = hs_smem_addr(hs_smem);
    float* al = reinterpret_cast<float*>(hs_smem + Sh::OFF_AL);
    const int t0 = (gridDim.x - 1 - blockIdx.x) * T, pair0 = blockIdx.y * NC, h = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wm = MT == 2 ? warp >> 2 : 0, wk = MT == 2 ? warp & 3 : warp, n_pairs = min(NC, P.n_pairs - pair0), s_end = min(t0 + T, P.S);
    auto request = [&](int s0) {
        hs_request<KT, 256>(base + Sh::OFF_K, P.K, s0, P.S, P.n_kv, h);
        hs_request<KT, 256>(base + Sh::OFF_V, P.V, s0, P.S, P.n_kv, h);
        hs_requested();
    };
#pragma unroll
    for (int g = 0; g < G; ++g) hs_request<T, 256>(base + g * T * 256, P.Q, t0, P.S, P.n_q, h * G + g);
    request(0);
#pragma unroll 2
    for (int item = tid; item < NC * T * 16; item += 256) {
        const int k = item / (T * 16), row = (item >> 4) % T, piece = item & 15;
        uint4 w[3] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
        if (t0 + row < P.S && k < n_pairs) {
            const float4* src = reinterpret_cast<const float4*>(P.U + ((static_cast<long long>(t0 + row) * P.n_kv + h) * P.n_pairs + pair0 + k) * D + 8 * piece);
            const float4 x = src[0], y = src[1];
            hs_split(x.x, x.y, w[0].x, w[1].x, w[2].x);
            hs_split(x.z, x.w, w[0].y, w[1].y, w[2].y);
            hs_split(y.x, y.y, w[0].z, w[1].z, w[2].z);
            hs_split(y.z, y.w, w[0].w, w[1].w, w[2].w);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) *reinterpret_cast<uint4*>(hs_smem + Sh::OFF_U + (k * 3 + i) * T * 256 + hs_piece(row, piece)) = w[i];
    }
    const int t_row = t0 + 16 * wm + (lane >> 2);        // this thread's positions: t_row, t_row + 8
    const int row0 = 16 * wm + (lane >> 2);
    // (maximum, 1 / sum) of each head and kappa of each pair for the tile's positions, read again where they are used
    float2* stat = reinterpret_cast<float2*>(hs_smem + Sh::OFF_STAT);
    float* kap = reinterpret_cast<float*>(hs_smem + Sh::OFF_KAPPA);
    for (int item = tid; item < (G + NC) * T; item += 256) {
        const int k = item / T, row = item % T;
        const long long t = min(t0 + row, P.S - 1);
        if (k < G) stat[item] = make_float2(P.row_m[t * P.n_q + h * G + k], P.row_linv[t * P.n_q + h * G + k]);
        else kap[item - G * T] = k - G < n_pairs ? P.kappa[(t * P.n_kv + h) * P.n_pairs + pair0 + k - G] : 0.f;
    }
    float asum[NC][2], wsum[NC][2];
#pragma unroll
    for (int k = 0; k < NC; ++k) asum[k][0] = asum[k][1] = wsum[k][0] = wsum[k][1] = 0.f;
    const unsigned a_row = hs_piece(16 * wm + (lane & 15), 0), a_xor = lane & 7, a_half = lane >> 4;       // piece p of the row: (p ^ a_xor) << 4 beyond its start
    const unsigned a_base = a_row - (a_xor << 4);
    for (int s0 = 0; s0 < s_end; s0 += KT) {
        const int key0 = 8 * NT * wk;                    // this warp's keys of the tile
        const bool active = s0 + key0 <= t0 + 16 * wm + 15;
        hs_landed<0>();
        for (int item = tid; item < NC * KT; item += 256) {
            const int k = item / KT, row = item % KT;
            al[item] = s0 + row < P.S && k < n_pairs ? P.alpha[(static_cast<long long>(s0 + row) * P.n_kv + h) * P.n_pairs + pair0 + k] : 0.f;
        }
        __syncthreads();
        float p[G][NT][4];
        unsigned v[8][NT][2];
        if (active) {
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int n = 0; n < NT; ++n) p[g][n][0] = p[g][n][1] = p[g][n][2] = p[g][n][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                unsigned b[NT][2];
#pragma unroll
                for (int n = 0; n < NT; n += 2) {
                    unsigned w[4];
                    hs_ldsm(base + Sh::OFF_K + hs_piece(key0 + 8 * n + (lane & 7) + ((lane >> 4) << 3), 2 * ks + ((lane >> 3) & 1)), w);
                    b[n][0] = w[0]; b[n][1] = w[1]; b[n + 1][0] = w[2]; b[n + 1][1] = w[3];
                    hs_ldsm(base + Sh::OFF_V + hs_piece(key0 + 8 * n + (lane & 7) + ((lane >> 4) << 3), 2 * ks + ((lane >> 3) & 1)), w);
                    v[ks][n][0] = w[0]; v[ks][n][1] = w[1]; v[ks][n + 1][0] = w[2]; v[ks][n + 1][1] = w[3];
                }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    unsigned a[4];
                    hs_ldsm(base + g * T * 256 + a_base + (((2 * ks + a_half) ^ a_xor) << 4), a);
#pragma unroll
                    for (int n = 0; n < NT; ++n) hs_mma_add(p[g][n], a, b[n][0], b[n][1]);
                }
            }
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float2 st = stat[g * T + row0 + 8 * r];
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int e = 2 * r; e < 2 * r + 2; ++e)
                            p[g][n][e] = s0 + key0 + 8 * n + 2 * (lane & 3) + (e & 1) <= t_row + 8 * r ? hs_ex2(fmaf(p[g][n][e], P.scale2, -st.x)) * st.y : 0.f;
                }
        }
        __syncthreads();
        if (s0 + KT < s_end) request(s0 + KT);
        if (active) {
            auto pair = [&](const int k, const float (&pa)[NT][4], const float (&pb)[NT][4]) {
                float rr[NT][4], small[NT][4];
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) rr[n][e] = small[n][e] = 0.f;
                const unsigned u0 = base + Sh::OFF_U + k * 3 * T * 256 + a_base;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const unsigned off = u0 + (((2 * ks + a_half) ^ a_xor) << 4);
                    unsigned a[3][4];
#pragma unroll
                    for (int i = 0; i < 3; ++i) hs_ldsm(off + i * T * 256, a[i]);
#pragma unroll
                    for (int i = 2; i >= 1; --i)
#pragma unroll
                        for (int n = 0; n < NT; ++n) hs_mma(small[n], a[i], v[ks][n][0], v[ks][n][1]);
#pragma unroll
                    for (int n = 0; n < NT; ++n) hs_mma_add(rr[n], a[0], v[ks][n][0], v[ks][n][1]);
                }
                const float kp[2] = {kap[k * T + row0], kap[k * T + row0 + 8]};
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const float2 av = *reinterpret_cast<const float2*>(al + k * KT + key0 + 8 * n + 2 * (lane & 3));
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float w = pa[n][e] * pb[n][e];
                        wsum[k][e >> 1] += w;
                        asum[k][e >> 1] = fmaf(w, ((e & 1 ? av.y : av.x) - (rr[n][e] + small[n][e])) + kp[e >> 1], asum[k][e >> 1]);
                    }
                }
            };
            // the chunk's pairs in order, each expanded with its heads known
            auto chunk = [&](auto tag) {
                constexpr int FIRST = decltype(tag)::value * NC;
                int index = 0;
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int gp = g; gp < G; ++gp, ++index)
                        if (index >= FIRST && index < FIRST + NC) pair(index - FIRST, p[g], p[gp]);
            };
            switch (blockIdx.y) {
                case 0: chunk(std::integral_constant<int, 0>{}); break;
                case 1: if constexpr (Sh::CHUNKS > 1) chunk(std::integral_constant<int, 1>{}); break;
                case 2: if constexpr (Sh::CHUNKS > 2) chunk(std::integral_constant<int, 2>{}); break;
                default: if constexpr (Sh::CHUNKS > 3) chunk(std::integral_constant<int, 3>{}); break;
            }
        }
        __syncthreads();                                 // alpha is read
    }
    // sums over the four lanes of a row, then over the warps' keys in order
    float* red = reinterpret_cast<float*>(hs_smem + Sh::OFF_K);       // [key warp][position][pair][A, W0]
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
            for (int off = 1; off <= 2; off <<= 1) {
                asum[k][r] += __shfl_xor_sync(0xffffffffu, asum[k][r], off);
                wsum[k][r] += __shfl_xor_sync(0xffffffffu, wsum[k][r], off);
            }
            if ((lane & 3) == 0) *reinterpret_cast<float2*>(red + ((wk * T + 16 * wm + (lane >> 2) + 8 * r) * NC + k) * 2) = make_float2(asum[k][r], wsum[k][r]);
        }
    __syncthreads();
    for (int item = tid; item < T * NC; item += 256) {
        const int row = item / NC, k = item % NC;
        if (t0 + row >= P.S || k >= n_pairs) continue;
        float a = 0.f, w = 0.f;
#pragma unroll
        for (int i = 0; i < KW; ++i) { const float2 x = *reinterpret_cast<const float2*>(red + (i * T * NC + item) * 2); a += x.x; w += x.y; }
        const long long o = (static_cast<long long>(t0 + row) * P.n_kv + h) * P.n_pairs + pair0 + k;
        P.A[o] = a;
        P.W0[o] = w;
    }
}

// One entry on or above the diagonal, and its mirror image.
__device__ __forceinline__ void add_key_entry(const HessParams& P, int h, int i, int j, double sum) {
    if (i > j) return;                                   // the other half of a block on the diagonal
    const double v = 2.0 * static_cast<double>(P.inv_tau) * static_cast<double>(P.inv_tau) * sum;
    double* H = P.H_K + static_cast<long long>(h) * D * D;
    H[i * D + j] += v;
    if (i != j) H[j * D + i] += v;
}

// H_K[h][i][j] += (2 / tau^2) sum_t sum_g q_{g,t}[i] (sum_g' A_{gg'}(t) q_{g',t}[j]): the 36 blocks of 16 x 16 entries on and above
// the diagonal, one per warp; the entries below are their mirror images (the sum is symmetric).  grid (slices of positions, n_kv, 3),
// 384 threads; lane (r, c) = (lane >> 2, lane & 3) holds rows 2 r .. and columns 4 c .. of its warp's block.  With one slice the
// sums go to H_K, else they are left in the workspace (over U and the head outputs, which nothing reads any more) and
// finish_kernel adds them up in the order of the slices: the same bits on every run.
// Three CTAs per slice keep short sequences from being one CTA's chain; what bounds it is shared-memory reads and fp32 issue alike
// (two wavefronts for eight multiply-adds per warp) and the conversions to float64: 57 us for 1024 tokens of 32 / 8 heads.  (With all 64 blocks, 512
// threads, loads waited for and float64 atomics the whole call, then 1344 us, took 8 us more, and 310 instead of 267 us for 300 tokens of 16 / 4.)
constexpr int KEY_SLICE = 64, KEY_BLOCKS = 36, KEY_WARPS = 12;
__device__ __forceinline__ void key_block(int k, int& bi, int& bj) { pair_heads(k, 8, bi, bj); }
template <int G>
__global__ void __launch_bounds__(32 * KEY_WARPS) key_kernel(HessParams P) {
    __shared__ __align__(16) float a_s[OUTER_K][HS_PITCH], b_s[OUTER_K][HS_PITCH];
    __shared__ float c_s[OUTER_K / G][G][G];
    constexpr int TG = OUTER_K / G;                      // positions per staged group (G = 1 .. 8: at least 2)
    const int h = blockIdx.y, tid = threadIdx.x, t_end = min(static_cast<int>(blockIdx.x + 1) * P.slice_len, P.S);
    const int block = blockIdx.z * KEY_WARPS + (tid >> 5), lane = tid & 31;
    int bi, bj;
    key_block(block, bi, bj);
    const int i0 = 16 * bi + 2 * (lane >> 2), j0 = 16 * bj + 4 * (lane & 3);
    double acc[2][4] = {};
    // the next group's queries and coefficients are requested while this one is multiplied
    constexpr int N_Q = (OUTER_K * 32 + 32 * KEY_WARPS - 1) / (32 * KEY_WARPS);
    static_assert(TG * G * G <= 32 * KEY_WARPS, "a coefficient per thread");
    uint2 q_next[N_Q];
    float c_next = 0.f;
    auto request = [&](int t0) {
#pragma unroll
        for (int n = 0; n < N_Q; ++n) {
            const int item = tid + n * 32 * KEY_WARPS, row = item >> 5, t = t0 + row / G;
            q_next[n] = row < TG * G && t < t_end
                            ? *reinterpret_cast<const uint2*>(P.Q + (static_cast<long long>(t) * P.n_q + h * G + row % G) * D + 4 * (item & 31)) : make_uint2(0u, 0u);
        }
        const int t = t0 + tid / (G * G), g = tid / G % G, gp = tid % G, lo = min(g, gp), hi = max(g, gp);
        c_next = tid < TG * G * G && t < t_end ? P.A[(static_cast<long long>(t) * P.n_kv + h) * P.n_pairs + lo * G - lo * (lo - 1) / 2 + hi - lo] : 0.f;
    };
    request(blockIdx.x * P.slice_len);
    for (int t0 = blockIdx.x * P.slice_len; t0 < t_end; t0 += TG) {
        __syncthreads();
        if (tid < TG * G * G) c_s[tid / (G * G)][tid / G % G][tid % G] = c_next;
#pragma unroll
        for (int n = 0; n < N_Q; ++n) {
            const int item = tid + n * 32 * KEY_WARPS;
            const uint2 w = q_next[n];
            if (item < OUTER_K * 32)
                *reinterpret_cast<float4*>(&a_s[item >> 5][4 * (item & 31)]) =
                    make_float4(bf16_bits_to_float(w.x & 0xffff), bf16_bits_to_float(w.x >> 16), bf16_bits_to_float(w.y & 0xffff), bf16_bits_to_float(w.y >> 16));
        }
        __syncthreads();
        request(t0 + TG);
        for (int item = tid; item < OUTER_K * D; item += 32 * KEY_WARPS) {
            const int row = item >> 7, ch = item & 127, tl = row / G, g = row % G;
            float x = 0.f;
            if (row < TG * G)
#pragma unroll
                for (int gp = 0; gp < G; ++gp) x = fmaf(c_s[tl][g][gp], a_s[tl * G + gp][ch], x);
            b_s[row][ch] = x;
        }
        __syncthreads();
#pragma unroll
        for (int tl = 0; tl < TG; ++tl) {                // a position's sum over the heads in fp32, beyond that float64
            float part[2][4] = {};
#pragma unroll
            for (int k = tl * G; k < tl * G + G; ++k) {
                const float2 av = *reinterpret_cast<const float2*>(&a_s[k][i0]);
                const float4 bv = *reinterpret_cast<const float4*>(&b_s[k][j0]);
                part[0][0] = fmaf(av.x, bv.x, part[0][0]); part[0][1] = fmaf(av.x, bv.y, part[0][1]);
                part[0][2] = fmaf(av.x, bv.z, part[0][2]); part[0][3] = fmaf(av.x, bv.w, part[0][3]);
                part[1][0] = fmaf(av.y, bv.x, part[1][0]); part[1][1] = fmaf(av.y, bv.y, part[1][1]);
                part[1][2] = fmaf(av.y, bv.z, part[1][2]); part[1][3] = fmaf(av.y, bv.w, part[1][3]);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[r][e] += static_cast<double>(part[r][e]);
        }
    }
    if (P.n_slices > 1) {
        double* dst = P.key_part + ((static_cast<long long>(blockIdx.x) * P.n_kv + h) * KEY_BLOCKS + block) * 256 + 32 * (lane >> 2) + 4 * (lane & 3);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            reinterpret_cast<double2*>(dst + 16 * r)[0] = make_double2(acc[r][0], acc[r][1]);
            reinterpret_cast<double2*>(dst + 16 * r)[1] = make_double2(acc[r][2], acc[r][3]);
        }
        return;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) add_key_entry(P, h, i0 + r, j0 + e, acc[r][e]);
}

// H_V[h] += 2 sum_{g<=g'} c_{gg'} sym(Gamma_{gg'}), c = sum_t W0(t), and the sums of key_kernel's slices: grid (16 row groups of H_V
// and, with several slices, the 36 blocks of H_K; n_kv), 256 threads.
__global__ void __launch_bounds__(256) finish_kernel(HessParams P) {
    __shared__ double c_s[36];
    const int h = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    if (blockIdx.x >= 16) {
        const int block = blockIdx.x - 16;
        int bi, bj;
        key_block(block, bi, bj);
        const double* src = P.key_part + (static_cast<long long>(h) * KEY_BLOCKS + block) * 256 + tid;
        double sum = 0.0;
#pragma unroll 8
        for (int k = 0; k < P.n_slices; ++k) sum += src[static_cast<long long>(k) * P.n_kv * KEY_BLOCKS * 256];
        add_key_entry(P, h, 16 * bi + (tid >> 4), 16 * bj + (tid & 15), sum);
        return;
    }
    for (int k = tid >> 5; k < P.n_pairs; k += 8) {
        double sum = 0.0;
#pragma unroll 8
        for (int t = lane; t < P.S; t += 32) sum += static_cast<double>(P.W0[(static_cast<long long>(t) * P.n_kv + h) * P.n_pairs + k]);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) c_s[k] = sum;
    }
    __syncthreads();
    double hv[D * D / 16 / 256] = {};                    // the thread's entries side by side: their loads are in flight together
    const int ij = blockIdx.x * (D * D / 16) + tid;
    int k = 0;
    for (int g = 0; g < P.G; ++g)
        for (int gp = g; gp < P.G; ++gp, ++k) {
            const float* up = P.gamma + (static_cast<long long>(h * P.G + g) * P.G + gp) * D * D + ij;
            const float* down = P.gamma + (static_cast<long long>(h * P.G + gp) * P.G + g) * D * D + ij;
#pragma unroll
            for (int e = 0; e < D * D / 16 / 256; ++e) {
                const double a = up[256 * e];
                hv[e] += c_s[k] * (g == gp ? a : a + static_cast<double>(down[256 * e]));
            }
        }
#pragma unroll
    for (int e = 0; e < D * D / 16 / 256; ++e) P.H_V[static_cast<long long>(h) * D * D + ij + 256 * e] += 2.0 * hv[e];
}

template <int G>
bool launch_pairs(const HessParams& P, cudaStream_t st) {
    using Sh = PairsShape<G>;
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(pairs_kernel<G>), Sh::SMEM)) return false;
    pairs_kernel<G><<<dim3((P.S + Sh::T - 1) / Sh::T, pair_chunks(G), P.n_kv), 256, Sh::SMEM, st>>>(P);
    key_kernel<G><<<dim3(P.n_slices, P.n_kv, KEY_BLOCKS / KEY_WARPS), 32 * KEY_WARPS, 0, st>>>(P);
    return true;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

struct HessLayout { size_t gamma, row_m, row_linv, Oh, U, alpha, A, W0, total; };
HessLayout hess_layout(int n_kv, int n_q, long long S) {
    const int G = n_q / n_kv, NP = G * (G + 1) / 2;
    HessLayout L;
    size_t off = 0;
    L.gamma = off;    off = align256(off + static_cast<size_t>(n_kv) * G * G * D * D * sizeof(float));
    L.row_m = off;    off = align256(off + static_cast<size_t>(S) * n_q * sizeof(float));
    L.row_linv = off; off = align256(off + static_cast<size_t>(S) * n_q * sizeof(float));
    L.Oh = off;       off = align256(off + static_cast<size_t>(S) * n_q * D * sizeof(float));
    L.U = off;        off = align256(off + static_cast<size_t>(S) * n_kv * NP * D * sizeof(float));
    L.alpha = off;    off = align256(off + static_cast<size_t>(S) * n_kv * NP * sizeof(float));
    L.A = off;        off = align256(off + static_cast<size_t>(S) * n_kv * NP * sizeof(float));
    L.W0 = off;       off = align256(off + static_cast<size_t>(S) * n_kv * NP * sizeof(float));
    L.total = off;
    return L;
}

}  // namespace
}  // namespace wushkv

using namespace wushkv;

extern "C" size_t wushkv_attention_hessians_workspace_bytes(int32_t n_kv, int32_t n_q, int32_t d, int64_t n_tokens) {
    if (d != D || n_kv <= 0 || n_q <= 0 || n_q % n_kv != 0 || n_q / n_kv > 8 || n_tokens <= 0) return 0;
    return hess_layout(n_kv, n_q, n_tokens).total;
}

extern "C" int wushkv_accumulate_attention_hessians_device(int32_t n_kv, int32_t n_q, int32_t d, int32_t d_model, int64_t n_tokens,
                                                           const uint16_t* K, const uint16_t* Q, const uint16_t* V, const float* W_O,
                                                           double tau, double* H_K, double* H_V,
                                                           void* workspace, size_t workspace_bytes, void* stream) {
    if (d != D || n_kv <= 0 || n_q <= 0 || n_q % n_kv != 0 || d_model <= 0 || n_tokens <= 0 || n_tokens > (1 << 24)) return WUSHKV_EINVAL;
    const int G = n_q / n_kv;
    if (G > 8) return WUSHKV_EINVAL;          // the library's group sizes: 1..8
    if (!K || !Q || !V || !W_O || !H_K || !H_V || !workspace || !(tau > 0.0)) return WUSHKV_EINVAL;
    if (!aligned(K, 16) || !aligned(Q, 16) || !aligned(V, 16) || !aligned(W_O, 16) || !aligned(workspace, 256)) return WUSHKV_EINVAL;
    const HessLayout L = hess_layout(n_kv, n_q, n_tokens);
    if (workspace_bytes < L.total) return WUSHKV_ECAPACITY;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    HessParams P;
    P.S = static_cast<int>(n_tokens); P.n_kv = n_kv; P.n_q = n_q; P.G = G; P.d_model = d_model; P.n_pairs = G * (G + 1) / 2;
    P.inv_tau = static_cast<float>(1.0 / tau);
    // (never 0: masked logits are -infinity when they meet it; at the smallest fp32 number any finite logit's exponential is 1)
    P.scale2 = std::max(static_cast<float>(1.4426950408889634 / tau), std::numeric_limits<float>::denorm_min());
    P.Q = Q; P.K = K; P.V = V; P.W_O = W_O;
    P.gamma = reinterpret_cast<float*>(ws + L.gamma);
    P.row_m = reinterpret_cast<float*>(ws + L.row_m); P.row_linv = reinterpret_cast<float*>(ws + L.row_linv);
    P.Oh = reinterpret_cast<float*>(ws + L.Oh); P.U = reinterpret_cast<float*>(ws + L.U);
    P.kappa = P.A = reinterpret_cast<float*>(ws + L.A);
    P.alpha = reinterpret_cast<float*>(ws + L.alpha); P.W0 = reinterpret_cast<float*>(ws + L.W0);
    P.H_K = H_K; P.H_V = H_V;
    // Slices of 64 positions or more: no more of them than give every SM two waves of CTAs, nor than fit over Oh and U.
    const long long room = static_cast<long long>(L.alpha - L.Oh) / (static_cast<long long>(n_kv) * KEY_BLOCKS * 256 * 8);
    const long long want = std::max<long long>(1, std::min<long long>({(n_tokens + KEY_SLICE - 1) / KEY_SLICE, room, 2LL * sm_count() / n_kv}));
    P.slice_len = static_cast<int>((n_tokens + want - 1) / want);
    P.n_slices = static_cast<int>((n_tokens + P.slice_len - 1) / P.slice_len);
    P.key_part = reinterpret_cast<double*>(ws + L.Oh);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(rows_kernel), ROWS_SMEM) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(project_kernel), PROJECT_SMEM))
        return WUSHKV_ECUDA;
    const unsigned tiles = (P.S + RT - 1) / RT;
    gamma_kernel<<<dim3(P.n_pairs, n_kv, D / 32), 128, 0, st>>>(P);
    rows_kernel<<<dim3(tiles, n_q), 128, ROWS_SMEM, st>>>(P);
    project_kernel<<<dim3((P.S + PROJECT_T - 1) / PROJECT_T, P.n_pairs, n_kv), 256, PROJECT_SMEM, st>>>(P);
    bool ok;
    switch (G) {
        case 1: ok = launch_pairs<1>(P, st); break;
        case 2: ok = launch_pairs<2>(P, st); break;
        case 3: ok = launch_pairs<3>(P, st); break;
        case 4: ok = launch_pairs<4>(P, st); break;
        case 5: ok = launch_pairs<5>(P, st); break;
        case 6: ok = launch_pairs<6>(P, st); break;
        case 7: ok = launch_pairs<7>(P, st); break;
        default: ok = launch_pairs<8>(P, st); break;
    }
    if (!ok) return WUSHKV_ECUDA;
    finish_kernel<<<dim3(16 + (P.n_slices > 1 ? KEY_BLOCKS : 0), n_kv), 256, 0, st>>>(P);
    return cudaGetLastError() == cudaSuccess ? WUSHKV_OK : WUSHKV_ECUDA;
}
