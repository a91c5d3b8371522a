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
// Every step is a contraction over 128 channels or over positions, done as register-blocked fp32 products out of shared
// memory (with a warp per row, a CTA per position and the sums over s as vectors of 128 channels per pair, 1024 tokens of 32 / 8
// heads took 6.0 ms, every value fetched being used for one or two multiplications; now 1.34 ms, pairs_kernel 0.59, rows_kernel 0.35.  In
// a capture of pairs_kernel two warps per scheduler keep the fp32 pipe busy 46 % of the cycles and the shared-memory pipe 52 %, and its
// last wave leaves SMs idle for a fifth of the time):
//   gamma_kernel      Gamma_{gg'}, 128 x 128 x d_model, float64 across groups of 16
//   rows_kernel       causal softmax statistics (max, 1 / sum) and head outputs o_{g,t}: 64 x 64 tiles
//   project_kernel    U, kappa and alpha: 64 x 128 tiles
//   pairs_kernel      logits and v_s . U for (position t; 4 keys s) per thread, all query heads and up to 10 pairs; A, W0
//   key_kernel        H_K: sum over (t, g) of q_{g,t} (sum_g' A_{gg'}(t) q_{g',t})^T, float64 across positions
//   finish_kernel     H_V = 2 sum_{gg'} (sum_t W0) Gamma_{gg'}; the slices of H_K added up in order
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "host_common.h"
#include "layout.cuh"

namespace wushkv {
namespace {

constexpr int HS_PITCH = D + 4;            // floats per staged row

struct HessParams {
    int S, n_kv, n_q, G, d_model, n_pairs;
    float inv_tau;
    const unsigned short* Q;     // [S][n_q][D] bf16
    const unsigned short* K;     // [S][n_kv][D]
    const unsigned short* V;     // [S][n_kv][D]
    const float* W_O;            // [n_q][D][d_model]
    float* gamma;                // [n_kv][G][G][D][D]
    float* row_m;                // [S][n_q] maximum of the logits (natural log domain)
    float* row_linv;             // [S][n_q] 1 / sum exp
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
__device__ __forceinline__ float4 bf16x4(const unsigned short* p) {
    const uint2 r = *reinterpret_cast<const uint2*>(p);
    return make_float4(bf16_bits_to_float(r.x & 0xffff), bf16_bits_to_float(r.x >> 16), bf16_bits_to_float(r.y & 0xffff), bf16_bits_to_float(r.y >> 16));
}
__device__ __forceinline__ void fma4(float& acc, const float4& a, const float4& b) { acc = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc)))); }

// C[i][j] += sum_k a[k][i] b[k][j] for one staged group of 16 k; thread: rows 4 (tid >> 4) .., columns (tid & 15) + 16 e.
constexpr int OUTER_K = 16;
__device__ __forceinline__ void outer_group(const float (*a)[HS_PITCH], const float (*b)[HS_PITCH], double (&acc)[4][8]) {
    const int i0 = 4 * (threadIdx.x >> 4), j0 = threadIdx.x & 15;
    float part[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int e = 0; e < 8; ++e) part[r][e] = 0.f;
#pragma unroll 4
    for (int k = 0; k < OUTER_K; ++k) {
        const float4 av = *reinterpret_cast<const float4*>(&a[k][i0]);
        float bv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) bv[e] = b[k][j0 + 16 * e];
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
__global__ void __launch_bounds__(128) gamma_kernel(HessParams P) {
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
    const int i0 = r0 + 4 * (tid >> 4), j0 = tid & 15;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float v = static_cast<float>(acc[r][e]);
            out[(i0 + r) * D + j0 + 16 * e] = v;
            if (g != gp) outT[(j0 + 16 * e) * D + i0 + r] = v;
        }
}

// Causal softmax statistics and o = sum_s p_s v_s of 64 positions of one query head, over tiles of 64 keys.  256 threads: thread
// (r, c) = (tid >> 4, tid & 15) holds the logits of positions 4 r .. and keys c + 16 e, then the outputs of the same positions
// and channels 4 c .., 64 + 4 c ...  grid (position tiles, n_q), the longest first.
constexpr int RT = 64;
struct RowsSmem { float q[RT][HS_PITCH], kv[RT][HS_PITCH], p[RT][RT + 4]; };
__global__ void __launch_bounds__(256, 2) rows_kernel(HessParams P) {
    extern __shared__ __align__(16) unsigned char hs_smem[];
    RowsSmem& sm = *reinterpret_cast<RowsSmem*>(hs_smem);
    const int t0 = (gridDim.x - 1 - blockIdx.x) * RT, j = blockIdx.y, h = j / P.G, tid = threadIdx.x, r = tid >> 4, c = tid & 15;
    for (int item = tid; item < RT * 32; item += 256) {
        const int row = item >> 5, piece = item & 31;
        *reinterpret_cast<float4*>(&sm.q[row][4 * piece]) =
            t0 + row < P.S ? bf16x4(P.Q + (static_cast<long long>(t0 + row) * P.n_q + j) * D + 4 * piece) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float m[4], l[4], o[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        m[a] = -INFINITY; l[a] = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) o[a][e] = 0.f;
    }
    for (int s0 = 0; s0 < min(t0 + RT, P.S); s0 += RT) {
        auto stage = [&](const unsigned short* X) {
            for (int item = tid; item < RT * 32; item += 256) {
                const int row = item >> 5, piece = item & 31;
                *reinterpret_cast<float4*>(&sm.kv[row][4 * piece]) =
                    s0 + row < P.S ? bf16x4(X + (static_cast<long long>(s0 + row) * P.n_kv + h) * D + 4 * piece) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        __syncthreads();
        stage(P.K);
        __syncthreads();
        float z[4][4] = {};
#pragma unroll 4
        for (int k = 0; k < D; k += 4) {
            float4 qa[4], kb[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) { qa[a] = *reinterpret_cast<const float4*>(&sm.q[4 * r + a][k]); kb[a] = *reinterpret_cast<const float4*>(&sm.kv[c + 16 * a][k]); }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int e = 0; e < 4; ++e) fma4(z[a][e], qa[a], kb[e]);
        }
        __syncthreads();
        stage(P.V);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int t = t0 + 4 * r + a;
            float mx = -INFINITY;
#pragma unroll
            for (int e = 0; e < 4; ++e) { z[a][e] = s0 + c + 16 * e <= t ? z[a][e] * P.inv_tau : -INFINITY; mx = fmaxf(mx, z[a][e]); }
#pragma unroll
            for (int off = 8; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float mn = fmaxf(m[a], mx), sc = __expf(m[a] - mn);        // every position sees a key of the first tile: mn is finite
            float sum = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) { const float p = __expf(z[a][e] - mn); sm.p[4 * r + a][c + 16 * e] = p; sum += p; }
            l[a] = l[a] * sc + sum;                                      // of this thread's keys
            m[a] = mn;
#pragma unroll
            for (int e = 0; e < 8; ++e) o[a][e] *= sc;
        }
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < RT; k += 4) {
            float4 pa[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) pa[a] = *reinterpret_cast<const float4*>(&sm.p[4 * r + a][k]);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float4 va = *reinterpret_cast<const float4*>(&sm.kv[k + kk][4 * c]), vb = *reinterpret_cast<const float4*>(&sm.kv[k + kk][64 + 4 * c]);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float p = kk == 0 ? pa[a].x : kk == 1 ? pa[a].y : kk == 2 ? pa[a].z : pa[a].w;
                    o[a][0] = fmaf(p, va.x, o[a][0]); o[a][1] = fmaf(p, va.y, o[a][1]); o[a][2] = fmaf(p, va.z, o[a][2]); o[a][3] = fmaf(p, va.w, o[a][3]);
                    o[a][4] = fmaf(p, vb.x, o[a][4]); o[a][5] = fmaf(p, vb.y, o[a][5]); o[a][6] = fmaf(p, vb.z, o[a][6]); o[a][7] = fmaf(p, vb.w, o[a][7]);
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) l[a] += __shfl_xor_sync(0xffffffffu, l[a], off);
        const int t = t0 + 4 * r + a;
        if (t >= P.S) continue;
        const float linv = 1.f / l[a];
        if (c == 0) { P.row_m[static_cast<long long>(t) * P.n_q + j] = m[a]; P.row_linv[static_cast<long long>(t) * P.n_q + j] = linv; }
        float* dst = P.Oh + (static_cast<long long>(t) * P.n_q + j) * D + 4 * c;
        *reinterpret_cast<float4*>(dst) = make_float4(o[a][0] * linv, o[a][1] * linv, o[a][2] * linv, o[a][3] * linv);
        *reinterpret_cast<float4*>(dst + 64) = make_float4(o[a][4] * linv, o[a][5] * linv, o[a][6] * linv, o[a][7] * linv);
    }
}

// U, kappa and alpha of 64 positions and one pair: y = Gamma x for 64 rows x, 256 threads; thread (r, c) holds positions 4 r .. and
// channels 4 c .., 64 + 4 c ...  grid (position tiles, pairs, n_kv).
struct ProjectSmem { float x[RT][HS_PITCH], gam[D][D]; };
__global__ void __launch_bounds__(256, 2) project_kernel(HessParams P) {
    extern __shared__ __align__(16) unsigned char hs_smem[];
    ProjectSmem& sm = *reinterpret_cast<ProjectSmem*>(hs_smem);
    int g, gp;
    pair_heads(blockIdx.y, P.G, g, gp);
    const int t0 = blockIdx.x * RT, h = blockIdx.z, tid = threadIdx.x, r = tid >> 4, c = tid & 15;
    float y[4][8];
    auto clear = [&] {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int e = 0; e < 8; ++e) y[a][e] = 0.f;
    };
    auto stage_gamma = [&](int ga, int gb) {             // Gamma_{ga gb} x = sum_j x_j Gamma_{gb ga}[j][.]: rows of the transpose
        const float4* src = reinterpret_cast<const float4*>(P.gamma + (static_cast<long long>(h * P.G + gb) * P.G + ga) * D * D);
        float4* dst = reinterpret_cast<float4*>(&sm.gam[0][0]);
#pragma unroll 4
        for (int k = tid; k < D * D / 4; k += 256) dst[k] = src[k];
    };
    auto stage_o = [&](int gx) {
#pragma unroll 4
        for (int item = tid; item < RT * 32; item += 256) {
            const int row = item >> 5, piece = item & 31;
            *reinterpret_cast<float4*>(&sm.x[row][4 * piece]) =
                t0 + row < P.S ? *reinterpret_cast<const float4*>(P.Oh + (static_cast<long long>(t0 + row) * P.n_q + h * P.G + gx) * D + 4 * piece) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto product = [&] {
#pragma unroll 2
        for (int k = 0; k < D; k += 4) {
            float4 xa[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) xa[a] = *reinterpret_cast<const float4*>(&sm.x[4 * r + a][k]);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float4 ga = *reinterpret_cast<const float4*>(&sm.gam[k + kk][4 * c]), gb = *reinterpret_cast<const float4*>(&sm.gam[k + kk][64 + 4 * c]);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float x = kk == 0 ? xa[a].x : kk == 1 ? xa[a].y : kk == 2 ? xa[a].z : xa[a].w;
                    y[a][0] = fmaf(x, ga.x, y[a][0]); y[a][1] = fmaf(x, ga.y, y[a][1]); y[a][2] = fmaf(x, ga.z, y[a][2]); y[a][3] = fmaf(x, ga.w, y[a][3]);
                    y[a][4] = fmaf(x, gb.x, y[a][4]); y[a][5] = fmaf(x, gb.y, y[a][5]); y[a][6] = fmaf(x, gb.z, y[a][6]); y[a][7] = fmaf(x, gb.w, y[a][7]);
                }
            }
        }
    };
    auto dot_rows = [&](float* out) {                    // out[t] = x_t . y_t with the staged rows
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float4 xa = *reinterpret_cast<const float4*>(&sm.x[4 * r + a][4 * c]), xb = *reinterpret_cast<const float4*>(&sm.x[4 * r + a][64 + 4 * c]);
            float d = 0.f;
            fma4(d, xa, make_float4(y[a][0], y[a][1], y[a][2], y[a][3]));
            fma4(d, xb, make_float4(y[a][4], y[a][5], y[a][6], y[a][7]));
#pragma unroll
            for (int off = 8; off >= 1; off >>= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
            if (c == 0 && t0 + 4 * r + a < P.S) out[(static_cast<long long>(t0 + 4 * r + a) * P.n_kv + h) * P.n_pairs + blockIdx.y] = d;
        }
    };
    // Gamma_{gg'} o_{g'}, its product with o_g, then + Gamma_{g'g} o_g
    clear();
    stage_gamma(g, gp);
    stage_o(gp);
    __syncthreads();
    product();
    __syncthreads();
    stage_o(g);
    if (g != gp) stage_gamma(gp, g);
    __syncthreads();
    dot_rows(P.kappa);
    product();                                           // (g = g': the same once more)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int t = t0 + 4 * r + a;
        if (t >= P.S) continue;
        float* dst = P.U + ((static_cast<long long>(t) * P.n_kv + h) * P.n_pairs + blockIdx.y) * D + 4 * c;
        *reinterpret_cast<float4*>(dst) = make_float4(y[a][0], y[a][1], y[a][2], y[a][3]);
        *reinterpret_cast<float4*>(dst + 64) = make_float4(y[a][4], y[a][5], y[a][6], y[a][7]);
    }
    __syncthreads();
    for (int item = tid; item < RT * 32; item += 256) {
        const int row = item >> 5, piece = item & 31;
        *reinterpret_cast<float4*>(&sm.x[row][4 * piece]) =
            t0 + row < P.S ? bf16x4(P.V + (static_cast<long long>(t0 + row) * P.n_kv + h) * D + 4 * piece) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    clear();
    product();                                           // v . Gamma_{g'g} v = v . Gamma_{gg'} v
    dot_rows(P.alpha);
}

// A and W0 of 16 positions and NC pairs (from pair0 on): thread (t, c) holds the logits of all heads and v . U of the pairs for its
// position and keys c + 16 e of a tile of 64.  grid (position tiles, pair chunks, n_kv), 256 threads.
template <int G, int NC>
struct PairsSmem { float q[G][16][HS_PITCH], u[NC][16][HS_PITCH], k[RT][HS_PITCH], v[RT][HS_PITCH], al[NC][RT]; };
constexpr int pair_chunks(int G) { return (G * (G + 1) / 2 + 9) / 10; }      // what fits in shared memory beside the heads' queries
constexpr int pairs_per_chunk(int G) { return (G * (G + 1) / 2 + pair_chunks(G) - 1) / pair_chunks(G); }
template <int G, int NC>
__global__ void __launch_bounds__(256, 1) pairs_kernel(HessParams P) {
    extern __shared__ __align__(16) unsigned char hs_smem[];
    PairsSmem<G, NC>& sm = *reinterpret_cast<PairsSmem<G, NC>*>(hs_smem);
    const int t0 = (gridDim.x - 1 - blockIdx.x) * 16, pair0 = blockIdx.y * NC, h = blockIdx.z, tid = threadIdx.x, tr = tid >> 4, c = tid & 15;
    const int t = t0 + tr, n_pairs = min(NC, P.n_pairs - pair0);
    for (int item = tid; item < G * 16 * 32; item += 256) {
        const int g = item >> 9, row = (item >> 5) & 15, piece = item & 31;
        *reinterpret_cast<float4*>(&sm.q[g][row][4 * piece]) =
            t0 + row < P.S ? bf16x4(P.Q + (static_cast<long long>(t0 + row) * P.n_q + h * G + g) * D + 4 * piece) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int item = tid; item < NC * 16 * 32; item += 256) {
        const int k = item >> 9, row = (item >> 5) & 15, piece = item & 31;
        *reinterpret_cast<float4*>(&sm.u[k][row][4 * piece]) =
            t0 + row < P.S && k < n_pairs ? *reinterpret_cast<const float4*>(P.U + ((static_cast<long long>(t0 + row) * P.n_kv + h) * P.n_pairs + pair0 + k) * D + 4 * piece)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float rm[G], rl[G], kap[NC], asum[NC], wsum[NC];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const long long row = static_cast<long long>(min(t, P.S - 1)) * P.n_q + h * G + g;
        rm[g] = P.row_m[row]; rl[g] = P.row_linv[row];
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        kap[k] = k < n_pairs ? P.kappa[(static_cast<long long>(min(t, P.S - 1)) * P.n_kv + h) * P.n_pairs + pair0 + k] : 0.f;
        asum[k] = wsum[k] = 0.f;
    }
    for (int s0 = 0; s0 < min(t0 + 16, P.S); s0 += RT) {
        __syncthreads();
#pragma unroll 2
        for (int item = tid; item < RT * 32; item += 256) {
            const int row = item >> 5, piece = item & 31;
            const bool in = s0 + row < P.S;
            const long long off = (static_cast<long long>(in ? s0 + row : 0) * P.n_kv + h) * D + 4 * piece;
            *reinterpret_cast<float4*>(&sm.k[row][4 * piece]) = in ? bf16x4(P.K + off) : make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4*>(&sm.v[row][4 * piece]) = in ? bf16x4(P.V + off) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int item = tid; item < NC * RT; item += 256) {
            const int k = item / RT, row = item % RT;
            sm.al[k][row] = s0 + row < P.S && k < n_pairs ? P.alpha[(static_cast<long long>(s0 + row) * P.n_kv + h) * P.n_pairs + pair0 + k] : 0.f;
        }
        __syncthreads();
        float p[G][4], rr[NC][4];
#pragma unroll
        for (int g = 0; g < G; ++g) p[g][0] = p[g][1] = p[g][2] = p[g][3] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) rr[k][0] = rr[k][1] = rr[k][2] = rr[k][3] = 0.f;
#pragma unroll 2
        for (int k4 = 0; k4 < D; k4 += 4) {
            float4 b[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) b[e] = *reinterpret_cast<const float4*>(&sm.k[c + 16 * e][k4]);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const float4 a = *reinterpret_cast<const float4*>(&sm.q[g][tr][k4]);
#pragma unroll
                for (int e = 0; e < 4; ++e) fma4(p[g][e], a, b[e]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) b[e] = *reinterpret_cast<const float4*>(&sm.v[c + 16 * e][k4]);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const float4 a = *reinterpret_cast<const float4*>(&sm.u[k][tr][k4]);
#pragma unroll
                for (int e = 0; e < 4; ++e) fma4(rr[k][e], a, b[e]);
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int e = 0; e < 4; ++e) p[g][e] = s0 + c + 16 * e <= t ? __expf(p[g][e] * P.inv_tau - rm[g]) * rl[g] : 0.f;
        // pairs in order, from the chunk's first one on (chunk boundaries are the same for every thread)
        int index = 0;
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int gp = g; gp < G; ++gp, ++index) {
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    if (NC < G * (G + 1) / 2 ? index == pair0 + k : index == k) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float w = p[g][e] * p[gp][e];
                            wsum[k] += w;
                            asum[k] = fmaf(w, (sm.al[k][c + 16 * e] - rr[k][e]) + kap[k], asum[k]);
                        }
                    }
                }
            }
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) { asum[k] += __shfl_xor_sync(0xffffffffu, asum[k], off); wsum[k] += __shfl_xor_sync(0xffffffffu, wsum[k], off); }
        if (c == 0 && t < P.S && k < n_pairs) {
            const long long o = (static_cast<long long>(t) * P.n_kv + h) * P.n_pairs + pair0 + k;
            P.A[o] = asum[k];
            P.W0[o] = wsum[k];
        }
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
// (two wavefronts for eight multiply-adds per warp) and the conversions to float64.  With all 64 blocks, 512 threads, loads waited for
// and float64 atomics the whole call took 1352 us for 1024 tokens of 32 / 8 heads and 310 us for 300 tokens of 16 / 4, now 1344 and 267.
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
        for (int t = lane; t < P.S; t += 32) sum += static_cast<double>(P.W0[(static_cast<long long>(t) * P.n_kv + h) * P.n_pairs + k]);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) c_s[k] = sum;
    }
    __syncthreads();
    for (int idx = tid; idx < D * D / 16; idx += 256) {
        const int ij = blockIdx.x * (D * D / 16) + idx;
        double hv = 0.0;
        int k = 0;
        for (int g = 0; g < P.G; ++g)
            for (int gp = g; gp < P.G; ++gp, ++k) {
                const double a = P.gamma[(static_cast<long long>(h * P.G + g) * P.G + gp) * D * D + ij];
                hv += c_s[k] * (g == gp ? a : a + static_cast<double>(P.gamma[(static_cast<long long>(h * P.G + gp) * P.G + g) * D * D + ij]));
            }
        P.H_V[static_cast<long long>(h) * D * D + ij] += 2.0 * hv;
    }
}

template <int G>
bool launch_pairs(const HessParams& P, cudaStream_t st) {
    constexpr int NC = pairs_per_chunk(G);
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(pairs_kernel<G, NC>), static_cast<int>(sizeof(PairsSmem<G, NC>)))) return false;
    pairs_kernel<G, NC><<<dim3((P.S + 15) / 16, pair_chunks(G), P.n_kv), 256, sizeof(PairsSmem<G, NC>), st>>>(P);
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
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(rows_kernel), static_cast<int>(sizeof(RowsSmem))) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(project_kernel), static_cast<int>(sizeof(ProjectSmem))))
        return WUSHKV_ECUDA;
    const unsigned tiles = (P.S + RT - 1) / RT;
    gamma_kernel<<<dim3(P.n_pairs, n_kv, D / 32), 128, 0, st>>>(P);
    rows_kernel<<<dim3(tiles, n_q), 256, sizeof(RowsSmem), st>>>(P);
    project_kernel<<<dim3(tiles, P.n_pairs, n_kv), 256, sizeof(ProjectSmem), st>>>(P);
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
