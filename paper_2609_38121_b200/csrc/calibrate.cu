// Calibration on the GPU (Algorithm 1): streaming Gram / Hessian accumulation over calibration sequences
// (lines 4-5, Eq. 4) and the WUSH transforms of all heads from the accumulated statistics (line 7, Eq. 1,
// Definition 1).  Same results as the host entry points wushkv_accumulate_gram / wushkv_build_transforms up to
// summation order; meant for calibration sets of millions of tokens, where the host loops take hours.
//
//   gram_kernel             X^T X of one head over a slice of tokens on tensor cores (bf16 operands are the inputs
//                           themselves, products exact, fp32 accumulation within the slice), added to the float64
//                           statistics with atomics.
//   build_transforms_kernel one CTA per head, float64 throughout: damping, Cholesky, L^T M L, one-sided Jacobi on its Cholesky
//                           factor with a round-robin ordering (64 disjoint rotations per step), canonical order / sign,
//                           T = c Had Lam^(-1/4) U^T L^T rounded to bf16, Gauss-Jordan inverse of the rounded matrix.
#include <cuda_runtime.h>

#include <cmath>

#include "host_common.h"
#include "layout.cuh"

namespace wushkv {
namespace {

constexpr int GR_TOK = 64;                 // tokens per staged tile
constexpr int GR_PITCH = D + 8;            // bf16 per staged row (272 bytes: conflict-free ldmatrix)
constexpr int GR_SLICE = 2048;             // tokens per CTA
constexpr int GR_FLUSH = 128;              // tokens whose products are summed in fp32 (8 tensor-core accumulations) before they move to float64

__device__ __forceinline__ unsigned saddr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void ldsm4t(unsigned addr, unsigned& a, unsigned& b, unsigned& c, unsigned& d) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_acc(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// grid (token slices, n_kv + n_q head slots), 256 threads: warp w owns output rows 16w .. 16w+15 (all 128 columns).  One CTA fits
// on an SM (64 float64 and 64 fp32 sums per thread), so the next tile is requested while this one is multiplied; the bound
// is the mma.sync rate.  32768 tokens of 32 / 8 heads: 575 us with the loads waited for, now 255 us.
__global__ void __launch_bounds__(256) gram_kernel(int n_kv, int n_q, long long n_tok, const unsigned short* __restrict__ K,
                                                   const unsigned short* __restrict__ Q, double* M, double* H) {
    __shared__ __align__(16) unsigned short xs2[2][GR_TOK][GR_PITCH];
    const int hs = blockIdx.y;
    const bool is_key = hs < n_kv;
    const int head = is_key ? hs : hs - n_kv, n_heads = is_key ? n_kv : n_q, G = n_q / n_kv;
    const unsigned short* X = is_key ? K : Q;
    double* out = is_key ? M + static_cast<long long>(head) * D * D : H + static_cast<long long>(head / G) * D * D;
    const double weight = is_key ? 1.0 : 2.0;                 // H = 2 sum_g sum_t q q^T (Eq. 4)
    const long long t0 = static_cast<long long>(blockIdx.x) * GR_SLICE, t1 = min(t0 + GR_SLICE, n_tok);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    float acc[16][4];
    double dacc[16][4];
#pragma unroll
    for (int nb = 0; nb < 16; ++nb) {
        acc[nb][0] = acc[nb][1] = acc[nb][2] = acc[nb][3] = 0.f;
        dacc[nb][0] = dacc[nb][1] = dacc[nb][2] = dacc[nb][3] = 0.0;
    }
    auto request = [&](long long base, int buf) {                        // 16-byte pieces; rows past the end are zero
#pragma unroll
        for (int item = tid; item < GR_TOK * 16; item += 256) {
            const int r = item >> 4, piece = item & 15;
            const bool in = base + r < t1;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr(&xs2[buf][r][8 * piece])),
                         "l"(X + ((in ? base + r : t0) * n_heads + head) * D + 8 * piece), "r"(in ? 16u : 0u) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    request(t0, 0);
    int buf = 0;
    for (long long base = t0; base < t1; base += GR_TOK, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                                 // this tile has landed; the other buffer has been read
        if (base + GR_TOK < t1) request(base + GR_TOK, buf ^ 1);
        const unsigned short (*xs)[GR_PITCH] = xs2[buf];
#pragma unroll
        for (int ks = 0; ks < GR_TOK / 16; ++ks) {
            // A = X^T (channel x token): registers (rows i0.., tokens lo), (rows i0+8.., lo), (rows i0.., hi), (rows i0+8.., hi)
            unsigned a0, a1, a2, a3;
            ldsm4t(saddr(&xs[16 * ks + 8 * (lane >> 4) + (lane & 7)][16 * warp + 8 * ((lane >> 3) & 1)]), a0, a1, a2, a3);
#pragma unroll
            for (int nb2 = 0; nb2 < 8; ++nb2) {
                unsigned b0, b1, b2, b3;                                 // B = X (token x channel): (tokens lo, cols), (hi, cols), (lo, cols+8), (hi, cols+8)
                ldsm4t(saddr(&xs[16 * ks + 8 * ((lane >> 3) & 1) + (lane & 7)][16 * nb2 + 8 * (lane >> 4)]), b0, b1, b2, b3);
                mma_bf16_acc(acc[2 * nb2], a0, a1, a2, a3, b0, b1);
                mma_bf16_acc(acc[2 * nb2 + 1], a0, a1, a2, a3, b2, b3);
            }
        }
        if (((base - t0) / GR_TOK) % (GR_FLUSH / GR_TOK) == GR_FLUSH / GR_TOK - 1 || base + GR_TOK >= t1) {
#pragma unroll
            for (int nb = 0; nb < 16; ++nb)
#pragma unroll
                for (int e = 0; e < 4; ++e) { dacc[nb][e] += static_cast<double>(acc[nb][e]); acc[nb][e] = 0.f; }
        }
    }
#pragma unroll
    for (int nb = 0; nb < 16; ++nb) {
        const int i0 = 16 * warp + g, j0 = 8 * nb + 2 * t;
        atomicAdd(out + i0 * D + j0, weight * dacc[nb][0]);
        atomicAdd(out + i0 * D + j0 + 1, weight * dacc[nb][1]);
        atomicAdd(out + (i0 + 8) * D + j0, weight * dacc[nb][2]);
        atomicAdd(out + (i0 + 8) * D + j0 + 1, weight * dacc[nb][3]);
    }
}

// ---- float64 helpers of the transform builder -----------------------------------------------------
__device__ __forceinline__ double round_double_to_bf16(double x) {     // nearest bf16, ties to even (values in the float range)
    unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
    u += ((1ull << 44) - 1ull) + ((u >> 45) & 1ull);
    u &= ~((1ull << 45) - 1ull);
    return __longlong_as_double(static_cast<long long>(u));
}

constexpr int BT_THREADS = 512;

__device__ double block_sum(double v, double* red) {
    const int tid = threadIdx.x;
    __syncthreads();
    red[tid] = v;
    __syncthreads();
    for (int s = BT_THREADS / 2; s > 0; s >>= 1) {
        if (tid < s) red[tid] += red[tid + s];
        __syncthreads();
    }
    return red[0];
}

constexpr int BT_PITCH = D + 4;                      // doubles per column (row) of the matrix in shared memory
constexpr int BT_PANEL = 16;                         // k values of a product that are staged together
constexpr size_t BT_SMEM = (static_cast<size_t>(D) * BT_PITCH + 2 * BT_PANEL * BT_PITCH) * sizeof(double);

// One thread's 4 x 8 block of a 128 x 128 product sum_k a(i, k) b(k, j): rows 4 (tid >> 4) .., columns (tid & 15) + 16 e.  The
// operands come through shared-memory panels of 16 k values: four elements per thread and panel.
template <class LoadA, class LoadB>
__device__ __forceinline__ void block_product(double (&acc)[4][8], double* panel, LoadA load_a, LoadB load_b) {
    const int tid = threadIdx.x, i0 = 4 * (tid >> 4), j0 = tid & 15;
    double* pa = panel;
    double* pb = panel + BT_PANEL * BT_PITCH;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[a][e] = 0.0;
#pragma unroll 1
    for (int k0 = 0; k0 < D; k0 += BT_PANEL) {
        double ta[4], tb[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) { ta[n] = load_a(k0, tid + n * BT_THREADS); tb[n] = load_b(k0, tid + n * BT_THREADS); }
        __syncthreads();                             // the previous panel has been read
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            load_a.store(pa, tid + n * BT_THREADS, ta[n]);
            load_b.store(pb, tid + n * BT_THREADS, tb[n]);
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < BT_PANEL; ++kk) {
            double av[4], bv[8];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = pa[kk * BT_PITCH + i0 + a];
#pragma unroll
            for (int e = 0; e < 8; ++e) bv[e] = pb[kk * BT_PITCH + j0 + 16 * e];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[a][e] = fma(av[a], bv[e], acc[a][e]);
        }
    }
}
// Panels of a row-major matrix X in global memory: element (k, x) of the panel is X[k][x] or X[x][k].
template <bool ROWS_ARE_K>
struct GlobalPanel {
    const double* X;
    __device__ __forceinline__ double operator()(int k0, int n) const {
        return ROWS_ARE_K ? X[(k0 + (n >> 7)) * D + (n & 127)] : X[(n >> 4) * D + k0 + (n & 15)];
    }
    __device__ __forceinline__ void store(double* p, int n, double v) const {
        if (ROWS_ARE_K) p[(n >> 7) * BT_PITCH + (n & 127)] = v; else p[(n & 15) * BT_PITCH + (n >> 4)] = v;
    }
};
struct PermutedPanel {                               // element (k, x) is X[x][perm[k]] of a row-major matrix in global memory
    const double* X;
    const int* perm;
    __device__ __forceinline__ double operator()(int k0, int n) const { return X[(n >> 4) * D + perm[k0 + (n & 15)]]; }
    __device__ __forceinline__ void store(double* p, int n, double v) const { p[(n & 15) * BT_PITCH + (n >> 4)] = v; }
};
struct ColumnPanel {                                 // element (k, x) is W[k] of column order[x] of the matrix in shared memory
    const double* W;
    const int* order;
    __device__ __forceinline__ double operator()(int k0, int n) const { return W[order[n >> 4] * BT_PITCH + k0 + (n & 15)]; }
    __device__ __forceinline__ void store(double* p, int n, double v) const { p[(n & 15) * BT_PITCH + (n >> 4)] = v; }
};

// Cholesky of the lower triangle of S (column j at S + j BT_PITCH), in place, the upper triangle set to zero.  False: not
// positive definite.
__device__ bool cholesky_columns(double* S, int* fail) {
    const int tid = threadIdx.x, i = tid & (D - 1), jg = tid >> 7;
#pragma unroll 1
    for (int k = 0; k < D; ++k) {
        const double piv = S[k * BT_PITCH + k];
        if (!(piv > 0.0) && tid == 0) *fail = 1;
        const double r = piv > 0.0 ? 1.0 / sqrt(piv) : 1.0;
        const double lik = i >= k ? S[k * BT_PITCH + i] * r : 0.0;
        __syncthreads();                             // every thread has read the column
        if (jg == 0) S[k * BT_PITCH + i] = lik;
        __syncthreads();
        for (int j = k + 1 + jg; j < D; j += 4)
            if (i >= j) S[j * BT_PITCH + i] = fma(-lik, S[k * BT_PITCH + j], S[j * BT_PITCH + i]);
        __syncthreads();
    }
    return *fail == 0;
}

// The same with diagonal pivoting, of a full symmetric S: C C^T = S with rows and columns taken in the order perm.  The columns of
// C then have falling lengths and are nearly orthogonal, which spares the Jacobi sweeps: 8 heads of 32768 tokens in 4.5 ms without the pivoting, 2.5 ms with it.
__device__ bool cholesky_pivoted(double* S, int* perm, int* pivot_s, int* fail) {
    const int tid = threadIdx.x, i = tid & (D - 1), jg = tid >> 7, lane = tid & 31;
    if (tid < D) perm[tid] = tid;
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < D; ++k) {
        if (tid < 32) {
            double best = -INFINITY;
            int at = k;
#pragma unroll
            for (int e = 0; e < D / 32; ++e) {
                const int j = lane + 32 * e;
                const double v = S[j * BT_PITCH + j];
                if (j >= k && v > best) { best = v; at = j; }
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const double v = __shfl_xor_sync(0xffffffffu, best, o);
                const int j = __shfl_xor_sync(0xffffffffu, at, o);
                if (v > best || (v == best && j < at)) { best = v; at = j; }
            }
            if (lane == 0) { *pivot_s = at; const int x = perm[k]; perm[k] = perm[at]; perm[at] = x; }
        }
        __syncthreads();
        const int p = *pivot_s;
        if (p != k) {                                // (the same for all threads)
            if (jg == 0) { const double x = S[k * BT_PITCH + i]; S[k * BT_PITCH + i] = S[p * BT_PITCH + i]; S[p * BT_PITCH + i] = x; }
            __syncthreads();
            if (jg == 0) { const double x = S[i * BT_PITCH + k]; S[i * BT_PITCH + k] = S[i * BT_PITCH + p]; S[i * BT_PITCH + p] = x; }
            __syncthreads();
        }
        const double piv = S[k * BT_PITCH + k];
        if (!(piv > 0.0) && tid == 0) *fail = 1;
        const double r = piv > 0.0 ? 1.0 / sqrt(piv) : 1.0;
        const double lik = i >= k ? S[k * BT_PITCH + i] * r : 0.0;
        __syncthreads();                             // every thread has read the column
        if (jg == 0) S[k * BT_PITCH + i] = lik;
        __syncthreads();
        if (i > k)
            for (int j = k + 1 + jg; j < D; j += 4) S[j * BT_PITCH + i] = fma(-lik, S[k * BT_PITCH + j], S[j * BT_PITCH + i]);
        __syncthreads();
    }
    return *fail == 0;
}

// One CTA per head, float64.  ws: 8 matrices of d x d float64 per head (3 are used; the first element of the fourth says how many
// sweeps the Jacobi took).
//   L L^T = H (damped);  A = L^T M L (M damped), scaled to trace 1;  C C^T = A with its rows and columns in pivot order.
//   One-sided Jacobi on the columns of C: rotations from the right until they are orthogonal, W = C V.  Then A = W W^T: the
//   eigenvectors of A are W's columns over their lengths, the eigenvalues the lengths' squares.
// What bounds it: 127 steps of 64 disjoint rotations per sweep.  A step reads and writes the whole matrix, 128 KB, in shared memory:
// 2048 cycles at 128 bytes per cycle, and behind the reads a chain of about 1000 cycles from the dot products to the rotated
// columns.  In a capture the shared-memory pipe is busy 65 % of the cycles of the eight SMs that work, the fp64 pipe 27 %.  A two-sided Jacobi on A with the
// rotations applied to A's columns, A's rows and the eigenvectors in global memory, four barriers per step, took 50.6 ms
// for 8 heads.
__global__ void __launch_bounds__(BT_THREADS) build_transforms_kernel(const double* Mall, const double* Hall, double gamma, float* Tall,
                                                                       float* Tinvall, double* wsall, int* status) {
    extern __shared__ __align__(16) double S[];      // the matrix, then two product panels
    double* panel = S + D * BT_PITCH;
    __shared__ double red[BT_THREADS];
    __shared__ double w_s[D], scale_s[D];
    __shared__ int order_s[D], piv_s[D], perm_s[D];      // perm_s: row k of the matrix is coordinate perm_s[k]
    __shared__ int fail_s, piv_row_s;
    const int h = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double* Mh = Mall + static_cast<long long>(h) * D * D;
    const double* Hh = Hall + static_cast<long long>(h) * D * D;
    double* ws = wsall + static_cast<long long>(h) * 8 * D * D;
    double *Md = ws, *L = ws + D * D, *B = ws + 2 * D * D;
    if (tid == 0) fail_s = 0;
    // ---- damping (Definition 1), Cholesky of the damped Hessian
    const double trM = block_sum(tid < D ? Mh[tid * D + tid] : 0.0, red);
    const double trH = block_sum(tid < D ? Hh[tid * D + tid] : 0.0, red);
    for (int idx = tid; idx < D * D; idx += BT_THREADS) {
        const int i = idx >> 7, j = idx & 127;
        Md[idx] = Mh[idx] + (i == j ? gamma * trM / D : 0.0);
        S[j * BT_PITCH + i] = Hh[idx] + (i == j ? gamma * trH / D : 0.0);
    }
    __syncthreads();
    if (!cholesky_columns(S, &fail_s)) { if (tid == 0) atomicOr(status, WUSHKV_ENOTPD); return; }
    for (int idx = tid; idx < D * D; idx += BT_THREADS) L[idx] = S[(idx & 127) * BT_PITCH + (idx >> 7)];
    // ---- A = L^T (Md L), symmetrised and scaled
    double acc[4][8];
    const int i0 = 4 * (tid >> 4), j0 = tid & 15;
    __syncthreads();
    block_product(acc, panel, GlobalPanel<false>{Md}, GlobalPanel<true>{L});
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 8; ++e) B[(i0 + a) * D + j0 + 16 * e] = acc[a][e];
    __syncthreads();
    block_product(acc, panel, GlobalPanel<true>{L}, GlobalPanel<true>{B});
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 8; ++e) S[(i0 + a) * BT_PITCH + j0 + 16 * e] = acc[a][e];
    __syncthreads();
    const double trA = block_sum(tid < D ? S[tid * BT_PITCH + tid] : 0.0, red);
    if (!(trA > 0.0)) { if (tid == 0) atomicOr(status, WUSHKV_ENOTPD); return; }
    for (int idx = tid; idx < D * D; idx += BT_THREADS) {
        const int i = idx >> 7, j = idx & 127;
        if (i >= j) {                                // (only this thread reads or writes the pair)
            const double v = 0.5 * (S[i * BT_PITCH + j] + S[j * BT_PITCH + i]) / trA;
            S[i * BT_PITCH + j] = v;
            S[j * BT_PITCH + i] = v;
        }
    }
    __syncthreads();
    if (!cholesky_pivoted(S, perm_s, &piv_row_s, &fail_s)) { if (tid == 0) atomicOr(status, WUSHKV_ENOTPD); return; }
    // ---- one-sided Jacobi, round-robin ordering.  Eight lanes own a pair of columns, 16 rows each (as 8 x 16 bytes: the eight lanes
    // read 128 consecutive bytes).  The angle is computed in fp32 (its error only delays convergence; where its operands leave the fp32
    // range, as for columns whose lengths differ by more than 1e5, in float64), the rotation from it in
    // float64, so that it is orthogonal to rounding; the longer column goes to the lower index, which speeds convergence up.
    int sweeps = 0;
    {
        constexpr double TOL2 = 1.6e-29;             // squared cosine below which a pair counts as orthogonal (its rounding is about 1e-30)
        const int pair = 4 * warp + (lane >> 3), l8 = lane & 7;
#pragma unroll 1
        for (; sweeps < 30; ++sweeps) {
            int rotated = 0;
#pragma unroll 1
            for (int step = 0; step < D - 1; ++step) {
                auto player = [&](int pos) { int x = pos - 1 - step; if (x < 0) x += D - 1; return pos == 0 ? 0 : 1 + x; };
                const int pa = player(pair), pb = player(D - 1 - pair);
                double2* P = reinterpret_cast<double2*>(S + min(pa, pb) * BT_PITCH) + l8;
                double2* Q = reinterpret_cast<double2*>(S + max(pa, pb) * BT_PITCH) + l8;
                double2 p[8], q[8];
                double alpha = 0.0, beta = 0.0, g = 0.0;
#pragma unroll
                for (int k = 0; k < 8; ++k) { p[k] = P[8 * k]; q[k] = Q[8 * k]; }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    alpha = fma(p[k].x, p[k].x, fma(p[k].y, p[k].y, alpha));
                    beta = fma(q[k].x, q[k].x, fma(q[k].y, q[k].y, beta));
                    g = fma(p[k].x, q[k].x, fma(p[k].y, q[k].y, g));
                }
#pragma unroll
                for (int o = 1; o <= 4; o <<= 1) {
                    alpha += __shfl_xor_sync(0xffffffffu, alpha, o);
                    beta += __shfl_xor_sync(0xffffffffu, beta, o);
                    g += __shfl_xor_sync(0xffffffffu, g, o);
                }
                if (g * g > TOL2 * (alpha * beta)) {
                    rotated = 1;
                    const float zeta = static_cast<float>(beta - alpha) / (2.f * static_cast<float>(g));
                    double t = static_cast<double>(copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.f))));
                    // zeta^2 overflows from 1.8e19 on, and zeta itself where g underflows: 1 / (2 zeta), and no more than 45 degrees
                    if (!(fabsf(zeta) < 1e15f)) t = fmin(fmax(g / (beta - alpha), -1.0), 1.0);
                    const double c = rsqrt(fma(t, t, 1.0)), s = c * t;
                    const bool swap = alpha - t * g < beta + t * g;
                    const double c1 = swap ? s : c, s1 = swap ? -c : s;       // first column: c1 p - s1 q, second: s2 p + c2 q
                    const double c2 = swap ? -s : c, s2 = swap ? c : s;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        P[8 * k] = make_double2(fma(c1, p[k].x, -s1 * q[k].x), fma(c1, p[k].y, -s1 * q[k].y));
                        Q[8 * k] = make_double2(fma(s2, p[k].x, c2 * q[k].x), fma(s2, p[k].y, c2 * q[k].y));
                    }
                }
                __syncthreads();
            }
            if (!__syncthreads_or(rotated)) break;
        }
    }
    if (tid == 0) ws[3 * D * D] = sweeps;            // for the tests: sweeps that rotated something
    // ---- canonical form: eigenvalues ascending, largest-magnitude entry of each eigenvector positive
    if (tid < D) {
        double len2 = 0.0, top = 0.0;
#pragma unroll 4
        for (int k = 0; k < D; ++k) {
            const double x = S[tid * BT_PITCH + k];
            len2 = fma(x, x, len2);
            if (fabs(x) > fabs(top)) top = x;
        }
        w_s[tid] = len2 * trA;
        if (!(len2 > 0.0)) fail_s = 1;
        red[tid] = (top < 0.0 ? -1.0 : 1.0) / sqrt(len2);
    }
    __syncthreads();
    if (fail_s) { if (tid == 0) atomicOr(status, WUSHKV_ENOTPD); return; }
    if (tid < D) {
        int rank = 0;
        for (int j = 0; j < D; ++j) rank += (w_s[j] < w_s[tid]) || (w_s[j] == w_s[tid] && j < tid);
        order_s[rank] = tid;
        scale_s[rank] = red[tid] * pow(w_s[tid], -0.25);         // sign and scale of row `rank` of Lam^(-1/4) U^T
    }
    const double sum_sqrt = block_sum(tid < D ? sqrt(w_s[tid]) : 0.0, red);
    const double hn = sqrt(1.0 + gamma) * sqrt(trM) / sqrt(sum_sqrt) / sqrt(static_cast<double>(D));
    // ---- Lam^(-1/4) U^T L^T: row i is scale_i sum_k W[k][order_i] L[j][perm_k]
    __syncthreads();
    block_product(acc, panel, ColumnPanel{S, order_s}, PermutedPanel{L, perm_s});
    __syncthreads();                                 // the eigenvectors have been read
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int e = 0; e < 8; ++e) S[(i0 + a) * BT_PITCH + j0 + 16 * e] = scale_s[i0 + a] * acc[a][e];
    __syncthreads();
    // ---- T = c Had (..): fast Walsh-Hadamard transform over the rows, rounded to bf16
    const int j = tid & (D - 1), grp = tid >> 7;
    {
        double x[32];
#pragma unroll
        for (int r = 0; r < 32; ++r) x[r] = S[(32 * grp + r) * BT_PITCH + j];
#pragma unroll
        for (int bit = 1; bit < 32; bit <<= 1)
#pragma unroll
            for (int r = 0; r < 32; ++r)
                if ((r & bit) == 0) { const double u = x[r], v = x[r | bit]; x[r] = u + v; x[r | bit] = u - v; }
#pragma unroll
        for (int r = 0; r < 32; ++r) S[(32 * grp + r) * BT_PITCH + j] = x[r];
    }
    __syncthreads();
    float* To = Tall + static_cast<long long>(h) * D * D;
#pragma unroll 2
    for (int r = 8 * grp; r < 8 * grp + 8; ++r) {
        const double x0 = S[r * BT_PITCH + j], x1 = S[(r + 32) * BT_PITCH + j], x2 = S[(r + 64) * BT_PITCH + j], x3 = S[(r + 96) * BT_PITCH + j];
        const double y[4] = {(x0 + x1) + (x2 + x3), (x0 - x1) + (x2 - x3), (x0 + x1) - (x2 + x3), (x0 - x1) - (x2 - x3)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const double v = round_double_to_bf16(hn * y[e]);
            S[(r + 32 * e) * BT_PITCH + j] = v;
            To[(r + 32 * e) * D + j] = static_cast<float>(v);
        }
    }
    __syncthreads();
    // ---- inverse of the rounded T: Gauss-Jordan with partial pivoting, in place; thread (j, grp) owns column j of rows grp + 4 m
#pragma unroll 1
    for (int col = 0; col < D; ++col) {
        if (warp == 0) {
            double best = -1.0;
            int at = col;
            for (int r = lane; r < D; r += 32)
                if (r >= col) { const double v = fabs(S[r * BT_PITCH + col]); if (v > best) { best = v; at = r; } }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const double v = __shfl_xor_sync(0xffffffffu, best, o);
                const int r = __shfl_xor_sync(0xffffffffu, at, o);
                if (v > best || (v == best && r < at)) { best = v; at = r; }
            }
            if (lane == 0) { piv_row_s = at; piv_s[col] = at; if (!(best > 0.0)) fail_s = 1; }
        }
        __syncthreads();
        if (fail_s) { if (tid == 0) atomicOr(status, WUSHKV_ENOTPD); return; }
        const int piv = piv_row_s;
        const double inv = 1.0 / S[piv * BT_PITCH + col];
        const double rowk = (j == col ? 1.0 : S[piv * BT_PITCH + j]) * inv, old_k = S[col * BT_PITCH + j];
        __syncthreads();
        if (grp == 0 && piv != col) S[piv * BT_PITCH + j] = old_k;       // row swap
        __syncthreads();
        if (tid < D) red[tid] = tid == col ? 0.0 : S[tid * BT_PITCH + col];      // the column being eliminated, before it changes
        __syncthreads();
#pragma unroll 8
        for (int i = grp; i < D; i += 4) {
            const double x = j == col ? 0.0 : S[i * BT_PITCH + j];
            S[i * BT_PITCH + j] = i == col ? rowk : fma(-red[i], rowk, x);
        }
        __syncthreads();
    }
#pragma unroll 1
    for (int col = D - 1; col >= 0; --col) {          // the row swaps, undone as column swaps in reverse
        const int piv = piv_s[col];
        if (piv != col && tid < D) { const double x = S[tid * BT_PITCH + col]; S[tid * BT_PITCH + col] = S[tid * BT_PITCH + piv]; S[tid * BT_PITCH + piv] = x; }
    }
    __syncthreads();
    float* Ti = Tinvall + static_cast<long long>(h) * D * D;
    for (int idx = tid; idx < D * D; idx += BT_THREADS) Ti[idx] = static_cast<float>(S[(idx & 127) * BT_PITCH + (idx >> 7)]);      // (T^-1)^T
}

}  // namespace
}  // namespace wushkv

using namespace wushkv;

extern "C" int wushkv_accumulate_gram_device(int32_t n_kv, int32_t n_q, int32_t d, int64_t n_tok, const uint16_t* K, const uint16_t* Q,
                                             double* M, double* H, void* stream) {
    if (!K || !Q || !M || !H || n_kv <= 0 || n_q <= 0 || d != D || n_tok < 0 || n_q % n_kv != 0) return WUSHKV_EINVAL;
    if (!aligned(K, 16) || !aligned(Q, 16) || !aligned(M, 8) || !aligned(H, 8)) return WUSHKV_EINVAL;
    if (n_tok == 0) return WUSHKV_OK;
    const long long slices = (n_tok + GR_SLICE - 1) / GR_SLICE;
    if (slices > 0x7fffffffLL) return WUSHKV_EINVAL;
    gram_kernel<<<dim3(static_cast<unsigned>(slices), n_kv + n_q), 256, 0, static_cast<cudaStream_t>(stream)>>>(n_kv, n_q, n_tok, K, Q, M, H);
    return cudaGetLastError() == cudaSuccess ? WUSHKV_OK : WUSHKV_ECUDA;
}

extern "C" size_t wushkv_build_transforms_workspace_bytes(int32_t n_heads, int32_t d) {
    if (n_heads <= 0 || d != D) return 0;
    return static_cast<size_t>(n_heads) * 8 * D * D * sizeof(double);
}

extern "C" int wushkv_build_transforms_device(int32_t n_heads, int32_t d, const double* M, const double* H, double gamma,
                                              float* T, float* T_invT, int32_t* dev_status, void* workspace, size_t workspace_bytes,
                                              void* stream) {
    if (!M || !H || !T || !T_invT || !dev_status || !workspace || n_heads <= 0 || d != D || !(gamma >= 0.0)) return WUSHKV_EINVAL;
    if (!aligned(M, 8) || !aligned(H, 8) || !aligned(workspace, 16)) return WUSHKV_EINVAL;
    if (workspace_bytes < wushkv_build_transforms_workspace_bytes(n_heads, d)) return WUSHKV_ECAPACITY;
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(build_transforms_kernel), static_cast<int>(BT_SMEM))) return WUSHKV_ECUDA;
    build_transforms_kernel<<<n_heads, BT_THREADS, BT_SMEM, static_cast<cudaStream_t>(stream)>>>(M, H, gamma, T, T_invT, static_cast<double*>(workspace), dev_status);
    return cudaGetLastError() == cudaSuccess ? WUSHKV_OK : WUSHKV_ECUDA;
}
