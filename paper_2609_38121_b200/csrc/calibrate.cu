// Calibration on the GPU (Algorithm 1): streaming Gram / Hessian accumulation over calibration sequences
// (lines 4-5, Eq. 4) and the WUSH transforms of all heads from the accumulated statistics (line 7, Eq. 1,
// Definition 1).  Same results as the host entry points wushkv_accumulate_gram / wushkv_build_transforms up to
// summation order; meant for calibration sets of millions of tokens, where the host loops take hours.
//
//   gram_kernel             X^T X of the heads on tensor cores (bf16 operands are the inputs themselves, products exact, fp32
//                           accumulation over 128 tokens, float64 beyond), added to the float64 statistics with atomics.
//   the transform builder   float64 throughout: damping, Cholesky, L^T M L, one-sided Jacobi on its Cholesky factor with a round-robin
//                           ordering (64 disjoint rotations per step), canonical order / sign, T = c Had Lam^(-1/4) U^T L^T
//                           rounded to bf16, Gauss-Jordan inverse of the rounded matrix.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "host_common.h"
#include "layout.cuh"

namespace wushkv {
namespace {

__device__ __forceinline__ unsigned saddr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

// ---- X^T X of all heads -------------------------------------------------------------------------------------------------
// A unit is 128 tokens of one head: a 128 x 128 tile of bf16 rows, fetched by two bulk tensor copies (64 channels each, 128-byte
// swizzle), which stands for both operands of 8 tcgen05.mma M128 N128 K16 (channels on M and N, tokens on K: both operands MN-major).  The
// fp32 sums over 128 tokens (8 accumulations) come back from tensor memory and move to float64 in registers.  One CTA per SM takes a
// consecutive part of the list (head, tokens); where the matrix changes, and at the end, a thread adds its 64 sums to the statistics
// with atomics (to the mirror image of their places, which makes a warp's addresses consecutive).
// Warps 0-7: float64 sums of the 32 tensor-memory lanes that their number allows, half the columns each.  Warp 8: copies, six tiles ahead.
// Warp 9: MMAs, into one of four accumulators.  32768 tokens of 32 / 8 heads: mma.sync with the sums in the same warps 255 us (its rate),
// this 92; with 32 columns loaded at a time, which spills, 106.  1.07 us per unit, and about 18 us for the launch and the atomics at the end.
// No unit of the SM binds alone (timing-only variants: tiles out of the L2 92 us, half the copies 91, one MMA instead of eight or no float64
// sums 88, both 82, all of it 80).
constexpr int GR_TOK = 128, GR_STAGES = 6, GR_ACC = 4, GR_THREADS = 320;
constexpr int GR_TILE_BYTES = GR_TOK * D * 2;
constexpr size_t GRAM_SMEM = static_cast<size_t>(GR_STAGES) * GR_TILE_BYTES + 1024;      // and alignment
constexpr unsigned GR_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((static_cast<unsigned>(D) >> 3) << 17) |
                              ((static_cast<unsigned>(D) >> 4) << 24);                   // fp32 <- bf16 x bf16, both MN-major
struct GramParams {
    int n_kv, n_q;
    long long groups, units;                         // groups of tokens; groups times heads (those of K, then those of Q)
    double *M, *H;
    const unsigned short *K, *Q;                     // read where there is no tensor map
    long long n_tok;
    int use_tma;
    int wait_limit;                                  // polls of about a microsecond each
    int drop;                                        // testing aid: 1 the first unit's products are never signalled, 2 one bulk copy is never issued
};
// False when the wait ran out, here or in another warp.
__device__ __forceinline__ bool gram_wait(unsigned bar, unsigned parity, int limit, volatile int* stop) {
#pragma unroll 1
    for (int n = 0; n < limit; ++n) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(bar), "r"(parity), "r"(1000u) : "memory");
        if (done) return true;
        if (stop && *stop) return false;
    }
    if (stop) *stop = 1;
    return false;
}
__device__ __forceinline__ void gram_commit(unsigned bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__global__ void __launch_bounds__(GR_THREADS, 1) gram_kernel(GramParams P, const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap q_map) {
    extern __shared__ __align__(16) unsigned char gram_smem[];
    __shared__ unsigned long long full_bar[GR_STAGES], free_bar[GR_STAGES], acc_bar[GR_ACC], read_bar[GR_ACC], drain_bar;
    __shared__ unsigned tmem_s;
    __shared__ int stop_s, copied_s;                // a wait ran out; tiles requested by bulk copies
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned tiles = (saddr(gram_smem) + 1023u) & ~1023u;
    const long long u0 = P.units * blockIdx.x / gridDim.x, u1 = P.units * (blockIdx.x + 1) / gridDim.x;
    const int n_units = static_cast<int>(u1 - u0);
    if (tid == 0) {
        auto init = [](unsigned long long* bar, unsigned count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory"); };
        for (int k = 0; k < GR_STAGES; ++k) { init(&full_bar[k], 1); init(&free_bar[k], 1); }
        for (int k = 0; k < GR_ACC; ++k) { init(&acc_bar[k], 1); init(&read_bar[k], 8); }
        init(&drain_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        stop_s = copied_s = 0;
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_s)), "r"(static_cast<unsigned>(GR_ACC * D)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = tmem_s;
    volatile int* stop = &stop_s;
    if (warp == 8 && !P.use_tma) {                   // the same tiles by 16-byte loads and stores of the warp's lanes
        int slot = static_cast<int>(u0 / P.groups);
        long long group = u0 % P.groups;
        for (int k = 0; k < n_units; ++k) {
            const int stage = k % GR_STAGES;
            if (!__all_sync(0xffffffffu, k < GR_STAGES || gram_wait(saddr(&free_bar[stage]), (k / GR_STAGES - 1) & 1, P.wait_limit, stop))) break;
            const bool key = slot < P.n_kv;
            const int head = key ? slot : slot - P.n_kv, heads = key ? P.n_kv : P.n_q;
            const unsigned short* X = (key ? P.K : P.Q) + static_cast<long long>(head) * D;
#pragma unroll 4
            for (int item = lane; item < GR_TOK * 16; item += 32) {
                const int r = item >> 4, piece = item & 15;
                const long long token = group * GR_TOK + r;
                const uint4 v = token < P.n_tok ? *reinterpret_cast<const uint4*>(X + token * heads * D + 8 * piece) : make_uint4(0, 0, 0, 0);
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                             ::"r"(tiles + stage * GR_TILE_BYTES + (piece >> 3) * (GR_TILE_BYTES / 2) + r * 128 + (((piece ^ r) & 7) << 4)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&full_bar[stage])) : "memory");
            if (++group == P.groups) { group = 0; ++slot; }
        }
    } else if (warp == 8) {
        if (lane == 0) {
            int slot = static_cast<int>(u0 / P.groups), k = 0;
            long long group = u0 % P.groups;
            for (; k < n_units; ++k) {
                const int stage = k % GR_STAGES;
                if (k >= GR_STAGES && !gram_wait(saddr(&free_bar[stage]), (k / GR_STAGES - 1) & 1, P.wait_limit, stop)) break;
                const unsigned bar = saddr(&full_bar[stage]), dst = tiles + stage * GR_TILE_BYTES;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(static_cast<unsigned>(GR_TILE_BYTES)) : "memory");
                const CUtensorMap* map = slot < P.n_kv ? &k_map : &q_map;
                const int head = slot < P.n_kv ? slot : slot - P.n_kv, row = static_cast<int>(group * GR_TOK);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (P.drop == 2 && k == 0 && half == 0) continue;
                    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                                 ::"r"(dst + half * (GR_TILE_BYTES / 2)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(64 * half), "r"(head), "r"(row), "r"(bar) : "memory");
                }
                if (++group == P.groups) { group = 0; ++slot; }
            }
            copied_s = k;
        }
    } else if (warp == 9) {
        if (lane == 0) {
            for (int k = 0; k < n_units; ++k) {
                const int stage = k % GR_STAGES, acc = k % GR_ACC;
                if (!gram_wait(saddr(&full_bar[stage]), (k / GR_STAGES) & 1, P.wait_limit, stop)) break;
                if (k >= GR_ACC && !gram_wait(saddr(&read_bar[acc]), (k / GR_ACC - 1) & 1, P.wait_limit, stop)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // rows of 128 bytes (64 channels of a token), groups of 8 tokens 1024 bytes apart, the other 64 channels half a tile behind
                const unsigned long long desc = (static_cast<unsigned long long>(((tiles + stage * GR_TILE_BYTES) >> 4) & 0x3FFFu)) |
                                                (static_cast<unsigned long long>((GR_TILE_BYTES / 2) >> 4) << 16) |
                                                (static_cast<unsigned long long>(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
#pragma unroll
                for (int ks = 0; ks < GR_TOK / 16; ++ks)
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
                                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %1, %2, {%4, %4, %4, %4}, p;\n\t}"
                                 ::"r"(tmem + acc * D), "l"(desc + static_cast<unsigned long long>(ks * 2048 >> 4)), "r"(GR_IDESC), "r"(ks), "r"(0u) : "memory");
                gram_commit(saddr(&free_bar[stage]));
                if (!(P.drop == 1 && k == 0)) gram_commit(saddr(&acc_bar[acc]));
            }
        }
    } else {
        double sum[64];
#pragma unroll
        for (int e = 0; e < 64; ++e) sum[e] = 0.0;
        const int i = 32 * (warp & 3) + lane, c0 = 64 * (warp >> 2), G = P.n_q / P.n_kv;
        int slot = static_cast<int>(u0 / P.groups);
        long long group = u0 % P.groups;
        for (int k = 0; k < n_units; ++k) {
            const int acc = k % GR_ACC;
            // (the lanes decide together whether to go on, but only after the loads: in front of them the vote takes 104 us instead of 92)
            const bool landed = gram_wait(saddr(&acc_bar[acc]), (k / GR_ACC) & 1, P.wait_limit, stop);
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int part = 0; part < 4; ++part) {
                unsigned v[16];
                const unsigned addr = tmem + acc * D + c0 + 16 * part + (static_cast<unsigned>(32 * (warp & 3)) << 16);
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                               "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                             : "r"(addr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (part == 3) {                     // the accumulator has been read
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&read_bar[acc])) : "memory");
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) sum[16 * part + e] += static_cast<double>(__uint_as_float(v[e]));
            }
            if (!__all_sync(0xffffffffu, landed)) break;
            const int matrix = slot < P.n_kv ? slot : P.n_kv + (slot - P.n_kv) / G;
            if (++group == P.groups) { group = 0; ++slot; }
            if (k == n_units - 1 || matrix != (slot < P.n_kv ? slot : P.n_kv + (slot - P.n_kv) / G)) {
                double* out = (matrix < P.n_kv ? P.M + static_cast<long long>(matrix) * D * D : P.H + static_cast<long long>(matrix - P.n_kv) * D * D) + c0 * D + i;
                const double weight = matrix < P.n_kv ? 1.0 : 2.0;       // H = 2 sum_g sum_t q q^T (Eq. 4)
#pragma unroll
                for (int e = 0; e < 64; ++e) { atomicAdd(out + e * D, weight * sum[e]); sum[e] = 0.0; }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (stop_s) {                                    // a wait ran out
        // no copy or product may be under way when the CTA has gone
        if (warp == 9 && lane == 0) {
            for (int n = max(copied_s - GR_STAGES, 0); n < copied_s; ++n) gram_wait(saddr(&full_bar[n % GR_STAGES]), (n / GR_STAGES) & 1, P.wait_limit, nullptr);
            gram_commit(saddr(&drain_bar));
            gram_wait(saddr(&drain_bar), 0, P.wait_limit, nullptr);
        }
        __syncwarp();
        // the statistics must not look usable: not a number on the diagonal of every matrix
        for (long long n = tid; n < static_cast<long long>(P.n_kv) * D; n += GR_THREADS) {
            const long long at = n / D * (D * D) + n % D * (D + 1);
            atomicAdd(P.M + at, static_cast<double>(NAN));
            atomicAdd(P.H + at, static_cast<double>(NAN));
        }
    }
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(static_cast<unsigned>(GR_ACC * D)) : "memory");
}

// ---- float64 helpers of the transform builder -----------------------------------------------------
__device__ __forceinline__ double round_double_to_bf16(double x) {     // nearest bf16, ties to even (values in the float range)
    unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
    u += ((1ull << 44) - 1ull) + ((u >> 45) & 1ull);
    u &= ~((1ull << 45) - 1ull);
    return __longlong_as_double(static_cast<long long>(u));
}

// ---- the transform builder: six kernels in a row, float64 throughout -------------------------------------------------
//   factor_kernel<false>   L L^T = H (damped), one CTA per head
//   congruence_kernel      A = L^T M L (M damped), 16 columns per CTA
//   factor_kernel<true>    C C^T = A, symmetrised and scaled to trace 1, with diagonal pivoting, one CTA per head
//   jacobi_kernel          one-sided Jacobi on the columns of C: rotations from the right until they are orthogonal, W = C V; a
//                          cluster of eight CTAs per head.  Then A = W W^T: the eigenvectors of A are W's columns over their
//                          lengths, the eigenvalues the lengths' squares
//   transform_kernel       canonical order and sign, T = c Had Lam^(-1/4) U^T L^T rounded to bf16, 16 columns per CTA
//   inverse_kernel         Gauss-Jordan inverse of the rounded T, one CTA per head
// A head that turns out not to be positive definite is marked in its workspace, and the later kernels leave it alone.
constexpr int BT_THREADS = 512;
constexpr int BT_PITCH = D + 4;                      // doubles per column of the matrix in shared memory
constexpr int BT_PANEL = 16;                         // columns factored together

// Workspace of a head: 8 matrices of d x d float64, of which three and a few numbers are used.
constexpr int WS_A = 0, WS_L = D * D, WS_W = 2 * D * D, WS_META = 3 * D * D;
constexpr int META_SWEEPS = WS_META;                 // for the tests: sweeps of the Jacobi that rotated something
constexpr int META_TR_M = WS_META + 1, META_TR_A = WS_META + 2, META_FAIL = WS_META + 3;
constexpr int META_EIG = WS_META + D, META_SCALE = WS_META + 2 * D;      // eigenvalues; sign / length of the columns of W
constexpr long long WS_HEAD = 8LL * D * D;
constexpr int BT_MAX_HEADS = 32768;                  // per launch

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double trace(const double* X) {                // by one warp
    const int lane = threadIdx.x & 31;
    return warp_sum((X[lane * (D + 1)] + X[(lane + 32) * (D + 1)]) + (X[(lane + 64) * (D + 1)] + X[(lane + 96) * (D + 1)]));
}

// Cholesky of a symmetric matrix, panels of 16 columns.  The lower triangle stands in shared memory (column j at S + j BT_PITCH); thread
// i < 128 holds row i of the panel in registers.  Within a panel a column is what the matrix had at the panel's start minus the
// products with the panel's columns so far, for which the pivot's row of them is handed round: one barrier of four warps
// per column.  All warps then subtract the panel from the rest of the matrix.  With PIVOT the pivot is the largest diagonal entry left
// (to 13 bits of its mantissa); rows are not moved, a row that has been a pivot is zero in later columns.  The columns
// then have falling lengths and are nearly orthogonal, which spares the Jacobi sweeps: 8 heads of 32768 tokens took 4.5 ms
// without the pivoting and 2.5 ms with it.  A chain of latencies bounds it: 8 heads 49 us,
// with the pivoting 63.
constexpr size_t FACTOR_SMEM = (static_cast<size_t>(D) * BT_PITCH + BT_PANEL * BT_PITCH) * sizeof(double);
template <bool PIVOT>
__global__ void __launch_bounds__(BT_THREADS) factor_kernel(const double* Mall, const double* Hall, double gamma, double* wsall, int* status) {
    extern __shared__ __align__(16) double S[];      // the matrix, then the panel: column c of it at P + c BT_PITCH
    double* P = S + D * BT_PITCH;
    __shared__ __align__(16) double row_s[2][4][BT_PANEL + 2];           // candidate of each warp (the pivot, if it is known): its row of the panel, its diagonal entry
    __shared__ __align__(16) unsigned key_s[2][4];
    const int h = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double* ws = wsall + h * WS_HEAD;
    double scale, lift = 1.0;
    if (PIVOT) {
        if (ws[META_FAIL] != 0.0) return;
        const double tr = trace(ws + WS_A);
        if (!(tr > 0.0)) {
            if (tid == 0) { atomicOr(status, WUSHKV_ENOTPD); ws[META_FAIL] = 1.0; }
            return;
        }
        if (tid == 0) ws[META_TR_A] = tr;
        if (!(tr > 0x1p-900 && tr < 0x1p900)) lift = tr < 1.0 ? 0x1p200 : 0x1p-200;      // where 1 / tr is beyond the range, or has lost bits
        scale = 0.5 / (lift * tr);
    } else {
        const double tr_m = trace(Mall + static_cast<long long>(h) * D * D);
        if (tid == 0) { ws[META_TR_M] = tr_m; ws[META_FAIL] = 0.0; }
        scale = gamma * trace(Hall + static_cast<long long>(h) * D * D) / D;          // the damping of Definition 1
    }
#pragma unroll 8
    for (int idx = tid; idx < D * D; idx += BT_THREADS) {
        const int i = idx >> 7, j = idx & 127;
        if (i < j) continue;
        S[j * BT_PITCH + i] = PIVOT ? scale * (lift * (ws[WS_A + idx] + ws[WS_A + j * D + i]))
                                    : Hall[static_cast<long long>(h) * D * D + idx] + (i == j ? scale : 0.0);
    }
    __syncthreads();
    bool fail = false, used = false;
    double diag = tid < D ? S[tid * BT_PITCH + tid] : 0.0;
#pragma unroll 1
    for (int k0 = 0; k0 < D; k0 += BT_PANEL) {
        if (tid < D) {
            double l[BT_PANEL];
#pragma unroll
            for (int c = 0; c < BT_PANEL; ++c) {
                // every warp's candidate for the pivot hands out its row; the warps agree on the best after the barrier
                bool mine;
                if (PIVOT) {
                    const unsigned key = !used && diag > 0.0 ? (static_cast<unsigned>(__double2hiint(diag)) & ~127u) | (127u - tid) : 0u;
                    const unsigned best = __reduce_max_sync(0xffffffffu, key);
                    mine = key == best && key != 0u;
                    if (lane == 0) key_s[c & 1][warp] = best;
                } else {
                    mine = tid == k0 + c;
                }
                double* mine_s = row_s[c & 1][PIVOT ? warp : 0];
                if (mine) {
#pragma unroll
                    for (int e = 0; e < c; ++e) mine_s[e] = l[e];
                    mine_s[BT_PANEL] = diag;
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                int piv = k0 + c;
                const double* row = row_s[c & 1][0];
                if (PIVOT) {
                    const uint4 k = *reinterpret_cast<const uint4*>(key_s[c & 1]);
                    const unsigned best = max(max(k.x, k.y), max(k.z, k.w));
                    if (best == 0u) { fail = true; piv = 0; } else piv = 127 - (best & 127u);
                    row = row_s[c & 1][piv >> 5];
                }
                const double d = row[BT_PANEL];
                fail |= !(d > 0.0);
                double v = S[min(piv, tid) * BT_PITCH + max(piv, tid)], w = 0.0;
#pragma unroll
                for (int e = 0; e + 1 < c; e += 2) { v = fma(-l[e], row[e], v); w = fma(-l[e + 1], row[e + 1], w); }
                if (c & 1) v = fma(-l[c - 1], row[c - 1], v);
                const double r = rsqrt(d);
                used |= tid == piv;
                l[c] = tid == piv ? d * r : (PIVOT ? used : tid < piv) ? 0.0 : (v + w) * r;
                if (tid != piv) diag = fma(-l[c], l[c], diag);
                P[c * BT_PITCH + tid] = l[c];
            }
        }
        __syncthreads();
        // the factor: L row by row, C column by column
        if (PIVOT) {
            for (int n = tid; n < BT_PANEL * D; n += BT_THREADS) ws[WS_W + (k0 + (n >> 7)) * D + (n & 127)] = P[(n >> 7) * BT_PITCH + (n & 127)];
        } else {
            for (int n = tid; n < BT_PANEL * D; n += BT_THREADS) ws[WS_L + (n >> 4) * D + k0 + (n & 15)] = P[(n & 15) * BT_PITCH + (n >> 4)];
        }
        // the rest of the matrix: a warp's unit is 64 rows x 4 columns of the lower triangle
        const int next = k0 + BT_PANEL;
#pragma unroll 1
        for (int unit = warp; unit < 48; unit += BT_THREADS / 32) {
            const int i = lane + (unit < 16 ? 0 : 64), j = 4 * (unit < 16 ? unit : unit - 16);
            if (next == D || (!PIVOT && (j < next || (unit < 16 && next >= 64)))) continue;
            double acc[2][4];
#pragma unroll
            for (int a = 0; a < 4; ++a) { acc[0][a] = S[(j + a) * BT_PITCH + i]; acc[1][a] = S[(j + a) * BT_PITCH + i + 32]; }
#pragma unroll 8
            for (int c = 0; c < BT_PANEL; ++c) {
                const double x = P[c * BT_PITCH + i], y = P[c * BT_PITCH + i + 32];
                const double2 u = *reinterpret_cast<const double2*>(P + c * BT_PITCH + j), w = *reinterpret_cast<const double2*>(P + c * BT_PITCH + j + 2);
                acc[0][0] = fma(-x, u.x, acc[0][0]); acc[0][1] = fma(-x, u.y, acc[0][1]); acc[0][2] = fma(-x, w.x, acc[0][2]); acc[0][3] = fma(-x, w.y, acc[0][3]);
                acc[1][0] = fma(-y, u.x, acc[1][0]); acc[1][1] = fma(-y, u.y, acc[1][1]); acc[1][2] = fma(-y, w.x, acc[1][2]); acc[1][3] = fma(-y, w.y, acc[1][3]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) { S[(j + a) * BT_PITCH + i] = acc[0][a]; S[(j + a) * BT_PITCH + i + 32] = acc[1][a]; }
        }
        __syncthreads();
    }
    if (fail && tid == 0) { atomicOr(status, WUSHKV_ENOTPD); ws[META_FAIL] = 1.0; }
}

// A = L^T (M + damping) L, columns 16 blockIdx.x ..; thread (i, quarter) sums a quarter of the products of row i, whose 32 factors it
// loads at once: the matrices come out of the L2, and a CTA has little to do but wait for them (two threads per row, 16 loads
// in flight: 40 us for 8 heads, this 16).  M may be read transposed, as A is symmetrised afterwards.  grid (8, heads), 512 threads.
constexpr int COLS = 16;                             // columns per CTA
constexpr size_t CONGRUENCE_SMEM = (static_cast<size_t>(D) * COLS + 4 * D * (COLS + 1)) * sizeof(double);
// y[i][c] = sum_k X[k][i] x[k][c] for a row-major X: partial sums of the four quarters of k to part
__device__ __forceinline__ void column_products(const double* __restrict__ X, const double* x, double* part) {
    const int i = threadIdx.x & (D - 1), quarter = threadIdx.x >> 7;
    double f[32], acc[COLS] = {};
#pragma unroll
    for (int n = 0; n < 32; ++n) f[n] = X[(32 * quarter + n) * D + i];
#pragma unroll
    for (int n = 0; n < 32; ++n) {
        const double2* b = reinterpret_cast<const double2*>(x + (32 * quarter + n) * COLS);
#pragma unroll
        for (int e = 0; e < COLS / 2; ++e) { const double2 v = b[e]; acc[2 * e] = fma(f[n], v.x, acc[2 * e]); acc[2 * e + 1] = fma(f[n], v.y, acc[2 * e + 1]); }
    }
#pragma unroll
    for (int e = 0; e < COLS; ++e) part[(quarter * D + i) * (COLS + 1) + e] = acc[e];
}
__device__ __forceinline__ double column_sum(const double* part, int i, int c) {
    const double* q = part + i * (COLS + 1) + c;
    constexpr int Q = D * (COLS + 1);
    return (q[0] + q[Q]) + (q[2 * Q] + q[3 * Q]);
}
__global__ void __launch_bounds__(BT_THREADS) congruence_kernel(const double* __restrict__ Mall, double gamma, double* wsall) {
    extern __shared__ __align__(16) double S[];
    double *x_s = S, *part = S + D * COLS;
    const int h = blockIdx.y, c0 = COLS * blockIdx.x, tid = threadIdx.x, i = tid & (D - 1), quarter = tid >> 7;
    double* ws = wsall + h * WS_HEAD;
    if (ws[META_FAIL] != 0.0) return;
    const double* L = ws + WS_L;
    const double damp = gamma * ws[META_TR_M] / D;
    for (int n = tid; n < D * COLS; n += BT_THREADS) x_s[n] = L[(n >> 4) * D + c0 + (n & 15)];
    __syncthreads();
    column_products(Mall + static_cast<long long>(h) * D * D, x_s, part);
    __syncthreads();
#pragma unroll
    for (int e = 4 * quarter; e < 4 * quarter + 4; ++e) x_s[i * COLS + e] = fma(damp, x_s[i * COLS + e], column_sum(part, i, e));
    __syncthreads();
    column_products(L, x_s, part);
    __syncthreads();
#pragma unroll
    for (int e = 4 * quarter; e < 4 * quarter + 4; ++e) ws[WS_A + (c0 + e) * D + i] = column_sum(part, i, e);
}

// One-sided Jacobi.  A sweep rotates every pair of the 128 columns once, in 127 steps of 64 disjoint pairs.  The columns stand in 16
// blocks of eight, two blocks in the shared memory of each of the cluster's CTAs.  A sweep is seven steps within the blocks, then 15
// rounds (round-robin) in which a CTA's two blocks meet, eight steps each; at a round's end the blocks go to their next CTA by
// stores to its shared memory, into the buffer that it read the round before, and one cluster barrier.  16 lanes own a pair of columns,
// 8 rows each; the column of the first block stays in registers for the round.
// The angle is computed in fp32 (its error only delays convergence; where its operands leave the fp32 range, as for columns
// whose lengths differ by more than 1e5, in float64), the rotation from it in float64, so that it is orthogonal to rounding; the longer
// column goes to the block with the lower number, which speeds convergence up.
// What bounds it: the chain of a step, from the loads through the dot product, its sum over the lanes and the rotation to the
// stores and the barrier, 0.5 us, and the cluster barrier of a round, about 0.7 us.  8 heads of 32768 tokens, 8 sweeps: 560 us; one CTA per
// head, every step reading and writing the whole matrix in shared memory, 2.1 us per step and 2.2 ms for 9 sweeps; clusters of four 680 us.
// All three lengths and the cosine in the chain, 200 instead of 148 instructions per step: 596 us.  Not kept: a warp meeting two
// columns with two, the second pair of rotations from inner products carried through the first, 680 us (four rotations' scalar code
// in a row in every warp).
constexpr int JC = 8, JB = D / (2 * JC), J_THREADS = 16 * JB, J_ROUNDS = 2 * JC - 1;     // CTAs per cluster, columns per block
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ float fast_rsqrt(float x) { asm("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(x)); return x; }
__device__ __forceinline__ float fast_sqrt(float x) { asm("sqrt.approx.ftz.f32 %0, %0;" : "+f"(x)); return x; }
__device__ __forceinline__ float fast_rcp(float x) { asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(x)); return x; }
struct JacobiState { unsigned rotated; float max_t, max_cos; };          // of a sweep: any rotation; largest tangent and cosine seen
// A column is kept as a scale times a vector: the rotation by the angle of tangent t then takes one multiply-add per row, and its cosine,
// which goes to the scale, is not waited for.  up and down: the scale and its reciprocal; norm2: the column's squared length, carried along
// from rotation to rotation and summed anew for every sweep (its error only changes the angle, and the lengths hardly
// change in the sweeps that decide what counts as orthogonal), which leaves one dot product to a step.
struct __align__(16) ColumnState { double up, down, norm2, pad; };
__device__ __forceinline__ double sum16(double v, unsigned mask) {
#pragma unroll
    for (int o = 1; o <= 8; o <<= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}
__device__ __forceinline__ double squared(const double2 (&p)[4]) {
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) { a = fma(p[k].x, p[k].x, a); b = fma(p[k].y, p[k].y, b); }
    return a + b;
}
__device__ __forceinline__ void jacobi_rotate(double2 (&p)[4], double2 (&q)[4], ColumnState& sp, ColumnState& sq, bool p_first, JacobiState& st) {
    constexpr float TOL = 4e-15f;                    // cosine below which a pair counts as orthogonal (its rounding is about 1e-15)
    const double r = sq.up * sp.down, ir = sp.up * sq.down, z = sq.norm2 - sp.norm2, both = sp.up * sq.up;
    const float zf = static_cast<float>(z), zz = zf * zf, len = fast_rsqrt(static_cast<float>(sp.norm2)) * fast_rsqrt(static_cast<float>(sq.norm2));
    double g0 = 0.0, g1 = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) { g0 = fma(p[k].x, q[k].x, g0); g1 = fma(p[k].y, q[k].y, g1); }
    const double g = sum16(g0 + g1, 0xffffffffu) * both;
    const float g2f = static_cast<float>(g + g);
    const float square = fmaf(g2f, g2f, zz);
    float cosine = 0.5f * fabsf(g2f) * len;
    const float ratio = g2f * fast_rcp(fabsf(zf) + fast_sqrt(square));
    float tf = zf < 0.f ? -ratio : ratio;
    double t = static_cast<double>(tf);
    bool turn = cosine > TOL;
    if (!(square > 1e-30f && square < 1e30f && fabsf(g2f) > 1e-35f && cosine <= 2.f)) {
        // nothing to turn by, columns of length 0, or numbers that fp32 does not hold: from tan = 1 / (zeta + sign sqrt(zeta^2 + 1))
        const unsigned half = 0xffffu << (threadIdx.x & 16);
        const double alpha = sum16(squared(p), half) * sp.up * sp.up, beta = sum16(squared(q), half) * sq.up * sq.up;
        turn = fabs(g) > static_cast<double>(TOL) * (sqrt(alpha) * sqrt(beta));
        if (turn) {
            const double zeta = z / (2.0 * g);
            t = fabs(zeta) < 1e150 ? copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0))) : fmin(fmax(g / z, -1.0), 1.0);
            tf = static_cast<float>(t);
        }
        cosine = 2.f;
    }
    if (!turn) return;
    st.rotated = 1u;
    st.max_t = fmaxf(st.max_t, fabsf(tf));
    st.max_cos = fmaxf(st.max_cos, cosine);
    const double tp = -t * r, tq = t * ir;           // p - t q and q + t p, of the scaled vectors
    const bool swap = (z >= 0.0) == p_first;         // the longer column is to be p, or q where the first block is q's
    if (swap) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 x = p[k], w = q[k];
            p[k] = make_double2(fma(tq, x.x, w.x), fma(tq, x.y, w.y));
            q[k] = make_double2(fma(tp, w.x, x.x), fma(tp, w.y, x.y));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 x = p[k], w = q[k];
            p[k] = make_double2(fma(tp, w.x, x.x), fma(tp, w.y, x.y));
            q[k] = make_double2(fma(tq, x.x, w.x), fma(tq, x.y, w.y));
        }
    }
    // c = a^(-1/2), a = 1 + t^2: an fp32 value y and one step of third order, which leaves the cube of its error.  With e = 1 - a y^2,
    // c = y (1 - e)^(-1/2), and the binomial series of that root begins 1 + e / 2 + 3 e^2 / 8.
    const double a = fma(t, t, 1.0), y = static_cast<double>(fast_rsqrt(fmaf(tf, tf, 1.f))), e = fma(-a * y, y, 1.0);
    const double c = fma(y * e, fma(0.375, e, 0.5), y), ic = a * c;
    const ColumnState np = {sp.up * c, sp.down * ic, fma(-t, g, sp.norm2), 0.0}, nq = {sq.up * c, sq.down * ic, fma(t, g, sq.norm2), 0.0};
    sp = swap ? nq : np;
    sq = swap ? np : nq;
}
constexpr size_t JACOBI_SMEM = 4 * JB * D * sizeof(double);
__global__ void __cluster_dims__(JC, 1, 1) __launch_bounds__(J_THREADS) jacobi_kernel(double* wsall, int* status) {
    extern __shared__ __align__(16) double S[];
    double2 (*buf)[2][JB][D / 2] = reinterpret_cast<double2 (*)[2][JB][D / 2]>(S);       // [parity][first, second block][column][rows]
    __shared__ ColumnState col_s[2][2][JB];
    __shared__ JacobiState state_s[2][32];                               // [sweep's parity][CTA and warp]
    static_assert(JC * J_THREADS == 1024, "a lane per warp of the cluster");
    const int h = blockIdx.x / JC, cta = blockIdx.x % JC, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, pair = tid >> 4, l16 = tid & 15;
    double* ws = wsall + h * WS_HEAD;
    if (ws[META_FAIL] != 0.0) return;                // (all CTAs of the cluster)
    const double2* C = reinterpret_cast<const double2*>(ws + WS_W);
    // CTA c holds positions c and 15 - c.  After a round the block at position 1 .. 14 moves one position up, that at 15 to 1.
    for (int n = tid; n < 2 * JB * D / 2; n += J_THREADS) {
        const int which = n / (JB * D / 2), block = which ? 2 * JC - 1 - cta : cta;
        (&buf[0][which][0][0])[n % (JB * D / 2)] = C[block * (JB * D / 2) + n % (JB * D / 2)];
    }
    cluster_barrier();
    const int first_cta = cta == 0 || cta == JC - 1 ? cta : cta + 1, first_which = cta == JC - 1 ? 1 : 0;
    const int second_cta = cta == 0 ? 1 : cta - 1, second_which = cta == 0 ? 0 : 1;
    int parity = 0, sweep = 0;
#pragma unroll 1
    for (;; ++sweep) {
        JacobiState st = {0u, 0.f, 0.f};
        double2 p[4], q[4];
#pragma unroll 1
        for (int which = 0; which < 2; ++which) {
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) p[k4] = buf[parity][which][pair][l16 + 16 * k4];
            const double norm2 = sum16(squared(p), 0xffffffffu);
            if (l16 == 0) col_s[parity][which][pair] = {1.0, 1.0, norm2, 0.0};
        }
        __syncthreads();
#pragma unroll 1
        for (int step = 0; step < JB - 1; ++step) {                      // within the blocks: pairs 0 .. 3 of the first, 4 .. 7 of the second
            auto player = [&](int pos) { int x = pos - 1 - step; if (x < 0) x += JB - 1; return pos == 0 ? 0 : 1 + x; };
            const int k = pair & (JB / 2 - 1), which = pair / (JB / 2), pa = player(k), pb = player(JB - 1 - k), lo = min(pa, pb), hi = max(pa, pb);
            double2 *pp = buf[parity][which][lo] + l16, *qq = buf[parity][which][hi] + l16;
            ColumnState sp = col_s[parity][which][lo], sq = col_s[parity][which][hi];
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) { p[k4] = pp[16 * k4]; q[k4] = qq[16 * k4]; }
            jacobi_rotate(p, q, sp, sq, true, st);
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) { pp[16 * k4] = p[k4]; qq[16 * k4] = q[k4]; }
            if (l16 == 0) { col_s[parity][which][lo] = sp; col_s[parity][which][hi] = sq; }
            __syncthreads();
        }
#pragma unroll 1
        for (int round = 0; round < J_ROUNDS; ++round, parity ^= 1) {
            auto block_at = [&](int pos) { int x = pos - 1 - round; if (x < 0) x += J_ROUNDS; return pos == 0 ? 0 : 1 + x; };
            const bool p_first = block_at(cta) < block_at(2 * JC - 1 - cta);
            ColumnState sp = col_s[parity][0][pair], sq;
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) p[k4] = buf[parity][0][pair][l16 + 16 * k4];
#pragma unroll 1
            for (int step = 0; step < JB; ++step) {
                const int column = (pair + step) & (JB - 1);
                double2* qq = buf[parity][1][column] + l16;
                sq = col_s[parity][1][column];
#pragma unroll
                for (int k4 = 0; k4 < 4; ++k4) q[k4] = qq[16 * k4];
                jacobi_rotate(p, q, sp, sq, p_first, st);
                if (step == JB - 1) break;
#pragma unroll
                for (int k4 = 0; k4 < 4; ++k4) qq[16 * k4] = q[k4];
                if (l16 == 0) col_s[parity][1][column] = sq;
                __syncthreads();
            }
            auto send = [&](const double2 (&x)[4], const ColumnState& s, int to, int which, int column) {
                const unsigned a = cluster_addr(&buf[parity ^ 1][which][column][l16], to);
#pragma unroll
                for (int k4 = 0; k4 < 4; ++k4)
                    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a + 256u * k4), "d"(s.up * x[k4].x), "d"(s.up * x[k4].y) : "memory");
                if (l16 == 0)
                    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %1};\nst.shared::cluster.f64 [%0 + 16], %2;"
                                 ::"r"(cluster_addr(&col_s[parity ^ 1][which][column], to)), "d"(1.0), "d"(s.norm2) : "memory");
            };
            send(p, sp, first_cta, first_which, pair);
            send(q, sq, second_cta, second_which, (pair + JB - 1) & (JB - 1));
            if (round == J_ROUNDS - 1) {             // what this warp saw, to every CTA of the cluster
                __syncwarp();
                const unsigned rot = __reduce_or_sync(0xffffffffu, st.rotated);
                const unsigned mt = __reduce_max_sync(0xffffffffu, __float_as_uint(st.max_t)), mc = __reduce_max_sync(0xffffffffu, __float_as_uint(st.max_cos));
                if (lane < JC) {
                    const unsigned a = cluster_addr(&state_s[sweep & 1][J_THREADS / 32 * cta + warp], lane);
                    asm volatile("st.shared::cluster.u32 [%0], %1;\nst.shared::cluster.u32 [%0 + 4], %2;\nst.shared::cluster.u32 [%0 + 8], %3;"
                                 ::"r"(a), "r"(rot), "r"(mt), "r"(mc) : "memory");
                }
            }
            cluster_barrier();
        }
        const JacobiState s = state_s[sweep & 1][lane];
        if (__reduce_or_sync(0xffffffffu, s.rotated) == 0u) break;
        // A pair that a sweep made orthogonal is disturbed by the sweep's later rotations of its columns: each adds less than
        // 2 max(t, cos) cos to its cosine.  Where 254 of them stay below the threshold there is nothing left to rotate.
        const float mt = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(s.max_t))), mc = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(s.max_cos)));
        if (sweep == 29 || 508.f * fmaxf(mt, mc) * mc < 4e-15f) { ++sweep; break; }
    }
    if (cta == 0 && tid == 0) ws[META_SWEEPS] = sweep;
    // eigenvalues, and the sign that makes an eigenvector's largest entry positive (of equal ones the first)
    const double tr = ws[META_TR_A];
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        const int slot = JB * (which ? 2 * JC - 1 - cta : cta) + pair;
        const double2* x = buf[parity][which][pair] + l16;
        double len2 = 0.0, top = -1.0;               // the largest magnitude, its row, whether it is negative
        int at = 0;
        bool negative = false;
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
            const double2 v = x[16 * k4];
            len2 = fma(v.x, v.x, fma(v.y, v.y, len2));
            const double mx = fabs(v.x), my = fabs(v.y);
            if (mx > top) { top = mx; at = 2 * (l16 + 16 * k4); negative = v.x < 0.0; }
            if (my > top) { top = my; at = 2 * (l16 + 16 * k4) + 1; negative = v.y < 0.0; }
        }
#pragma unroll
        for (int o = 1; o <= 8; o <<= 1) {
            len2 += __shfl_xor_sync(0xffffffffu, len2, o);
            const double v = __shfl_xor_sync(0xffffffffu, top, o);
            const int row = __shfl_xor_sync(0xffffffffu, at, o), sign = __shfl_xor_sync(0xffffffffu, static_cast<int>(negative), o);
            if (v > top || (v == top && row < at)) { top = v; at = row; negative = sign != 0; }
        }
        if (l16 == 0) {
            ws[META_EIG + slot] = len2 * tr;
            ws[META_SCALE + slot] = (negative ? -1.0 : 1.0) / sqrt(len2);
            if (!(len2 > 0.0)) { atomicOr(status, WUSHKV_ENOTPD); ws[META_FAIL] = 1.0; }
        }
    }
    // W row by row: transform_kernel's threads own columns
    for (int n = tid; n < 2 * JB * D; n += J_THREADS) {
        const int which = n / (JB * D), k = n / JB % D, column = n % JB;
        ws[WS_A + k * D + JB * (which ? 2 * JC - 1 - cta : cta) + column] = reinterpret_cast<const double*>(buf[parity][which][column])[k];
    }
}

// Columns 16 blockIdx.x .. of T = c Had Lam^(-1/4) U^T L^T, rounded to bf16: thread (i, half) holds row i of eight of them, which is
// scale_i sum_k W[k][order_i] L[j][k]; then a fast Walsh-Hadamard transform over the rows.  grid (8, heads), 256 threads.
__global__ void __launch_bounds__(256) transform_kernel(double gamma, const double* __restrict__ wsall, float* __restrict__ Tall) {
    __shared__ __align__(16) double l_s[D][COLS];
    __shared__ double y_s[D][COLS + 1], eig_s[D];
    __shared__ int order_s[D];
    __shared__ double sum_s;
    const int h = blockIdx.y, c0 = COLS * blockIdx.x, tid = threadIdx.x, i = tid & (D - 1), half = tid >> 7, lane = tid & 31;
    const double* ws = wsall + h * WS_HEAD;
    if (ws[META_FAIL] != 0.0) return;
    if (tid < D) eig_s[tid] = ws[META_EIG + tid];
    for (int n = tid; n < D * COLS; n += 256) l_s[n & (D - 1)][n >> 7] = ws[WS_L + (c0 + (n >> 7)) * D + (n & (D - 1))];
    __syncthreads();
    if (tid < D) {
        const double mine = eig_s[tid];
        int rank = 0;
#pragma unroll 16
        for (int j = 0; j < D; ++j) rank += (eig_s[j] < mine) || (eig_s[j] == mine && j < tid);
        order_s[rank] = tid;
    }
    if (tid >= 224) {
        const double sum = warp_sum((sqrt(eig_s[lane]) + sqrt(eig_s[lane + 32])) + (sqrt(eig_s[lane + 64]) + sqrt(eig_s[lane + 96])));
        if (lane == 0) sum_s = sum;
    }
    __syncthreads();
    const int slot = order_s[i];
    const double hn = sqrt(1.0 + gamma) * sqrt(ws[META_TR_M]) / sqrt(sum_s) / sqrt(static_cast<double>(D));
    const double scale = ws[META_SCALE + slot] * pow(eig_s[slot], -0.25);
    const double* W = ws + WS_A + slot;
    double acc[8] = {};
#pragma unroll
    for (int k0 = 0; k0 < D; k0 += 32) {
        double f[32];
#pragma unroll
        for (int n = 0; n < 32; ++n) f[n] = W[(k0 + n) * D];
#pragma unroll
        for (int n = 0; n < 32; ++n) {
            const double2* b = reinterpret_cast<const double2*>(&l_s[k0 + n][8 * half]);
#pragma unroll
            for (int e = 0; e < 4; ++e) { const double2 v = b[e]; acc[2 * e] = fma(f[n], v.x, acc[2 * e]); acc[2 * e + 1] = fma(f[n], v.y, acc[2 * e + 1]); }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        double x = scale * acc[e];
#pragma unroll
        for (int o = 1; o <= 16; o <<= 1) {
            const double y = __shfl_xor_sync(0xffffffffu, x, o);
            x = lane & o ? y - x : x + y;
        }
        y_s[i][8 * half + e] = x;
    }
    __syncthreads();
    float* T = Tall + static_cast<long long>(h) * D * D + i * D + c0 + 8 * half;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int column = 8 * half + e;
        const double x0 = y_s[lane][column], x1 = y_s[lane + 32][column], x2 = y_s[lane + 64][column], x3 = y_s[lane + 96][column];
        const double u = i & 32 ? x0 - x1 : x0 + x1, v = i & 32 ? x2 - x3 : x2 + x3;
        T[e] = static_cast<float>(round_double_to_bf16(hn * (i & 64 ? u - v : u + v)));
    }
}

// (T^-1)^T by Gauss-Jordan elimination in place, pivots within columns, panels of 16 columns.  The matrix stands in shared memory column
// by column.  Thread i < 128 eliminates with row i of the panel in registers; every warp's candidate for a pivot hands out its row of the
// panel and the warps agree on the best after the barrier, one per column.  What the panel has become are the factors by which the pivots'
// rows are added to all other columns: a 128 x 112 x 16 product of all warps.  Rows are not moved: row piv[c] stands for row c of
// the permuted matrix, whose inverse has its columns in the order piv.  One CTA per head; bound by the chain of a column's steps.  (Column by column,
// the matrix in registers, with two barriers of 16 warps for each: 165 to 185 us for 8 heads, this 75.)
constexpr int INV_PITCH = D + 1;
constexpr size_t INVERSE_SMEM = (static_cast<size_t>(BT_PANEL) * BT_PITCH + static_cast<size_t>(D) * INV_PITCH) * sizeof(double);
__global__ void __launch_bounds__(BT_THREADS) inverse_kernel(const float* __restrict__ Tall, float* __restrict__ Tinvall, const double* wsall, int* status) {
    extern __shared__ __align__(16) double R[];      // the pivots' rows as they were before the panel, then the matrix
    double* S = R + BT_PANEL * BT_PITCH;
    __shared__ __align__(16) double row_s[2][4][BT_PANEL];
    __shared__ __align__(16) unsigned key_s[2][4];
    __shared__ int piv_s[D], pos_s[D], fail_s;
    const int h = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (wsall[h * WS_HEAD + META_FAIL] != 0.0) return;
    const float* T = Tall + static_cast<long long>(h) * D * D;
#pragma unroll 16
    for (int idx = tid; idx < D * D; idx += BT_THREADS) S[(idx & 127) * INV_PITCH + (idx >> 7)] = static_cast<double>(T[idx]);
    if (tid < D) pos_s[tid] = -1;
    if (tid == 0) fail_s = 0;
    __syncthreads();
    bool used = false;
#pragma unroll 1
    for (int k0 = 0; k0 < D; k0 += BT_PANEL) {
        if (tid < D) {
            double a[BT_PANEL];
#pragma unroll
            for (int e = 0; e < BT_PANEL; ++e) a[e] = S[(k0 + e) * INV_PITCH + tid];
#pragma unroll
            for (int c = 0; c < BT_PANEL; ++c) {
                const unsigned key = used ? 0u : (static_cast<unsigned>(__double2hiint(a[c])) & 0x7fffff80u) | (127u - tid);
                const unsigned mine = __reduce_max_sync(0xffffffffu, key);
                if (key == mine) {                   // (several where the warp has no row left, or row 127's key is 0: then it does not matter)
#pragma unroll
                    for (int e = 0; e < BT_PANEL; ++e) row_s[c & 1][warp][e] = a[e];
                }
                if (lane == 0) key_s[c & 1][warp] = mine;
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const uint4 k = *reinterpret_cast<const uint4*>(key_s[c & 1]);
                const unsigned best = max(max(k.x, k.y), max(k.z, k.w));
                const int piv = 127 - (best & 127u); // the largest entry to 13 bits of its mantissa
                if (best < 0x80u || best >= 0x7ff00000u) fail_s = 1;     // zero or not finite
                const double* row = row_s[c & 1][piv >> 5];
                const double inv = 1.0 / row[c];
                if (tid == piv) {
                    used = true;
                    piv_s[k0 + c] = piv;
                    pos_s[piv] = k0 + c;
#pragma unroll
                    for (int e = 0; e < BT_PANEL; ++e) a[e] *= inv;
                    a[c] = inv;
                } else {
                    const double f = a[c] * inv;
#pragma unroll
                    for (int e = 0; e < BT_PANEL; ++e) a[e] = fma(-f, row[e], a[e]);
                    a[c] = -f;
                }
            }
#pragma unroll
            for (int e = 0; e < BT_PANEL; ++e) S[(k0 + e) * INV_PITCH + tid] = a[e];
        }
        __syncthreads();
        if (fail_s) {                                // (the same for all threads)
            if (tid == 0) atomicOr(status, WUSHKV_ENOTPD);
            return;
        }
        for (int n = tid; n < BT_PANEL * D; n += BT_THREADS) R[(n >> 7) * BT_PITCH + (n & 127)] = S[(n & 127) * INV_PITCH + piv_s[k0 + (n >> 7)]];
        __syncthreads();
        bool pivot[4];                               // rows lane + 32 r
#pragma unroll
        for (int r = 0; r < 4; ++r) pivot[r] = pos_s[lane + 32 * r] >= k0;
#pragma unroll 1
        for (int unit = warp; unit < (D - BT_PANEL) / 4; unit += BT_THREADS / 32) {      // all rows of four columns
            const int j = 4 * unit < k0 ? 4 * unit : 4 * unit + BT_PANEL;
            double acc[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[r][e] = pivot[r] ? 0.0 : S[(j + e) * INV_PITCH + lane + 32 * r];
#pragma unroll 4
            for (int c = 0; c < BT_PANEL; ++c) {
                const double2 u = *reinterpret_cast<const double2*>(R + c * BT_PITCH + j), v = *reinterpret_cast<const double2*>(R + c * BT_PITCH + j + 2);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const double x = S[(k0 + c) * INV_PITCH + lane + 32 * r];
                    acc[r][0] = fma(x, u.x, acc[r][0]); acc[r][1] = fma(x, u.y, acc[r][1]); acc[r][2] = fma(x, v.x, acc[r][2]); acc[r][3] = fma(x, v.y, acc[r][3]);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int e = 0; e < 4; ++e) S[(j + e) * INV_PITCH + lane + 32 * r] = acc[r][e];
        }
        __syncthreads();
    }
    // entry (c, piv[j]) of the inverse stands in row piv[c], column j
    float* Ti = Tinvall + static_cast<long long>(h) * D * D;
#pragma unroll 8
    for (int idx = tid; idx < D * D; idx += BT_THREADS) Ti[idx] = static_cast<float>(S[pos_s[idx >> 7] * INV_PITCH + piv_s[idx & 127]]);
}

}  // namespace
}  // namespace wushkv

using namespace wushkv;

extern "C" int wushkv_accumulate_gram_device(int32_t n_kv, int32_t n_q, int32_t d, int64_t n_tok, const uint16_t* K, const uint16_t* Q,
                                             double* M, double* H, void* stream) {
    if (!K || !Q || !M || !H || n_kv <= 0 || n_q <= 0 || d != D || n_tok < 0 || n_q % n_kv != 0) return WUSHKV_EINVAL;
    if (!aligned(K, 16) || !aligned(Q, 16) || !aligned(M, 8) || !aligned(H, 8)) return WUSHKV_EINVAL;
    if (n_tok == 0) return WUSHKV_OK;
    if (n_tok > 0x7fffffffLL * 2048) return WUSHKV_EINVAL;
    GramParams P;
    P.n_kv = n_kv; P.n_q = n_q; P.M = M; P.H = H;
    P.wait_limit = knobs().wait_limit > 0 ? static_cast<int>(std::min(knobs().wait_limit, 1LL << 20)) : 1 << 20;      // about a second
    P.drop = knobs().drop_gram;
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(gram_kernel), static_cast<int>(GRAM_SMEM))) return WUSHKV_ECUDA;
    constexpr long long LAUNCH_TOK = 1LL << 29;      // keeps rows and a CTA's units within 32 bits
    for (long long t0 = 0; t0 < n_tok; t0 += LAUNCH_TOK) {
        P.K = K + t0 * n_kv * D; P.Q = Q + t0 * n_q * D;
        P.n_tok = std::min(LAUNCH_TOK, n_tok - t0);
        P.groups = (P.n_tok + GR_TOK - 1) / GR_TOK;
        P.units = P.groups * (static_cast<long long>(n_kv) + n_q);
        CUtensorMap k_map, q_map;
        const bool mk = make_row_tensor_map(k_map, true, P.K, n_kv, P.n_tok, GR_TOK), mq = make_row_tensor_map(q_map, true, P.Q, n_q, P.n_tok, GR_TOK);
        P.use_tma = mk && mq && !knobs().gram_no_tma;
        const unsigned ctas = static_cast<unsigned>(P.units < sm_count() ? P.units : sm_count());
        gram_kernel<<<ctas, GR_THREADS, GRAM_SMEM, static_cast<cudaStream_t>(stream)>>>(P, k_map, q_map);
    }
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
    if (!opt_in_dynamic_smem(reinterpret_cast<const void*>(factor_kernel<false>), static_cast<int>(FACTOR_SMEM)) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(factor_kernel<true>), static_cast<int>(FACTOR_SMEM)) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(jacobi_kernel), static_cast<int>(JACOBI_SMEM)) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(congruence_kernel), static_cast<int>(CONGRUENCE_SMEM)) ||
        !opt_in_dynamic_smem(reinterpret_cast<const void*>(inverse_kernel), static_cast<int>(INVERSE_SMEM)))
        return WUSHKV_ECUDA;
    double* ws = static_cast<double*>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (int h0 = 0; h0 < n_heads; h0 += BT_MAX_HEADS) {                 // (the heads are a grid's second dimension in two kernels)
        const int n = n_heads - h0 < BT_MAX_HEADS ? n_heads - h0 : BT_MAX_HEADS;
        const long long m = static_cast<long long>(h0) * D * D;
        double* w = ws + h0 * WS_HEAD;
        factor_kernel<false><<<n, BT_THREADS, FACTOR_SMEM, st>>>(M + m, H + m, gamma, w, dev_status);
        congruence_kernel<<<dim3(D / COLS, n), BT_THREADS, CONGRUENCE_SMEM, st>>>(M + m, gamma, w);
        factor_kernel<true><<<n, BT_THREADS, FACTOR_SMEM, st>>>(M + m, H + m, gamma, w, dev_status);
        jacobi_kernel<<<n * JC, J_THREADS, JACOBI_SMEM, st>>>(w, dev_status);
        transform_kernel<<<dim3(D / COLS, n), 256, 0, st>>>(gamma, w, T + m);
        inverse_kernel<<<n, BT_THREADS, INVERSE_SMEM, st>>>(T + m, T_invT + m, w, dev_status);
    }
    return cudaGetLastError() == cudaSuccess ? WUSHKV_OK : WUSHKV_ECUDA;
}
