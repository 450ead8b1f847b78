// CUR assembly (Section 1.1: C = A(:,J), U = A(I,J)^dagger, R = A(I,:)) and the
// residual of the cross (Theorem 1's Chebyshev norm max|A - CUR| and the relative
// Frobenius error of Section 3.1).
//
// The residual reads A exactly once. W = U R (r x n) is formed first in FP64 and
// rounded to the arithmetic type; each CTA then owns a 128-row panel, keeps its
// C rows in shared memory and walks the panel's column tiles: E = A - C W on a
// 128 x 128 tile, with |E| max, sum E^2 and sum A^2 folded in the epilogue.

#include <algorithm>
#include <climits>
#include <cstring>

#include "common.cuh"
#include "gj.cuh"
#include "internal.h"

namespace curk {

constexpr double kEpsR = 2.220446049250313e-16;

template <typename TA>
__global__ void gather_C_k(const TA* __restrict__ A, int64_t m, int64_t n, int64_t ld,
                           const int32_t* __restrict__ J, int r, TA* __restrict__ C, int* status) {
    const int64_t total = m * r;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / r;
        const int64_t j = J[e - i * r];
        if (j < 0 || j >= n) { set_status(status, CUR_ERR_ARG); C[e] = A[0]; continue; }
        C[e] = A[i * ld + j];
    }
}

template <typename TA>
__global__ void gather_R_k(const TA* __restrict__ A, int64_t m, int64_t n, int64_t ld,
                           const int32_t* __restrict__ I, int r, TA* __restrict__ R, int* status) {
    const int64_t total = (int64_t)r * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = e / n, j = e - k * n;
        const int64_t i = I[k];
        if (i < 0 || i >= m) { set_status(status, CUR_ERR_ARG); R[e] = A[0]; continue; }
        R[e] = A[i * ld + j];
    }
}

// The usual case of the assembly above r = 44: U = A(I,J)^-1 in FP64 by one cluster (gj.cuh), its rcond in
// the 1-norm. Where the inverse does not stand (a singular or ill-conditioned M, indices out of
// range, data that are not finite) *redo is set and assemble_inv_k decides. colsum: r doubles.
// r = 128: 1220 us in assemble_inv_k.
template <typename TA, int RU, int CPW>
__global__ void __launch_bounds__(32 * kGjWarps) assemble_gj_k(const TA* __restrict__ A, int64_t m, int64_t n, int64_t ld,
                                                               const int32_t* __restrict__ I, const int32_t* __restrict__ J,
                                                               int r, double* __restrict__ U, double* rcond_out,
                                                               double* __restrict__ colsum, int* redo) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const GjSmem gs(smem_raw, r);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const unsigned rank = gj_rank();
    // every CTA: max |M|, the largest column sum (a warp per column) and whether M is usable
    double mx = 0.0, n1 = 0.0;
    int bad = 0;
    for (int b = tid >> 5; b < r; b += nt >> 5) {
        const int64_t j = J[b];
        double s = 0.0;
        for (int a = lane; a < r; a += 32) {
            const int64_t i = I[a];
            if (i < 0 || i >= m || j < 0 || j >= n) { bad = 1; continue; }
            const double x = fabs(to_d(A[i * ld + j]));
            if (!isfinite(x)) bad = 1;
            mx = fmax(mx, x);
            s += x;
        }
        n1 = fmax(n1, warp_sum(s));
    }
    bad = __syncthreads_or(bad);
    mx = block_max(mx);
    n1 = block_max(n1);
    if (bad) {   // every CTA of the cluster alike
        if (rank == 0 && tid == 0) *redo = 1;
        return;
    }
    int c0, nw;
    gj_columns(r, CPW, c0, nw);
    double v[CPW][RU];
#pragma unroll
    for (int q = 0; q < CPW; ++q)
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int i = lane + 32 * u;
            v[q][u] = q < nw && i < r ? to_d(A[(int64_t)I[i] * ld + J[c0 + q]]) : 0.0;
        }
    const int res = gj_flow<RU, CPW>(gs, r, (double)r * kEpsR * mx, v, c0, nw, nullptr);
    if (!res) {
#pragma unroll
        for (int q = 0; q < CPW; ++q)
            if (q < nw) {
                const int c = gs.perm[c0 + q];
                double s = 0.0;
#pragma unroll
                for (int u = 0; u < RU; ++u) {
                    const int i = lane + 32 * u;
                    if (i < r) U[(int64_t)i * r + c] = v[q][u];
                    if (i < r) s += fabs(v[q][u]);
                }
                s = warp_sum(s);
                if (lane == 0) colsum[c0 + q] = s;
            }
    }
    __threadfence();
    gj_cluster_sync();
    if (rank == 0) {
        double cs = 0.0;
        if (!res)
            for (int c = tid; c < r; c += nt) cs = fmax(cs, __ldcg(colsum + c));
        cs = block_max(cs);
        const double rc = 1.0 / (n1 * cs);
        if (tid == 0) {
            *redo = res != 0 || !(rc >= 1e-13);
            if (!*redo) *rcond_out = rc;
        }
    }
}

// Where *redo is set (or redo is null: always), one CTA: M = A(I,J) in FP64, LU with partial pivoting, inverse, rcond; if
// rcond < 1e-13 (or M is singular) the pseudo-inverse from a one-sided Jacobi SVD
// (round-robin pair order, one warp per pair) with cutoff r eps s_max.
// work: 3 r^2 doubles (global scratch).
template <typename TA>
__global__ void __launch_bounds__(256) assemble_inv_k(const TA* __restrict__ A, int64_t m,
                                                      int64_t n, int64_t ld,
                                                      const int32_t* __restrict__ I,
                                                      const int32_t* __restrict__ J, int r,
                                                      double* __restrict__ U, double* rcond_out,
                                                      double* __restrict__ work, int* status,
                                                      const int* __restrict__ redo) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (redo && !*redo) return;
    const int tid = threadIdx.x, nt = blockDim.x;
    double* M = reinterpret_cast<double*>(smem_raw);  // r x r, inverted in place
    double* colk = M + r * r;
    int* piv = reinterpret_cast<int*>(colk + r);
    double* X = work + r * r;    // r x r (Jacobi V)
    double* M0 = work + 2 * r * r;
    __shared__ int s_bad;
    __shared__ double s_max, s_n1, s_ni;
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int e = tid; e < r * r; e += nt) {
        const int a = e / r, b = e - a * r;
        const int64_t i = I[a], j = J[b];
        double x = 0.0;
        if (i < 0 || i >= m || j < 0 || j >= n) s_bad = 1;
        else x = to_d(A[i * ld + j]);
        if (!isfinite(x)) s_bad = 2;
        M[e] = x;
        M0[e] = x;
    }
    __syncthreads();
    if (s_bad) {
        if (tid == 0) {
            set_status(status, s_bad == 2 ? CUR_ERR_NONFINITE : CUR_ERR_ARG);
            *rcond_out = 0.0;
        }
        return;
    }
    {
        // max |M| and the 1-norm (largest column sum), one column per thread
        double mx = 0.0, cs = 0.0;
        for (int c = tid; c < r; c += nt) {
            double s = 0.0;
            for (int a = 0; a < r; ++a) { mx = fmax(mx, fabs(M[a * r + c])); s += fabs(M[a * r + c]); }
            cs = fmax(cs, s);
        }
        mx = block_max(mx);
        cs = block_max(cs);
        if (tid == 0) { s_max = mx; s_n1 = cs; }
        __syncthreads();
    }
    const int sing = gj_inverse(M, r, colk, piv, (double)r * kEpsR * s_max, nullptr);
    bool use_pinv = sing != 0;
    if (!use_pinv) {
        double cs = 0.0;
        for (int c = tid; c < r; c += nt) {
            double s = 0.0;
            for (int a = 0; a < r; ++a) s += fabs(M[a * r + c]);
            cs = fmax(cs, s);
        }
        cs = block_max(cs);
        if (tid == 0) {
            s_ni = cs;
            *rcond_out = 1.0 / (s_n1 * cs);
        }
        __syncthreads();
        use_pinv = !(1.0 / (s_n1 * s_ni) >= 1e-13);
        if (!use_pinv) {
            for (int e = tid; e < r * r; e += nt) U[e] = M[e];
            return;
        }
    } else if (tid == 0) {
        *rcond_out = 0.0;
    }
    // ---- pseudo-inverse: one-sided Jacobi on the columns of M0, V accumulates rotations
    double* Aj = M0;
    double* V = X;
    for (int e = tid; e < r * r; e += nt) V[e] = ((e / r) == (e % r)) ? 1.0 : 0.0;
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    const int rr = (r % 2 == 0) ? r : r + 1;  // round-robin over an even count (phantom column)
    __shared__ int s_rot;
    for (int sweep = 0; sweep < 80; ++sweep) {
        if (tid == 0) s_rot = 0;
        __syncthreads();
        for (int step = 0; step < rr - 1; ++step) {
            for (int pr = warp; pr < rr / 2; pr += nw) {
                // pairs (a, b) of the round-robin schedule: position 0 fixed, others rotate
                int a, b;
                {
                    const int i1 = pr, i2 = rr - 1 - pr;
                    auto pos = [&](int i) { return i == 0 ? 0 : 1 + (i - 1 + step) % (rr - 1); };
                    a = pos(i1);
                    b = pos(i2);
                }
                if (a > b) { const int t = a; a = b; b = t; }
                if (b >= r) continue;
                double al = 0.0, be = 0.0, ga = 0.0;
                for (int i = lane; i < r; i += 32) {
                    const double x = Aj[i * r + a], y = Aj[i * r + b];
                    al = fma(x, x, al);
                    be = fma(y, y, be);
                    ga = fma(x, y, ga);
                }
                al = warp_sum(al);
                be = warp_sum(be);
                ga = warp_sum(ga);
                if (ga == 0.0 || fabs(ga) <= 1e-15 * sqrt(al * be)) continue;
                if (lane == 0) s_rot = 1;
                const double zeta = (be - al) / (2.0 * ga);
                const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
                for (int i = lane; i < r; i += 32) {
                    const double x = Aj[i * r + a], y = Aj[i * r + b];
                    Aj[i * r + a] = c * x - s * y;
                    Aj[i * r + b] = s * x + c * y;
                    const double vx = V[i * r + a], vy = V[i * r + b];
                    V[i * r + a] = c * vx - s * vy;
                    V[i * r + b] = s * vx + c * vy;
                }
            }
            __syncthreads();
        }
        const int rot = s_rot;
        __syncthreads();
        if (!rot) break;
    }
    // singular values, cutoff, U = V diag(1/s) Uhat^T with Uhat = Aj / s
    __shared__ double sv[128];
    for (int k = tid; k < r; k += nt) {
        double s = 0.0;
        for (int i = 0; i < r; ++i) s = fma(Aj[i * r + k], Aj[i * r + k], s);
        sv[k] = sqrt(s);
    }
    __syncthreads();
    if (tid == 0) {
        double smax = 0.0;
        for (int k = 0; k < r; ++k) smax = fmax(smax, sv[k]);
        s_max = (double)r * kEpsR * smax;
    }
    __syncthreads();
    for (int e = tid; e < r * r; e += nt) {
        const int i = e / r, j = e - i * r;
        double s = 0.0;
        for (int k = 0; k < r; ++k)
            if (sv[k] > s_max) s += V[i * r + k] * (Aj[j * r + k] / sv[k]) / sv[k];
        U[e] = s;
    }
}

// W = U R (r x n) in FP64, rounded to TW. One thread per column.
template <typename TA, typename TW>
__global__ void __launch_bounds__(256) residual_w_k(const double* __restrict__ U,
                                                   const TA* __restrict__ R, int r, int64_t n,
                                                   TW* __restrict__ W) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* Us = reinterpret_cast<double*>(smem_raw);
    for (int e = threadIdx.x; e < r * r; e += blockDim.x) Us[e] = U[e];
    __syncthreads();
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        double rc[128];
        for (int l = 0; l < r; ++l) rc[l] = to_d(R[(int64_t)l * n + j]);
        for (int k = 0; k < r; ++k) {
            double s = 0.0;
            for (int l = 0; l < r; ++l) s = fma(Us[k * r + l], rc[l], s);
            W[(int64_t)k * n + j] = (TW)s;
        }
    }
}

// N consecutive elements from 16-byte aligned memory as 16-byte loads.
template <typename T, int N>
__device__ __forceinline__ void ld_vec(const T* p, T (&x)[N]) {
    static_assert((N * sizeof(T)) % 16 == 0, "16-byte multiple");
    const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
    for (int c = 0; c < (int)(N * sizeof(T) / 16); ++c) {
        const uint4 v = q[c];
        memcpy(&x[c * (16 / sizeof(T))], &v, 16);
    }
}

// Residual tiles. TM x TN outputs per thread, 16 x 16 threads, tile (16 TM) x (16 TN).
// Grid: (panels, segments); CTA (p, s) takes rows [p*BM, p*BM+BM) and column tiles
// s, s + segs, ... Partials per CTA: max|E|, sum E^2, sum A^2, non-finite flag.
template <typename TA, typename TW, int TM, int TN>
__global__ void __launch_bounds__(256, 2) residual_k(const TA* __restrict__ A, int64_t m, int64_t n,
                                                  int64_t ld, const TA* __restrict__ C,
                                                  const TW* __restrict__ W, int r,
                                                  double* __restrict__ part, int vec) {
    constexpr int BM = 16 * TM, BN = 16 * TN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TW* Ct = reinterpret_cast<TW*>(smem_raw);  // r x BM (transposed C panel)
    TW* Ws = Ct + (size_t)r * BM;              // r x BN
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t r0 = (int64_t)blockIdx.x * BM;
    const int segs = gridDim.y;
    for (int e = threadIdx.x; e < BM * r; e += blockDim.x) {
        const int k = e / BM, i = e - k * BM;
        Ct[k * BM + i] = (r0 + i < m) ? (TW)to_d(C[(r0 + i) * r + k]) : (TW)0;
    }
    double mx = 0.0, se = 0.0, sa = 0.0;
    int bad = 0;
    const int64_t ntile = (n + BN - 1) / BN;
    for (int64_t tn = blockIdx.y; tn < ntile; tn += segs) {
        const int64_t c0 = tn * BN;
        __syncthreads();
        for (int e = threadIdx.x; e < BN * r; e += blockDim.x) {
            const int k = e / BN, j = e - k * BN;
            Ws[k * BN + j] = (c0 + j < n) ? W[(int64_t)k * n + c0 + j] : (TW)0;
        }
        __syncthreads();
        TW acc[TM][TN];
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int b = 0; b < TN; ++b) acc[a][b] = (TW)0;
#pragma unroll 4
        for (int k = 0; k < r; ++k) {
            TW x[TM], y[TN];
            ld_vec<TW, TM>(Ct + k * BM + ty * TM, x);
            // column pairs 2 tx + 32 b (+1): a half-warp reads 128 contiguous bytes per load
#pragma unroll
            for (int b = 0; b < TN / 2; ++b) {
                const TW* q = Ws + k * BN + 2 * tx + 32 * b;
                y[2 * b] = q[0];
                y[2 * b + 1] = q[1];
            }
#pragma unroll
            for (int a = 0; a < TM; ++a)
#pragma unroll
                for (int b = 0; b < TN; ++b) acc[a][b] = fma(x[a], y[b], acc[a][b]);
        }
        TW tmx = (TW)0, tse = (TW)0, tsa = (TW)0;
#pragma unroll
        for (int a = 0; a < TM; ++a) {
            const int64_t i = r0 + ty * TM + a;
            if (i >= m) continue;
            const TA* arow = A + i * ld + c0;
            TA araw[TN];
#pragma unroll
            for (int b = 0; b < TN; ++b) {
                const int64_t cc = 2 * tx + 32 * (b >> 1) + (b & 1);
                araw[b] = (c0 + cc < n) ? arow[cc] : arow[0];
            }
#pragma unroll
            for (int b = 0; b < TN; ++b) {
                if (c0 + 2 * tx + 32 * (b >> 1) + (b & 1) >= n) continue;
                const TW av = (TW)to_d(araw[b]);
                const TW e = av - acc[a][b];
                if (!(fabs(e) <= (TW)INFINITY)) bad = 1;
                tmx = fmax(tmx, fabs(e));
                tse = fma(e, e, tse);
                tsa = fma(av, av, tsa);
            }
        }
        mx = fmax(mx, (double)tmx);
        se += (double)tse;
        sa += (double)tsa;
    }
    // CTA reduction
    __shared__ double rmx[8], rse[8], rsa[8];
    __shared__ int rbad;
    if (threadIdx.x == 0) rbad = 0;
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        se += __shfl_xor_sync(0xffffffffu, se, o);
        sa += __shfl_xor_sync(0xffffffffu, sa, o);
    }
    __syncthreads();
    if (bad) rbad = 1;
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { rmx[warp] = mx; rse[warp] = se; rsa[warp] = sa; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a1 = 0.0, a2 = 0.0, a3 = 0.0;
        for (int w = 0; w < 8; ++w) { a1 = fmax(a1, rmx[w]); a2 += rse[w]; a3 += rsa[w]; }
        const int64_t cta = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
        part[cta * 4 + 0] = a1;
        part[cta * 4 + 1] = a2;
        part[cta * 4 + 2] = a3;
        part[cta * 4 + 3] = rbad ? 1.0 : 0.0;
    }
}

// ---- the same residual for FP32 and BF16 data at the FP32 FMA rate
//
// Every element is the FP32 FMA chain over k of residual_k and every 8 x 8 group of a tile folds
// the same 64 elements in the same order, so max|E| and the tile sums are bit-identical to it.
// What bounds it is the FMA pipe: m n r FMAs, 14.7 ms at 262144 x 16384, r = 128 (residual_k
// took 77.6 ms: it staged W with plain loads between barriers, one CTA per SM at r = 128, so
// that the loads, the FMAs and the reads of A followed one another). Here
//   * two CTAs per SM: one CTA's reads of A and its partial sums run under the other's FMAs;
//   * W comes by cp.async in chunks of 32 k, two stages, during the chunk before;
//   * a thread has two of residual_k's groups, 16 rows x 8 columns, and its FMAs are pairs
//     (fma.rn.f32x2, each half rounded as fmaf) of two rows of C times one column of W: per k
//     64 of them for 4 + 4 loads from shared memory. (With 8 x 8 per thread and W stored
//     twice over for ready pairs, 2 + 4 16-byte loads per 32 pairs, the loads took 1.2 times
//     the FMAs' time: 28.5 ms.)
//   * CTAs walk contiguous ranges of tiles along row panels and keep the C panel.
constexpr int kRfB = 128;    // rows and columns of a tile; 8 x 16 threads, 16 x 8 each
constexpr int kRfKC = 32;    // k per stage of W
constexpr int kRfT = 128;    // threads

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// W = U R summed in FP64 (one chain over l) and rounded to FP32 as residual_w_k does, rows of
// npad columns, zeros past n. A block takes 32 columns and kRfWK rows k; a thread 4 k x 2 j
// (eight FP64 chains; the FP64 pipe bounds it: r^2 n DFMAs).
constexpr int kRfWK = 64;
template <typename TA>
__global__ void __launch_bounds__(256) residual_w2_k(const double* __restrict__ U, const TA* __restrict__ R, int r,
                                                     int64_t n, int64_t npad, float* __restrict__ W) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* Us = reinterpret_cast<double*>(smem_raw);   // Us[l * 64 + k] = U(k0 + k, l)
    double* Rs = Us + (size_t)r * kRfWK;                // Rs[l * 32 + jj] = R(l, j0 + jj)
    const int64_t j0 = (int64_t)blockIdx.x * 32;
    const int k0 = blockIdx.y * kRfWK;
    for (int e = threadIdx.x; e < r * kRfWK; e += blockDim.x) {
        const int k = e / r, l = e - k * r;
        Us[l * kRfWK + k] = k0 + k < r ? U[(int64_t)(k0 + k) * r + l] : 0.0;
    }
    for (int e = threadIdx.x; e < r * 32; e += blockDim.x) {
        const int l = e >> 5, jj = e & 31;
        Rs[e] = j0 + jj < n ? to_d(R[(int64_t)l * n + j0 + jj]) : 0.0;
    }
    __syncthreads();
    const int jg = threadIdx.x & 15, kg = threadIdx.x >> 4;
    double acc[4][2] = {};
    for (int l = 0; l < r; ++l) {
        const double2 ua = *reinterpret_cast<const double2*>(Us + l * kRfWK + 4 * kg);
        const double2 ub = *reinterpret_cast<const double2*>(Us + l * kRfWK + 4 * kg + 2);
        const double2 rr = *reinterpret_cast<const double2*>(Rs + l * 32 + 2 * jg);
        const double u4[4] = {ua.x, ua.y, ub.x, ub.y};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i][0] = fma(u4[i], rr.x, acc[i][0]);
            acc[i][1] = fma(u4[i], rr.y, acc[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = k0 + 4 * kg + i;
        const int64_t j = j0 + 2 * jg;
        if (k >= r || j >= npad) continue;
        const float a = j < n ? (float)acc[i][0] : 0.f, b = j + 1 < n ? (float)acc[i][1] : 0.f;
        *reinterpret_cast<float2*>(W + (int64_t)k * npad + j) = make_float2(a, b);
    }
}

// WHOLE: m and n are multiples of the tile and A lies on pairs, so that the kernel has no code for ends and
// keeps its registers for the sums: 262144 x 16384 BF16, r = 128, 21.9 ms, with ends 23.8; FP32
// 65536 x 8192, r = 100, 2.44 and 2.60.
template <typename TA, bool WHOLE>
__global__ void __launch_bounds__(kRfT, 2) residual_fma_k(const TA* __restrict__ A, int64_t m, int64_t n, int64_t ld,
                                                          const TA* __restrict__ C, const float* __restrict__ W,
                                                          int64_t npad, int r, int64_t ntile_n, int64_t ntiles,
                                                          double* __restrict__ part, int pairs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* Ws = reinterpret_cast<float*>(smem_raw);   // two stages of kRfKC x 128
    float* Ct = Ws + 2 * kRfKC * kRfB;                // r x 128 (transposed C panel)
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = ntiles * blockIdx.x / gridDim.x, t1 = ntiles * (blockIdx.x + 1) / gridDim.x;
    const int nchunk = (r + kRfKC - 1) / kRfKC;
    double mx = 0.0, se = 0.0, sa = 0.0;
    int bad = 0;
    // chunk c of the column tile ct into stage s: row k is 512 bytes, one warp's 16-byte copies
    auto load = [&](int64_t ct, int c, int s) {
        const float* src = W + ct * kRfB + 4 * lane;
#pragma unroll
        for (int x = 0; x < kRfKC / 4; ++x) {
            const int kk = 4 * x + warp, k = c * kRfKC + kk;
            if (k < r) cp_async16(Ws + (s * kRfKC + kk) * kRfB + 4 * lane, src + (int64_t)k * npad);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int64_t panel = -1;
    int stage = 0;
    if (t0 < t1) load(t0 % ntile_n, 0, 0);
    for (int64_t t = t0; t < t1; ++t) {
        const int64_t pn = t / ntile_n, ct = t - pn * ntile_n;
        const int64_t r0 = pn * kRfB, c0 = ct * kRfB;
        if (pn != panel) {
            panel = pn;
            __syncthreads();
            for (int e = tid; e < kRfB * r; e += kRfT) {
                const int k = e / kRfB, i = e - k * kRfB;
                Ct[e] = r0 + i < m ? to_f(C[(r0 + i) * r + k]) : 0.f;
            }
        }
        uint64_t acc[8][8];   // rows 2 a, 2 a + 1 of the thread's sixteen, column b
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = 0ull;
        for (int c = 0; c < nchunk; ++c, stage ^= 1) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();   // this chunk has landed, and the other stage has been read
            if (c + 1 < nchunk) load(ct, c + 1, stage ^ 1);
            else if (t + 1 < t1) load((t + 1) % ntile_n, 0, stage ^ 1);
            const float* ws = Ws + stage * kRfKC * kRfB + 2 * tx;
            const float* cs = Ct + c * kRfKC * kRfB + 16 * ty;
            const int kc = min(kRfKC, r - c * kRfKC);
            // operands of the next k are loaded before the FMAs of this one
            ulonglong2 x[4], xn[4];
            float2 y[4], yn[4];
            auto fetch = [&](int kk, ulonglong2* xx, float2* yy) {
#pragma unroll
                for (int q = 0; q < 4; ++q) xx[q] = *reinterpret_cast<const ulonglong2*>(cs + kk * kRfB + 4 * q);
#pragma unroll
                for (int q = 0; q < 4; ++q) yy[q] = *reinterpret_cast<const float2*>(ws + kk * kRfB + 32 * q);
            };
            auto step = [&](const ulonglong2* xx, const float2* yy) {
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const float wf = b & 1 ? yy[b >> 1].y : yy[b >> 1].x;
                    const uint64_t w = pk(wf, wf);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        acc[2 * q][b] = fma2(xx[q].x, w, acc[2 * q][b]);
                        acc[2 * q + 1][b] = fma2(xx[q].y, w, acc[2 * q + 1][b]);
                    }
                }
            };
            fetch(0, x, y);
            int kk = 0;
            for (; kk + 2 <= kc; kk += 2) {
                fetch(kk + 1, xn, yn);
                step(x, y);
                fetch(min(kk + 2, kc - 1), x, y);
                step(xn, yn);
            }
            if (kk < kc) step(x, y);
        }
        const bool whole = WHOLE || (pairs && c0 + kRfB <= n);
#pragma unroll
        for (int grp = 0; grp < 2; ++grp) {
            float tmx = 0.f, tse = 0.f, tsa = 0.f;
            auto fold = [&](float av, float d) {
                const float e = av - d;
                if (!(fabsf(e) <= INFINITY)) bad = 1;
                tmx = fmaxf(tmx, fabsf(e));
                tse = fmaf(e, e, tse);
                tsa = fmaf(av, av, tsa);
            };
#pragma unroll
            for (int a0 = 0; a0 < 8; a0 += 4) {
                const int64_t i0 = r0 + ty * 16 + grp * 8 + a0;
                if (WHOLE || (whole && i0 + 4 <= m)) {   // two elements per load, sixteen loads in flight
                    uint64_t raw[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const TA* p = A + (i0 + a) * ld + c0 + 2 * tx + 32 * b;
                            if constexpr (sizeof(TA) == 4)
                                raw[a][b] = __ldcs(reinterpret_cast<const unsigned long long*>(p));
                            else
                                raw[a][b] = __ldcs(reinterpret_cast<const unsigned*>(p));
                        }
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            const uint64_t v = raw[a][b >> 1];
                            const uint32_t bits = sizeof(TA) == 4 ? (uint32_t)(b & 1 ? v >> 32 : v)
                                                                  : (b & 1 ? (uint32_t)v & 0xffff0000u : (uint32_t)v << 16);
                            const int row = grp * 8 + a0 + a;
                            const uint64_t d = acc[row >> 1][b];
                            fold(__uint_as_float(bits), __uint_as_float((uint32_t)(row & 1 ? d >> 32 : d)));
                        }
                } else if constexpr (!WHOLE) {
                    // A's last rows or columns, or rows off the pairs' grid: one element per load, the
                    // 32 loads issued before they are folded, and an entry past A's end folds as zeros
                    // (loaded and folded one by one: BF16 113763 x 393, r = 16, 240 us; residual_k 169,
                    // this 136). BF16 loads some valid address instead of a predicate: its conversions
                    // otherwise wait for each load in turn (228 us); FP32 is faster with one (119 and 148)
                    const int rr = (int)min((int64_t)4, m - i0), rc = (int)min((int64_t)kRfB, n - c0);   // what A has here
                    TA raw[4][8];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const TA* p = A + min(i0 + a, m - 1) * ld + c0;
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            const int cc = 2 * tx + 32 * (b >> 1) + (b & 1);
                            if constexpr (sizeof(TA) == 4) raw[a][b] = a < rr && cc < rc ? p[cc] : 0.f;
                            else raw[a][b] = p[cc < rc ? cc : 0];
                        }
                    }
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            const int row = grp * 8 + a0 + a;
                            const uint64_t d = acc[row >> 1][b];
                            const bool in = a < rr && 2 * tx + 32 * (b >> 1) + (b & 1) < rc;
                            fold(in ? to_f(raw[a][b]) : 0.f, in ? __uint_as_float((uint32_t)(row & 1 ? d >> 32 : d)) : 0.f);
                        }
                }
            }
            mx = fmax(mx, (double)tmx);
            se += (double)tse;
            sa += (double)tsa;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __shared__ double rmx[kRfT / 32], rse[kRfT / 32], rsa[kRfT / 32];
    __shared__ int rbad;
    if (tid == 0) rbad = 0;
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        se += __shfl_xor_sync(0xffffffffu, se, o);
        sa += __shfl_xor_sync(0xffffffffu, sa, o);
    }
    __syncthreads();
    if (bad) rbad = 1;
    if (lane == 0) { rmx[warp] = mx; rse[warp] = se; rsa[warp] = sa; }
    __syncthreads();
    if (tid == 0) {
        double a1 = 0.0, a2 = 0.0, a3 = 0.0;
        for (int w = 0; w < kRfT / 32; ++w) { a1 = fmax(a1, rmx[w]); a2 += rse[w]; a3 += rsa[w]; }
        part[(int64_t)blockIdx.x * 4 + 0] = a1;
        part[(int64_t)blockIdx.x * 4 + 1] = a2;
        part[(int64_t)blockIdx.x * 4 + 2] = a3;
        part[(int64_t)blockIdx.x * 4 + 3] = rbad ? 1.0 : 0.0;
    }
}

// Combines the per-CTA partials in a fixed order (one CTA of 256 threads).
__global__ void residual_final_k(const double* part, int64_t nparts, double* cheb, double* fro,
                                 int* status, double* sums = nullptr) {
    __shared__ double s1[256], s2[256], s3[256];
    __shared__ int sb[256];
    const int tid = threadIdx.x;
    double a1 = 0.0, a2 = 0.0, a3 = 0.0;
    int bad = 0;
    for (int64_t c = tid; c < nparts; c += blockDim.x) {
        a1 = fmax(a1, part[c * 4 + 0]);
        a2 += part[c * 4 + 1];
        a3 += part[c * 4 + 2];
        bad |= part[c * 4 + 3] != 0.0;
    }
    s1[tid] = a1; s2[tid] = a2; s3[tid] = a3; sb[tid] = bad;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (tid < o) {
            s1[tid] = fmax(s1[tid], s1[tid + o]);
            s2[tid] += s2[tid + o];
            s3[tid] += s3[tid + o];
            sb[tid] |= sb[tid + o];
        }
        __syncthreads();
    }
    if (tid != 0) return;
    a1 = s1[0];
    if (sb[0]) {
        set_status(status, CUR_ERR_NONFINITE);
        a1 = NAN;
    }
    *cheb = a1;
    if (fro) *fro = s3[0] > 0.0 ? sqrt(s2[0] / s3[0]) : 0.0;
    if (sums) { sums[0] = s2[0]; sums[1] = s3[0]; }
}

static inline unsigned nb(int64_t n, int t = 256) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + t - 1) / t, 65535));
}

template <typename TA>
static cur_status assemble_t(cur_handle* h, const cur_mat* Am, const int32_t* I, const int32_t* J,
                             int r, void* C_out, double* U_out, void* R_out, double* rcond_out,
                             Arena& ar, cudaStream_t st) {
    const TA* A = static_cast<const TA*>(Am->data);
    double* work = ar.get<double>((size_t)3 * r * r);   // its first r doubles: assemble_gj_k's column sums
    int* redo = ar.get<int>(1);
    if (!ar.ok) return CUR_ERR_NOMEM;
    if (C_out) {
        gather_C_k<TA><<<nb(Am->rows * r), 256, 0, st>>>(A, Am->rows, Am->cols, Am->ld, J, r, static_cast<TA*>(C_out), h->status);
        CUR_CK(cudaGetLastError());
    note_launch();
    }
    if (R_out) {
        gather_R_k<TA><<<nb(Am->cols * r), 256, 0, st>>>(A, Am->rows, Am->cols, Am->ld, I, r, static_cast<TA*>(R_out), h->status);
        CUR_CK(cudaGetLastError());
    note_launch();
    }
    // Up to r = 44 assemble_inv_k alone is the faster (us an assembly of 600 x 500, with assemble_gj_k
    // before it and alone: r = 4 26.7 and 22.6, 16 43.0 and 39.0, 33 86 and 68, 44 98.3 and 96.4, 48 106 and
    // 117, 64 112 and 209): a cluster's launch, and the second kernel's that then finds nothing to do
    if (r > 44) {
        int nc, cpw;
        gj_plan(r, &nc, &cpw);
#define ASSEMBLE(RU, CPW) assemble_gj_k<TA, RU, CPW>
        CUR_TRY(gj_launch(GJ_KERNEL(r, cpw, ASSEMBLE), nc, nc, GjSmem::bytes(r), st, A, Am->rows, Am->cols, Am->ld, I, J, r,
                          U_out, rcond_out, work, redo));
#undef ASSEMBLE
    } else {
        redo = nullptr;
    }
    const size_t sm = ((size_t)r * r + r) * sizeof(double) + (size_t)r * sizeof(int) + 64;
    CUR_TRY(smem_attr((const void*)assemble_inv_k<TA>, sm));
    assemble_inv_k<TA><<<1, 256, sm, st>>>(A, Am->rows, Am->cols, Am->ld, I, J, r, U_out, rcond_out, work, h->status, redo);
    CUR_CK(cudaGetLastError());
    note_launch();
    return CUR_OK;
}

// CUR_ERR_ARG where the workspace cannot hold W padded to whole tiles (the caller then takes
// residual_k, which needs up to 512 r bytes less).
template <typename TA>
static cur_status residual_fma_t(cur_handle* h, const cur_mat* Am, const void* C, const double* U, const void* R,
                                 int r, double* cheb, double* fro, Arena& ar, cudaStream_t st, double* sums) {
    const int64_t m = Am->rows, n = Am->cols;
    const int64_t ntile_n = (n + kRfB - 1) / kRfB, npad = ntile_n * kRfB, ntiles = (m + kRfB - 1) / kRfB * ntile_n;
    float* W = ar.get<float>((size_t)r * npad);
    const int grid = (int)std::min<int64_t>(2LL * h->num_sms, ntiles);
    double* part = ar.get<double>((size_t)grid * 4);
    if (!ar.ok || npad / 32 > INT_MAX) return CUR_ERR_ARG;
    const size_t smw = (size_t)r * (kRfWK + 32) * sizeof(double);
    CUR_TRY(smem_attr((const void*)residual_w2_k<TA>, smw));
    residual_w2_k<TA><<<dim3((unsigned)(npad / 32), (unsigned)((r + kRfWK - 1) / kRfWK)), 256, smw, st>>>(
        U, static_cast<const TA*>(R), r, n, npad, W);
    CUR_CK(cudaGetLastError());
    note_launch();
    const size_t sm = (size_t)(2 * kRfKC + r) * kRfB * sizeof(float);
    const int pairs = (reinterpret_cast<uintptr_t>(Am->data) % (2 * sizeof(TA))) == 0 && Am->ld % 2 == 0;
    auto kernel = pairs && m % kRfB == 0 && n % kRfB == 0 ? residual_fma_k<TA, true> : residual_fma_k<TA, false>;
    CUR_TRY(smem_attr((const void*)kernel, sm));
    kernel<<<grid, kRfT, sm, st>>>(static_cast<const TA*>(Am->data), m, n, Am->ld, static_cast<const TA*>(C),
                                               W, npad, r, ntile_n, ntiles, part, pairs);
    CUR_CK(cudaGetLastError());
    note_launch();
    residual_final_k<<<1, 256, 0, st>>>(part, grid, cheb, fro, h->status, sums);
    CUR_CK(cudaGetLastError());
    note_launch();
    return CUR_OK;
}

template <typename TA, typename TW, int TM, int TN>
static cur_status residual_t(cur_handle* h, const cur_mat* Am, const void* C, const double* U,
                             const void* R, int r, double* cheb, double* fro, Arena& ar,
                             cudaStream_t st, double* sums) {
    const int64_t m = Am->rows, n = Am->cols;
    TW* W = ar.get<TW>((size_t)r * n);
    constexpr int BM = 16 * TM, BN = 16 * TN;
    const int64_t panels = (m + BM - 1) / BM;
    const int64_t ntile = (n + BN - 1) / BN;
    const size_t sm = (size_t)r * (BM + BN) * sizeof(TW);
    CUR_TRY(smem_attr((const void*)residual_k<TA, TW, TM, TN>, sm));
    int occ = 1;
    CUR_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, residual_k<TA, TW, TM, TN>, 256, sm));
    const int64_t want = (int64_t)h->num_sms * std::max(1, occ) * 4;
    int64_t segs = std::max<int64_t>(1, std::min<int64_t>(ntile, (want + panels - 1) / panels));
    segs = std::min<int64_t>(segs, 65535);
    if (panels > 2147483647LL) return CUR_ERR_ARG;
    double* part = ar.get<double>((size_t)panels * segs * 4);
    if (!ar.ok) return CUR_ERR_NOMEM;
    const size_t smw = (size_t)r * r * sizeof(double);
    CUR_TRY(smem_attr((const void*)residual_w_k<TA, TW>, smw));
    residual_w_k<TA, TW><<<nb(n), 256, smw, st>>>(U, static_cast<const TA*>(R), r, n, W);
    CUR_CK(cudaGetLastError());
    note_launch();
    const uintptr_t base = reinterpret_cast<uintptr_t>(Am->data);
    const int vec = (base % 16 == 0) && ((size_t)Am->ld * sizeof(TA)) % 16 == 0 ? 1 : 0;
    residual_k<TA, TW, TM, TN><<<dim3((unsigned)panels, (unsigned)segs), 256, sm, st>>>(
        static_cast<const TA*>(Am->data), m, n, Am->ld, static_cast<const TA*>(C), W, r, part, vec);
    CUR_CK(cudaGetLastError());
    note_launch();
    residual_final_k<<<1, 256, 0, st>>>(part, panels * segs, cheb, fro, h->status, sums);
    CUR_CK(cudaGetLastError());
    note_launch();
    return CUR_OK;
}

}  // namespace curk

cur_status assemble_impl(cur_handle* h, const cur_mat* A, const int32_t* I, const int32_t* J,
                         int r, void* C_out, double* U_out, void* R_out, double* rcond_out,
                         Arena& ar, cudaStream_t st) {
    switch (A->dtype) {
        case CUR_F64: return curk::assemble_t<double>(h, A, I, J, r, C_out, U_out, R_out, rcond_out, ar, st);
        case CUR_F32: return curk::assemble_t<float>(h, A, I, J, r, C_out, U_out, R_out, rcond_out, ar, st);
        case CUR_BF16: return curk::assemble_t<__nv_bfloat16>(h, A, I, J, r, C_out, U_out, R_out, rcond_out, ar, st);
    }
    return CUR_ERR_ARG;
}

cur_status residual_impl(cur_handle* h, const cur_mat* A, const void* C, const double* U,
                         const void* R, int r, double* cheb_out, double* fro_out, Arena& ar,
                         cudaStream_t st, double* sums_out) {
    if (A->dtype == CUR_F32) {
        // tensor-core (tcgen05) form where it applies; CUR_ERR_ARG means it does not
        const size_t mark = ar.off;
        const cur_status s = residual_tc_impl(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out);
        if (s != CUR_ERR_ARG) return s;
        ar.off = mark;
        ar.ok = true;
    }
    if (A->dtype != CUR_F64) {
        const size_t mark = ar.off;
        const cur_status s = A->dtype == CUR_F32
            ? curk::residual_fma_t<float>(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out)
            : curk::residual_fma_t<__nv_bfloat16>(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out);
        if (s != CUR_ERR_ARG) return s;
        ar.off = mark;
        ar.ok = true;
    }
    switch (A->dtype) {
        case CUR_F64: return curk::residual_t<double, double, 4, 4>(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out);
        case CUR_F32: return curk::residual_t<float, float, 8, 8>(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out);
        case CUR_BF16: return curk::residual_t<__nv_bfloat16, float, 8, 8>(h, A, C, U, R, r, cheb_out, fro_out, ar, st, sums_out);
    }
    return CUR_ERR_ARG;
}

// ---------------------------------------------------------------- allocation-free residual
//
// cur_residual_cheb needs a handle, and a handle allocates its workspace with cudaMalloc.
// Some callers cannot do that where they need the residual: code that runs after its
// device memory has been handed to a pool or allocator of its own, or a loop that must
// not hit cudaMalloc's implicit device synchronisation. For them
// cur_residual_cheb_noalloc keeps its scratch (W = U R and the per-CTA partial sums) in
// one array compiled into this library. The array's device address is looked up once
// per device, on the first call made with that device current, and kept until the
// process exits; a device reset after that first call is not supported (the kept
// address would no longer be valid).

#include <mutex>

namespace curk {
constexpr size_t kNoallocScratchBytes = (size_t)16 << 20;  // 16 MiB on every device
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];
}  // namespace curk

static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[256] = {};

// Device address of the scratch array on the current device (set up on first use).
static cur_status noalloc_scratch(void** out) {
    int dev = 0;
    CUR_CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) return CUR_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, curk::g_noalloc_scratch) != cudaSuccess || !p) return CUR_ERR_CUDA;
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return CUR_OK;
}

template <typename TA, typename TW, int TM, int TN>
static cur_status residual_noalloc_t(const cur_mat* Am, const void* C, const double* U,
                                     const void* R, int r, double* cheb, double* fro,
                                     cudaStream_t st) {
    using namespace curk;
    const int64_t m = Am->rows, n = Am->cols;
    constexpr int BM = 16 * TM, BN = 16 * TN;
    const int64_t panels = (m + BM - 1) / BM;
    const int64_t ntile = (n + BN - 1) / BN;
    if (panels > 65535LL * 32768LL) return CUR_ERR_ARG;
    int dev = 0, sms = 0;
    CUR_CK(cudaGetDevice(&dev));
    CUR_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t sm = (size_t)r * (BM + BN) * sizeof(TW);
    CUR_TRY(smem_attr((const void*)residual_k<TA, TW, TM, TN>, sm));
    int occ = 1;
    CUR_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, residual_k<TA, TW, TM, TN>, 256, sm));
    const int64_t want = (int64_t)sms * std::max(1, occ) * 4;
    int64_t segs = std::max<int64_t>(1, std::min<int64_t>(ntile, (want + panels - 1) / panels));
    segs = std::min<int64_t>(segs, 65535);
    if (panels > 2147483647LL) return CUR_ERR_ARG;
    // scratch: W (r x n) then the partials (4 doubles per CTA), 256-byte aligned
    const size_t w_bytes = ((size_t)r * n * sizeof(TW) + 255) / 256 * 256;
    const size_t p_bytes = (size_t)panels * segs * 4 * sizeof(double);
    if (w_bytes + p_bytes > kNoallocScratchBytes) return CUR_ERR_NOMEM;
    void* base = nullptr;
    CUR_TRY(noalloc_scratch(&base));
    TW* W = static_cast<TW*>(base);
    double* part = reinterpret_cast<double*>(static_cast<unsigned char*>(base) + w_bytes);
    const size_t smw = (size_t)r * r * sizeof(double);
    CUR_TRY(smem_attr((const void*)residual_w_k<TA, TW>, smw));
    residual_w_k<TA, TW><<<nb(n), 256, smw, st>>>(U, static_cast<const TA*>(R), r, n, W);
    CUR_CK(cudaGetLastError());
    const uintptr_t abase = reinterpret_cast<uintptr_t>(Am->data);
    const int vec = (abase % 16 == 0) && ((size_t)Am->ld * sizeof(TA)) % 16 == 0 ? 1 : 0;
    residual_k<TA, TW, TM, TN><<<dim3((unsigned)panels, (unsigned)segs), 256, sm, st>>>(
        static_cast<const TA*>(Am->data), m, n, Am->ld, static_cast<const TA*>(C), W, r, part, vec);
    CUR_CK(cudaGetLastError());
    residual_final_k<<<1, 256, 0, st>>>(part, panels * segs, cheb, fro, nullptr);
    CUR_CK(cudaGetLastError());
    return CUR_OK;
}

extern "C" cur_status cur_residual_cheb_noalloc(const cur_mat* A, const void* C, const double* U,
                                                const void* R, int32_t r, double* cheb_out,
                                                double* fro_rel_out, cudaStream_t stream) {
    if (!A || !A->data || A->rows < 1 || A->cols < 1 || A->ld < A->cols) return CUR_ERR_ARG;
    if (!C || !U || !R || !cheb_out || r < 1 || r > 128) return CUR_ERR_ARG;
    switch (A->dtype) {
        case CUR_F64: return residual_noalloc_t<double, double, 4, 4>(A, C, U, R, r, cheb_out, fro_rel_out, stream);
        case CUR_F32: return residual_noalloc_t<float, float, 8, 8>(A, C, U, R, r, cheb_out, fro_rel_out, stream);
        case CUR_BF16: return residual_noalloc_t<__nv_bfloat16, float, 8, 8>(A, C, U, R, r, cheb_out, fro_rel_out, stream);
    }
    return CUR_ERR_ARG;
}
