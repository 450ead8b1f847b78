// Algorithm 1 of the paper (Section 1.3): adaptive cross approximation with full
// pivoting, the sequential baseline that Algorithm 3 is set against.
//
// Step k picks (i, j) = argmax |R_k(i,j)| over the whole residual (ties: smallest
// row-major index) and eliminates R_{k+1} = R_k - R_k(:,j) R_k(i,:) / R_k(i,j). The
// residual is kept explicitly in a caller-owned m x n buffer (FP32 for FP32/BF16 data,
// FP64 for FP64 data), so a step is one streaming pass that reads and writes R once:
//   a1_update : R <- R - u v^T with u = R_k(:,j)/R_k(i,j), v = R_k(i,:), row i and
//               column j set to zero (exactly zero in exact arithmetic), and each
//               CTA's (max |R_{k+1}|, lowest index) in the same pass
//   a1_pick   : every CTA combines the CTA maxima and applies the rounding stop
//               (|pivot| <= max(m,n) eps max|A|); CTA 0 records I, J and the pivot, all of
//               them write u and v of the new pivot for the next update
// a1_init copies A into R and finds the first pivot's candidates. All steps are
// enqueued without host synchronisation; after a stop the remaining kernels return
// at once.

#include <algorithm>
#include <climits>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace curk {

struct A1State {
    double amax;      // max |A|
    double piv;       // pivot value of the current step
    long long idx;    // its row-major index i n + j
    int stop;         // 1 once the loop has ended
};

constexpr int kA1Threads = 256;

// (value, index): larger value wins, then the smaller index
__device__ __forceinline__ void a1_better(double v, long long i, double& bv, long long& bi) {
    if (v > bv || (v == bv && i < bi)) { bv = v; bi = i; }
}

__device__ __forceinline__ void a1_block_argmax(double& bv, long long& bi, double* pv, long long* pi) {
    __shared__ double sv[32];
    __shared__ long long si[32];
    for (int o = 16; o > 0; o >>= 1) {
        const double v2 = __shfl_xor_sync(0xffffffffu, bv, o);
        const long long i2 = __shfl_xor_sync(0xffffffffu, bi, o);
        a1_better(v2, i2, bv, bi);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) { sv[w] = bv; si[w] = bi; }
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        bv = lane < nw ? sv[lane] : -1.0;
        bi = lane < nw ? si[lane] : LLONG_MAX;
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xffffffffu, bv, o);
            const long long i2 = __shfl_xor_sync(0xffffffffu, bi, o);
            a1_better(v2, i2, bv, bi);
        }
        if (lane == 0) { pv[blockIdx.x] = bv; pi[blockIdx.x] = bi; }
    }
}

template <typename TR> struct Vec;
template <> struct Vec<float> { using T = float4; static constexpr int W = 4; };
template <> struct Vec<double> { using T = double2; static constexpr int W = 2; };

template <typename TR>
__device__ __forceinline__ void vload(const TR* p, TR* x) {
    if constexpr (sizeof(TR) == 4) {
        const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
        const double2 t = __ldcs(reinterpret_cast<const double2*>(p));
        x[0] = t.x; x[1] = t.y;
    }
}
template <typename TR>
__device__ __forceinline__ void vstore(TR* p, const TR* x) {
    if constexpr (sizeof(TR) == 4) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(x[0], x[1], x[2], x[3]));
    } else {
        __stcs(reinterpret_cast<double2*>(p), make_double2(x[0], x[1]));
    }
}

template <typename TR, typename TA>
__device__ __forceinline__ TR a1_conv(TA x) {
    if constexpr (sizeof(TR) == 8) return to_d(x); else return to_f(x);
}

// The residual is contiguous, so the passes walk it as one flat array in groups of W elements
// (16 bytes) whatever n is: with n % W != 0 a group may run over the end of a row. (Element by
// element, the form for such n before, moved 4 bytes per access with 64-bit index arithmetic
// for each: 1.7 TB/s of the update pass against 6.4 at 16383 x 4099.)
//
// A thread's groups: e = first element of the group, (i, c) its row and column.
struct A1Walk {
    int64_t i, c, di, dc, n, e, de;
    __device__ __forceinline__ A1Walk(int64_t n_, int W) : n(n_) {
        e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
        de = (int64_t)gridDim.x * blockDim.x * W;
        i = e / n;
        c = e - i * n;
        di = de / n;
        dc = de - di * n;
    }
    __device__ __forceinline__ void next() {
        e += de;
        c += dc;
        i += di;
        if (c >= n) { c -= n; ++i; }
    }
};

// R = A (converted), CTA argmax of |A|; non-finite data stops the loop. The scan
// compares in the residual's type; a thread visits increasing indices, so a strict
// '>' keeps the lowest index of its equal maxima. FLAT: A is contiguous too (ld = n), of R's
// type and 16-byte aligned: vector loads.
template <typename TA, typename TR, bool VEC, bool FLAT>
__global__ void __launch_bounds__(kA1Threads) a1_init(const TA* __restrict__ A, int64_t m, int64_t n,
                                                      int64_t ld, TR* __restrict__ R, double* pv,
                                                      long long* pi, int* status) {
    constexpr int W = VEC ? Vec<TR>::W : 1;
    constexpr int U = 4;
    TR bv = (TR)-1;
    long long bi = LLONG_MAX;
    int bad = 0;
    const int64_t total = m * n;
    A1Walk w(n, W);
    while (w.e < total) {
        int64_t e[U];
        TR x[U][W];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            e[q] = w.e;
            if (FLAT && w.e + W <= total) {
                vload<TR>(reinterpret_cast<const TR*>(A) + w.e, x[q]);
            } else if (w.e < total) {
                int64_t i = w.i, c = w.c;
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    x[q][k] = w.e + k < total ? a1_conv<TR>(A[i * ld + c]) : (TR)0;
                    if (++c == n) { c = 0; ++i; }
                }
            }
            w.next();
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (e[q] >= total) break;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const TR ax = fabs(x[q][k]);
                if (!(ax <= (TR)INFINITY)) bad = 1;
                if (ax > bv && e[q] + k < total) { bv = ax; bi = e[q] + k; }
            }
            if (VEC && e[q] + W <= total) {
                if constexpr (VEC) vstore<TR>(R + e[q], x[q]);
            } else {
#pragma unroll
                for (int k = 0; k < W; ++k)
                    if (e[q] + k < total) R[e[q] + k] = x[q][k];
            }
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(status, CUR_ERR_NONFINITE);
    double dv = (double)bv;
    a1_block_argmax(dv, bi, pv, pi);
}

// One step's pivot and its vectors: every CTA combines the CTA maxima (~1200, from L2) and
// takes the same decision; CTA 0 records it, and each CTA writes its share of u = R(:, j) /
// R(i, j) and v = R(i, :). (One CTA that picked and a second kernel for u and v took 14 us a
// step at 16383 x 4099.) What CTA 0 writes here is not read by the others: amax and stop are
// taken from their own copies of the same values.
template <typename TR>
__global__ void __launch_bounds__(256) a1_pick(const TR* __restrict__ R, int64_t m, int64_t n, int k, int r,
                                               const double* __restrict__ pv, const long long* __restrict__ pi,
                                               int nparts, const A1State* prev, A1State* s, int32_t* I, int32_t* J,
                                               double* piv_out, TR* __restrict__ u, TR* __restrict__ v, int* status) {
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (prev->stop) {
        if (first) s->stop = 1;
        return;
    }
    const bool nonfinite = *status == CUR_ERR_NONFINITE;
    double bv = -1.0;
    long long bi = LLONG_MAX;
    for (int c = threadIdx.x; c < nparts; c += blockDim.x) a1_better(pv[c], pi[c], bv, bi);
    unsigned long long bk = dkey(bv);
    block_argmax_key(bk, bi);
    bv = dkey_value(bk);
    const double amax = k == 0 ? bv : prev->amax;
    const double tol = (double)max(m, n) * 2.220446049250313e-16 * amax;
    const double p = (bi >= 0 && bi < m * n) ? (double)R[bi] : 0.0;
    if (nonfinite || !(fabs(p) > tol) || !(bv > tol)) {
        if (first) {
            s->stop = 1;
            for (int q = k; q < r; ++q) { I[q] = -1; J[q] = -1; if (piv_out) piv_out[q] = 0.0; }
            if (!nonfinite) set_status(status, CUR_WARN_RANK);
        }
        return;
    }
    const int64_t i0 = bi / n, j0 = bi - i0 * n;
    if (first) {
        I[k] = (int32_t)i0;
        J[k] = (int32_t)j0;
        if (piv_out) piv_out[k] = p;
        s->amax = amax;
        s->piv = p;
        s->idx = bi;
        s->stop = 0;
    }
    const TR pt = (TR)p;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m + n; e += (int64_t)gridDim.x * blockDim.x) {
        if (e < m) u[e] = R[e * n + j0] / pt;
        else v[e - m] = R[i0 * n + (e - m)];
    }
}

// R <- R - u v^T with row i0 and column j0 zeroed; CTA argmax of the new |R|.
// VEC: W consecutive elements per access (R 16-byte aligned), else 1; VROW: n % W == 0 too, so
// that a group lies in one row and v is read by vectors. A thread takes U groups a grid stride
// apart per iteration and issues their U loads before any store, so each SM keeps U x 16 bytes
// per thread in flight. Within a thread the indices increase, so a strict '>' keeps the lowest
// index of equal maxima. HBM: 2 m n sizeof(TR) bytes.
template <typename TR, bool VEC, bool VROW>
__global__ void __launch_bounds__(kA1Threads) a1_update(TR* __restrict__ R, int64_t m, int64_t n,
                                                        const A1State* s, const TR* __restrict__ u,
                                                        const TR* __restrict__ v, double* pv,
                                                        long long* pi) {
    if (s->stop) return;
    constexpr int W = VEC ? Vec<TR>::W : 1;
    constexpr int U = 4;
    const int64_t i0 = s->idx / n, j0 = s->idx - i0 * n, total = m * n;
    TR bv = (TR)-1;
    long long bi = LLONG_MAX;
    A1Walk w(n, W);
    while (w.e < total) {
        int64_t ri[U], rc[U], re[U];
        TR x[U][W];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            ri[q] = w.i;
            rc[q] = w.c;
            re[q] = w.e;
            if (VEC && w.e + W <= total) {
                if constexpr (VEC) vload<TR>(R + w.e, x[q]);
            } else {
#pragma unroll
                for (int k = 0; k < W; ++k) x[q][k] = w.e + k < total ? __ldcs(R + w.e + k) : (TR)0;
            }
            w.next();
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (re[q] >= total) break;
            if (VROW || rc[q] + W <= n) {
                const TR ui = u[ri[q]];
                const bool zrow = ri[q] == i0;
                TR vv[W];
                if constexpr (VROW && VEC) {
                    memcpy(vv, __builtin_assume_aligned(v + rc[q], 16), sizeof(vv));
                } else {
#pragma unroll
                    for (int k = 0; k < W; ++k) vv[k] = v[rc[q] + k];
                }
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    TR y = fma(-ui, vv[k], x[q][k]);
                    if (zrow || rc[q] + k == j0) y = (TR)0;
                    x[q][k] = y;
                    const TR ay = fabs(y);
                    if (ay > bv) { bv = ay; bi = re[q] + k; }
                }
            } else {   // over the end of a row, or of R
                int64_t i = ri[q], c = rc[q];
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    if (re[q] + k < total) {
                        TR y = fma(-u[i], v[c], x[q][k]);
                        if (i == i0 || c == j0) y = (TR)0;
                        x[q][k] = y;
                        const TR ay = fabs(y);
                        if (ay > bv) { bv = ay; bi = re[q] + k; }
                        if (++c == n) { c = 0; ++i; }
                    }
                }
            }
            if (VEC && re[q] + W <= total) {
                if constexpr (VEC) vstore<TR>(R + re[q], x[q]);
            } else {
#pragma unroll
                for (int k = 0; k < W; ++k)
                    if (re[q] + k < total) __stcs(R + re[q] + k, x[q][k]);
            }
        }
    }
    double dv = (double)bv;
    a1_block_argmax(dv, bi, pv, pi);
}

template <typename TA, typename TR>
static cur_status aca_full_t(cur_handle* h, const cur_mat* A, int r, TR* R, int32_t* I, int32_t* J,
                             double* piv, Arena& ar, cudaStream_t st) {
    const int64_t m = A->rows, n = A->cols;
    constexpr int W = Vec<TR>::W;
    const bool vec = (reinterpret_cast<uintptr_t>(R) % 16) == 0, vrow = vec && n % W == 0;
    auto update = vrow ? a1_update<TR, true, true> : (vec ? a1_update<TR, true, false> : a1_update<TR, false, false>);
    // one wave of the update pass: every CTA resident (no tail wave)
    int occ = 0;
    CUR_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, update, kA1Threads, 0));
    const int G = h->num_sms * std::max(1, occ);
    double* pv = ar.get<double>(G);
    long long* pi = ar.get<long long>(G);
    TR* u = ar.get<TR>((size_t)m);
    TR* v = ar.get<TR>((size_t)n);
    A1State* s = ar.get<A1State>(2);   // step k reads s[k & 1] and writes s[(k + 1) & 1]
    if (!ar.ok) return CUR_ERR_NOMEM;
    CUR_CK(cudaMemsetAsync(s, 0, 2 * sizeof(A1State), st));
    const bool flat = vec && std::is_same<TA, TR>::value && A->ld == n &&
                      (reinterpret_cast<uintptr_t>(A->data) % 16) == 0;
    auto init = flat ? a1_init<TA, TR, true, std::is_same<TA, TR>::value>
                     : (vec ? a1_init<TA, TR, true, false> : a1_init<TA, TR, false, false>);
    init<<<G, kA1Threads, 0, st>>>(static_cast<const TA*>(A->data), m, n, A->ld, R, pv, pi, h->status);
    CUR_CK(cudaGetLastError());
    note_launch();
    const unsigned ge = (unsigned)std::min<int64_t>((m + n + 255) / 256, (int64_t)h->num_sms);
    for (int k = 0; k < r; ++k) {
        A1State* now = s + ((k + 1) & 1);
        a1_pick<TR><<<ge, 256, 0, st>>>(R, m, n, k, r, pv, pi, G, s + (k & 1), now, I, J, piv, u, v, h->status);
        CUR_CK(cudaGetLastError());
        const bool ev = h->prof && h->prof_n < 4096;
        if (ev) CUR_CK(cudaEventRecord(h->prof_ev[2 * h->prof_n], st));
        update<<<G, kA1Threads, 0, st>>>(R, m, n, now, u, v, pv, pi);
        CUR_CK(cudaGetLastError());
        if (ev) CUR_CK(cudaEventRecord(h->prof_ev[2 * h->prof_n + 1], st));
        if (ev) ++h->prof_n;
        note_launch(2);
    }
    return CUR_OK;
}

}  // namespace curk

cur_status aca_full_impl(cur_handle* h, const cur_mat* A, int r, void* R, int32_t* I, int32_t* J,
                         double* piv, Arena& ar, cudaStream_t st) {
    switch (A->dtype) {
        case CUR_F64:
            return curk::aca_full_t<double, double>(h, A, r, static_cast<double*>(R), I, J, piv, ar, st);
        case CUR_F32:
            return curk::aca_full_t<float, float>(h, A, r, static_cast<float*>(R), I, J, piv, ar, st);
        case CUR_BF16:
            return curk::aca_full_t<__nv_bfloat16, float>(h, A, r, static_cast<float*>(R), I, J, piv, ar, st);
    }
    return CUR_ERR_ARG;
}
