// Algorithm 3 (Section 2.2) on the columns of every matrix of a batch, one launch.
//
// The batch holds many small matrices of uneven shapes (up to a few thousand rows and a
// thousand columns, each a few MB), so each one is taken whole by one CTA: a persistent
// grid walks the batch, and a CTA runs all r rounds of its matrix with no grid-wide
// synchronisation. The rounds are those of the full-matrix kernels (the implicit
// residual nu_j = ||a_j||^2 - sum_k (q_k^T a_j)^2, one read of the matrix per round):
//   pass   : w_j = a_j^T q_t for every column (Dot2 with q as FP32 hi/lo pairs), the
//            512 threads split into n/4 four-column groups x as many row groups as fit
//            (2 for n = 1024, 16 for n = 128); the rows come through shared memory, one or
//            two CTAs per SM
//   pick   : nu_j -= w_j^2, masked argmax (lowest index on ties)
//   vector : v = a_p - Q W(:,p) with W = the passes' q^T a (the first Gram-Schmidt sweep
//            needs no Q^T a_p of its own), orthogonalised once more against q_1..q_t
//            (double-float), the early stop
//            on the recomputed ||v||^2 <= (max(m,n) eps ||A||_F)^2, q = v / ||v||
// Q lives in the CTA's slice of the workspace (r x m hi and lo floats); everything else
// in shared memory. Supports FP32 data, r <= 64, m <= 4096, n <= 1024.

#include <algorithm>
#include <climits>

#include "common.cuh"
#include "df64.cuh"
#include "internal.h"
#include "tc.cuh"

namespace curk {

constexpr int kBA_T = 512;      // threads per CTA
constexpr int kBA_RG = kBA_T / 256;   // partial-sum rows per column in shared memory: RG n <= kBA_RG kBA_MaxN
constexpr int kBA_MaxM = 4096;
constexpr int kBA_MaxN = 1024;
constexpr int kBA_MaxR = 64;

struct BatAcaItem {
    int64_t aoff, m, n, ld;   // matrix at data + aoff, row-major with leading dimension ld
    int32_t r;
    int64_t joff;             // its J0 at J + joff (r entries)
};

// The pass's rows on their way: kBA_Slots slots of consecutive rows, of 16 KB each with two CTAs on
// an SM, of three times that with one. Loaded HBM answers after ~2700 cycles, so an SM's share of it (23
// bytes per cycle) wants 64 KB in flight; and a slot costs a warp about a hundred instructions beside its
// sums, so large ones are worth more than a second CTA: 1024 matrices of 2150 x 580 on average take
// 81 ms with 2 x 3 x 16 KB, 52 with 4 x 32 KB and 48 with 3 x 48 KB (sums in nine operations; eleven: 53).
constexpr int kBA_Slots = 3;
constexpr int kBA_Rows = 16384;
constexpr int bat_slot_bytes(int per_sm) { return (per_sm == 1 ? 3 : 1) * kBA_Rows + 32; }

// shared-memory layout (bytes): part RG x n x 8 | nu n x 8 | v m x 8 (the direction in the making, then q: high and low words) | s kBA_MaxR x 8 |
// mask n | ring
constexpr size_t bat_aca_smem(int per_sm) {
    return (size_t)kBA_Slots * bat_slot_bytes(per_sm) + (size_t)kBA_RG * kBA_MaxN * 8 + (size_t)kBA_MaxN * 8 + (size_t)kBA_MaxM * 8 +
           (size_t)kBA_MaxR * 8 + kBA_MaxN;
}

// (key, index) maximum over the CTA, integer keys (dkey order): no FP64 comparisons.
__device__ __forceinline__ void bat_argmax(unsigned long long& k, int& i) {
    long long li = i;
    block_argmax_key(k, li);
    i = (int)li;
}

__device__ __forceinline__ df64 bat_df_sum(df64 x) {
    __shared__ df64 sw[32];
    for (int o = 16; o > 0; o >>= 1)
        x = df_add(x, df64{__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.l, o)});
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sw[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        df64 s{0.f, 0.f};
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s = df_add(s, sw[q]);
        sw[0] = s;
    }
    __syncthreads();
    const df64 out = sw[0];
    __syncthreads();
    return out;
}

// v - sum_{k < t} Q(k, i) qs[k] for the rows ia and ib: the entries of eight directions are loaded
// before their sums (a chain over k would otherwise wait for memory at each pair), two chains a row.
__device__ __forceinline__ void bat_minus_q(const float* Qh, const float* Ql, int64_t m, int t, int64_t ia, int64_t ib,
                                            const df64* qs, df64& va, df64& vb) {
    constexpr int B = 8;
    df64 a1{0.f, 0.f}, b1{0.f, 0.f};
    for (int k0 = 0; k0 < t; k0 += B) {
        float ha[B], la[B], hb[B], lb[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const int64_t o = (int64_t)min(k0 + u, t - 1) * m;   // past t: a valid entry, not used
            ha[u] = Qh[o + ia];
            la[u] = Ql[o + ia];
            hb[u] = Qh[o + ib];
            lb[u] = Ql[o + ib];
        }
#pragma unroll
        for (int u = 0; u < B; u += 2) {
            if (k0 + u < t) {
                const df64 s = qs[k0 + u];
                va = df_sub(va, df_mul(df64{ha[u], la[u]}, s));
                vb = df_sub(vb, df_mul(df64{hb[u], lb[u]}, s));
            }
            if (k0 + u + 1 < t) {
                const df64 s = qs[k0 + u + 1];
                a1 = df_sub(a1, df_mul(df64{ha[u + 1], la[u + 1]}, s));
                b1 = df_sub(b1, df_mul(df64{hb[u + 1], lb[u + 1]}, s));
            }
        }
    }
    va = df_add(va, a1);
    vb = df_add(vb, b1);
}

// qs[k] = sum_i Q(k, i) v(i) for k < t (one warp per direction, double-float, sixteen loads in
// flight per lane), then v(i) -= sum_k Q(k, i) qs[k].
__device__ void bat_project(const float* Qh, const float* Ql, int64_t m, int t, df64* v, df64* qs) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int k = warp; k < t; k += nw) {
        const float* qh = Qh + (int64_t)k * m;
        const float* ql = Ql + (int64_t)k * m;
        df64 a0{0.f, 0.f}, a1{0.f, 0.f};
        constexpr int B = 8;
        for (int i = lane; i < m; i += 32 * B) {
            float h[B], l[B];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int ii = i + 32 * u < m ? i + 32 * u : i;
                h[u] = qh[ii];
                l[u] = ql[ii];
            }
#pragma unroll
            for (int u = 0; u < B; u += 2) {
                const int ia = i + 32 * u, ib = ia + 32;
                if (ia < m) a0 = df_add(a0, df_mul(df64{h[u], l[u]}, v[ia]));
                if (ib < m) a1 = df_add(a1, df_mul(df64{h[u + 1], l[u + 1]}, v[ib]));
            }
        }
        df64 s = df_add(a0, a1);
        for (int o = 16; o > 0; o >>= 1)
            s = df_add(s, df64{__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.l, o)});
        if (lane == 0) qs[k] = s;
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < m; i += 2 * blockDim.x) {
        const int64_t ib = i + blockDim.x;
        df64 a{0.f, 0.f}, b{0.f, 0.f};
        bat_minus_q(Qh, Ql, m, t, i, ib < m ? ib : i, qs, a, b);
        v[i] = df_add(v[i], a);
        if (ib < m) v[ib] = df_add(v[ib], b);
    }
    __syncthreads();
}

// A row's terms of a thread's four columns, in Dot2's eleven operations: the picks of a thousand
// matrices, some among nearly equal columns, stay those of the scalar sums.
template <bool DOT>
__device__ __forceinline__ void bat_add(Dot2x2 (&acc)[2], const float (&x)[4], df64 q) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint64_t a = pk(x[2 * k], x[2 * k + 1]);
        if (DOT) acc[k].add(a, pk(q.h, q.h), pk(q.l, q.l));
        else acc[k].c = add2(acc[k].c, acc[k].term_sq(a));
    }
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t done;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(done) : "r"(su32(b)), "r"(parity) : "memory");
    return done != 0;
}

// One round's pass over a matrix: part[rg n + j] = sum over the row group rg's rows i of a_ij q_i
// (DOT) or a_ij^2. A thread sums the columns cg + cgn c, c = 0..3, of its group's rows: neighbouring
// lanes take neighbouring words whatever the row's alignment. The rows come by bulk copies of
// their 16-byte lines, a slot of consecutive rows each; a warp releases a slot when it has summed its
// part, and no barrier holds the others back. (Loads of every entry to registers: 81 ms for the
// batch above; 16-byte cp.async with a barrier per slot: 95.) What bounds it is the issue
// slots: eleven FMA-pipe operations per element and about half as many instructions beside the packed sums. Words of the first
// and last line that lie outside the matrix are not touched. `next` is the slot that fills
// next and `phase` its parity. False: a copy did not arrive in time (*feed 0: none is made, for
// the self-test).
template <bool DOT>
__device__ __forceinline__ bool bat_pass(const float* __restrict__ A, int64_t m, int64_t n, int64_t ld, int cgn, int RG,
                                         const df64* q, unsigned char* ring, int slot_b, const int* feed, uint64_t* bars, uint64_t* freed,
                                         unsigned& next, unsigned& phase, df64* part) {
    const int tid = threadIdx.x, cg = tid % cgn, rg = tid / cgn;
    const bool active = rg < RG;
    int co[4];   // a column past n: the group's first, its sum is not stored
#pragma unroll
    for (int c = 0; c < 4; ++c) co[c] = cg + cgn * c < n ? cg + cgn * c : cg;
    Dot2x2 acc[2];
    int per = (int)(kBA_Rows / (ld * 4)) / RG * RG;   // rows per slot
    if (slot_b > 3 * kBA_Rows) per *= 3;
    if (per > 0) {
        const int stages = (int)((m + per - 1) / per);
        const uintptr_t base = reinterpret_cast<uintptr_t>(A), end = base + ((m - 1) * ld + n) * 4;
        auto fill = [&](int s, unsigned slot) {   // thread 0
            const int64_t r0 = (int64_t)s * per, r1 = min(m, r0 + per);
            const uintptr_t a0 = base + r0 * ld * 4, a1 = base + ((r1 - 1) * ld + n) * 4;
            uintptr_t lo = a0 & ~(uintptr_t)15, hi = (a1 + 15) & ~(uintptr_t)15;
            unsigned char* d = ring + slot * slot_b;
            const uintptr_t d0 = lo;   // the address at the slot's start
            if (lo < base) {
                lo += 16;
                for (uintptr_t x = a0; x < min(lo, a1); x += 4) *reinterpret_cast<float*>(d + (x - d0)) = *reinterpret_cast<const float*>(x);
            }
            if (hi > end) {
                hi = max(hi - 16, lo);
                for (uintptr_t x = hi; x < a1; x += 4) *reinterpret_cast<float*>(d + (x - d0)) = *reinterpret_cast<const float*>(x);
            }
            hi = max(hi, lo);
            mbar_expect_tx(&bars[slot], (uint32_t)(hi - lo));
            if (hi > lo) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             :: "r"(su32(d + (lo - d0))), "l"(lo), "r"((uint32_t)(hi - lo)), "r"(su32(&bars[slot])) : "memory");
            }
        };
        if (tid == 0 && *feed)
            for (int s = 0; s < min(stages, kBA_Slots); ++s) fill(s, (next + s) % kBA_Slots);
        // addresses by addition only: the loop's issue slots are the sums'
        const int step = RG * (int)(ld * 4), first = active ? rg * (int)(ld * 4) : 0, bytes = per * (int)(ld * 4);
        const int o0 = first + 4 * co[0], o1 = first + 4 * co[1], o2 = first + 4 * co[2], o3 = first + 4 * co[3];
        unsigned slot = next, parity = phase;
        int shift = (int)(base & 15), left = (int)m;
        const df64* qr = q + rg;
        // no barrier of the CTA between slots: a slot is filled again once every warp has released it
        bool ok = true;
        unsigned last = 0, last_parity = 0;
        int s = 0;
        for (; s < stages; ++s) {
            ok = __all_sync(0xffffffffu, mbar_try(&bars[slot], parity) || mbar_wait(&bars[slot], parity));
            if (!ok) break;
            if (tid == 0 && s > 0 && s - 1 + kBA_Slots < stages && mbar_wait(&freed[last], last_parity)) fill(s - 1 + kBA_Slots, last);
            if (active) {
                const unsigned char* f = ring + slot * slot_b + shift;
                const df64* qs = qr;
                const int rows = min(per, left);
                auto row = [&](const unsigned char* x, float (&y)[4]) {
                    y[0] = *reinterpret_cast<const float*>(x + o0);
                    y[1] = *reinterpret_cast<const float*>(x + o1);
                    y[2] = *reinterpret_cast<const float*>(x + o2);
                    y[3] = *reinterpret_cast<const float*>(x + o3);
                };
                int u = rg;
                for (; u + RG < rows; u += 2 * RG) {
                    float x[4], y[4];
                    row(f, x);
                    row(f + step, y);
                    bat_add<DOT>(acc, x, DOT ? qs[0] : df64{0.f, 0.f});
                    bat_add<DOT>(acc, y, DOT ? qs[RG] : df64{0.f, 0.f});
                    f += 2 * step;
                    qs += 2 * RG;
                }
                if (u < rows) {
                    float x[4];
                    row(f, x);
                    bat_add<DOT>(acc, x, DOT ? qs[0] : df64{0.f, 0.f});
                }
            }
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(&freed[slot]);
            last = slot;
            last_parity = parity;
            left -= per;
            qr += per;
            shift = (shift + bytes) & 15;
            if (++slot == kBA_Slots) { slot = 0; parity ^= 1u; }
        }
        if (!__syncthreads_and(ok)) {   // wait for the copies in flight, with the same limit, and give up
            for (int w = s; w < min(stages, s + kBA_Slots); ++w) {
                mbar_wait(&bars[slot], parity);
                if (++slot == kBA_Slots) { slot = 0; parity ^= 1u; }
            }
            return false;
        }
        next = slot;
        phase = parity;
    } else if (active) {   // rows too far apart for a slot
        for (int64_t i = rg; i < m; i += 4 * RG) {
            float x[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < 4; ++c) x[u][c] = i + u * RG < m ? __ldcs(A + (i + u * RG) * ld + co[c]) : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * RG < m) bat_add<DOT>(acc, x[u], DOT ? q[i + u * RG] : df64{0.f, 0.f});
        }
    }
    if (active)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int64_t j = cg + (int64_t)cgn * c;
            const Dot2 d = acc[c >> 1].half(c & 1);
            if (j < n) part[rg * n + j] = fast_two_sum(d.s, d.c);
        }
    __syncthreads();
    return true;
}

// order: the matrices by decreasing cost (r m n); queue: a zeroed counter. A CTA takes
// the next matrix of the order when it finishes one (largest first, so the tail is short). A CTA
// whose wait ran out records it and ends its matrix and what is left of the queue without picks: counts
// and J hold valid entries or -1 for every matrix whatever happens, and the padding and the gathers that
// follow rely on that. drop: the matrix whose copies are withheld, `count` for all of them, < 0 for none.
__global__ void __launch_bounds__(kBA_T, 2) bat_aca_k(const float* __restrict__ data, const BatAcaItem* items,
                                                       const int32_t* order, int* queue, int count, int32_t* J,
                                                       int32_t* counts, float* Qws, int slot_b, int drop, int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    df64* part = reinterpret_cast<df64*>(smem_raw);                      // RG x n
    double* nu = reinterpret_cast<double*>(part + kBA_RG * kBA_MaxN);
    df64* v = reinterpret_cast<df64*>(nu + kBA_MaxN);                    // m
    df64* qs = v + kBA_MaxM;                                             // r
    unsigned char* mask = reinterpret_cast<unsigned char*>(qs + kBA_MaxR);
    __shared__ double s_frob2;
    __shared__ int s_next, s_feed;
    unsigned char* ring = mask + kBA_MaxN;
    __shared__ __align__(8) uint64_t bars[kBA_Slots], freed[kBA_Slots];
    const int tid = threadIdx.x;
    unsigned next = 0, phase = 0;
    if (tid == 0) {
        for (int s = 0; s < kBA_Slots; ++s) {
            mbar_init(&bars[s], 1);
            mbar_init(&freed[s], kBA_T / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    float* Qh = Qws + (int64_t)blockIdx.x * 2 * kBA_MaxR * kBA_MaxM;
    float* Ql = Qh + (int64_t)kBA_MaxR * kBA_MaxM;
    // W(t, j) = q_t^T a_j from the passes (the CTA's slice after all CTAs' Q slices)
    df64* W = reinterpret_cast<df64*>(Qws + (int64_t)gridDim.x * 2 * kBA_MaxR * kBA_MaxM) +
              (int64_t)blockIdx.x * kBA_MaxR * kBA_MaxN;

    while (true) {
        if (tid == 0) s_next = atomicAdd(queue, 1);
        __syncthreads();
        const int q = s_next;
        __syncthreads();
        if (q >= count) break;
        const int it = order[q];
        const BatAcaItem b = items[it];
        const float* A = data + b.aoff;
        const int64_t m = b.m, n = b.n, ld = b.ld;
        const int r = b.r;
        // column groups of 4 columns; as many row groups as the CTA's threads cover, so every
        // thread streams (a narrow matrix would otherwise leave most of them idle)
        const int cgn = (int)((n + 3) / 4);
        const int RG = max(1, min((int)blockDim.x / cgn, (int)(kBA_RG * kBA_MaxN / n)));
        for (int j = tid; j < n; j += blockDim.x) mask[j] = 0;
        int picked = 0, bad = 0;
        if (tid == 0) s_feed = drop < 0 || (drop < count && drop != it);
        for (int t = -1; t < r - 1; ++t) {
            // ---- pass: squared norms (t = -1) or w = A^T q_t
            if (!(t < 0 ? bat_pass<false>(A, m, n, ld, cgn, RG, v, ring, slot_b, &s_feed, bars, freed, next, phase, part)
                        : bat_pass<true>(A, m, n, ld, cgn, RG, v, ring, slot_b, &s_feed, bars, freed, next, phase, part))) {
                if (tid != 0) return;
                set_status(status, CUR_ERR_TIMEOUT);
                int end = it, k0 = picked;
                while (true) {
                    const BatAcaItem e = items[end];
                    counts[end] = k0;
                    for (int k = k0; k < e.r; ++k) J[e.joff + k] = -1;
                    const int at = atomicAdd(queue, 1);
                    if (at >= count) return;
                    end = order[at];
                    k0 = 0;
                }
            }
            // ---- pick
            unsigned long long bk = dkey(-INFINITY);
            int bi = INT_MAX;
            double fs = 0.0;
            for (int j = tid; j < n; j += blockDim.x) {
                df64 w = part[j];
                for (int g = 1; g < RG; ++g) w = df_add(w, part[g * n + j]);
                const double wd = df_to_d(w);
                double nuj;
                if (t < 0) {
                    nuj = wd;
                    fs += wd;
                    if (!isfinite(wd)) bad = 1;
                } else {
                    nuj = nu[j] - wd * wd;
                    W[(int64_t)t * n + j] = w;
                }
                nu[j] = nuj;
                const unsigned long long kj = dkey(nuj);
                if (!mask[j] && (kj > bk || (kj == bk && j < bi))) { bk = kj; bi = j; }
            }
            bad = __syncthreads_or(bad);
            if (t < 0) {
                const df64 f = bat_df_sum(df64{(float)fs, (float)(fs - (double)(float)fs)});
                if (tid == 0) s_frob2 = df_to_d(f);
            }
            bat_argmax(bk, bi);
            if (bad) {
                if (tid == 0) set_status(status, CUR_ERR_NONFINITE);
                break;
            }
            if (bi == INT_MAX) break;
            const int p = bi;
            // ---- vector: v = a_p - Q W(:,p) (the first projection's coefficients q^T a_p are
            // the passes' w, as in the full-matrix kernel), then orthogonalised once more
            const int k = t + 1;
            for (int kk = tid; kk < k; kk += blockDim.x) qs[kk] = W[(int64_t)kk * n + p];
            __syncthreads();
            for (int64_t i = tid; i < m; i += 2 * blockDim.x) {
                const int64_t ib = i + blockDim.x;
                df64 a{A[i * ld + p], 0.f}, b{ib < m ? A[ib * ld + p] : 0.f, 0.f};
                bat_minus_q(Qh, Ql, m, k, i, ib < m ? ib : i, qs, a, b);
                v[i] = a;
                if (ib < m) v[ib] = b;
            }
            __syncthreads();
            bat_project(Qh, Ql, m, k, v, qs);
            df64 nv{0.f, 0.f};
            for (int64_t i = tid; i < m; i += blockDim.x) nv = df_add(nv, df_mul(v[i], v[i]));
            const double s_tot = df_to_d(bat_df_sum(nv));
            const double mx = (double)max(m, n) * 2.220446049250313e-16;
            if (!(s_tot > mx * mx * s_frob2)) break;
            if (tid == 0) {
                J[b.joff + k] = p;
                mask[p] = 1;
            }
            picked = k + 1;
            if (k == r - 1) break;
            const df64 inv = df_from_d(1.0 / sqrt(s_tot));
            for (int64_t i = tid; i < m; i += blockDim.x) {
                const df64 q = df_mul(v[i], inv);
                Qh[(int64_t)k * m + i] = q.h;
                Ql[(int64_t)k * m + i] = q.l;
                v[i] = q;
            }
            __syncthreads();
        }
        if (tid == 0) {
            counts[it] = picked;
            for (int k = picked; k < r; ++k) J[b.joff + k] = -1;
        }
        __syncthreads();
    }
}

}  // namespace curk

size_t bat_aca_workspace(int grid) {
    return (size_t)grid * 2 * curk::kBA_MaxR * curk::kBA_MaxM * sizeof(float) +
           (size_t)grid * curk::kBA_MaxR * curk::kBA_MaxN * sizeof(double);
}

cur_status bat_aca_launch(const float* data, const void* items_dev, const int32_t* order, int* queue, int count,
                          int32_t* J, int32_t* counts, float* Qws, int per_sm, int grid, int drop, int* status,
                          cudaStream_t st) {
    using namespace curk;
    CUR_TRY(smem_attr((const void*)bat_aca_k, bat_aca_smem(1)));
    CUR_CK(cudaMemsetAsync(queue, 0, sizeof(int), st));
    bat_aca_k<<<grid, kBA_T, bat_aca_smem(per_sm), st>>>(data, static_cast<const BatAcaItem*>(items_dev), order, queue,
                                                         count, J, counts, Qws, bat_slot_bytes(per_sm), drop, status);
    CUR_CK(cudaGetLastError());
    note_launch();
    return CUR_OK;
}

size_t bat_aca_item_size() { return sizeof(curk::BatAcaItem); }
