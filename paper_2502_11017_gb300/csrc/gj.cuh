// FP64 Gauss-Jordan inverse of an r x r matrix (r <= 128) with partial pivoting, as a dataflow
// over the warps of one CTA or of a thread-block cluster.
//
// What bounds an inverse: r dependent steps (pivot search, one FP64 division, the elimination of
// the next column), and r^3 FP64 multiply-adds on a pipe that does two per clock and SM (0.55 ms
// for r = 128 on one SM). gj_inverse (common.cuh) keeps the matrix in shared memory and meets
// two block barriers a step; here a warp holds whole columns in registers (lane = row, rows
// lane + 32 u) and nothing but the step's message is shared: the warp that holds column k + 1
// brings it up to date first, finds its pivot, and posts (pivot row, pivot, reciprocal, the
// column after the interchange) into every CTA's shared memory, one slot and one mbarrier per
// step, so that no slot is ever reused and no warp waits for another but through the messages.
// A row interchange is two shuffles. With NC CTAs in the cluster the columns, and the FP64 work,
// are spread over NC SMs; consecutive columns mostly stay on one CTA, so the chain of pivots
// crosses SMs only NC - 1 times.
// Same pivots (first maximum, integer keys) and the same operation per element as gj_inverse:
// bit-identical inverses. Kernel times: r = 64 203 -> 101 us (assembly, four SMs), r = 128
// 1218 -> 240 us (eight SMs); r = 16 31 -> 27 us (the chain alone).
#pragma once

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace curk {

constexpr int kGjWarps = 16;   // 512 threads per CTA

__device__ __forceinline__ unsigned gj_rank() { unsigned x; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(x)); return x; }
__device__ __forceinline__ unsigned gj_size() { unsigned x; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(x)); return x; }
__device__ __forceinline__ void gj_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t gj_mapa(uint32_t addr, unsigned rank) {
    uint32_t x;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(x) : "r"(addr), "r"(rank));
    return x;
}
__device__ __forceinline__ void gj_st(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void gj_st(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
// Arrival on a CTA's mbarrier (release at cluster scope).
__device__ __forceinline__ void gj_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ bool gj_wait(uint64_t* b) {
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0; selp.u32 %0, 1, 0, p; }"
                     : "=r"(done) : "r"(su32(b)) : "memory");
        if (done) return true;
        if (clock64() - t0 > kTcWait) return false;
    }
}

// Shared memory: the steps' columns (r x r), pivots, reciprocals, pivot rows, mbarriers, and the
// final place of each column.
struct GjSmem {
    double* col;
    double* d;
    double* dinv;
    uint64_t* bar;
    int* p;
    int* perm;
    __host__ __device__ static size_t bytes(int r) { return ((size_t)r * r + 3 * (size_t)r) * 8 + 2 * (size_t)r * 4 + 16; }
    __device__ GjSmem(unsigned char* base, int r) {
        col = reinterpret_cast<double*>(base);
        d = col + (size_t)r * r;
        dinv = d + r;
        bar = reinterpret_cast<uint64_t*>(dinv + r);
        p = reinterpret_cast<int*>(bar + r);
        perm = p + r;
    }
};

// The columns of a warp: [c0, c0 + n), n <= CPW.
__device__ __forceinline__ void gj_columns(int r, int cpw, int& c0, int& n) {
    const int cw = (r + (int)gj_size() - 1) / (int)gj_size();
    const int first = (int)gj_rank() * cw, end = min(r, first + cw);
    c0 = first + (int)(threadIdx.x >> 5) * cpw;
    n = max(0, min(cpw, end - c0));
}

// a = i == j ? b : a. (A chain of '?:' over an array is turned into an indexed load, and the
// columns then live in local memory instead of registers.)
__device__ __forceinline__ void gj_pick(double& a, double b, int i, int j) {
    asm("{ .reg .pred p; setp.eq.s32 p, %2, %3; selp.f64 %0, %1, %0, p; }" : "+d"(a) : "d"(b), "r"(i), "r"(j));
}
template <int RU>
__device__ __forceinline__ double gj_row(const double (&v)[RU], int i) {   // entry of row i, on every lane
    double x = v[0];
#pragma unroll
    for (int u = 1; u < RU; ++u) gj_pick(x, v[u], i >> 5, u);
    return __shfl_sync(0xffffffffu, x, i & 31);
}

// The pivot of column k (this warp's v, final up to step k - 1), posted to every CTA (but, for the
// self-test, the last step's not to CTA `mute`).
template <int RU>
__device__ __forceinline__ void gj_post(const GjSmem& s, const double (&v)[RU], int k, int r, int mute) {
    const int lane = threadIdx.x & 31;
    unsigned long long bk = 0ull;
    long long bi = k;
#pragma unroll
    for (int u = 0; u < RU; ++u) {
        const int i = lane + 32 * u;
        if (i >= k && i < r) {
            const unsigned long long x = dkey(fabs(v[u]));
            if (x > bk) { bk = x; bi = i; }
        }
    }
    warp_argmax_key(bk, bi);
    const int p = (int)bi;
    const double d = gj_row<RU>(v, p), vk = gj_row<RU>(v, k);
    double ck[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
        const int i = lane + 32 * u;
        ck[u] = i == k ? d : (i == p ? vk : v[u]);
        if (i < r) s.col[(size_t)k * r + i] = ck[u];
    }
    const double dinv = 1.0 / d;
    if (lane == 0) {
        s.d[k] = d;
        s.dinv[k] = dinv;
        s.p[k] = p;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s.bar[k]);
    const unsigned nc = gj_size(), me = gj_rank();
    if (nc == 1) return;
    auto muted = [&](unsigned q) { return mute >= 0 && k == r - 1 && (int)q == mute; };
    for (unsigned q = 0; q < nc; ++q) {
        if (q == me || muted(q)) continue;
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int i = lane + 32 * u;
            if (i < r) gj_st(gj_mapa(su32(s.col + (size_t)k * r + i), q), ck[u]);
        }
        if (lane == 0) {
            gj_st(gj_mapa(su32(s.d + k), q), d);
            gj_st(gj_mapa(su32(s.dinv + k), q), dinv);
            gj_st(gj_mapa(su32(s.p + k), q), p);
        }
    }
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
    __syncwarp();
    if ((unsigned)lane < nc && (unsigned)lane != me && !muted((unsigned)lane)) gj_arrive(gj_mapa(su32(s.bar + k), (unsigned)lane));
}

// Step k on one column c (RU rows per lane): interchange of rows k and p, elimination.
template <int RU>
__device__ __forceinline__ void gj_step(double (&v)[RU], const double (&ck)[RU], int c, int k, int p, double dinv) {
    const int lane = threadIdx.x & 31;
    const double ap = gj_row<RU>(v, p), ak = gj_row<RU>(v, k);
    const double pr = (c == k ? 1.0 : ap) * dinv;
#pragma unroll
    for (int u = 0; u < RU; ++u) {
        const int i = lane + 32 * u;
        const double base = c == k ? 0.0 : (i == p ? ak : v[u]);
        v[u] = i == k ? pr : fma(-ck[u], pr, base);
    }
}

// In-place inverse of the matrix whose columns c0 .. c0 + n - 1 this warp holds in v (v[s][u] =
// row lane + 32 u of column c0 + s; rows past r zero). All threads of every CTA of the cluster
// call it with 512 threads per CTA. A pivot with !(|pivot| > thresh) ends it: returns 1
// (singular), 2 after a wait that ran out (in any CTA: what the others hold is then not a whole
// inverse), else 0; the same value in every thread of the cluster. After 0 column c0 + s belongs
// at column s.perm[c0 + s] of the inverse.
// logabsdet (may be null): log|det|, in the threads of each CTA's first warp.
template <int RU, int CPW>
__device__ __forceinline__ int gj_flow(const GjSmem& s, int r, double thresh, double (&v)[CPW][RU], int c0, int n,
                                       double* logabsdet, int mute = -1) {
    const int lane = threadIdx.x & 31;
    __shared__ int s_out, s_lost;   // s_lost: a wait ran out in some CTA of the cluster
    if (threadIdx.x == 0) s_out = s_lost = 0;
    for (int k = threadIdx.x; k < r; k += blockDim.x) mbar_init(&s.bar[k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    gj_cluster_sync();
    int out = 0;
    if (c0 == 0 && n > 0) gj_post<RU>(s, v[0], 0, r, mute);
    if (n > 0) {
        for (int k = 0; k < r; ++k) {
            if (!__all_sync(0xffffffffu, gj_wait(&s.bar[k]))) { out = 2; break; }
            const double d = s.d[k], dinv = s.dinv[k];
            const int p = s.p[k];
            if (!(fabs(d) > thresh)) { out = 1; break; }
            double ck[RU];
#pragma unroll
            for (int u = 0; u < RU; ++u) ck[u] = lane + 32 * u < r ? s.col[(size_t)k * r + lane + 32 * u] : 0.0;
            const int nx = k + 1 - c0;   // slot of column k + 1
            if (nx >= 0 && nx < n) {
                double t[RU];   // selected and put back by constant indices: v stays in registers
#pragma unroll
                for (int u = 0; u < RU; ++u) t[u] = v[0][u];
#pragma unroll
                for (int q = 1; q < CPW; ++q)
#pragma unroll
                    for (int u = 0; u < RU; ++u) gj_pick(t[u], v[q][u], q, nx);
                gj_step<RU>(t, ck, k + 1, k, p, dinv);
                gj_post<RU>(s, t, k + 1, r, mute);
#pragma unroll
                for (int q = 0; q < CPW; ++q)
#pragma unroll
                    for (int u = 0; u < RU; ++u) gj_pick(v[q][u], t[u], q, nx);
            }
#pragma unroll
            for (int q = 0; q < CPW; ++q)
                if (q != nx && q < n) gj_step<RU>(v[q], ck, c0 + q, k, p, dinv);
        }
    }
    if (out && lane == 0) atomicMax(&s_out, out);
    __syncthreads();
    if (threadIdx.x == 0 && s_out == 0) {   // (a CTA whose warps hold no column follows the messages here)
        for (int k = 0; k < r && s_out == 0; ++k) {
            if (!gj_wait(&s.bar[k])) s_out = 2;
            else if (!(fabs(s.d[k]) > thresh)) s_out = 1;
        }
    }
    __syncthreads();
    if (s_out == 0) {
        // the row interchanges undone on the columns, from the last to the first
        for (int c = threadIdx.x; c < r; c += blockDim.x) {
            int at = c;
            for (int k = r - 1; k >= 0; --k) {
                const int p = s.p[k];
                at = at == k ? p : (at == p ? k : at);
            }
            s.perm[c] = at;
        }
        if (logabsdet && threadIdx.x < 32) {   // |det|: four pivots per lane in order, then a tree
            LogAcc acc;
            acc.init();
            const int per = (r + 31) / 32;
            for (int k = lane * per; k < min(r, (lane + 1) * per); ++k) acc.mul(df_from_d(s.d[k]));
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const df64 m{__shfl_xor_sync(0xffffffffu, acc.mant.h, o), __shfl_xor_sync(0xffffffffu, acc.mant.l, o)};
                const int e = __shfl_xor_sync(0xffffffffu, acc.expo, o);
                acc.mul(m);
                acc.expo += e;
            }
            *logabsdet = acc.log_value();
        }
    }
    if (threadIdx.x < gj_size() && s_out == 2) gj_st(gj_mapa(su32(&s_lost), threadIdx.x), 1);
    gj_cluster_sync();   // no CTA leaves while another may still write to its shared memory
    return s_lost ? 2 : s_out;
}

inline int gj_cpw(int r, int nc) {   // columns per warp with nc CTAs
    const int cw = (r + nc - 1) / nc, w = (cw + kGjWarps - 1) / kGjWarps;
    return w <= 1 ? 1 : (w <= 2 ? 2 : (w <= 4 ? 4 : 8));
}

// CTAs and columns per warp of a single inverse. A step's FP64 work on one SM is r^2 / 2 clocks, its
// chain of dependent operations ~600: SMs are added until the work is the shorter (r = 64:
// four, 128: eight, the portable cluster size).
inline void gj_plan(int r, int* nc, int* cpw) {
    int c = 1;
    while (c < 8 && r * r > 1200 * c) c *= 2;
    *nc = c;
    *cpw = gj_cpw(r, c);
}

// CTAs per inverse for a stage of P, 0 for one CTA each with the matrix in shared memory (gj_inverse).
// Clusters win while all of them run at once; a stage that fills the GPU is bound by the FP64 pipe, which
// gj_inverse keeps busier (it has no padded columns and fits several CTAs on an SM). us a stage, with
// clusters of the size taken and with one CTA each in shared memory:
//   r = 16   P = 152 26 and 32, 1024 108 and 137     r = 32   P = 152 55 and 59, 304 76 and 72, 1024 294 and 254
//   r = 48   P = 76 83 and 95                        r = 64   P = 36 90 and 140, 76 120 and 140
//   r = 72   P = 19 140 and 174                      r = 80   P = 36 203 and 230
//   r = 96   P = 76 328 and 353                      r = 128  P = 16 474 and 726, 76 524 and 726
// One CTA each in registers is the slower one above r = 32 (r = 64: P = 152 169 and 142, 1024 955 and 763;
// r = 96: 484 and 351, 3352 and 2051), as are two CTAs at 65 <= r <= 88 (252 and 230 at 80) and four at
// r <= 74 (162 and 140 at 65). 36 clusters of four run at once, not 38 (r = 96: 247 and 490).
inline int gj_stage_plan(int r, int P, int num_sms) {
    if (r <= 32) return r > 24 && P > num_sms ? 0 : 1;
    if (r > 64 && 8LL * P <= num_sms) return 8;
    if (r > 48 && (r <= 64 || r > 74) && 4LL * P <= num_sms - 8) return 4;
    if (r > 34 && (r <= 64 || r > 88) && 2LL * P <= num_sms) return 2;
    return 0;
}

// KERNEL<..., RU, CPW> for a rank and a plan; X(RU, CPW) names it.
#define GJ_KERNEL(r, cpw, X)                                                             \
    ((r) <= 32   ? ((cpw) == 1 ? X(1, 1) : X(1, 2))                                      \
     : (r) <= 64 ? ((cpw) == 1 ? X(2, 1) : ((cpw) == 2 ? X(2, 2) : X(2, 4)))             \
                 : ((cpw) == 1 ? X(4, 1) : ((cpw) == 2 ? X(4, 2) : ((cpw) == 4 ? X(4, 4) : X(4, 8)))))

// Launches a kernel of clusters of nc CTAs, 512 threads each.
template <typename... K, typename... A>
inline cur_status gj_launch(void (*kernel)(K...), int ctas, int nc, size_t smem, cudaStream_t st, A... args) {
    CUR_TRY(smem_attr(reinterpret_cast<const void*>(kernel), smem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(32 * kGjWarps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    CUR_CK(cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...));
    note_launch();
    return CUR_OK;
}

}  // namespace curk
