// pa_cluster.cuh -- the weight arithmetic of one resampling over a population
// (or one rank's shard of it) in a single thread-block cluster: every step's
// resampling (k_rs_step) and the resampling entry points on caller buffers,
// where a launch does all of it by itself.
//
// n slots, padded with zero weights to L = NT K C: CTA c of the C <= 8 CTAs of
// NT threads holds the aligned range of L / C slots, thread t of it K
// consecutive ones in registers. So the pairwise tree (s_i <- s_2i + s_2i+1) runs inside the thread,
// over the lanes, over the warps and over the CTAs, in the order of the
// level-by-level tree, and the integer prefix likewise; two cluster barriers
// replace the passes over global memory.
#pragma once

#include <cooperative_groups.h>

#include "pa_internal.cuh"

namespace pa {

constexpr int CL_THREADS = 1024;  // where the resampling is the whole call
constexpr int CL_CTAS = 8;        // portable cluster size
constexpr int CL_LOW = 8;         // low bits of E - E_min whose products are tabled

struct QPow {
    double v[32];   // squarings of q = exp(-(beta_k - beta_prev))
};

// CTAs and slots per thread for n slots (n <= 65536).
struct ClusterShape {
    int ctas, k;
};
__host__ inline ClusterShape cluster_shape(int32_t n, int threads) {
    int L = threads;
    while (L < n) L <<= 1;
    ClusterShape s;
    s.ctas = L / threads < CL_CTAS ? L / threads : CL_CTAS;
    s.k = L / (threads * s.ctas);
    return s;
}

struct ClusterShared {
    double tab[1 << CL_LOW];          // products of the squarings over the bits of the index
    double wsum[32];
    unsigned long long tsum[32];
    int32_t mn[32];
    double ctaA;
    unsigned long long ctaT;
    int32_t ctaMin;
    double A;                          // totals over the cluster (every CTA has them)
    unsigned long long T, before;      // before: total of the lower CTAs
    int32_t emin;
};

// Products over the low bits, multiplied in ascending bit order from 1.0, so a
// weight that starts from its entry is rounded as the plain product is.
__device__ __forceinline__ void cluster_table(ClusterShared &sh, const double *q) {
    for (int i = threadIdx.x; i < (1 << CL_LOW); i += blockDim.x) {
        double w = 1.0;
#pragma unroll
        for (int b = 0; b < CL_LOW; ++b)
            if ((i >> b) & 1) w = __dmul_rn(w, q[b]);
        sh.tab[i] = w;
    }
}

__device__ __forceinline__ double cluster_weight(const ClusterShared &sh, const double *q, uint32_t d) {
    double w = sh.tab[d & ((1u << CL_LOW) - 1u)];
    d >>= CL_LOW;
    while (d) {
        w = __dmul_rn(w, q[CL_LOW + __ffs(d) - 1]);
        d &= d - 1u;
    }
    return w;
}

// E_min over the cluster of each thread's minimum.
__device__ __forceinline__ int32_t cluster_min(ClusterShared &sh, int32_t v) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = __reduce_min_sync(0xFFFFFFFFu, v);
    if (lane == 0) sh.mn[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = __reduce_min_sync(0xFFFFFFFFu, sh.mn[lane]);
        if (lane == 0) sh.ctaMin = v;
    }
    cl.sync();
    if (warp == 0) {
        const int C = (int)cl.num_blocks();
        v = *cl.map_shared_rank(&sh.ctaMin, lane < C ? lane : 0);
        v = __reduce_min_sync(0xFFFFFFFFu, v);
        if (lane == 0) sh.emin = v;
    }
    __syncthreads();
    return sh.emin;
}

// Tree sum A, integer total T and each thread's exclusive prefix of t (over the
// cluster) from the K weights a thread holds. Ends with sh.A, sh.T set in every
// CTA; the caller closes with a cluster barrier before any CTA leaves.
template <int NT, int K>
__device__ __forceinline__ unsigned long long cluster_sums(ClusterShared &sh, const double (&w)[K],
                                                           const unsigned long long (&t)[K]) {
    constexpr int NW = NT / 32;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double s[K];
    unsigned long long loc = 0ull;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        s[i] = w[i];
        loc += t[i];
    }
#pragma unroll
    for (int h = 1; h < K; h <<= 1)
#pragma unroll
        for (int i = 0; i < K; i += 2 * h) s[i] = __dadd_rn(s[i], s[i + h]);
    double a = s[0];
    unsigned long long inc = loc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        a = __dadd_rn(a, __shfl_xor_sync(0xFFFFFFFFu, a, off));
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += y;
    }
    if (lane == 31) {
        sh.wsum[warp] = a;
        sh.tsum[warp] = inc;
    }
    __syncthreads();
    if (warp == 0) {
        double b = lane < NW ? sh.wsum[lane] : 0.0;
        unsigned long long u = lane < NW ? sh.tsum[lane] : 0ull;
        const unsigned long long mine = u;
#pragma unroll
        for (int off = 1; off < NW; off <<= 1) {
            b = __dadd_rn(b, __shfl_xor_sync(0xFFFFFFFFu, b, off));
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, u, off);
            if (lane >= off) u += y;
        }
        if (lane < NW) sh.tsum[lane] = u - mine;   // exclusive over the warps
        if (lane == NW - 1) {
            sh.ctaA = b;
            sh.ctaT = u;
        }
    }
    cl.sync();
    if (warp == 0) {
        const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
        double b = lane < C ? *cl.map_shared_rank(&sh.ctaA, lane < C ? lane : 0) : 0.0;
        unsigned long long T = lane < C ? *cl.map_shared_rank(&sh.ctaT, lane < C ? lane : 0) : 0ull;
        unsigned long long before = lane < rank ? T : 0ull;
#pragma unroll
        for (int off = 1; off < CL_CTAS; off <<= 1) {
            b = __dadd_rn(b, __shfl_xor_sync(0xFFFFFFFFu, b, off));
            T += __shfl_xor_sync(0xFFFFFFFFu, T, off);
            before += __shfl_xor_sync(0xFFFFFFFFu, before, off);
        }
        if (lane == 0) {
            sh.A = b;
            sh.T = T;
            sh.before = before;
        }
    }
    __syncthreads();
    return sh.before + sh.tsum[warp] + (inc - loc);
}

// Slots [lo, hi) of `parent` get r on every lane of the warp: short runs by the
// lane itself, runs above eight slots (few replicas carry the weight late in an
// anneal) by the whole warp, so that one long run does not serialise it.
__device__ __forceinline__ void fill_parents(int32_t *__restrict__ parent, int32_t lo, int32_t hi, int32_t r) {
    const int lane = threadIdx.x & 31;
    const bool many = hi - lo > 8;
    if (!many)
        for (int32_t q = lo; q < hi; ++q) parent[q] = r;
    for (uint32_t b = __ballot_sync(0xFFFFFFFFu, many); b; b &= b - 1u) {
        const int src = __ffs(b) - 1;
        const int32_t l = __shfl_sync(0xFFFFFFFFu, lo, src), h = __shfl_sync(0xFFFFFFFFu, hi, src);
        const int32_t v = __shfl_sync(0xFFFFFFFFu, r, src);
        for (int32_t q = l + lane; q < h; q += 32) parent[q] = v;
    }
}

// Launches a cluster kernel of `shape` on st; early: see wait_previous.
template <class... P, class... A>
cudaError_t launch_cluster(void (*kernel)(P...), const ClusterShape &shape, int threads, cudaStream_t st, bool early, A... args) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(shape.ctas);
    lc.blockDim = dim3(threads);
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = shape.ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    early_attribute(at[1]);
    lc.attrs = at;
    lc.numAttrs = early ? 2 : 1;
    return cudaLaunchKernelEx(&lc, kernel, args...);
}

}  // namespace pa
