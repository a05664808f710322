// pa_noalloc.cu -- pa_resample_noalloc(): one resampling step that allocates
// no memory. For callers that cannot call cudaMalloc: a host framework that
// owns the device-memory budget through its own pool, and latency-critical
// loops where an allocator call may block, synchronise or fail. The caller
// passes the energies and receives the parents and copy counts in its own
// device buffers; every intermediate value lives in registers and shared
// memory, and the four results the host may ask for in one file-scope
// __device__ record shared by all calls.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "../../include/pa.h"
#include "pa_cluster.cuh"

namespace {

using pa::QPow;

constexpr int NA_MAX_R = PA_NOALLOC_MAX_R;   // 32768 replicas

// Every GPU that loads the library holds this record until the process exits.
// Each call writes all of it.
static __device__ pa_resample_result g_noalloc_result;

// One cluster: minimum, weights, tree sum and prefix (pa_cluster.cuh),
// systematic copy counts and parents: the arithmetic of the resampling inside
// pa_anneal. Bound by latency: one launch, three cluster barriers, FP64
// products. R = 16384 (8 CTAs, K = 2 slots per thread in registers): the call
// with its host result takes 29 us; with one CTA that kept weights, tree levels
// and integer weights in global memory (92 us) and four result copies it took
// 141 us.
template <int K>
__global__ void __launch_bounds__(pa::CL_THREADS) k_resample_noalloc(const int32_t *__restrict__ E, int32_t R,
                                                                     const QPow qp, uint32_t key0, uint32_t key1,
                                                                     uint32_t k, int32_t *__restrict__ parent,
                                                                     int32_t *__restrict__ counts,
                                                                     pa_resample_result *__restrict__ result) {
    namespace cg = cooperative_groups;
    __shared__ pa::ClusterShared sh;
    const int r0 = ((int)cg::this_cluster().block_rank() * pa::CL_THREADS + (int)threadIdx.x) * K;
    int32_t e[K], mn = 0x7FFFFFFF;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        e[i] = r0 + i < R ? E[r0 + i] : 0x7FFFFFFF;
        mn = min(mn, e[i]);
    }
    pa::cluster_table(sh, qp.v);
    const int32_t emin = pa::cluster_min(sh, mn);
    double w[K];
    unsigned long long t[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        w[i] = r0 + i < R ? pa::cluster_weight(sh, qp.v, (uint32_t)(e[i] - emin)) : 0.0;
        t[i] = (unsigned long long)__dmul_rn(w[i], 4294967296.0);
    }
    unsigned long long P = pa::cluster_sums<pa::CL_THREADS, K>(sh, w, t);
    const unsigned long long T = sh.T, m = ~0ull / T;
    const uint32_t o = pa::philox10(make_uint4(0u, 0u, k, pa::TAG_RESAMPLE), key0, key1).x;
    int32_t lo = pa::systematic_count_m(P, R, T, m, o);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        P += t[i];
        const int32_t hi = pa::systematic_count_m(P, R, T, m, o);
        if (r0 + i < R) {
            if (counts) counts[r0 + i] = hi - lo;
        }
        pa::fill_parents(parent, lo, r0 + i < R ? hi : lo, r0 + i);
        lo = hi;
    }
    if (r0 == 0) {
        pa_resample_result res;
        res.A = sh.A;
        res.T = T;
        res.emin = emin;
        res.o = o;
        *result = res;
    }
    cg::this_cluster().sync();   // no CTA leaves while another may read its totals
}

std::mutex g_noalloc_mutex;
void *g_noalloc_ptr[64] = {};

}  // namespace

extern "C" int pa_resample_noalloc(const int32_t *energies, int32_t R, double beta_prev, double beta_k,
                                   uint64_t seed, int32_t k, int32_t *parent, int32_t *counts,
                                   pa_resample_result *out, void *stream) {
    if (!energies || !parent || R < 1 || R > NA_MAX_R || k < 0) return PA_EINVAL;
    if (!std::isfinite(beta_prev) || !std::isfinite(beta_k) || beta_prev < 0.0 || beta_k < beta_prev)
        return PA_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return PA_ECUDA;
    void *base = nullptr;
    {
        // Set-up once per device, with that device current: host code only has a
        // stand-in for the __device__ array, so its device address is looked up.
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_result) != cudaSuccess || !p) {
                cudaGetLastError();
                return PA_ECUDA;
            }
            g_noalloc_ptr[dev] = p;
        }
        base = g_noalloc_ptr[dev];
    }
    pa_resample_result *result = reinterpret_cast<pa_resample_result *>(base);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    QPow qp;
    double sq = std::exp(-(beta_k - beta_prev));
    for (int b = 0; b < 32; ++b) {
        qp.v[b] = sq;
        sq = sq * sq;
    }
    const pa::ClusterShape shape = pa::cluster_shape(R, pa::CL_THREADS);
    auto *kernel = shape.k == 1 ? &k_resample_noalloc<1> : shape.k == 2 ? &k_resample_noalloc<2> : &k_resample_noalloc<4>;
    if (pa::launch_cluster(kernel, shape, pa::CL_THREADS, st, false, energies, R, qp, (uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)k, parent,
                           counts, result) != cudaSuccess) {
        cudaGetLastError();
        return PA_ECUDA;
    }
    if (out) {
        pa_resample_result res;
        if (cudaMemcpyAsync(&res, result, sizeof(res), cudaMemcpyDeviceToHost, st) != cudaSuccess) return PA_ECUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return PA_ECUDA;
        *out = res;
    }
    return PA_OK;
}
