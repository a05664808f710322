// pa_shard.cu -- resampling of one population split over G ranks (replica
// sharding). Each rank holds the aligned power-of-two slot range
// [g R/G, (g+1) R/G) of a population of R = 2^a replicas, so its slots form
// one subtree of the pairwise weight tree of the single-population resampling
// (Sec. 3 names population annealing; the reweighting and systematic
// resampling follow the library's reading: weights q^(E - E_min) as FP64
// products of squarings, pairwise tree sum A, integer weights floor(2^32 w),
// copies F(P + t) - F(P) with F(P) = floor((P R 2^32 + o T) / (T 2^32))).
//
// One step on rank g:
//   1. pa_shard_min       E_min,g of the rank's energies; the caller reduces
//                         E_min = min over ranks;
//   2. pa_shard_partials  weights with that E_min, the subtree sum A_g, the
//                         integer weights t_r, their total T_g and local
//                         exclusive prefix, in caller scratch;
//   3. the caller gathers (A_h, T_h) of every rank;
//   4. pa_shard_plan      (host) A = pairwise tree over the A_h in rank order,
//                         which is the top of the single-population tree, so A
//                         is bitwise the single-population value; T = sum T_h;
//                         P_base = sum_{h<g} T_h; the new slots this rank's
//                         parents fill, [F(P_base), F(P_base + T_g)) (systematic
//                         resampling keeps parent order, so they are contiguous),
//                         and how many rows go to and come from every rank;
//   5. pa_shard_parents   for each of those new slots, its local parent;
//   6. pa_shard_gather    the rows (spins, energy) in new-slot order, ready
//                         for an all-to-all whose send counts pa_shard_plan
//                         gave; received rows arrive in new-slot order.
// All integer sums are exact, so counts, parents and rows equal the
// single-population resampling bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "../../include/pa.h"
#include "pa_cluster.cuh"

namespace {

constexpr int SH_THREADS = 1024;

using pa::QPow;

__global__ void __launch_bounds__(SH_THREADS) k_shard_min(const int32_t *__restrict__ E, int32_t n,
                                                          int32_t *__restrict__ out) {
    __shared__ int32_t sh[SH_THREADS / 32];
    int v = 0x7FFFFFFF;
    for (int r = threadIdx.x; r < n; r += SH_THREADS) v = min(v, E[r]);
    v = __reduce_min_sync(0xFFFFFFFFu, v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = sh[0];
        for (int w = 1; w < SH_THREADS / 32; ++w) m = min(m, sh[w]);
        *out = m;
    }
}

// Scratch (caller device memory, pa_shard_scratch_bytes(n)): t[n] and pre[n]
// (exclusive prefix) as 64-bit integers, then A and T, after an unused part of
// 3/2 L doubles (L = n rounded up to a power of two) that belongs to the size
// callers were told.
struct ShardScratch {
    unsigned long long *t, *pre;
    double *A;
    unsigned long long *T;
};

__host__ __device__ inline int32_t pow2_ceil(int32_t n) {
    int32_t L = 1;
    while (L < n) L <<= 1;
    return L;
}

__host__ __device__ inline ShardScratch scratch_view(void *base, int32_t n) {
    const int32_t L = pow2_ceil(n);
    ShardScratch s;
    s.t = reinterpret_cast<unsigned long long *>(base) + L + (L > 1 ? L / 2 : 1);
    s.pre = s.t + n;
    s.A = reinterpret_cast<double *>(s.pre + n);
    s.T = reinterpret_cast<unsigned long long *>(s.A + 1);
    return s;
}

// Weights, tree sum, integer weights and their prefix in one cluster
// (pa_cluster.cuh). n = 16384: 88 us with one CTA and the tree in global
// memory, 8.8 us now.
template <int K>
__global__ void __launch_bounds__(pa::CL_THREADS) k_shard_partials(const int32_t *__restrict__ E, int32_t n,
                                                                   int32_t emin, const QPow qp, ShardScratch s) {
    namespace cg = cooperative_groups;
    __shared__ pa::ClusterShared sh;
    const int r0 = ((int)cg::this_cluster().block_rank() * pa::CL_THREADS + (int)threadIdx.x) * K;
    pa::cluster_table(sh, qp.v);
    __syncthreads();
    double w[K];
    unsigned long long t[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        w[i] = r0 + i < n ? pa::cluster_weight(sh, qp.v, (uint32_t)(E[r0 + i] - emin)) : 0.0;
        t[i] = (unsigned long long)__dmul_rn(w[i], 4294967296.0);
    }
    unsigned long long P = pa::cluster_sums<pa::CL_THREADS, K>(sh, w, t);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        if (r0 + i < n) {
            s.t[r0 + i] = t[i];
            s.pre[r0 + i] = P;
        }
        P += t[i];
    }
    if (r0 == 0) {
        *s.A = sh.A;
        *s.T = sh.T;
    }
    cg::this_cluster().sync();   // no CTA leaves while another may read its totals
}

// floor((P R 2^32 + o T) / (T 2^32)) for R <= 65536 (P R < 2^64): written as
// floor(P R / T) + [(P R mod T) 2^32 >= T (2^32 - o)].
__host__ __device__ inline int32_t shard_count(unsigned long long P, int32_t R, unsigned long long T, uint32_t o) {
    if (P >= T) return R;
    const unsigned long long X = P * (unsigned long long)R;
    const unsigned long long q = X / T, r = X - q * T;
    const unsigned __int128 lhs = (unsigned __int128)r << 32;
    const unsigned __int128 rhs = (unsigned __int128)T * (0x100000000ull - (unsigned long long)o);
    return (int32_t)(q + (lhs >= rhs ? 1ull : 0ull));
}

__global__ void k_shard_parents(ShardScratch s, int32_t n, unsigned long long P_base, unsigned long long T,
                                int32_t R, uint32_t o, int32_t new_lo, int32_t *__restrict__ src,
                                int32_t *__restrict__ counts) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        const unsigned long long P = P_base + s.pre[r];
        const int32_t lo = shard_count(P, R, T, o), hi = shard_count(P + s.t[r], R, T, o);
        for (int32_t q = lo; q < hi; ++q) src[q - new_lo] = r;
        if (counts) counts[r] = hi - lo;
    }
}

// Rows in new-slot order, one CTA (short rows: one warp) per row: bound by the
// copy's bandwidth. VEC: rows of whole 16-byte units at 16-byte boundaries move
// four units per thread at a time, otherwise byte by byte where the start or the
// end of a row is not at a word boundary and word by word in between (the source
// words shifted into place). 16384 rows of 7008 bytes from a flushed L2: 216 us byte by byte, 40 us in
// units (14,803 distinct rows read, 5.5 TB/s; identity 42 us).
constexpr int GATHER_THREADS = 128;

template <bool VEC, int NT>
__global__ void __launch_bounds__(GATHER_THREADS) k_shard_gather(const int8_t *__restrict__ spins,
                                                                 const int32_t *__restrict__ E, int32_t ncols,
                                                                 const int32_t *__restrict__ src, int32_t nout,
                                                                 int8_t *__restrict__ spins_out,
                                                                 int32_t *__restrict__ E_out) {
    constexpr int ROWS = GATHER_THREADS / NT;   // rows of the CTA at a time
    const int tid = threadIdx.x % NT;
    for (int j = (int)blockIdx.x * ROWS + (int)threadIdx.x / NT; j < nout; j += (int)gridDim.x * ROWS) {
        const int32_t r = src[j];
        const int8_t *in = spins + (size_t)r * ncols;
        int8_t *out = spins_out + (size_t)j * ncols;
        if (VEC) {
            const uint4 *vi = reinterpret_cast<const uint4 *>(in);
            uint4 *vo = reinterpret_cast<uint4 *>(out);
            const int nv = ncols >> 4;
            for (int c0 = tid; c0 < nv; c0 += 4 * NT) {
                uint4 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c0 + q * NT < nv) v[q] = __ldg(&vi[c0 + q * NT]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c0 + q * NT < nv) vo[c0 + q * NT] = v[q];
            }
        } else {
            // Output words [w0, w1) whose source words lie wholly inside the row.
            const uintptr_t ob = reinterpret_cast<uintptr_t>(out), ib = reinterpret_cast<uintptr_t>(in);
            const int head = (int)((4 - (ob & 3)) & 3) + 4;
            const int words = ncols > head + 8 ? (ncols - head - 4) >> 2 : 0;
            const int sh = (int)((ib + head) & 3);
            const uint32_t *wi = reinterpret_cast<const uint32_t *>(ib + head - sh);
            uint32_t *wo = reinterpret_cast<uint32_t *>(ob + head);
            for (int c = tid; c < words; c += NT)
                wo[c] = sh ? __funnelshift_r(__ldg(&wi[c]), __ldg(&wi[c + 1]), 8 * sh) : __ldg(&wi[c]);
            const int tail = words ? head + 4 * words : 0;
            if (words && tid < head) out[tid] = in[tid];
            for (int c = tail + tid; c < ncols; c += NT) out[c] = in[c];
        }
        if (tid == 0 && E) E_out[j] = E[r];
    }
}

bool is_pow2(int32_t x) { return x > 0 && (x & (x - 1)) == 0; }

}  // namespace

extern "C" {

size_t pa_shard_scratch_bytes(int32_t n) {
    if (n < 1) return 0;
    const size_t L = (size_t)pow2_ceil(n);
    return 8 * (L + (L > 1 ? L / 2 : 1) + 2 * (size_t)n + 2);
}

int pa_shard_min(const int32_t *energies, int32_t n, int32_t *scratch, int32_t *emin, void *stream) {
    if (!energies || !scratch || !emin || n < 1) return PA_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    k_shard_min<<<1, SH_THREADS, 0, st>>>(energies, n, scratch);
    if (cudaGetLastError() != cudaSuccess) return PA_ECUDA;
    if (cudaMemcpyAsync(emin, scratch, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return PA_ECUDA;
    return PA_OK;
}

int pa_shard_partials(const int32_t *energies, int32_t n, int32_t emin, double beta_prev, double beta_k,
                      void *scratch, double *A, uint64_t *T, void *stream) {
    if (!energies || !scratch || !A || !T || n < 1 || n > PA_SHARD_MAX_SLOTS) return PA_EINVAL;
    if (!std::isfinite(beta_prev) || !std::isfinite(beta_k) || beta_prev < 0.0 || beta_k < beta_prev) return PA_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    QPow qp;
    double sq = std::exp(-(beta_k - beta_prev));
    for (int b = 0; b < 32; ++b) {
        qp.v[b] = sq;
        sq = sq * sq;
    }
    const ShardScratch s = scratch_view(scratch, n);
    const pa::ClusterShape shape = pa::cluster_shape(n, pa::CL_THREADS);
    auto *kernel = shape.k == 1   ? &k_shard_partials<1>
                   : shape.k == 2 ? &k_shard_partials<2>
                   : shape.k == 4 ? &k_shard_partials<4>
                                  : &k_shard_partials<8>;
    if (pa::launch_cluster(kernel, shape, pa::CL_THREADS, st, false, energies, n, emin, qp, s) != cudaSuccess) {
        cudaGetLastError();
        return PA_ECUDA;
    }
    struct {
        double A;
        unsigned long long T;
    } res;   // A and T lie side by side
    if (cudaMemcpyAsync(&res, s.A, sizeof(res), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return PA_ECUDA;
    *A = res.A;
    *T = res.T;
    return PA_OK;
}

int pa_shard_plan(int32_t G, int32_t g, int32_t R, const double *A_all, const uint64_t *T_all, uint32_t o,
                  pa_shard_step *out) {
    if (!A_all || !T_all || !out || !is_pow2(G) || G > PA_SHARD_MAX_RANKS || g < 0 || g >= G || !is_pow2(R) ||
        R > 65536 || R < G)
        return PA_EINVAL;
    // Top of the pairwise tree: rank subtrees combined in rank order.
    double lvl[PA_SHARD_MAX_RANKS];
    for (int h = 0; h < G; ++h) lvl[h] = A_all[h];
    for (int len = G; len > 1; len >>= 1)
        for (int i = 0; i < len / 2; ++i) lvl[i] = lvl[2 * i] + lvl[2 * i + 1];
    unsigned long long T = 0, base[PA_SHARD_MAX_RANKS + 1];
    for (int h = 0; h < G; ++h) {
        base[h] = T;
        T += T_all[h];
    }
    base[G] = T;
    if (T == 0) return PA_EINVAL;   // every weight underflowed: impossible with E_min from the data
    const int32_t width = R / G;
    out->A = lvl[0];
    out->T = T;
    out->P_base = base[g];
    out->new_lo = shard_count(base[g], R, T, o);
    out->new_hi = shard_count(base[g + 1], R, T, o);
    for (int h = 0; h < PA_SHARD_MAX_RANKS; ++h) out->send[h] = out->recv[h] = 0;
    for (int h = 0; h < G; ++h) {
        // rows this rank sends to rank h, and rows rank h's parents send here
        const int32_t lo = h * width, hi = lo + width;
        out->send[h] = (int32_t)std::max(0, std::min(out->new_hi, hi) - std::max(out->new_lo, lo));
        const int32_t hlo = shard_count(base[h], R, T, o), hhi = shard_count(base[h + 1], R, T, o);
        out->recv[h] = (int32_t)std::max(0, std::min(hhi, g * width + width) - std::max(hlo, g * width));
    }
    return PA_OK;
}

int pa_shard_parents(const void *scratch, int32_t n, int32_t R, uint32_t o, const pa_shard_step *step,
                     int32_t *src, int32_t *counts, void *stream) {
    if (!scratch || !step || (!src && step->new_hi > step->new_lo) || n < 1 || n > PA_SHARD_MAX_SLOTS || R < 1 || R > 65536) return PA_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const ShardScratch s = scratch_view(const_cast<void *>(scratch), n);
    k_shard_parents<<<(n + 255) / 256, 256, 0, st>>>(s, n, step->P_base, step->T, R, o, step->new_lo, src, counts);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ECUDA;
}

int pa_shard_gather(const int8_t *spins, const int32_t *energies, int32_t ncols, const int32_t *src, int32_t nout,
                    int8_t *spins_out, int32_t *energies_out, void *stream) {
    if (nout == 0) return PA_OK;   // a rank whose parents fill no new slot sends nothing
    if (!spins || !src || !spins_out || ncols < 1 || nout < 0 || (energies && !energies_out)) return PA_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const uintptr_t mis = reinterpret_cast<uintptr_t>(spins) | reinterpret_cast<uintptr_t>(spins_out) | (uintptr_t)ncols;
    // Rows of less than 768 bytes: a warp each, four in a CTA, and no more CTAs than
    // fill the GPU a few times; a CTA for each costs more than its copy. us of the
    // call, 65,536 rows, a CTA each / a warp each: 1 byte 52 / 25, 90 bytes 53 / 28,
    // 600 bytes 52 / 29.
    const bool vec = (mis & 15) == 0, brief = ncols < 768;
    const int ctas = brief ? (nout - 1) / 4 + 1 : nout, most = brief ? 4096 : 65536;
    auto *kernel = brief ? (vec ? &k_shard_gather<true, 32> : &k_shard_gather<false, 32>)
                         : (vec ? &k_shard_gather<true, GATHER_THREADS> : &k_shard_gather<false, GATHER_THREADS>);
    kernel<<<ctas < most ? ctas : most, GATHER_THREADS, 0, st>>>(spins, energies, ncols, src, nout, spins_out, energies_out);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ECUDA;
}

uint32_t pa_resample_offset(uint64_t seed, int32_t k) {
    return pa::philox10(make_uint4(0u, 0u, (uint32_t)k, pa::TAG_RESAMPLE), (uint32_t)seed, (uint32_t)(seed >> 32)).x;
}

}  // extern "C"
