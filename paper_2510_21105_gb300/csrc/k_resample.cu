// k_resample.cu -- population initialisation, local fields / energies, and the
// per-temperature-step reweighting + resampling of PAMC (Sec. 3 of arXiv
// 2510.21105 names population annealing; the scheme below is the library's
// reading of it).
//
// Resampling of step k (energies E_r of the R replicas entering the step):
//   E_min = min_r E_r, d_r = E_r - E_min
//   w_r   = q^{d_r}, q = exp(-(beta_k - beta_{k-1})), as the product of the
//           host-computed squarings q^(2^b) over the set bits b of d_r in
//           ascending b (FP64, round to nearest, no fused operations)
//   A     = sum of w_r as a pairwise tree over slots padded to a power of two
//   t_r   = floor(2^32 w_r) (integer weights), T = sum t_r, P_r = sum_{s<r} t_s
//   new slots [F(P_r), F(P_r + t_r)) copy replica r, with the systematic
//   count F(P) = floor((P R 2^32 + o T) / (T 2^32)) and o the Philox word of
//   (0, 0, k, tag 1). Sum of copies is exactly R.
// The sweep kernels leave E_min of the next step; k_rs_min finds it where the
// energies came another way. k_rs_step does the rest.
#include "pa_cluster.cuh"

namespace pa {
namespace {

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void k_init_spins(GraphDev g, int8_t *spins, int32_t Rpad, uint32_t k0, uint32_t k1) {
    const int nchunk = g.np >> 2;
    const long total = (long)(Rpad >> 2) * nchunk;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (long)gridDim.x * blockDim.x) {
        const int grp = (int)(idx / nchunk), c = (int)(idx % nchunk);
        uint32_t out[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = 4 * c + j;
            if (p < g.n) {
                const uint4 u = philox10(make_uint4(g.vid[p], (uint32_t)grp, 0u, TAG_INIT), k0, k1);
                const uint32_t uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) out[q] |= ((uu[q] >> 31) ? 0x01u : 0xFFu) << (8 * j);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint32_t *>(spins + (size_t)(4 * grp + q) * g.np + 4 * c) = out[q];
    }
}

constexpr int ROW_STATIC = 256;   // bytes of static shared memory a kernel may use beside a row

// One CTA per replica: h_p = sum_j w_pj x_j and E = 1/2 sum_p x_p h_p. The
// replica's row is read once into shared memory, where the neighbours' spins are
// gathered (N = 18001, R = 1024: 89 us; gathered from global memory 162 us).
__global__ void k_fields_energy(GraphDev g, const int8_t *spins, int16_t *fields, int32_t *E) {
    extern __shared__ __align__(16) int8_t x[];   // [np]
    const int r = blockIdx.x;
    int16_t *h = fields + (size_t)r * g.np;
    const uint4 *row = reinterpret_cast<const uint4 *>(spins + (size_t)r * g.np);
    for (int i = threadIdx.x; i < (g.np >> 4); i += blockDim.x) reinterpret_cast<uint4 *>(x)[i] = row[i];
    __syncthreads();
    long long acc = 0;
    for (int p = threadIdx.x; p < g.np; p += blockDim.x) {
        int hp = 0;
        if (p < g.n) {
            const uint32_t e1 = g.rp[p + 1];
            for (uint32_t e = g.rp[p]; e < e1; ++e) {
                const int xj = x[g.col[e]];
                hp += g.wt ? (int)g.wt[e] * xj : xj;
            }
            acc += (long long)x[p] * hp;
        }
        h[p] = (int16_t)hp;
    }
    __shared__ long long red[ROW_STATIC / 8];
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        E[r] = (int32_t)(t / 2);
    }
}

__global__ void __launch_bounds__(RS_CHUNK) k_rs_min(ResampleArgs a) {
    const int r = blockIdx.x * RS_CHUNK + threadIdx.x;
    int v = r < a.R ? a.E[r] : 0x7FFFFFFF;
    v = __reduce_min_sync(0xFFFFFFFFu, v);
    if ((threadIdx.x & 31) == 0) atomicMin(&a.emin[a.k], v);
}

// Weights, sums and parents in one cluster (pa_cluster.cuh) of CTAs small enough
// to find room beside other work. Bound by latency and the FP64 rate (about two
// results per SM and cycle). With the minimum left by the sweep a step needs one
// launch instead of three (minimum, weights, parents); us per step: R = 2048
// 3.9 against 6.9 and two launch gaps, R = 32768 with long runs of one parent
// 20.2 against 21.0. Whole anneals: n = 800, R = 256 6.40 -> 5.72 ms (100 steps),
// ESS-adaptive R = 2048 56.7 -> 53.4 ms (384 steps).
constexpr int RS_THREADS = 256;

template <int K>
__global__ void __launch_bounds__(RS_THREADS) k_rs_step(ResampleArgs a) {
    namespace cg = cooperative_groups;
    __shared__ ClusterShared sh;
    __shared__ double qs[32];
    const int rank = (int)cg::this_cluster().block_rank();
    wait_previous();
    ready_for_next();
    if (rank == 0 && threadIdx.x == 0) a.stamp[a.k] = gtimer();
    if (a.active && !a.active[a.k]) return;   // the whole cluster
    const int row = a.qsel ? a.qsel[a.k] : a.k;
    if (threadIdx.x < 32) qs[threadIdx.x] = a.qpow[(size_t)row * 32 + threadIdx.x];
    const int r0 = (rank * RS_THREADS + (int)threadIdx.x) * K;
    const int32_t emin = a.emin[a.k];
    int32_t e[K];
#pragma unroll
    for (int i = 0; i < K; ++i) e[i] = r0 + i < a.R ? a.E[r0 + i] : emin;
    __syncthreads();
    cluster_table(sh, qs);
    __syncthreads();
    double w[K];
    unsigned long long t[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        w[i] = r0 + i < a.R ? cluster_weight(sh, qs, (uint32_t)(e[i] - emin)) : 0.0;
        t[i] = (unsigned long long)__dmul_rn(w[i], 4294967296.0);
    }
    unsigned long long P = cluster_sums<RS_THREADS, K>(sh, w, t);
    const unsigned long long T = sh.T, m = ~0ull / T;
    const uint32_t o = philox10(make_uint4(0u, 0u, (uint32_t)a.k, TAG_RESAMPLE), a.key0, a.key1).x;
    // Slot r fills new slots [F(P_r), F(P_r + t_r)).
    int32_t lo = systematic_count_m(P, a.R, T, m, o);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        P += t[i];
        const int32_t hi = systematic_count_m(P, a.R, T, m, o);
        const bool real = r0 + i < a.R;
        if (real && a.counts) a.counts[(size_t)a.k * a.R + r0 + i] = hi - lo;
        fill_parents(a.parent, lo, real ? hi : lo, r0 + i);
        lo = hi;
    }
    if (r0 == 0) {
        a.recA[a.k] = sh.A;
        a.recT[a.k] = T;
        a.reco[a.k] = o;
    }
    cg::this_cluster().sync();   // no CTA leaves while another may read its totals
}

// Rows <-> configurations in vertex order: one CTA per row, the row in shared
// memory, so that both global sides are read and written in order. 1024 rows of
// 18001 spins: 19 us out, 23 us in; the host loops they replace took
// 16 ms each way.
constexpr int ROWS_THREADS = 256;

template <bool BITS>
__global__ void __launch_bounds__(ROWS_THREADS) k_rows_out(int32_t n, int32_t np, int32_t nbw,
                                                           const int32_t *__restrict__ pos,
                                                           const int8_t *__restrict__ rows, int8_t *__restrict__ raw) {
    extern __shared__ __align__(16) int8_t x[];   // the row: [np] bytes or [nbw] words
    const uint32_t *xw = reinterpret_cast<const uint32_t *>(x);
    const int units = BITS ? nbw >> 2 : np >> 4;
    const uint4 *row = reinterpret_cast<const uint4 *>(rows) + (size_t)blockIdx.x * units;
    for (int i = threadIdx.x; i < units; i += ROWS_THREADS) reinterpret_cast<uint4 *>(x)[i] = row[i];
    __syncthreads();
    auto spin = [&](int p) {
        return BITS ? (uint8_t)((xw[p >> 5] >> (p & 31)) & 1u ? 0x01 : 0xFF) : (uint8_t)x[p];
    };
    int8_t *out = raw + (size_t)blockIdx.x * n;
    // Rows start at any byte: whole words at word boundaries, bytes at the ends.
    const int head = min(n, (int)((4 - (reinterpret_cast<uintptr_t>(out) & 3)) & 3)), words = (n - head) >> 2;
    for (int c = threadIdx.x; c < words; c += ROWS_THREADS) {
        uint32_t v = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) v |= (uint32_t)spin(__ldg(&pos[head + 4 * c + j])) << (8 * j);
        *reinterpret_cast<uint32_t *>(out + head + 4 * c) = v;
    }
    const int rest = n - 4 * words;   // head and tail bytes
    for (int t = threadIdx.x; t < rest; t += ROWS_THREADS) {
        const int i = t < head ? t : 4 * words + t;
        out[i] = (int8_t)spin(__ldg(&pos[i]));
    }
}

template <bool BITS>
__global__ void __launch_bounds__(ROWS_THREADS) k_rows_in(int32_t n, int32_t np, int32_t nbw,
                                                          const uint32_t *__restrict__ vid,
                                                          const int8_t *__restrict__ raw, int8_t *__restrict__ rows,
                                                          int32_t R) {
    extern __shared__ __align__(16) int8_t x[];   // [n]
    const int8_t *in = raw + (size_t)min((int)blockIdx.x, R - 1) * n;
    for (int i = threadIdx.x; i < n; i += ROWS_THREADS) x[i] = in[i];
    __syncthreads();
    if (BITS) {
        uint32_t *out = reinterpret_cast<uint32_t *>(rows) + (size_t)blockIdx.x * nbw;
        for (int p = threadIdx.x; p < 32 * nbw; p += ROWS_THREADS) {   // whole warps
            const uint32_t w = __ballot_sync(0xFFFFFFFFu, p < n && x[__ldg(&vid[min(p, n - 1)])] == 1);
            if ((p & 31) == 0) out[p >> 5] = w;
        }
        return;
    }
    uint32_t *out = reinterpret_cast<uint32_t *>(rows + (size_t)blockIdx.x * np);
    for (int c = threadIdx.x; c < (np >> 2); c += ROWS_THREADS) {
        uint32_t v = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * c + j < n) v |= (uint32_t)(uint8_t)x[__ldg(&vid[4 * c + j])] << (8 * j);
        out[c] = v;
    }
}

__global__ void k_check(const int8_t *__restrict__ raw, size_t bytes, int32_t *__restrict__ bad) {
    const size_t units = bytes >> 4, step = (size_t)gridDim.x * blockDim.x;   // raw is 16-byte aligned
    bool wrong = false;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < units; i += step) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(raw) + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // 0x01 or 0xFF in every byte: odd, and the upper seven bits equal
            const uint32_t t = (w[j] & ~0x01010101u);
            wrong |= (w[j] & 0x01010101u) != 0x01010101u || t != ((w[j] >> 7) & 0x01010101u) * 0xFEu;
        }
    }
    for (size_t i = (units << 4) + (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < bytes; i += step)
        wrong |= raw[i] != 1 && raw[i] != -1;
    if (wrong) *bad = 1;
}

__global__ void k_stamp(unsigned long long *stamp) { *stamp = gtimer(); }

}  // namespace

namespace {
// A row in dynamic shared memory: up to 65,536 bytes. Without the attribute the
// 48 KB hold the kernel's static part as well.
cudaError_t allow_row(const void *fn, int32_t np) {
    return np + ROW_STATIC <= 48 * 1024 ? cudaSuccess : cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536);
}
}  // namespace

cudaError_t launch_rows_out(const GraphDev &g, const int32_t *pos, const int8_t *rows, bool bits, int8_t *raw,
                            int32_t R, cudaStream_t st) {
    auto *fn = bits ? &k_rows_out<true> : &k_rows_out<false>;
    if (cudaError_t e = allow_row(reinterpret_cast<const void *>(fn), g.np)) return e;
    fn<<<R, ROWS_THREADS, bits ? 4 * g.nbw : g.np, st>>>(g.n, g.np, g.nbw, pos, rows, raw);
    return cudaGetLastError();
}

cudaError_t launch_rows_in(const GraphDev &g, const int8_t *raw, int8_t *rows, bool bits, int32_t R, int32_t Rpad,
                           cudaStream_t st) {
    auto *fn = bits ? &k_rows_in<true> : &k_rows_in<false>;
    if (cudaError_t e = allow_row(reinterpret_cast<const void *>(fn), g.np)) return e;
    fn<<<Rpad, ROWS_THREADS, g.np, st>>>(g.n, g.np, g.nbw, g.vid, raw, rows, R);
    return cudaGetLastError();
}

cudaError_t launch_check(const int8_t *raw, size_t bytes, int32_t *bad, cudaStream_t st) {
    const size_t blocks = (bytes / 16 + 255) / 256 + 1;
    k_check<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(raw, bytes, bad);
    return cudaGetLastError();
}

cudaError_t launch_init(const GraphDev &g, int8_t *spins, int32_t Rpad, uint32_t key0,
                        uint32_t key1, cudaStream_t st) {
    const long total = (long)(Rpad >> 2) * (g.np >> 2);
    long blocks = (total + 255) / 256;
    if (blocks > 65535L * 16) blocks = 65535L * 16;
    k_init_spins<<<(unsigned)blocks, 256, 0, st>>>(g, spins, Rpad, key0, key1);
    return cudaGetLastError();
}

cudaError_t launch_fields(const GraphDev &g, const int8_t *spins, int16_t *fields, int32_t *E,
                          int32_t Rpad, cudaStream_t st) {
    if (cudaError_t e = allow_row(reinterpret_cast<const void *>(&k_fields_energy), g.np)) return e;
    k_fields_energy<<<Rpad, 256, g.np, st>>>(g, spins, fields, E);
    return cudaGetLastError();
}

cudaError_t launch_rs_min(const ResampleArgs &a, cudaStream_t st) {
    k_rs_min<<<a.nch, RS_CHUNK, 0, st>>>(a);
    return cudaGetLastError();
}

int rs_step_ctas(int32_t R) { return cluster_shape(R, RS_THREADS).ctas; }

cudaError_t launch_rs_step(const ResampleArgs &a, cudaStream_t st, bool early) {
    const ClusterShape shape = cluster_shape(a.R, RS_THREADS);
    auto *kernel = shape.k == 1   ? &k_rs_step<1>
                   : shape.k == 2 ? &k_rs_step<2>
                   : shape.k == 4 ? &k_rs_step<4>
                   : shape.k == 8 ? &k_rs_step<8>
                   : shape.k == 16 ? &k_rs_step<16>
                                   : &k_rs_step<32>;
    return launch_cluster(kernel, shape, RS_THREADS, st, early, a);
}

cudaError_t launch_stamp(unsigned long long *stamp, cudaStream_t st) {
    k_stamp<<<1, 1, 0, st>>>(stamp);
    return cudaGetLastError();
}

}  // namespace pa
