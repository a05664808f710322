// k_sweep.cu -- colour-ordered Metropolis sweeps of PAMC (Sec. 3 of arXiv
// 2510.21105; the paper names the method but not the sweep, so the rule is
// the library's reading: standard Metropolis on the Ising form of Eq. 1).
//
// One CTA holds a block of B = 4G replicas in shared memory while it runs all
// S sweeps of one temperature step on them:
//   S_sm[p][g]  uint32: int8 spins of replicas 4g..4g+3 at position p
//   H_sm[p][g]  local fields of the same replicas, biased to unsigned:
//               16-bit: two uint32 words (replicas 0,1 | 2,3), h + 32768
//                8-bit: one uint32 word, h + 128 (max degree <= 127)
// A colour class is an independent set, so all of its positions update in
// parallel (one thread per (position, group)); the accepted flips push
// +-2 into the neighbours' fields with one packed 32-bit shared atomic per
// neighbour and group (the bias keeps every lane non-negative, so the packed
// add never carries across lanes). The top bytes of the group's four
// uniforms are the bytes of one word of Philox(counter = (vertex, slot/16,
// step, sweep)): byte q of word (slot/4) % 4 belongs to slot 4*(slot/4) + q;
// the low 24 bits are drawn only when a top byte ties with the threshold's.
// The block is loaded from the parents chosen by the resampling (the copy of
// the resampling is fused into this load) and written to the next buffers.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <unordered_map>

#include "pa_internal.cuh"

namespace pa {
namespace {

// Allows a kernel `smem` bytes of dynamic shared memory. The attribute belongs
// to the kernel function, not to a context: only ever raise it, so that
// contexts configured earlier keep launching.
cudaError_t raise_smem(void *fn, size_t smem) {
    static std::mutex mu;
    static std::unordered_map<void *, size_t> raised;
    std::lock_guard<std::mutex> lock(mu);
    size_t &cur = raised[fn];
    if (smem > cur) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        cur = smem;
    }
    return cudaSuccess;
}

__device__ __forceinline__ void transpose4x4_bytes(uint32_t w0, uint32_t w1, uint32_t w2,
                                                   uint32_t w3, uint32_t o[4]) {
    const uint32_t a_lo = __byte_perm(w0, w1, 0x5140);
    const uint32_t a_hi = __byte_perm(w0, w1, 0x7362);
    const uint32_t b_lo = __byte_perm(w2, w3, 0x5140);
    const uint32_t b_hi = __byte_perm(w2, w3, 0x7362);
    o[0] = __byte_perm(a_lo, b_lo, 0x5410);
    o[1] = __byte_perm(a_lo, b_lo, 0x7632);
    o[2] = __byte_perm(a_hi, b_hi, 0x5410);
    o[3] = __byte_perm(a_hi, b_hi, 0x7632);
}

// Byte permute with sign replication: each selector nibble with bit 3 set
// fills its result byte with the top bit of the selected byte.
__device__ __forceinline__ uint32_t prmt_sign(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// Entry of m in the packed kernel's decision table: E(m) in both 16-bit
// halves. Two replicas are decided by one 32-bit multiply-add in 16-bit lanes,
// lane = 128 top + E(m) with the top byte of the uniform (t8 = T[m] >> 24):
//   E = 0x8000 - 128 t8:  lane < 0x8000 iff top < t8 (accept),
//                         lane = 0x8000 iff top = t8 (tie),
//   + 64 when T[m] has no low bits (a tie rejects), 0x8040 when T[m] = 0,
//   1 for m <= 0 (always accepted).
// Every lane stays in [1, 0xFFC0], so lanes never carry into each other; bit
// 15 of a lane is "reject or tie" and bit 15 of lane - 1 is "reject".
__device__ __forceinline__ uint32_t pk_entry(int m, const uint32_t *tab, int mmax) {
    uint32_t e = 1u;   // m <= 0: always accepted
    if (m > 0) {
        const uint32_t T = m <= mmax ? tab[m] : 0u;
        e = T == 0u ? 0x8040u : 0x8000u - 128u * (T >> 24) + ((T & 0xFFFFFFu) == 0u ? 64u : 0u);
    }
    return e * 0x00010001u;
}

// ---------------------------------------------------------------------------
// Field updates of accepted items, shared by the layouts that keep fields: an
// accepted item (a position of one group of four replicas) adds its change to
// every neighbour's field. The items of a round go to a queue of the block, and
// after a barrier all threads of the block walk their rows, 2^lt lanes per row
// with 2^lt the largest power of two that gives every queued item its lanes (so
// few items on long rows still use the whole block). Bound: latency. n = 500,
// mean degree 250, R = 1024, us per step of 4 sweeps: 765 with one thread per
// row, 375 with the queue (512 threads).
// Counters of three rounds and entries of two, so that one barrier per round
// is enough: the counter a round uses was cleared after the barrier two rounds
// before, and its entries were read before the barrier one round before.
struct SweepQueue {
    uint4 *ent;        // [2][threads]
    int32_t *count;    // [3], zero at the start
    int round;

    __device__ __forceinline__ void push(bool have, const uint4 &e, int lane) {
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, have);
        if (!bal) return;
        int base = 0;
        if (lane == 0) base = atomicAdd(&count[round % 3], __popc(bal));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (have) ent[(size_t)(round & 1) * blockDim.x + base + __popc(bal & ((1u << lane) - 1u))] = e;
    }
    // Closes the round for the whole block; walk(entry, lane of the row, lanes per row).
    template <class F>
    __device__ __forceinline__ void drain(F walk) {
        __syncthreads();
        const int total = count[round % 3];
        if (threadIdx.x == 0) count[(round + 2) % 3] = 0;
        if (total) {
            const int lt = min(31 - __clz((int)blockDim.x / total), 7);
            for (int t = threadIdx.x; t < (total << lt); t += blockDim.x)
                walk(ent[(size_t)(round & 1) * blockDim.x + (t >> lt)], t & ((1 << lt) - 1), 1 << lt);
        }
        ++round;
    }
};
__host__ __device__ inline size_t sweep_queue_bytes(int threads) { return (size_t)threads * 32 + 16; }

// Top bytes of the four uniforms of group c1 at vertex vid: word c1 & 3 of the
// call of slots 16 (c1 >> 2) ..
__device__ __forceinline__ uint32_t group_uniforms(const SweepArgs &a, uint32_t vid, uint32_t c1, uint32_t c3) {
    return word_of(philox10(make_uint4(vid, c1 >> 2, (uint32_t)a.k, c3), a.key0, a.key1), c1 & 3u);
}

// Decides the four replicas of an item and applies its own part; returns
// whether any flipped, with the packed field changes D0, D1 of its neighbours.
template <int G, int FB>
__device__ __forceinline__ bool sweep_item(uint32_t *__restrict__ Ssm, const uint32_t *__restrict__ Hsm,
                                           const uint32_t *__restrict__ Tt, const SweepArgs &a, int p, int g,
                                           uint32_t vid, uint32_t uw, uint32_t c1, uint32_t c3, uint32_t vmask,
                                           int dE[4], uint32_t &nacc, uint32_t &D0, uint32_t &D1) {
    const int widx = p * G + g;
    const uint32_t sw = Ssm[widx];
    uint32_t hw0, hw1 = 0;
    if (FB == 16) {
        const uint2 hv = reinterpret_cast<const uint2 *>(Hsm)[widx];
        hw0 = hv.x;
        hw1 = hv.y;
    } else {
        hw0 = Hsm[widx];
    }
    int m[4], x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        x[q] = (int)(int8_t)(sw >> (8 * q));
        int h;
        if (FB == 16)
            h = (int)(((q < 2 ? hw0 : hw1) >> (16 * (q & 1))) & 0xFFFFu) - 32768;
        else
            h = (int)((hw0 >> (8 * q)) & 0xFFu) - 128;
        m[q] = x[q] > 0 ? -h : h;   // dE = -2 x h = 2m
    }
    uint32_t acc = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool ok = (m[q] <= 0) || accept_by_top_byte((uw >> (8 * q)) & 0xFFu, Tt[min(m[q], a.g.mmax)], vid,
                                                          4u * c1 + q, (uint32_t)a.k, c3, a.key0, a.key1);
        acc |= (uint32_t)ok << q;
    }
    if (!acc) return false;
    uint32_t flip = 0;
    int d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool f = (acc >> q) & 1u;
        flip |= f ? (0xFEu << (8 * q)) : 0u;
        dE[q] += f ? 2 * m[q] : 0;
        d[q] = f ? -2 * x[q] : 0;
    }
    Ssm[widx] = sw ^ flip;
    nacc += __popc(acc & vmask);
    if (FB == 16) {
        D0 = (uint32_t)(d[0] + d[1] * 65536);
        D1 = (uint32_t)(d[2] + d[3] * 65536);
    } else {
        D0 = (uint32_t)(d[0] + d[1] * 256 + d[2] * 65536 + d[3] * 16777216);
    }
    return true;
}

template <int G, int FB, bool WEIGHTED, bool QUEUED>
__global__ void __launch_bounds__(1024) k_sweep(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    wait_previous();
    // A step after the adaptive schedule has ended only carries the population over.
    const bool act = !a.active || a.active[a.k];
    const int nsweeps = act ? a.S : 0;
    const int np = a.g.np;
    constexpr int HW = (FB == 16) ? 2 : 1;
    uint32_t *Ssm = reinterpret_cast<uint32_t *>(smem);
    uint32_t *Hsm = Ssm + (size_t)np * G;
    uint32_t *Tt = Hsm + (size_t)np * G * HW;
    const int tsz = (a.g.mmax + 1 + 3) & ~3;
    int32_t *cls = reinterpret_cast<int32_t *>(Tt + tsz);
    const int csz = (a.g.ncol + 1 + 3) & ~3;
    int32_t *Eacc = cls + csz;          // [4G]
    int32_t *PS = Eacc + 4 * G;         // [4G] parent slot of each replica
    int32_t *misc = PS + 4 * G;         // best E, step, sweep, slot, copy-from (q+1), changed
    SweepQueue Q{reinterpret_cast<uint4 *>(misc + 8), nullptr, 0};
    Q.count = reinterpret_cast<int32_t *>(Q.ent + 2 * blockDim.x);

    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
    const uint32_t *tab = a.tables + (size_t)a.tidx[a.k] * (a.g.mmax + 1);
    for (int i = tid; i <= a.g.mmax; i += NT) Tt[i] = tab[i];
    for (int i = tid; i <= a.g.ncol; i += NT) cls[i] = a.g.cls[i];
    if (QUEUED && tid < 3) Q.count[tid] = 0;
    const int gthr = tid % G;   // NT is a multiple of 32, so each thread keeps one group

    for (int blk = blockIdx.x; blk < a.nblk; blk += gridDim.x) {
        const int slot0 = blk * 4 * G;
        if (tid < 4 * G) PS[tid] = act ? a.parent[slot0 + tid] : slot0 + tid;
        if (tid == 0) {
            const int4 br = a.best_rec[blk];
            misc[0] = br.x; misc[1] = br.y; misc[2] = br.z; misc[3] = br.w;
            misc[4] = 0; misc[5] = 0;
        }
        __syncthreads();
        if (tid < 4 * G) Eacc[tid] = a.E_in[PS[tid]];
        // Load the block, transposing replica rows into position-major words.
        for (int idx = tid; idx < (np >> 2) * G; idx += NT) {
            const int g = idx % G, c = idx / G;
            uint32_t w[4];
            uint2 f[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)PS[4 * g + q] * np + 4 * c;
                w[q] = __ldcg(reinterpret_cast<const uint32_t *>(a.spins_in + row));
                f[q] = __ldcg(reinterpret_cast<const uint2 *>(a.fields_in + row));
            }
            uint32_t o[4];
            transpose4x4_bytes(w[0], w[1], w[2], w[3], o);
#pragma unroll
            for (int j = 0; j < 4; ++j) Ssm[(4 * c + j) * G + g] = o[j];
            if (FB == 16) {
                uint2 *H2 = reinterpret_cast<uint2 *>(Hsm);
                H2[(4 * c + 0) * G + g] = make_uint2(__byte_perm(f[0].x, f[1].x, 0x5410) ^ 0x80008000u,
                                                     __byte_perm(f[2].x, f[3].x, 0x5410) ^ 0x80008000u);
                H2[(4 * c + 1) * G + g] = make_uint2(__byte_perm(f[0].x, f[1].x, 0x7632) ^ 0x80008000u,
                                                     __byte_perm(f[2].x, f[3].x, 0x7632) ^ 0x80008000u);
                H2[(4 * c + 2) * G + g] = make_uint2(__byte_perm(f[0].y, f[1].y, 0x5410) ^ 0x80008000u,
                                                     __byte_perm(f[2].y, f[3].y, 0x5410) ^ 0x80008000u);
                H2[(4 * c + 3) * G + g] = make_uint2(__byte_perm(f[0].y, f[1].y, 0x7632) ^ 0x80008000u,
                                                     __byte_perm(f[2].y, f[3].y, 0x7632) ^ 0x80008000u);
            } else {
                const uint32_t px01 = __byte_perm(f[0].x, f[1].x, 0x6420);
                const uint32_t px23 = __byte_perm(f[2].x, f[3].x, 0x6420);
                const uint32_t py01 = __byte_perm(f[0].y, f[1].y, 0x6420);
                const uint32_t py23 = __byte_perm(f[2].y, f[3].y, 0x6420);
                Hsm[(4 * c + 0) * G + g] = __byte_perm(px01, px23, 0x6420) ^ 0x80808080u;
                Hsm[(4 * c + 1) * G + g] = __byte_perm(px01, px23, 0x7531) ^ 0x80808080u;
                Hsm[(4 * c + 2) * G + g] = __byte_perm(py01, py23, 0x6420) ^ 0x80808080u;
                Hsm[(4 * c + 3) * G + g] = __byte_perm(py01, py23, 0x7531) ^ 0x80808080u;
            }
        }
        __syncthreads();

        uint32_t vmask = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) vmask |= (slot0 + 4 * gthr + q < a.R) ? (1u << q) : 0u;
        const uint32_t c1 = (uint32_t)(blk * G + gthr);
        uint32_t nacc = 0;
        // With the queue the uniforms of a thread's first item of the next class are
        // drawn while the present class is finished (they depend on no spin).
        uint32_t vid = 0, uw = 0;
        auto draw = [&](int p, uint32_t c3) {
            vid = __ldg(&a.g.vid[p]);
            uw = group_uniforms(a, vid, c1, c3);
        };
        if (QUEUED && nsweeps && tid < cls[1] * G) draw(tid / G, TAG_SWEEP);
        for (int s = 0; s < nsweeps; ++s) {
            const uint32_t c3 = TAG_SWEEP | (uint32_t)s;
            int dE[4] = {0, 0, 0, 0};
            for (int c = 0; c < a.g.ncol; ++c) {
                const int p0 = cls[c], cnt = (cls[c + 1] - p0) * G;
                auto walk = [&](const uint4 &e, int sub, int lanes) {
                    const uint32_t pe = e.x & 0xFFFFu, ge = e.x >> 16;
                    const uint32_t e1 = __ldg(&a.g.rp[pe + 1]);
                    for (uint32_t i = __ldg(&a.g.rp[pe]) + sub; i < e1; i += lanes) {
                        const int j = __ldg(&a.g.col[i]);
                        uint32_t s0 = e.y, s1 = e.z;
                        if (WEIGHTED && __ldg(&a.g.wt[i]) < 0) {
                            s0 = 0u - s0;
                            s1 = 0u - s1;
                        }
                        if (FB == 16) {
                            atomicAdd(&Hsm[2 * (j * G + ge)], s0);
                            atomicAdd(&Hsm[2 * (j * G + ge) + 1], s1);
                        } else {
                            atomicAdd(&Hsm[j * G + ge], s0);
                        }
                    }
                };
                if (QUEUED) {
                    for (int base = 0; base < cnt; base += NT) {   // uniform over the block
                        const int idx = base + tid;
                        bool have = false;
                        uint4 ent = make_uint4(0u, 0u, 0u, 0u);
                        if (idx < cnt) {
                            const int p = p0 + idx / G;
                            if (base) draw(p, c3);
                            have = sweep_item<G, FB>(Ssm, Hsm, Tt, a, p, gthr, vid, uw, c1, c3, vmask, dE, nacc, ent.y, ent.z);
                            ent.x = (uint32_t)p | (uint32_t)gthr << 16;
                        }
                        Q.push(have, ent, lane);
                        if (base + NT >= cnt) {
                            const int cn = c + 1 < a.g.ncol ? c + 1 : 0;
                            if (tid < (cls[cn + 1] - cls[cn]) * G)
                                draw(cls[cn] + tid / G, TAG_SWEEP | (uint32_t)(cn ? s : s + 1));
                        }
                        Q.drain(walk);
                    }
                } else {
                    for (int idx = tid; idx < cnt; idx += NT) {
                        const int p = p0 + idx / G;
                        uint4 ent = make_uint4((uint32_t)p | (uint32_t)gthr << 16, 0u, 0u, 0u);
                        draw(p, c3);
                        if (sweep_item<G, FB>(Ssm, Hsm, Tt, a, p, gthr, vid, uw, c1, c3, vmask, dE, nacc, ent.y, ent.z)) walk(ent, 0, 1);
                    }
                }
                __syncthreads();
            }
            // Energies after sweep s: reduce the per-thread changes of each replica.
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                int v = dE[q];
#pragma unroll
                for (int off = G; off < 32; off <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
                if (lane < G && v != 0) atomicAdd(&Eacc[4 * lane + q], v);
            }
            __syncthreads();
            if (tid == 0) {
                int bq = -1, bE = 0x7FFFFFFF;
                for (int q = 0; q < 4 * G; ++q)
                    if (slot0 + q < a.R && Eacc[q] < bE) { bE = Eacc[q]; bq = q; }
                misc[4] = 0;
                if (bq >= 0) {
                    atomicMin(&a.sweep_emin[(size_t)a.k * a.S + s], bE);
                    if (bE < misc[0]) {
                        misc[0] = bE; misc[1] = a.k; misc[2] = s; misc[3] = slot0 + bq;
                        misc[4] = bq + 1; misc[5] = 1;
                    }
                }
            }
            __syncthreads();
            if (misc[4]) {   // block-uniform: copy the new best configuration
                const int q = misc[4] - 1, g = q >> 2, sh = 8 * (q & 3);
                uint32_t *dst = reinterpret_cast<uint32_t *>(a.best_cfg + (size_t)blk * np);
                for (int c = tid; c < (np >> 2); c += NT) {
                    uint32_t v = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) v |= ((Ssm[(4 * c + j) * G + g] >> sh) & 0xFFu) << (8 * j);
                    dst[c] = v;
                }
                __syncthreads();
            }
        }
        // Store the block to the next population buffers.
        for (int idx = tid; idx < (np >> 2) * G; idx += NT) {
            const int g = idx % G, c = idx / G;
            uint32_t o[4];
            transpose4x4_bytes(Ssm[(4 * c + 0) * G + g], Ssm[(4 * c + 1) * G + g],
                               Ssm[(4 * c + 2) * G + g], Ssm[(4 * c + 3) * G + g], o);
            uint2 f[4];
            if (FB == 16) {
                const uint2 *H2 = reinterpret_cast<const uint2 *>(Hsm);
                const uint2 h0 = H2[(4 * c + 0) * G + g], h1 = H2[(4 * c + 1) * G + g];
                const uint2 h2 = H2[(4 * c + 2) * G + g], h3 = H2[(4 * c + 3) * G + g];
                const uint32_t L0 = h0.x ^ 0x80008000u, L1 = h1.x ^ 0x80008000u;
                const uint32_t L2 = h2.x ^ 0x80008000u, L3 = h3.x ^ 0x80008000u;
                const uint32_t U0 = h0.y ^ 0x80008000u, U1 = h1.y ^ 0x80008000u;
                const uint32_t U2 = h2.y ^ 0x80008000u, U3 = h3.y ^ 0x80008000u;
                f[0] = make_uint2(__byte_perm(L0, L1, 0x5410), __byte_perm(L2, L3, 0x5410));
                f[1] = make_uint2(__byte_perm(L0, L1, 0x7632), __byte_perm(L2, L3, 0x7632));
                f[2] = make_uint2(__byte_perm(U0, U1, 0x5410), __byte_perm(U2, U3, 0x5410));
                f[3] = make_uint2(__byte_perm(U0, U1, 0x7632), __byte_perm(U2, U3, 0x7632));
            } else {
                uint32_t P[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) P[j] = Hsm[(4 * c + j) * G + g] ^ 0x80808080u;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    int h[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) h[j] = (int)(int8_t)(P[j] >> (8 * q));
                    f[q] = make_uint2(((uint32_t)h[0] & 0xFFFFu) | ((uint32_t)h[1] << 16),
                                      ((uint32_t)h[2] & 0xFFFFu) | ((uint32_t)h[3] << 16));
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)(slot0 + 4 * g + q) * np + 4 * c;
                *reinterpret_cast<uint32_t *>(a.spins_out + row) = o[q];
                *reinterpret_cast<uint2 *>(a.fields_out + row) = f[q];
            }
        }
        if (tid < 4 * G) {
            a.E_out[slot0 + tid] = Eacc[tid];
            if (a.emin_next && slot0 + tid < a.R) atomicMin(a.emin_next, Eacc[tid]);
        }
        if (tid == 0 && misc[5]) a.best_rec[blk] = make_int4(misc[0], misc[1], misc[2], misc[3]);
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, nacc);
        if (act && lane == 0 && wsum) atomicAdd(&a.accepts[a.k], (unsigned long long)wsum);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Packed variant: one byte per (position, replica) holds the spin in bit 0 and
// the biased local field in bits 1..7. Because h_p = sum of deg(p) terms +-1,
// h_p + 128 has the parity of deg(p), so its low bit is redundant and is
// replaced by the spin bit:  byte = ((h + 128) & ~1) | s,  s = (x == +1).
// Needs max degree <= 127. Flipping a spin toggles bit 0; a neighbour flip
// adds +-2 to the byte (bit 0 untouched), four replicas per packed atomic.
// With m = -x h and mb = m + 128 per byte:
//   hb = (b & 0xFE..) | par,  M = s * 0xFF,  mb = (hb ^ M) + s
// (for s = 1 this is the bytewise negation 256 - hb; hb >= 1 so no carry).
// A move is accepted iff mb <= 128 (m <= 0) or u < T[m].
struct PkItem {
    uint32_t b, mb, smask, acc;
};

// Ties of the top byte in a packed item (rare): the low 24 bits of the
// uniform decide.
__device__ __forceinline__ uint32_t pk_settle_ties(const SweepArgs &a, uint32_t acc, uint32_t tie, uint32_t mb,
                                                uint32_t vid, uint32_t c1, uint32_t c3) {
    const uint32_t *tab = a.tables + (size_t)a.tidx[a.k] * (a.g.mmax + 1);
    do {
        const int q = __ffs(tie) - 1;
        tie &= tie - 1u;
        const uint32_t T = __ldg(&tab[(int)((mb >> (8 * q)) & 0xFFu) - 128]);
        if (sweep_tail_bits(vid, 4u * c1 + q, (uint32_t)a.k, c3, a.key0, a.key1) < (T & 0xFFFFFFu)) acc |= 1u << q;
    } while (tie);
    return acc;
}

__device__ __forceinline__ void pk_decide(const uint32_t *__restrict__ Bsm, const uint32_t *__restrict__ T256,
                                          const uint32_t *__restrict__ Psm, const SweepArgs &a, int p,
                                          uint32_t vid, uint32_t uw, uint32_t c1, uint32_t c3, PkItem &it) {
    const uint32_t b = Bsm[p];
    const uint32_t par = (Psm[p >> 5] >> (p & 31)) & 1u;
    const uint32_t smask = b & 0x01010101u;
    const uint32_t hb = (b & 0xFEFEFEFEu) | (par * 0x01010101u);
    const uint32_t mb = (hb ^ (smask * 0xFFu)) + smask;
    // The four decisions in 16-bit lanes (pk_entry).
    const uint32_t e0 = T256[mb & 0xFFu], e1 = T256[(mb >> 8) & 0xFFu];
    const uint32_t e2 = T256[(mb >> 16) & 0xFFu], e3 = T256[mb >> 24];
    const uint32_t slo = __byte_perm(uw, 0u, 0x4140u) * 128u + __byte_perm(e0, e1, 0x5410u);
    const uint32_t shi = __byte_perm(uw, 0u, 0x4342u) * 128u + __byte_perm(e2, e3, 0x5410u);
    const uint32_t RT = prmt_sign(slo, shi, 0xFDB9u);                               // reject or tie
    const uint32_t RS = prmt_sign(slo - 0x00010001u, shi - 0x00010001u, 0xFDB9u);   // reject
    uint32_t acc = (((~RT >> 7) & 0x01010101u) * 0x01020408u) >> 24;       // bit q: replica q accepted
    uint32_t tie = ((((RT & ~RS) >> 7) & 0x01010101u) * 0x01020408u) >> 24;
    if (tie) acc = pk_settle_ties(a, acc, tie, mb, vid, c1, c3);   // rare
    it.b = b;
    it.mb = mb;
    it.smask = smask;
    it.acc = acc;
}

// Own word, energy and acceptance bookkeeping of an item; returns the packed
// field change D of its neighbours (0 if nothing was accepted).
__device__ __forceinline__ uint32_t pk_commit_self(uint32_t *__restrict__ Bsm, int p, const PkItem &it,
                                                   uint32_t vmask, int dE[4], uint32_t &nacc) {
    if (!it.acc) return 0u;
    const uint32_t a01 = (it.acc * 0x00204081u) & 0x01010101u;   // bit q -> bit 8q
    Bsm[p] = it.b ^ a01;
    nacc += __popc(it.acc & vmask);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        dE[q] += ((it.acc >> q) & 1u) ? 2 * ((int)((it.mb >> (8 * q)) & 0xFFu) - 128) : 0;
    // field change of the neighbours: -2 x_q per accepted replica q
    return ((a01 & ~it.smask) << 1) - ((a01 & it.smask) << 1);
}

// Per-warp ring of accepted items (position, D) awaiting their neighbour
// updates; a full round gives every lane one item, so the row walks run with
// all lanes busy instead of with the few lanes that happened to accept.
constexpr int PK_QCAP = 64;   // backlog < 32 + 32 after each drain

__device__ __forceinline__ void pk_enqueue(uint2 *__restrict__ Q, uint32_t &qtail, int p, uint32_t D,
                                           int lane) {
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, D != 0u);
    if (D) {
        const uint32_t rank = __popc(bal & ((1u << lane) - 1u));
        Q[(qtail + rank) & (PK_QCAP - 1)] = make_uint2((uint32_t)p, D);
    }
    qtail += __popc(bal);
}

// Adds D to the fields of the four neighbours of one row unit.
template <bool WEIGHTED>
__device__ __forceinline__ void pk_add4(uint32_t *__restrict__ Bsm, const uint2 &v, uint32_t D) {
    const uint32_t idx[4] = {v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        if (WEIGHTED)
            atomicAdd(&Bsm[idx[t] & 0x7FFFu], (idx[t] & 0x8000u) ? 0u - D : D);
        else
            atomicAdd(&Bsm[idx[t]], D);
    }
}

template <bool WEIGHTED>
__device__ __forceinline__ void pk_round(uint32_t *__restrict__ Bsm, const uint2 *__restrict__ Q,
                                         uint32_t qhead, uint32_t count, const SweepArgs &a, int lane) {
    __syncwarp();
    if ((uint32_t)lane < count) {
        const uint2 ent = Q[(qhead + lane) & (PK_QCAP - 1)];
        const uint32_t D = ent.y;
        const uint32_t e0 = __ldg(&a.g.prp[ent.x]), e1 = __ldg(&a.g.prp[ent.x + 1]);
        for (uint32_t e = e0; e < e1; ++e) pk_add4<WEIGHTED>(Bsm, __ldg(&a.g.pcol[e]), D);
    }
    __syncwarp();
}

template <bool WEIGHTED, int NTB, int MINB>
__global__ void __launch_bounds__(NTB, MINB) k_sweep_packed(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    wait_previous();
    const bool act = !a.active || a.active[a.k];
    const int nsweeps = act ? a.S : 0;
    const int np = a.g.np;
    uint32_t *Bsm = reinterpret_cast<uint32_t *>(smem);          // [np + 32], last 32 are scratch
    uint32_t *T256 = Bsm + np + 32;                                 // [256] decision entries by m + 128
    int32_t *cls = reinterpret_cast<int32_t *>(T256 + 256);
    const int csz = (a.g.ncol + 1 + 3) & ~3;
    int32_t *Eacc = cls + csz;      // [4]
    int32_t *PS = Eacc + 4;         // [4]
    int32_t *misc = PS + 4;         // best E, step, sweep, slot, copy-from (q+1), changed
    uint32_t *Psm = reinterpret_cast<uint32_t *>(misc + 8);         // degree parity bits
    const int npw = (np + 31) >> 5;
    uint2 *Qall = reinterpret_cast<uint2 *>(Psm + ((npw + 3) & ~3));  // [NT/32][PK_QCAP]

    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
    uint2 *Q = Qall + (size_t)(tid >> 5) * PK_QCAP;
    const uint32_t *tab = a.tables + (size_t)a.tidx[a.k] * (a.g.mmax + 1);
    for (int i = tid; i < 256; i += NT) T256[i] = pk_entry(i - 128, tab, a.g.mmax);   // by m + 128
    for (int i = tid; i <= a.g.ncol; i += NT) cls[i] = a.g.cls[i];
    for (int i = tid; i < npw; i += NT) Psm[i] = a.g.parity[i];

    for (int blk = blockIdx.x; blk < a.nblk; blk += gridDim.x) {
        const int slot0 = blk * 4;
        if (tid < 4) PS[tid] = act ? a.parent[slot0 + tid] : slot0 + tid;
        if (tid == 0) {
            const int4 br = a.best_rec[blk];
            misc[0] = br.x; misc[1] = br.y; misc[2] = br.z; misc[3] = br.w;
            misc[4] = 0; misc[5] = 0;
        }
        __syncthreads();
        if (tid < 4) Eacc[tid] = a.E_in[PS[tid]];
        // Load: int8 spins + int16 fields of four replica rows -> packed bytes.
        for (int c = tid; c < (np >> 2); c += NT) {
            uint32_t w[4];
            uint2 f[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)PS[q] * np + 4 * c;
                w[q] = __ldcg(reinterpret_cast<const uint32_t *>(a.spins_in + row));
                f[q] = __ldcg(reinterpret_cast<const uint2 *>(a.fields_in + row));
            }
            uint32_t o[4];
            transpose4x4_bytes(w[0], w[1], w[2], w[3], o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t word = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t hv = j < 2 ? f[q].x : f[q].y;
                    const uint32_t h128 = ((hv >> (16 * (j & 1))) + 128u) & 0xFFu;   // h + 128
                    const uint32_t sbit = ((o[j] >> (8 * q)) & 0xFFu) == 1u ? 1u : 0u;
                    word |= ((h128 & 0xFEu) | sbit) << (8 * q);
                }
                Bsm[4 * c + j] = word;
            }
        }
        __syncthreads();

        uint32_t vmask = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) vmask |= (slot0 + q < a.R) ? (1u << q) : 0u;
        const uint32_t c1 = (uint32_t)blk;
        uint32_t nacc = 0;
        for (int s = 0; s < nsweeps; ++s) {
            const uint32_t c3 = TAG_SWEEP | (uint32_t)s;
            int dE[4] = {0, 0, 0, 0};
            for (int c = 0; c < a.g.ncol; ++c) {
                const int p0 = cls[c], p1 = cls[c + 1];
                uint32_t qhead = 0, qtail = 0;   // warp-uniform
                for (int base = p0; base < p1; base += 2 * NT) {   // trip count uniform in the CTA
                    const int pA = base + tid, pB = pA + NT;
                    PkItem A, Bi;
                    A.acc = 0;
                    Bi.acc = 0;
                    if (pA < p1) {
                        const uint32_t vA = __ldg(&a.g.vid[pA]);
                        pk_decide(Bsm, T256, Psm, a, pA, vA, group_uniforms(a, vA, c1, c3), c1, c3, A);
                    }
                    if (pB < p1) {
                        const uint32_t vB = __ldg(&a.g.vid[pB]);
                        pk_decide(Bsm, T256, Psm, a, pB, vB, group_uniforms(a, vB, c1, c3), c1, c3, Bi);
                    }
                    const uint32_t DA = pk_commit_self(Bsm, pA, A, vmask, dE, nacc);
                    const uint32_t DB = pk_commit_self(Bsm, pB, Bi, vmask, dE, nacc);
                    pk_enqueue(Q, qtail, pA, DA, lane);
                    if (qtail - qhead >= 32u) {
                        pk_round<WEIGHTED>(Bsm, Q, qhead, 32u, a, lane);
                        qhead += 32u;
                    }
                    pk_enqueue(Q, qtail, pB, DB, lane);
                    if (qtail - qhead >= 32u) {
                        pk_round<WEIGHTED>(Bsm, Q, qhead, 32u, a, lane);
                        qhead += 32u;
                    }
                }
                if (qtail != qhead) pk_round<WEIGHTED>(Bsm, Q, qhead, qtail - qhead, a, lane);
                __syncthreads();
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int v = __reduce_add_sync(0xFFFFFFFFu, dE[q]);
                if (lane == 0 && v != 0) atomicAdd(&Eacc[q], v);
            }
            __syncthreads();
            if (tid == 0) {
                int bq = -1, bE = 0x7FFFFFFF;
                for (int q = 0; q < 4; ++q)
                    if (slot0 + q < a.R && Eacc[q] < bE) { bE = Eacc[q]; bq = q; }
                misc[4] = 0;
                if (bq >= 0) {
                    atomicMin(&a.sweep_emin[(size_t)a.k * a.S + s], bE);
                    if (bE < misc[0]) {
                        misc[0] = bE; misc[1] = a.k; misc[2] = s; misc[3] = slot0 + bq;
                        misc[4] = bq + 1; misc[5] = 1;
                    }
                }
            }
            __syncthreads();
            if (misc[4]) {
                const int sh = 8 * (misc[4] - 1);
                uint32_t *dst = reinterpret_cast<uint32_t *>(a.best_cfg + (size_t)blk * np);
                for (int c = tid; c < (np >> 2); c += NT) {
                    uint32_t v = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t sb = (Bsm[4 * c + j] >> sh) & 1u;
                        const bool real = 4 * c + j < a.g.n;
                        v |= (real ? (sb ? 0x01u : 0xFFu) : 0u) << (8 * j);
                    }
                    dst[c] = v;
                }
                __syncthreads();
            }
        }
        // Store: packed bytes -> int8 spins + int16 fields of the next buffers.
        for (int c = tid; c < (np >> 2); c += NT) {
            uint32_t sp[4] = {0u, 0u, 0u, 0u};
            uint32_t fx[4] = {0u, 0u, 0u, 0u}, fy[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = 4 * c + j;
                const uint32_t word = Bsm[p];
                const uint32_t pb = (Psm[p >> 5] >> (p & 31)) & 1u;
                const bool real = p < a.g.n;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t byte = (word >> (8 * q)) & 0xFFu;
                    const uint32_t sv = real ? ((byte & 1u) ? 0x01u : 0xFFu) : 0u;
                    const int h = real ? (int)((byte & 0xFEu) | pb) - 128 : 0;
                    sp[q] |= sv << (8 * j);
                    if (j < 2) fx[q] |= ((uint32_t)h & 0xFFFFu) << (16 * j);
                    else fy[q] |= ((uint32_t)h & 0xFFFFu) << (16 * (j - 2));
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)(slot0 + q) * np + 4 * c;
                *reinterpret_cast<uint32_t *>(a.spins_out + row) = sp[q];
                *reinterpret_cast<uint2 *>(a.fields_out + row) = make_uint2(fx[q], fy[q]);
            }
        }
        if (tid < 4) {
            a.E_out[slot0 + tid] = Eacc[tid];
            if (a.emin_next && slot0 + tid < a.R) atomicMin(a.emin_next, Eacc[tid]);
        }
        if (tid == 0 && misc[5]) a.best_rec[blk] = make_int4(misc[0], misc[1], misc[2], misc[3]);
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, nacc);
        if (act && lane == 0 && wsum) atomicAdd(&a.accepts[a.k], (unsigned long long)wsum);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Small graphs in the layouts that keep fields (packed byte, FB = 7, or int8
// spins with int16 fields, FB = 16): every colour class fits one round of the
// block. With a few positions per class nothing is left but the latency of the
// class's chain, and this kernel takes out of it what does not depend on spins:
//   - all uniforms of a sweep are drawn before it (both Philox calls, so the
//     full 32-bit uniform: no tie path), 16 bytes per position;
//   - half of the warps decide (one lane per replica), the other half walk the
//     rows (a power of two of lanes per position, fixed by the class size, no
//     queue), and each half reads what it needs for its next turn while the
//     other one works.
// What stays per class: decide, barrier, field updates, barrier.
// Bound: that latency, and shared-memory atomics with many neighbours. Measured
// on GB300, us per step of 4 sweeps, general kernel / this one: n = 800, mean
// degree 48 (packed): R = 256 100 / 50, R = 2048 98 / 80, R = 3000 106 / 90,
// R = 4096 117 / 141; n = 96, degree 14, R = 24 35 / 24; n = 500, degree 250
// (int16, the general kernel with its queue and 128 threads): R = 1024 388 / 149,
// R = 4096 404 / 314, R = 8192 780 / 553. So it runs up to 5 (packed) or 16
// (int16) blocks per SM, with half the threads from 3 on.
// NH: deciding and walking threads, each.
constexpr int SMALL_MAX_HALF = 256;
constexpr int SMALL_UNITS = 3;   // row units a thread reads ahead

template <int FB>
__host__ __device__ inline size_t small_smem_words(int np, int ncol, int mmax, int half) {
    // uniforms, words of the layout, field changes, row starts, thresholds, class bounds, records, parities
    return 4 * (size_t)np + (FB == 7 ? (size_t)(np + 32) : 3 * (size_t)np + 64) + 2 * (size_t)half + (size_t)np + 4 +
           (size_t)((mmax + 4) & ~3) + (size_t)((ncol + 4) & ~3) + 16 + (FB == 7 ? (size_t)((np + 127) >> 7) * 4 : 0);
}

template <int FB, bool WEIGHTED, int NH>
__global__ void __launch_bounds__(2 * NH) k_sweep_small(const SweepArgs a) {
    constexpr int NT = 2 * NH;
    extern __shared__ __align__(16) unsigned char smem[];
    const int np = a.g.np, n = a.g.n, ncol = a.g.ncol;
    uint32_t *U = reinterpret_cast<uint32_t *>(smem);              // [np][4] uniforms of the sweep
    uint32_t *Bsm = U + 4 * np;                                    // FB 7: [np + 32] bytes; FB 16: [2 (np + 32)] fields
    uint32_t *Ssm = Bsm + 2 * (np + 32);                           // FB 16: [np] spins
    uint32_t *Dsm = FB == 7 ? Bsm + np + 32 : Ssm + np;            // [NH][2] field changes of the class
    uint32_t *rows = Dsm + 2 * NH;                                 // [np + 4] row starts in units
    uint32_t *T = rows + np + 4;                                   // thresholds by m
    int32_t *cls = reinterpret_cast<int32_t *>(T + ((a.g.mmax + 4) & ~3));
    int32_t *Eacc = cls + ((ncol + 4) & ~3);   // [4]
    int32_t *PS = Eacc + 4;                    // [4]
    int32_t *misc = PS + 4;                    // best E, step, sweep, slot, copy-from (q+1), changed
    uint32_t *Psm = reinterpret_cast<uint32_t *>(misc + 8);        // FB 7: degree parity bits
    const int tid = threadIdx.x, lane = tid & 31, ht = tid & (NH - 1);   // ht: thread of its half
    const bool decides = tid < NH;
    for (int i = tid; i <= n; i += NT) rows[i] = a.g.prp[i];
    if (FB == 7)
        for (int i = tid; i < (np + 31) >> 5; i += NT) Psm[i] = a.g.parity[i];
    for (int i = tid; i <= ncol; i += NT) cls[i] = a.g.cls[i];
    wait_previous();
    const bool act = !a.active || a.active[a.k];
    const int nsweeps = act ? a.S : 0;
    const uint32_t *tab = a.tables + (size_t)a.tidx[a.k] * (a.g.mmax + 1);
    for (int i = tid; i <= a.g.mmax; i += NT) T[i] = tab[i];

    for (int blk = blockIdx.x; blk < a.nblk; blk += gridDim.x) {
        const int slot0 = blk * 4;
        if (tid < 4) PS[tid] = act ? a.parent[slot0 + tid] : slot0 + tid;
        if (tid == 0) {
            const int4 br = a.best_rec[blk];
            misc[0] = br.x; misc[1] = br.y; misc[2] = br.z; misc[3] = br.w;
            misc[4] = 0; misc[5] = 0;
        }
        __syncthreads();
        if (tid < 4) Eacc[tid] = a.E_in[PS[tid]];
        for (int c = tid; c < (np >> 2); c += NT) {
            uint32_t w[4];
            uint2 f[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)PS[q] * np + 4 * c;
                w[q] = __ldcg(reinterpret_cast<const uint32_t *>(a.spins_in + row));
                f[q] = __ldcg(reinterpret_cast<const uint2 *>(a.fields_in + row));
            }
            uint32_t o[4];
            transpose4x4_bytes(w[0], w[1], w[2], w[3], o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t h[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) h[q] = ((j < 2 ? f[q].x : f[q].y) >> (16 * (j & 1))) & 0xFFFFu;
                if (FB == 7) {
                    uint32_t word = 0;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        word |= (((h[q] + 128u) & 0xFEu) | (((o[j] >> (8 * q)) & 0xFFu) == 1u ? 1u : 0u)) << (8 * q);
                    Bsm[4 * c + j] = word;
                } else {
                    Ssm[4 * c + j] = o[j];
                    Bsm[2 * (4 * c + j)] = (h[0] | h[1] << 16) ^ 0x80008000u;
                    Bsm[2 * (4 * c + j) + 1] = (h[2] | h[3] << 16) ^ 0x80008000u;
                }
            }
        }
        __syncthreads();
        const int q = tid & 3;   // the thread's replica
        const uint32_t live = slot0 + q < a.R ? 1u : 0u;
        const uint32_t c1 = (uint32_t)blk;
        uint32_t nacc = 0;
        // A walking thread's share of the class's rows: item, its first units and
        // where the rest would be.
        int li = 0;
        uint32_t nu = 0, enext = 0, lanes = 1;
        uint2 un[SMALL_UNITS];
        auto ahead = [&](int c) {
            const int p0 = cls[c], P = cls[c + 1] - p0;
            const int lt = P > 1 ? __clz(P - 1) - __clz(NH - 1) : 32 - __clz(NH - 1);   // log2(NH) less that of P rounded up
            li = ht >> lt;
            lanes = 1u << lt;
            nu = 0;
            if (li >= P) return;
            const uint32_t e0 = rows[p0 + li] + (ht & (lanes - 1u)), e1 = rows[p0 + li + 1];
            nu = e0 < e1 ? (e1 - e0 + lanes - 1u) >> lt : 0u;
            enext = e0 + SMALL_UNITS * lanes;
#pragma unroll
            for (int i = 0; i < SMALL_UNITS; ++i)
                if ((uint32_t)i < nu) un[i] = __ldg(&a.g.pcol[e0 + i * lanes]);
        };
        auto add4 = [&](const uint2 &v, const uint2 &D) {
            const uint32_t idx[4] = {v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const bool neg = WEIGHTED && (idx[t] & 0x8000u);
                const uint32_t j = idx[t] & 0x7FFFu;
                if (FB == 7) {
                    atomicAdd(&Bsm[j], neg ? 0u - D.x : D.x);
                } else {
                    atomicAdd(&Bsm[2 * j], neg ? 0u - D.x : D.x);
                    atomicAdd(&Bsm[2 * j + 1], neg ? 0u - D.y : D.y);
                }
            }
        };
        auto draw = [&](int s) {   // top bytes and tail bits of the four uniforms of every position
            const uint32_t c3 = TAG_SWEEP | (uint32_t)s;
            for (int p = tid; p < n; p += NT) {
                const uint32_t vid = __ldg(&a.g.vid[p]);
                const uint4 top = philox10(make_uint4(vid, c1 >> 2, (uint32_t)a.k, c3), a.key0, a.key1);
                const uint4 tl = philox10(make_uint4(vid, c1, (uint32_t)a.k, TAG_TAIL | (uint32_t)s), a.key0, a.key1);
                const uint32_t uw = word_of(top, c1 & 3u);
                *reinterpret_cast<uint4 *>(U + 4 * p) =
                    make_uint4(uw << 24 | tl.x >> 8, (uw >> 8) << 24 | tl.y >> 8, (uw >> 16) << 24 | tl.z >> 8,
                               (uw >> 24) << 24 | tl.w >> 8);
            }
        };
        // A deciding thread's first attempt of the next class: all but the spin
        // and the field.
        int idx = 0, cnt = 0;   // 4 position + replica, attempts of the class
        uint32_t u = 0, par = 0;
        auto load = [&](int i) {
            u = U[i];
            if (FB == 7) par = (Psm[i >> 7] >> ((i >> 2) & 31)) & 1u;
        };
        auto first = [&](int c) {
            idx = 4 * cls[c] + ht;
            cnt = 4 * (cls[c + 1] - cls[c]);
            if (ht < cnt) load(idx);
        };
        int dE = 0;
        if (nsweeps) {
            draw(0);
            __syncthreads();
            if (decides) first(0);
        }
        for (int s = 0; s < nsweeps; ++s) {
            for (int c = 0; c < ncol; ++c) {
                if (decides) {
                    for (int base = 0; base < cnt; base += NH) {   // uniform over the deciding half
                        const int i = idx + base, it = (base + ht) >> 2;
                        int d = 0;   // change of the neighbours' fields: -2 x if the replica flips
                        if (base + ht < cnt) {
                            if (base) load(i);
                            int h;
                            unsigned char *byte;
                            uint32_t up;   // x = +1
                            if (FB == 7) {
                                byte = reinterpret_cast<unsigned char *>(Bsm) + i;
                                const uint32_t b = *byte;
                                up = b & 1u;
                                h = (int)((b & 0xFEu) | par) - 128;
                            } else {
                                byte = reinterpret_cast<unsigned char *>(Ssm) + i;
                                h = (int)reinterpret_cast<const uint16_t *>(Bsm)[i] - 32768;
                                up = *byte == 1u;
                            }
                            const int m = up ? -h : h;   // dE = -2 x h = 2m
                            if (m <= 0 || u < T[min(m, a.g.mmax)]) {
                                *byte ^= FB == 7 ? 1u : 0xFEu;
                                d = up ? -2 : 2;
                                dE += 2 * m;
                                nacc += live;
                            }
                        }
                        if (FB == 7) {
                            int v = d * (1 << (8 * q));
                            v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                            v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
                            if (q == 0) Dsm[2 * it] = (uint32_t)v;
                        } else {
                            int v = d * (1 << (16 * (q & 1)));
                            v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                            if ((q & 1) == 0) Dsm[2 * it + (q >> 1)] = (uint32_t)v;
                        }
                    }
                } else {
                    ahead(c);
                }
                __syncthreads();
                if (decides) {
                    if (c + 1 < ncol) {
                        first(c + 1);
                    } else {   // the energies after the sweep
#pragma unroll
                        for (int off = 4; off < 32; off <<= 1) dE += __shfl_xor_sync(0xFFFFFFFFu, dE, off);
                        if (lane < 4 && dE != 0) atomicAdd(&Eacc[lane], dE);
                        dE = 0;
                    }
                } else if (nu) {
                    const uint2 D = make_uint2(Dsm[2 * li], FB == 7 ? 0u : Dsm[2 * li + 1]);
                    if (D.x | D.y) {
#pragma unroll
                        for (int i = 0; i < SMALL_UNITS; ++i)
                            if ((uint32_t)i < nu) add4(un[i], D);
                        for (uint32_t i = SMALL_UNITS, e = enext; i < nu; ++i, e += lanes) add4(__ldg(&a.g.pcol[e]), D);
                    }
                }
                __syncthreads();
            }
            if (tid < 32) {   // lowest energy of the sweep, the lowest slot first
                const int v = lane < 4 && slot0 + lane < a.R ? Eacc[lane] : 0x7FFFFFFF;
                const int bE = __reduce_min_sync(0xFFFFFFFFu, v);
                const int bq = __ffs(__ballot_sync(0xFFFFFFFFu, v == bE)) - 1;
                if (lane == 0) {
                    misc[4] = 0;
                    if (slot0 < a.R) atomicMin(&a.sweep_emin[(size_t)a.k * a.S + s], bE);
                    if (slot0 < a.R && bE < misc[0]) {
                        misc[0] = bE; misc[1] = a.k; misc[2] = s; misc[3] = slot0 + bq;
                        misc[4] = bq + 1; misc[5] = 1;
                    }
                }
            }
            if (s + 1 < nsweeps) draw(s + 1);
            __syncthreads();
            if (misc[4]) {   // block-uniform: copy the new best configuration
                const int sh = 8 * (misc[4] - 1);
                for (int c = tid; c < np; c += NT) {
                    const uint32_t w = FB == 7 ? Bsm[c] >> sh : Ssm[c] >> sh;
                    a.best_cfg[(size_t)blk * np + c] =
                        (int8_t)(FB == 16 ? (w & 0xFFu) : c < n ? ((w & 1u) ? 0x01u : 0xFFu) : 0u);
                }
                __syncthreads();   // before the next sweep changes the words
            }
            if (decides) first(0);
        }
        if (blk + (int)gridDim.x >= a.nblk) ready_for_next();
        // Store to the next population buffers.
        for (int c = tid; c < (np >> 2); c += NT) {
            uint32_t sp[4] = {0u, 0u, 0u, 0u}, fx[4] = {0u, 0u, 0u, 0u}, fy[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = 4 * c + j;
                const bool real = p < n;
                const uint32_t word = FB == 7 ? Bsm[p] : Ssm[p];
                const uint32_t pb = FB == 7 ? (Psm[p >> 5] >> (p & 31)) & 1u : 0u;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t byte = (word >> (8 * q)) & 0xFFu;
                    uint32_t h, sv;
                    if (FB == 7) {
                        sv = real ? ((byte & 1u) ? 0x01u : 0xFFu) : 0u;
                        h = real ? (uint32_t)((int)((byte & 0xFEu) | pb) - 128) & 0xFFFFu : 0u;
                    } else {
                        sv = byte;
                        h = ((Bsm[2 * p + (q >> 1)] ^ 0x80008000u) >> (16 * (q & 1))) & 0xFFFFu;
                    }
                    sp[q] |= sv << (8 * j);
                    if (j < 2) fx[q] |= h << (16 * j);
                    else fy[q] |= h << (16 * (j - 2));
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t row = (size_t)(slot0 + q) * np + 4 * c;
                *reinterpret_cast<uint32_t *>(a.spins_out + row) = sp[q];
                *reinterpret_cast<uint2 *>(a.fields_out + row) = make_uint2(fx[q], fy[q]);
            }
        }
        if (tid < 4) {
            a.E_out[slot0 + tid] = Eacc[tid];
            if (a.emin_next && slot0 + tid < a.R) atomicMin(a.emin_next, Eacc[tid]);
        }
        if (tid == 0 && misc[5]) a.best_rec[blk] = make_int4(misc[0], misc[1], misc[2], misc[3]);
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, nacc);
        if (act && lane == 0 && wsum) atomicAdd(&a.accepts[a.k], (unsigned long long)wsum);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Multi-spin-coded variant: W[p] holds the spins of 32 replicas (slots
// 32*blk .. 32*blk+31) at position p, 1 for +1. Replica 4g + q (byte q of
// word g of its Philox calls) sits at bit 8q + g. No fields are kept.
//
// An item (p, word) makes 32 attempts with bit-sliced arithmetic from the
// neighbour words to the decisions; a plane is one word holding one binary
// digit of a number for each of the 32 replicas.
//   count     XOR with each neighbour's word (and with all ones for a -1
//             weight) gives the frustrated-bond bits; carry-save adders count
//             them. The counter starts at -(deg/2 + 1), so it ends as
//             e = c - deg/2 - 1 in N-bit two's complement: its top plane says
//             m <= 0, and m = 2e + 1 (odd degree) or 2e + 2 (even degree).
//   uniforms  the 32 top bytes of the two Philox calls are turned into eight
//             planes by an 8 x 8 bit transpose in every byte lane.
//   decision  the planes of the threshold's top byte are OR-ed together from
//             the values of m whose T[m] has a non-zero top byte (from none
//             above beta = 2.8 to about 2.8 / beta); one comparison of eight
//             planes then gives "below" (accepted) and "equal" (a tie, which
//             the low 24 bits decide) for all 32 replicas.
//   energy    m of the accepted replicas is added to bit-sliced accumulators.
// What it replaces: the counts were transposed to one byte per replica, each
// group of four replicas was decided by two look-ups in a pair table and two
// multiply-adds in 16-bit lanes, and the energies went to byte counters
// flushed after every colour class: about 200 of 560 instructions per item.
// Bound: the ALU pipe (three-input logic and shifts) and, with few large
// colour classes' worth of warps per SM, latency. Measured per step of 10
// sweeps, means over beta 0.2 .. 3.6, R = 16384: G63-shaped (N = 7000) 0.981 ->
// 0.872 ms, signed torus (N = 10000) 1.030 -> 0.843 ms; with bit rows, round
// keys for the ties and narrower accumulators since, whole anneals of 200 steps
// G63-shaped 199 -> 161 ms and, R = 32768, 80 steps of 8 sweeps, torus 140 -> 110.
//
// A tie (probability 1/256 per uncertain attempt) is queued with its counter
// planes, and the ties of a warp's items are settled by all 32 lanes together
// before the class barrier (one tail Philox call per lane). Accepted replicas
// flip with one XOR.
__device__ __forceinline__ int msc_bit(int r) {   // bit of replica r = 4g + q in a word
    return 8 * (r & 3) + (r >> 2);
}

// 32 x 32 bit transpose over a warp: bit b of lane l goes to bit l of lane b.
__device__ __forceinline__ uint32_t msc_transpose32(uint32_t x, int lane) {
#pragma unroll
    for (int s = 16; s; s >>= 1) {
        const uint32_t m = 0xFFFFFFFFu / ((1u << s) + 1u);   // bits b with (b & s) == 0
        const bool hi = lane & s;
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
        const uint32_t keep = hi ? ~m : m, rot = __funnelshift_l(y, y, hi ? 32 - s : s);
        x = (keep & x) | (~keep & rot);
    }
    return x;
}

// Bit rows <-> words: a warp takes 128 positions of the word's 32 replicas, lane
// l the row of the replica at bit l (msc_bit), 16 bytes of it, and transposes
// them. Against int8 rows (32 loads and about 800 instructions per 4 positions
// of a thread and step) a step without sweeps went from 50 to 22 us (G63-
// shaped, R = 16384) and from 167 to 48 us (torus, R = 32768).
__device__ __forceinline__ int msc_lane_replica(int lane) { return 4 * (lane & 7) + (lane >> 3); }

// row: this lane's row; group of 128 positions q.
__device__ __forceinline__ void msc_load_words(const uint32_t *row, uint32_t *Wsm, int np, int q, int lane) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(row) + q);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t t = msc_transpose32(w[j], lane);
        const int p = 128 * q + 32 * j + lane;
        if (p < np) Wsm[p] = t;
    }
}

__device__ __forceinline__ void msc_store_words(const uint32_t *Wsm, uint32_t *row, int np, int q, int lane) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int p = 128 * q + 32 * j + lane;
        w[j] = msc_transpose32(p < np ? Wsm[p] : 0u, lane);
    }
    reinterpret_cast<uint4 *>(row)[q] = make_uint4(w[0], w[1], w[2], w[3]);
}

// Philox4x32-10 for the counters (c0, c1_g, c2, c3) of one item, which differ
// only in word 1: the products of rounds 1-3 whose inputs do not depend on c1
// are computed once (the result is identical to philox10 of each counter).
struct PhiloxShared {
    uint32_t u1;      // round 1: hi(M1 c2) ^ k0        (uniform)
    uint32_t l1;      // round 1: lo(M1 c2)              (uniform)
    uint32_t a, b;    // round 1: hi(M0 c0) ^ c3 ^ k1, lo(M0 c0)
    uint32_t s0, s1;  // round 2: hi(M1 a) ^ l1 ^ k0', lo(M1 a)
    uint32_t h3, l3;  // round 3: hi(M0 s0), lo(M0 s0)
};

__device__ __forceinline__ PhiloxShared philox_shared(uint32_t c0, uint32_t c2, uint32_t c3, uint32_t k0,
                                                      uint32_t k1) {
    PhiloxShared p;
    uint32_t hi;
    mul_wide(0xCD9E8D57u, c2, p.l1, hi);
    p.u1 = hi ^ k0;
    mul_wide(0xD2511F53u, c0, p.b, hi);
    p.a = hi ^ c3 ^ k1;
    mul_wide(0xCD9E8D57u, p.a, p.s1, hi);
    p.s0 = hi ^ p.l1 ^ (k0 + 0x9E3779B9u);
    mul_wide(0xD2511F53u, p.s0, p.l3, p.h3);
    return p;
}

// Philox4x32-10 of two counters of one item (word 1 = c1a, c1b), finished
// from the shared round-1-3 products and advanced round by round together,
// so that the two dependency chains interleave. The round keys come
// precomputed in the kernel arguments (rk0[r] = key0 + r * 0x9E3779B9,
// rk1[r] = key1 + r * 0xBB67AE85), so they are operands, not additions. Round 1: only word 0 depends
// on c1. Round 2: the word-2 product (s0, s1) is shared, the word-0 product
// is per counter. Round 3: the word-0 product (h3, l3) is shared.
__device__ __forceinline__ void philox_from_shared2(const PhiloxShared &p, uint32_t c1a, uint32_t c1b,
                                                    const uint32_t (&rk0)[10], const uint32_t (&rk1)[10], uint4 &ra,
                                                    uint4 &rb) {
    uint32_t lo, hi, lo2, hi2;
    mul_wide(0xD2511F53u, p.u1 ^ c1a, lo, hi);
    mul_wide(0xD2511F53u, p.u1 ^ c1b, lo2, hi2);
    uint4 a = make_uint4(p.s0, p.s1, hi ^ p.b ^ rk1[1], lo);
    uint4 b = make_uint4(p.s0, p.s1, hi2 ^ p.b ^ rk1[1], lo2);
    mul_wide(0xCD9E8D57u, a.z, lo, hi);
    mul_wide(0xCD9E8D57u, b.z, lo2, hi2);
    a = make_uint4(hi ^ a.y ^ rk0[2], lo, p.h3 ^ a.w ^ rk1[2], p.l3);
    b = make_uint4(hi2 ^ b.y ^ rk0[2], lo2, p.h3 ^ b.w ^ rk1[2], p.l3);
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        uint32_t alo0, ahi0, alo1, ahi1, blo0, bhi0, blo1, bhi1;
        mul_wide(0xD2511F53u, a.x, alo0, ahi0);
        mul_wide(0xD2511F53u, b.x, blo0, bhi0);
        mul_wide(0xCD9E8D57u, a.z, alo1, ahi1);
        mul_wide(0xCD9E8D57u, b.z, blo1, bhi1);
        a = make_uint4(ahi1 ^ a.y ^ rk0[r], alo1, ahi0 ^ a.w ^ rk1[r], alo0);
        b = make_uint4(bhi1 ^ b.y ^ rk0[r], blo1, bhi0 ^ b.w ^ rk1[r], blo0);
    }
    ra = a;
    rb = b;
}

// One three-input logic instruction; LUT is the function of 0xF0, 0xCC, 0xAA.
// Written out, because the compiler does not always find the single
// instruction for a majority or a bit select.
template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return d;
}
constexpr int L_MAJ = 0xE8, L_XOR = 0x96, L_SEL = 0xCA;   // a b + b c + c a; a ^ b ^ c; a ? b : c

// philox10 with the round keys of the kernel arguments.
__device__ __forceinline__ uint4 philox10_keys(uint4 c, const uint32_t (&rk0)[10], const uint32_t (&rk1)[10]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t lo0, hi0, lo1, hi1;
        mul_wide(0xD2511F53u, c.x, lo0, hi0);
        mul_wide(0xCD9E8D57u, c.z, lo1, hi1);
        c = make_uint4(hi1 ^ c.y ^ rk0[r], lo1, hi0 ^ c.w ^ rk1[r], lo0);
    }
    return c;
}

// Full adder of the planes a, b, c: returns the carry, a becomes the sum.
__device__ __forceinline__ uint32_t msc_fa(uint32_t &a, uint32_t b, uint32_t c) {
    const uint32_t k = lop3<L_MAJ>(a, b, c);
    a = lop3<L_XOR>(a, b, c);
    return k;
}

// Adds one carry plane into counters kept in complemented form (below), from
// plane FROM upwards: full adders whose third input is a zero, that is x.
template <int N, int FROM>
__device__ __forceinline__ void msc_ripple(uint32_t (&A)[N], uint32_t x, uint32_t c) {
#pragma unroll
    for (int b = FROM; b < N; ++b) c = msc_fa(A[b], c, x);
}

// Adds four or eight bonds to counters kept in complemented form A_b =
// plane_b ^ x, where the input words are the raw neighbour words w_j. A full
// adder keeps the form: (a^x) ^ (p^x) ^ (q^x) = (a^p^q) ^ x and, majority
// being self-dual, maj(a^x, p^x, q^x) = maj(a, p, q) ^ x. Eight bonds: seven
// full adders (four on the ones, two on the twos, one on the fours) and one
// carry to ripple, 14 + 2 (N - 3) - 1 operations against 2 (6 + 2 (N - 2) - 1)
// for two steps of four.
template <int N>
__device__ __forceinline__ void msc_step4x(uint32_t (&A)[N], uint32_t x, const uint32_t (&w)[4]) {
    const uint32_t c1 = msc_fa(A[0], w[0], w[1]);
    const uint32_t c2 = msc_fa(A[0], w[2], w[3]);
    msc_ripple<N, 2>(A, x, msc_fa(A[1], c1, c2));
}

template <int N>
__device__ __forceinline__ void msc_step8x(uint32_t (&A)[N], uint32_t x, const uint32_t (&w)[4],
                                           const uint32_t (&v)[4]) {
    const uint32_t c1 = msc_fa(A[0], w[0], w[1]);
    const uint32_t c2 = msc_fa(A[0], w[2], w[3]);
    const uint32_t c3 = msc_fa(A[0], v[0], v[1]);
    const uint32_t c4 = msc_fa(A[0], v[2], v[3]);
    const uint32_t d1 = msc_fa(A[1], c1, c2);
    const uint32_t d2 = msc_fa(A[1], c3, c4);
    msc_ripple<N, 3>(A, x, msc_fa(A[2], d1, d2));
}

// 8 x 8 bit transpose in every byte lane: bit i of byte q of r[j] goes to bit
// j of byte q of r[i]. Words NZ..7 are zero on input (their swaps fold).
template <int NZ>
__device__ __forceinline__ void msc_transpose8(uint32_t (&r)[8]) {
    auto swap = [](uint32_t &x, uint32_t &y, int s, uint32_t M, bool zx, bool zy) {
        if (zx && zy) return;
        const uint32_t lo = zy ? (x & M) : lop3<L_SEL>(M, x, y << s);
        y = zy ? ((x >> s) & M) : lop3<L_SEL>(M, x >> s, y);
        x = lo;
    };
#pragma unroll
    for (int b = 0; b < 4; ++b) swap(r[b], r[b + 4], 4, 0x0F0F0F0Fu, b >= NZ, b + 4 >= NZ);
#pragma unroll
    for (int b = 0; b < 8; b += (b & 1) ? 3 : 1)   // 0, 1, 4, 5
        swap(r[b], r[b + 2], 2, 0x33333333u, (b & 3) >= NZ, ((b + 2) & 3) >= NZ);
#pragma unroll
    for (int b = 0; b < 8; b += 2)
        swap(r[b], r[b + 1], 1, 0x55555555u, (b & 3) >= NZ && ((b ^ 2) & 3) >= NZ,
             ((b + 1) & 3) >= NZ && (((b + 1) ^ 2) & 3) >= NZ);
}

// Shape of the multi-spin-coded tables for N counter planes (max degree below
// 2^N). lvl: masks of the eight bits of T[m] >> 24 for every m = 2e + 1
// (odd degree) and 2e + 2 (even degree) in that order, as words (N <= 5) or,
// to keep the table small at wide degrees, as bytes. init: the
// planes 0 .. N-2 of -(deg/2 + 1) as masks by degree (the top plane is always
// set; wider counters derive them from the number).
template <int N>
struct MscShape {
    static constexpr bool wide = N > 5;
    static constexpr int nm = 1 << N;                        // values of m in the table
    static constexpr int lvl_words = wide ? 2 * nm : 8 * nm;
    static constexpr int init_words = wide ? 0 : 4 * nm;
    // Energy accumulators and the items they hold: 2^k (2^N - 1) < 2^(N + k).
    // More planes flush less often and cost two operations per item each.
    static constexpr int flush_items = N > 4 ? 32 : 64;
    static constexpr int acc_planes = N + (N > 4 ? 6 : 7);
    static constexpr int entry = (N + 3) & ~1;               // words of a tie-queue entry: 3 and N - 1 planes, made even
};

// Words of shared memory a block may use beside the words of the positions
// and the class bounds: fixed by the degree class, so that the largest graph
// that fits does not move when the tables change. The tie queues take what the
// tables leave, and more when the graph leaves room.
__host__ __device__ inline int msc_reserved_words(int mmax) {
    return 256 + (mmax <= 7 ? 256 : mmax <= 15 ? 1024 : mmax <= 31 ? 4096 : 0) + 72 + 512;
}

__host__ __device__ inline int msc_planes(int mmax) {
    return mmax <= 7 ? 3 : mmax <= 15 ? 4 : mmax <= 31 ? 5 : mmax <= 63 ? 6 : 7;
}

__host__ __device__ inline int msc_entry_words(int mmax) { return (msc_planes(mmax) + 3) & ~1; }

__host__ __device__ inline int msc_table_words(int mmax) {   // lvl, init, thresholds
    const int nm = 1 << msc_planes(mmax);
    return (nm > 32 ? 2 * nm : 12 * nm) + nm;
}

// Uniform parameters of a step's decisions, found once per block.
struct MscLevels {
    int top;    // values e >= top have thresholds with a zero top byte
    int zero;   // values e >= zero have a zero threshold: their ties reject
};

// One unit (four bonds) of a lane's row: the neighbours' words, complemented
// for weight -1. BIG: 32-bit entries (byte offset | sign); otherwise pairs of
// 16-bit byte offsets with the pair's signs in the low bits of the first.
template <bool BIG>
using MscUnit = std::conditional_t<BIG, uint4, uint2>;

template <bool WEIGHTED>
__device__ __forceinline__ void msc_unit_words(const unsigned char *Wb, const uint2 &v, uint32_t (&w)[4]) {
    const uint32_t vv[2] = {v.x, v.y};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        w[2 * j] = *reinterpret_cast<const uint32_t *>(Wb + (vv[j] & 0xFFFCu));
        w[2 * j + 1] = *reinterpret_cast<const uint32_t *>(Wb + (vv[j] >> 16));
        if (WEIGHTED) {
            w[2 * j] ^= (uint32_t)((int32_t)(vv[j] << 31) >> 31);
            w[2 * j + 1] ^= (uint32_t)((int32_t)(vv[j] << 30) >> 31);
        }
    }
}

template <bool WEIGHTED>
__device__ __forceinline__ void msc_unit_words(const unsigned char *Wb, const uint4 &v, uint32_t (&w)[4]) {
    const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w[j] = *reinterpret_cast<const uint32_t *>(Wb + (WEIGHTED ? vv[j] & ~3u : vv[j]));
        if (WEIGHTED) w[j] ^= (uint32_t)((int32_t)(vv[j] << 31) >> 31);
    }
}

// One slice as a warp sees it.
struct MscSlice {
    uint32_t vd;            // vertex | degree << 16 | 1 << 31 on lanes past the class
    uint32_t off, units;    // byte offset of the lane's first unit; units of the slice (uniform)
};

template <bool BIG>
__device__ __forceinline__ MscUnit<BIG> msc_unit(const void *mcol, uint32_t off, uint32_t u) {
    constexpr uint32_t bytes = 32u * sizeof(MscUnit<BIG>);
    return __ldg(reinterpret_cast<const MscUnit<BIG> *>(reinterpret_cast<const char *>(mcol) + (off + u * bytes)));
}

// One (position, word) item: 32 attempts. Returns the mask of accepted
// replicas; `tie` are the undecided ones, E the counter planes of e. Lanes past
// their class run along and accept nothing.
// The first two units are read before the random numbers are drawn, which
// covers their latency.
template <int N, bool WEIGHTED, bool BIG>
__device__ __forceinline__ uint32_t msc_item(const SweepArgs &a, const uint32_t *Wsm, const uint32_t *lvl,
                                             const uint32_t *init, const MscLevels &L, const MscSlice &sl,
                                             uint32_t x, uint32_t c3, int blk, uint32_t (&E)[N],
                                             uint32_t (&S)[MscShape<N>::acc_planes], uint32_t &tie,
                                             uint32_t &odd_out) {
    const uint32_t vid = sl.vd & 0xFFFFu, deg = (sl.vd >> 16) & 0x7Fu;
    const MscUnit<BIG> v0 = msc_unit<BIG>(a.g.mcol, sl.off, 0u), v1 = msc_unit<BIG>(a.g.mcol, sl.off, sl.units > 1u ? 1u : 0u);
    // Both Philox calls of the item (slots 32 blk .. +15 and +16 .. +31).
    uint4 u0, u1;
    philox_from_shared2(philox_shared(vid, (uint32_t)a.k, c3, a.key0, a.key1), 2u * blk, 2u * blk + 1u, a.rk0, a.rk1,
                        u0, u1);
    uint32_t U[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
    if (L.top) msc_transpose8<8>(U);
    // Counter planes of -(deg/2 + 1), complemented by x.
    uint32_t A[N];
    if (MscShape<N>::wide) {
        const uint32_t k = ~(deg >> 1);   // -(deg/2 + 1)
#pragma unroll
        for (int b = 0; b < N - 1; ++b) A[b] = x ^ (uint32_t)((int32_t)(k << (31 - b)) >> 31);
    } else {
        const uint4 i4 = *reinterpret_cast<const uint4 *>(init + 4 * deg);
        const uint32_t iv[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
        for (int b = 0; b < N - 1; ++b) A[b] = x ^ iv[b];
    }
    A[N - 1] = ~x;
    {
        const unsigned char *Wb = reinterpret_cast<const unsigned char *>(Wsm);
        uint32_t w[4], v[4];
        msc_unit_words<WEIGHTED>(Wb, v0, w);
        if (sl.units > 1) {
            msc_unit_words<WEIGHTED>(Wb, v1, v);
            msc_step8x<N>(A, x, w, v);
            uint32_t u = 2;
            for (; u + 2 <= sl.units; u += 2) {
                msc_unit_words<WEIGHTED>(Wb, msc_unit<BIG>(a.g.mcol, sl.off, u), w);
                msc_unit_words<WEIGHTED>(Wb, msc_unit<BIG>(a.g.mcol, sl.off, u + 1u), v);
                msc_step8x<N>(A, x, w, v);
            }
            if (u < sl.units) {
                msc_unit_words<WEIGHTED>(Wb, msc_unit<BIG>(a.g.mcol, sl.off, u), w);
                msc_step4x<N>(A, x, w);
            }
        } else {
            msc_step4x<N>(A, x, w);
        }
    }
#pragma unroll
    for (int b = 0; b < N; ++b) E[b] = A[b] ^ x;
    const uint32_t neg = E[N - 1];
    uint32_t high = 0u;   // e >= 4 (or negative)
#pragma unroll
    for (int b = 2; b < N; ++b) high |= E[b];
    uint32_t lt = 0u, eq;
    if (L.top == 0) {
        // Every threshold has a zero top byte: only a zero byte can accept. The
        // OR of each byte's bits, folded in the steps of the transpose (35
        // operations against 48 and 4; steps with beta above 2.8: -8%).
        auto fold = [](uint32_t x, uint32_t y, int s, uint32_t M) {
            return lop3<L_SEL>(M, x | (x >> s), y | (y << s));
        };
        const uint32_t f0 = fold(U[0], U[4], 4, 0x0F0F0F0Fu), f1 = fold(U[1], U[5], 4, 0x0F0F0F0Fu);
        const uint32_t f2 = fold(U[2], U[6], 4, 0x0F0F0F0Fu), f3 = fold(U[3], U[7], 4, 0x0F0F0F0Fu);
        eq = ~fold(fold(f0, f2, 2, 0x33333333u), fold(f1, f3, 2, 0x33333333u), 1, 0x55555555u);
    } else {
        // Planes of the threshold's top byte: for every value of e below L.top,
        // the replicas with that e take the bits of their own parity's m.
        uint32_t TP[8];
        const uint32_t *lv = lvl + ((deg & 1u) ? 0 : MscShape<N>::wide ? 2 : 8);
        auto take = [&](int e, uint32_t who, bool first) {
            uint32_t v[8];
            if (MscShape<N>::wide) {
                const uint2 q = *reinterpret_cast<const uint2 *>(lv + 4 * e);
#pragma unroll
                for (int b = 0; b < 8; ++b) v[b] = __byte_perm(b < 4 ? q.x : q.y, 0u, 0x1111u * (b & 3));
            } else {
                const uint4 q0 = *reinterpret_cast<const uint4 *>(lv + 16 * e);
                const uint4 q1 = *reinterpret_cast<const uint4 *>(lv + 16 * e + 4);
                v[0] = q0.x; v[1] = q0.y; v[2] = q0.z; v[3] = q0.w;
                v[4] = q1.x; v[5] = q1.y; v[6] = q1.z; v[7] = q1.w;
            }
#pragma unroll
            for (int b = 0; b < 8; ++b) TP[b] = first ? (who & v[b]) : lop3<0xF8>(TP[b], who, v[b]);   // | who & v
        };
        take(0, ~(high | E[0] | E[1]), true);
        if (L.top > 1) {
            take(1, lop3<0x10>(E[0], E[1], high) , false);   // E0 & ~E1 & ~high
            if (L.top > 2) {
                take(2, lop3<0x04>(E[0], E[1], high), false);   // ~E0 & E1 & ~high
                if (L.top > 3) take(3, lop3<0x40>(E[0], E[1], high), false);   // E0 & E1 & ~high
            }
#pragma unroll 1
            for (int j = 1; N > 3 && 4 * j < L.top; ++j) {
                uint32_t no = neg;   // not in this group of four values
#pragma unroll
                for (int b = 2; b < N - 1; ++b) no |= ((j >> (b - 2)) & 1) ? ~E[b] : E[b];
                take(4 * j, ~(no | E[0] | E[1]), false);
                take(4 * j + 1, lop3<0x10>(E[0], E[1], no), false);
                take(4 * j + 2, lop3<0x04>(E[0], E[1], no), false);
                take(4 * j + 3, lop3<0x40>(E[0], E[1], no), false);
            }
        }
        eq = ~0u;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            lt = lop3<0xB2>(TP[b], U[b], lt);   // T & ~U | ~(T ^ U) & lt
            eq = lop3<0x82>(TP[b], U[b], eq);   // ~(T ^ U) & eq
        }
    }
    const uint32_t live = ~(uint32_t)((int32_t)sl.vd >> 31);
    const uint32_t acc = (neg | lt) & live;
    // Ties of a zero threshold reject: e >= 4 (e >= 2) where no such threshold is left.
    tie = eq & ~neg & live;
    if (L.zero <= 4) tie &= ~high;
    if (L.zero <= 2) tie &= ~E[1];
    // Energies: S += m = 2e + 1 + (even degree) of the accepted replicas, in
    // two's complement (the carry-in is the 1).
    const uint32_t odd = 0u - (deg & 1u);
    odd_out = odd;
    uint32_t c = lop3<0xD0>(acc, S[0], odd);   // acc & (S0 | ~odd)
    S[0] = lop3<0x78>(S[0], acc, odd);         // S0 ^ (acc & odd)
#pragma unroll
    for (int b = 0; b < N; ++b) c = msc_fa(S[b + 1], E[b] & acc, c);
    const uint32_t sign = neg & acc;
#pragma unroll
    for (int b = N + 1; b < MscShape<N>::acc_planes; ++b) c = msc_fa(S[b], sign, c);
    return acc;
}

// Adds the accumulated m of the warp's lanes to the energies (dE = 2m) and
// clears them: the planes become bytes by transposes (the low eight planes,
// then the rest with the sign plane inverted, that is plus 2^(W-1)), which sum
// over the lanes in 16-bit halves without carries. Runs after at most 64 (32) items
// per lane, so once or a few times per sweep.
template <int N>
__device__ __forceinline__ void msc_flush_energy(uint32_t (&S)[MscShape<N>::acc_planes], int32_t *Eacc, int lane) {
    constexpr int W = MscShape<N>::acc_planes, NH = W - 8;
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        lo[b] = S[b];
        hi[b] = b < NH ? (b == NH - 1 ? ~S[b + 8] : S[b + 8]) : 0u;
    }
    msc_transpose8<8>(lo);
    msc_transpose8<NH>(hi);
    uint32_t mlo = 0u, mhi = 0u;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        const uint32_t a0 = __reduce_add_sync(0xFFFFFFFFu, lo[g] & 0x00FF00FFu);          // bytes 0, 2
        const uint32_t a1 = __reduce_add_sync(0xFFFFFFFFu, (lo[g] >> 8) & 0x00FF00FFu);   // bytes 1, 3
        const uint32_t b0 = __reduce_add_sync(0xFFFFFFFFu, hi[g] & 0x00FF00FFu);
        const uint32_t b1 = __reduce_add_sync(0xFFFFFFFFu, (hi[g] >> 8) & 0x00FF00FFu);
        if ((lane >> 2) == g) {
            mlo = (lane & 1) ? a1 : a0;
            mhi = (lane & 1) ? b1 : b0;
        }
    }
    const int sh = (lane & 2) ? 16 : 0;
    const int m = (int)((mlo >> sh) & 0xFFFFu) + 256 * (int)((mhi >> sh) & 0xFFFFu) - (32 << (W - 1));
    if (m) atomicAdd(&Eacc[lane], 2 * m);
#pragma unroll
    for (int b = 0; b < W; ++b) S[b] = 0u;
}

// Copies of the word array that a block writes besides its own: the other
// CTAs of its cluster (none outside a cluster).
template <bool CL>
struct MscPeers {
    uint32_t *Wsm;
    int rank, size;
    __device__ __forceinline__ void store(int p, uint32_t v) const {
        Wsm[p] = v;
        if (CL)
            for (int d = 1; d < size; ++d) cooperative_groups::this_cluster().map_shared_rank(Wsm, rank ^ d)[p] = v;
    }
    __device__ __forceinline__ void flip(int p, uint32_t bits) const {
        atomicXor(&Wsm[p], bits);
        if (CL)
            for (int d = 1; d < size; ++d)
                atomicXor(&cooperative_groups::this_cluster().map_shared_rank(Wsm, rank ^ d)[p], bits);
    }
};

// Ties queued by the items of a warp (entry: tie mask, position | vertex << 16,
// odd-degree mask, planes of e) are settled together: each lane takes one entry, draws
// the low 24 bits of its uniforms and applies an accepted flip to the word
// (and its copies), the energy and the accept count. Items of one colour class
// never read each other's words, so a flip applied after the other items of
// the class is the same as one applied at once; every queue is emptied before
// the class barrier.
template <int N, bool CL>
__device__ __forceinline__ void msc_drain_ties(const SweepArgs &a, const uint32_t *Tt, const uint32_t *TQ, int qc,
                                               const MscPeers<CL> &W, int32_t *Eacc, int blk, uint32_t c3,
                                               uint32_t vmask, uint32_t &nacc, int lane) {
    __syncwarp();
    for (int i = lane; i < qc; i += 32) {
        const uint32_t *q = TQ + MscShape<N>::entry * i;
        uint32_t tie = q[0];
        const int p = (int)(q[1] & 0xFFFFu), odd = (int)(q[2] & 1u);
        const uint32_t vid = q[1] >> 16;
        do {
            const int bit = __ffs(tie) - 1;
            tie &= tie - 1u;
            uint32_t e = 0u;
#pragma unroll
            for (int b = 0; b < N - 1; ++b) e |= ((q[3 + b] >> bit) & 1u) << b;
            const int m = 2 * (int)e + 2 - odd;
            const int rep = 4 * (bit & 7) + (bit >> 3);
            const uint4 u = philox10_keys(make_uint4(vid, (32u * blk + rep) >> 2, (uint32_t)a.k, TAG_TAIL | c3), a.rk0,
                                          a.rk1);
            if ((word_of(u, rep & 3u) >> 8) < (Tt[m] & 0xFFFFFFu)) {
                W.flip(p, 1u << bit);
                atomicAdd(&Eacc[rep], 2 * m);
                nacc += (vmask >> bit) & 1u;
            }
        } while (tie);
    }
    __syncwarp();
}

// Sweeps of multi-spin-coded words. CL: a thread-block cluster (2, 4 or
// 8 CTAs) shares a word. Every CTA keeps a full copy of the word array; inside a
// colour class the CTAs take the positions in turns of 32, every changed word
// is stored into all copies (the others' through distributed shared memory),
// and a cluster barrier closes each class. The 32 energies live in CTA 0,
// which also does the best tracking; the others add their changes there
// remotely. Halving the work unit lets the SMs balance the words that do not
// divide over them.
template <int N, bool WEIGHTED, bool BIG, bool CL>
__global__ void __launch_bounds__(512, 2) k_sweep_msc(const SweepArgs a) {
    namespace cg = cooperative_groups;
    using Sh = MscShape<N>;
    extern __shared__ __align__(16) unsigned char smem[];
    wait_previous();
    const bool act = !a.active || a.active[a.k];
    const int nsweeps = act ? a.S : 0;
    const int np = a.g.np, n = a.g.n;
    uint32_t *lvl = reinterpret_cast<uint32_t *>(smem);            // top-byte masks by m
    uint32_t *init = lvl + Sh::lvl_words;                           // counter start by degree
    uint32_t *Tt = init + Sh::init_words;                           // [2^N] thresholds by m
    uint32_t *Wsm = Tt + Sh::nm;                                    // [np]
    int32_t *cls = reinterpret_cast<int32_t *>(Wsm + np);
    const int csz = (a.g.ncol + 1 + 3) & ~3;
    int32_t *Eacc = cls + csz;      // [32] (in a cluster: CTA 0's)
    int32_t *PS = Eacc + 32;        // [32]
    int32_t *misc = PS + 32;        // best E, step, sweep, slot, copy-from (r+1), changed, level bounds
    const int NT = blockDim.x;   // 256 or 512
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    uint32_t *TQ = reinterpret_cast<uint32_t *>(misc + 8) + (size_t)warp * a.qcap * Sh::entry;   // this warp's tie queue
    int rank = 0, csize = 1;
    if (CL) {
        rank = (int)cg::this_cluster().block_rank();
        csize = (int)cg::this_cluster().num_blocks();
    }
    const MscPeers<CL> W{Wsm, rank, csize};
    int32_t *E0 = CL ? cg::this_cluster().map_shared_rank(Eacc, 0) : Eacc;
    auto barrier = [&]() {
        if (CL) cg::this_cluster().sync();
        else __syncthreads();
    };

    if (tid < 2) misc[6 + tid] = 0;
    __syncthreads();
    const uint32_t *tab = a.tables + (size_t)a.tidx[a.k] * (a.g.mmax + 1);
    for (int m = tid; m < Sh::nm; m += NT) {
        const uint32_t Tm = m > 0 && m <= a.g.mmax ? tab[m] : 0u;
        Tt[m] = Tm;
        if (Tm >> 24) atomicMax(&misc[6], (m + 1) >> 1);   // e + 1 of this m
        if (Tm) atomicMax(&misc[7], (m + 1) >> 1);
        const uint32_t T = m + 1 <= a.g.mmax ? tab[m + 1] : 0u;   // entry m: m + 1 = 2e + 1 or 2e + 2
        if (Sh::wide) {
            uint32_t lo = 0u, hi = 0u;
            for (int b = 0; b < 4; ++b) {
                lo |= ((T >> (24 + b)) & 1u) * (0xFFu << (8 * b));
                hi |= ((T >> (28 + b)) & 1u) * (0xFFu << (8 * b));
            }
            lvl[2 * m] = lo;
            lvl[2 * m + 1] = hi;
        } else {
            for (int b = 0; b < 8; ++b) lvl[8 * m + b] = 0u - ((T >> (24 + b)) & 1u);
            for (int b = 0; b < 4; ++b) init[4 * m + b] = 0u - ((~((uint32_t)m >> 1) >> b) & 1u);   // m: a degree here
        }
    }
    for (int i = tid; i <= a.g.ncol; i += NT) cls[i] = a.g.csl[i];   // slices of each class

    const int nunits = (int)gridDim.x / csize;
    for (int lb = (int)blockIdx.x / csize; lb < a.nblk; lb += nunits) {   // uniform within a cluster
        const int blk = a.blk_base + lb;
        const int slot0 = blk * 32;
        if (tid < 32) PS[tid] = act ? a.parent[slot0 + tid] : slot0 + tid;
        if (tid == 0) {
            const int4 br = a.best_rec[blk];
            misc[0] = br.x; misc[1] = br.y; misc[2] = br.z; misc[3] = br.w;
            misc[4] = 0; misc[5] = 0;
        }
        __syncthreads();
        if (tid < 32 && rank == 0) Eacc[tid] = a.E_in[PS[tid]];
        {   // bit rows of the parents -> one word per position
            const uint32_t *row = reinterpret_cast<const uint32_t *>(a.spins_in) +
                                  (size_t)PS[msc_lane_replica(lane)] * a.g.nbw;
            for (int q = warp; 4 * q < a.g.nbw; q += NT / 32) msc_load_words(row, Wsm, np, q, lane);
        }
        barrier();   // all copies loaded, energies in place
        const MscLevels L{misc[6], misc[7]};
        uint32_t vmask = 0u;   // bits of the live replicas
        for (int r = 0; r < 32; ++r) vmask |= (slot0 + r < a.R ? 1u : 0u) << msc_bit(r);
        uint32_t nacc = 0;
        uint32_t S[Sh::acc_planes];
#pragma unroll
        for (int b = 0; b < Sh::acc_planes; ++b) S[b] = 0u;
        int cnt = 0;   // items per lane in S
        const int w0 = warp * csize + rank, nw = (NT >> 5) * csize;
        // Descriptor and vertices of the warp's next slice, read one slice ahead.
        uint2 d = make_uint2(0u, 0u);
        uint32_t vd = 0u;
        auto ahead = [&](int k) {
            d = __ldg(&a.g.msl[k]);
            vd = __ldg(&a.g.mvd[32 * k + lane]);
        };
        if (w0 < cls[1]) ahead(w0);
        for (int s = 0; s < nsweeps; ++s) {
            const uint32_t c3 = TAG_SWEEP | (uint32_t)s;
            for (int c = 0; c < a.g.ncol; ++c) {
                const int k1 = cls[c + 1];
                int qc = 0;   // entries in this warp's tie queue
                for (int k = cls[c] + w0; k < k1; k += nw) {
                    constexpr uint32_t bytes = sizeof(MscUnit<BIG>);
                    const MscSlice sl{vd, (d.x & 0xFFFFFFu) * (32u * bytes) + bytes * (uint32_t)lane,
                                      __shfl_sync(0xFFFFFFFFu, d.x >> 24, 0)};
                    const uint32_t p = d.y + (uint32_t)lane;   // past the class: still inside the block's memory
                    const uint32_t x = Wsm[p];
                    if (k + nw < k1) ahead(k + nw);
                    uint32_t tie, odd, E[N];
                    const uint32_t acc = msc_item<N, WEIGHTED, BIG>(a, Wsm, lvl, init, L, sl, x, c3, blk, E, S, tie, odd);
                    if (acc) {
                        W.store(p, x ^ acc);
                        nacc += __popc(acc & vmask);
                    }
                    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, tie != 0u);
                    const int nt = __popc(bal);
                    if (qc + nt > a.qcap) {
                        msc_drain_ties<N, CL>(a, Tt, TQ, qc, W, E0, blk, c3, vmask, nacc, lane);
                        qc = 0;
                    }
                    int rk = qc + __popc(bal & ((1u << lane) - 1u));
                    qc += nt;
                    for (;;) {   // once, unless the queue is shorter than the ties of one slice
                        if (tie && (uint32_t)rk < (uint32_t)a.qcap) {
                            uint32_t *q = TQ + Sh::entry * rk;
                            uint32_t v[10] = {tie, p | sl.vd << 16, odd, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
                            for (int b = 0; b < N - 1; ++b) v[3 + b] = E[b];
                            if (Sh::entry == 8) {
                                *reinterpret_cast<uint4 *>(q) = make_uint4(v[0], v[1], v[2], v[3]);
                                *reinterpret_cast<uint4 *>(q + 4) = make_uint4(v[4], v[5], v[6], v[7]);
                            } else {
#pragma unroll
                                for (int b = 0; b < Sh::entry; b += 2)
                                    *reinterpret_cast<uint2 *>(q + b) = make_uint2(v[b], v[b + 1]);
                            }
                        }
                        if (qc <= a.qcap) break;
                        msc_drain_ties<N, CL>(a, Tt, TQ, a.qcap, W, E0, blk, c3, vmask, nacc, lane);
                        rk -= a.qcap;
                        qc -= a.qcap;
                    }
                    if (++cnt == Sh::flush_items) {
                        msc_flush_energy<N>(S, E0, lane);
                        cnt = 0;
                    }
                }
                {
                    const int cn = c + 1 < a.g.ncol ? c + 1 : 0, kc = cls[cn] + w0;
                    if (kc < cls[cn + 1]) ahead(kc);
                }
                if (qc) msc_drain_ties<N, CL>(a, Tt, TQ, qc, W, E0, blk, c3, vmask, nacc, lane);
                if (c + 1 == a.g.ncol && cnt) {
                    msc_flush_energy<N>(S, E0, lane);
                    cnt = 0;
                }
                barrier();
            }
            if (rank == 0 && warp == 0) {   // lowest energy of the sweep, the lowest slot first
                const int v = slot0 + lane < a.R ? Eacc[lane] : 0x7FFFFFFF;
                const int bE = __reduce_min_sync(0xFFFFFFFFu, v);
                const int bq = __ffs(__ballot_sync(0xFFFFFFFFu, v == bE)) - 1;
                if (lane == 0) {
                    misc[4] = 0;
                    atomicMin(&a.sweep_emin[(size_t)a.k * a.S + s], bE);
                    if (bE < misc[0]) {
                        misc[0] = bE; misc[1] = a.k; misc[2] = s; misc[3] = slot0 + bq;
                        misc[4] = bq + 1; misc[5] = 1;
                    }
                }
            }
            __syncthreads();
            if (misc[4]) {   // in a cluster: CTA 0 only (the others never set it)
                const int rq = misc[4] - 1;
                uint32_t *dst = reinterpret_cast<uint32_t *>(a.best_cfg + (size_t)blk * np);
                for (int c = tid; c < (np >> 2); c += NT) {
                    uint32_t v = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool real = 4 * c + j < n;
                        v |= (real ? (((Wsm[4 * c + j] >> msc_bit(rq)) & 1u) ? 0x01u : 0xFFu) : 0u) << (8 * j);
                    }
                    dst[c] = v;
                }
                if (!CL) __syncthreads();
            }
            if (CL) barrier();   // the copy reads CTA 0's words before the next sweep changes them
        }
        if (lb + nunits >= a.nblk) ready_for_next();
        {   // words -> bit rows; the CTAs of a cluster share the columns
            uint32_t *row = reinterpret_cast<uint32_t *>(a.spins_out) +
                            (size_t)(slot0 + msc_lane_replica(lane)) * a.g.nbw;
            for (int q = warp * csize + rank; 4 * q < a.g.nbw; q += (NT / 32) * csize)
                msc_store_words(Wsm, row, np, q, lane);
        }
        if (rank == 0) {
            if (warp == 0) {
                a.E_out[slot0 + lane] = Eacc[lane];
                const int v = __reduce_min_sync(0xFFFFFFFFu, slot0 + lane < a.R ? Eacc[lane] : 0x7FFFFFFF);
                if (lane == 0 && a.emin_next) atomicMin(a.emin_next, v);
            }
            if (tid == 0 && misc[5]) a.best_rec[blk] = make_int4(misc[0], misc[1], misc[2], misc[3]);
        }
        const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, nacc);
        if (act && lane == 0 && wsum) atomicAdd(&a.accepts[a.k], (unsigned long long)wsum);
        barrier();   // no copy is reused before all CTAs are done with this word
    }
}

// Energies of 32 configurations at a time, one CTA per word, for graphs with
// slice rows: the configurations become words, the frustrated bonds of every
// position are counted as in the sweep (7 planes for any degree) and summed in
// bit-sliced accumulators; E = (stored entries / 2) - sum of the counts. SRC:
//   WORDS_INIT  spins of the initial population: +1 iff bit 31 of its Philox
//               word is set; written to the population's bit rows
//   WORDS_POP   bit rows of a population
//   WORDS_RAW   configurations in vertex order (n bytes each, any alignment);
//               a byte other than +1 / -1 sets *bad (null: checked already)
// Against a byte per neighbour and replica from global memory the rows are read
// once per 32 replicas. Torus, N = 10000, R = 32768: initial spins, fields and
// energies took 1320 us, spins and energies alone (the multi-spin-coded layouts
// read no fields) take 287 us; bound by the Philox calls.
inline size_t word_energy_smem(const GraphDev &g) { return ((size_t)g.np + 32 + 32) * 4; }

constexpr int WORDS_INIT = 0, WORDS_POP = 1, WORDS_RAW = 2;

template <bool WEIGHTED, bool BIG, int SRC>
__global__ void __launch_bounds__(256, 3) k_word_energy(GraphDev g, const int8_t *__restrict__ in,
                                                        const int32_t *__restrict__ pos, int8_t *__restrict__ rows,
                                                        int32_t *__restrict__ E, int32_t R, uint32_t key0,
                                                        uint32_t key1, int32_t *__restrict__ bad) {
    constexpr int N = 7, NT = 256;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *Wsm = reinterpret_cast<uint32_t *>(smem);             // [np]
    int32_t *Eacc = reinterpret_cast<int32_t *>(Wsm + g.np + 32);   // [32]; the 32 words before are read past a class
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const int slot0 = (int)blockIdx.x * 32;
    if (tid < 32) Eacc[tid] = 0;
    if (SRC == WORDS_RAW) {
        // Four positions a thread at a time, and of a ragged word only the
        // configurations that exist (the bits of the others stay 0, their energies
        // are not written). us of a call, against one position at a time and 32 loads
        // for it whatever R: n = 57,000, R = 1 403 -> 191, R = 33 608 -> 347; N = 7000,
        // R = 300 136 -> 113.
        const int live = min(32, R - slot0);
        bool wrong = false;
        for (int i0 = tid; i0 < g.n; i0 += 4 * NT) {
            uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll 8
            for (int r = 0; r < live; ++r) {
                const int8_t *x = in + (size_t)(slot0 + r) * g.n;
                const int b = msc_bit(r);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int v = i0 + j * NT < g.n ? __ldg(&x[i0 + j * NT]) : 1;
                    w[j] |= (uint32_t)(v == 1) << b;
                    wrong |= v != 1 && v != -1;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j * NT < g.n) Wsm[pos[i0 + j * NT]] = w[j];
        }
        if (wrong && bad) *bad = 1;
    } else {
        uint32_t *row = reinterpret_cast<uint32_t *>(rows) + (size_t)(slot0 + msc_lane_replica(lane)) * g.nbw;
        for (int q = warp; 4 * q < g.nbw; q += NT / 32) {
            if (SRC == WORDS_POP) {
                msc_load_words(row, Wsm, g.np, q, lane);
                continue;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = 128 * q + 32 * j + lane;
                uint32_t w = 0u;
                if (p < g.n) {
                    const uint32_t vid = __ldg(&g.vid[p]);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint4 u = philox10(make_uint4(vid, (uint32_t)(slot0 >> 2) + i, 0u, TAG_INIT), key0, key1);
                        w |= ((u.x >> 31) | (u.y >> 31) << 8 | (u.z >> 31) << 16 | (u.w >> 31) << 24) << i;
                    }
                }
                if (p < g.np) Wsm[p] = w;
            }
            __syncwarp();
            msc_store_words(Wsm, row, g.np, q, lane);
        }
    }
    __syncthreads();
    uint32_t S[MscShape<N>::acc_planes];
#pragma unroll
    for (int b = 0; b < MscShape<N>::acc_planes; ++b) S[b] = 0u;
    int cnt = 0;
    const unsigned char *Wb = reinterpret_cast<const unsigned char *>(Wsm);
    const int nsl = g.csl[g.ncol];
    for (int k = warp; k < nsl; k += NT / 32) {
        const uint2 d = __ldg(&g.msl[k]);
        const bool live = !(__ldg(&g.mvd[32 * k + lane]) >> 31);
        const uint32_t x = Wsm[d.y + (uint32_t)lane], units = d.x >> 24;
        const uint32_t off = ((d.x & 0xFFFFFFu) * 32u + (uint32_t)lane) * (uint32_t)sizeof(MscUnit<BIG>);
        uint32_t A[N];
#pragma unroll
        for (int b = 0; b < N; ++b) A[b] = x;
        for (uint32_t u = 0; u < units; ++u) {
            uint32_t w[4];
            msc_unit_words<WEIGHTED>(Wb, msc_unit<BIG>(g.mcol, off, u), w);
            msc_step4x<N>(A, x, w);
        }
        uint32_t c = 0u;
#pragma unroll
        for (int b = 0; b < N; ++b) c = msc_fa(S[b], live ? A[b] ^ x : 0u, c);
#pragma unroll
        for (int b = N; b < MscShape<N>::acc_planes; ++b) c = msc_fa(S[b], c, 0u);
        if (++cnt == MscShape<N>::flush_items) {
            msc_flush_energy<N>(S, Eacc, lane);
            cnt = 0;
        }
    }
    if (cnt) msc_flush_energy<N>(S, Eacc, lane);   // adds twice the sums
    __syncthreads();
    if (tid < 32 && (SRC != WORDS_RAW || slot0 + tid < R)) E[slot0 + tid] = (int32_t)(((int64_t)g.m2 - Eacc[tid]) / 2);
}

template <bool W, bool BIG>
const void *word_energy_kernel(int src) {
    return src == WORDS_INIT  ? reinterpret_cast<const void *>(&k_word_energy<W, BIG, WORDS_INIT>)
           : src == WORDS_POP ? reinterpret_cast<const void *>(&k_word_energy<W, BIG, WORDS_POP>)
                              : reinterpret_cast<const void *>(&k_word_energy<W, BIG, WORDS_RAW>);
}

cudaError_t launch_word_energy(int src, GraphDev g, const int8_t *in, const int32_t *pos, int8_t *rows, int32_t *E,
                               int32_t R, int32_t words, uint32_t key0, uint32_t key1, int32_t *bad, cudaStream_t st) {
    // Unsigned graphs have 32-bit entries at every size.
    const void *fn = !g.wt ? word_energy_kernel<false, true>(src)
                     : g.mbig ? word_energy_kernel<true, true>(src) : word_energy_kernel<true, false>(src);
    const size_t smem = word_energy_smem(g);
    if (cudaError_t e = raise_smem(const_cast<void *>(fn), smem)) return e;
    void *args[] = {&g, &in, &pos, &rows, &E, &R, &key0, &key1, &bad};
    return cudaLaunchKernel(fn, dim3(words), dim3(256), args, smem, st);
}

template <bool W, bool BIG, bool CL>
void *msc_kernel(int mmax) {
    switch (msc_planes(mmax)) {
        case 3: return reinterpret_cast<void *>(&k_sweep_msc<3, W, BIG, CL>);
        case 4: return reinterpret_cast<void *>(&k_sweep_msc<4, W, BIG, CL>);
        case 5: return reinterpret_cast<void *>(&k_sweep_msc<5, W, BIG, CL>);
        case 6: return reinterpret_cast<void *>(&k_sweep_msc<6, W, BIG, CL>);
        default: return reinterpret_cast<void *>(&k_sweep_msc<7, W, BIG, CL>);
    }
}

template <bool W, bool BIG>
void *msc_kernel(int mmax, bool cluster) {
    return cluster ? msc_kernel<W, BIG, true>(mmax) : msc_kernel<W, BIG, false>(mmax);
}

template <int FB, bool W>
void *small_kernel(int threads) {
    return threads == 512 ? reinterpret_cast<void *>(&k_sweep_small<FB, W, 256>)
                          : reinterpret_cast<void *>(&k_sweep_small<FB, W, 128>);
}

template <bool W>
void *packed_kernel(int threads) {
    switch (threads) {
        // 64 registers a thread (at least 1024 threads per SM): the packed item
        // with its lane decisions spills at 40 registers.
        case 128: return reinterpret_cast<void *>(&k_sweep_packed<W, 128, 8>);
        case 256: return reinterpret_cast<void *>(&k_sweep_packed<W, 256, 4>);
        case 384: return reinterpret_cast<void *>(&k_sweep_packed<W, 384, 2>);
        case 512: return reinterpret_cast<void *>(&k_sweep_packed<W, 512, 2>);
        default: return reinterpret_cast<void *>(&k_sweep_packed<W, 1024, 1>);
    }
}

template <int G, int FB, bool W>
void *kernel_ptr(bool queued) {
    return queued ? reinterpret_cast<void *>(&k_sweep<G, FB, W, true>) : reinterpret_cast<void *>(&k_sweep<G, FB, W, false>);
}

void *select_kernel(int G, int fb, bool weighted, int threads, int mmax, bool big, bool small, bool queued) {
    if (fb == 1 || fb == 2) {
        if (!weighted) return msc_kernel<false, true>(mmax, fb == 2);   // 32-bit entries at every size
        return big ? msc_kernel<true, true>(mmax, fb == 2) : msc_kernel<true, false>(mmax, fb == 2);
    }
    if (small) {
        if (fb == 7) return weighted ? small_kernel<7, true>(threads) : small_kernel<7, false>(threads);
        return weighted ? small_kernel<16, true>(threads) : small_kernel<16, false>(threads);
    }
    if (fb == 7) return weighted ? packed_kernel<true>(threads) : packed_kernel<false>(threads);
    if (G == 1) {
        if (fb == 16) return weighted ? kernel_ptr<1, 16, true>(queued) : kernel_ptr<1, 16, false>(queued);
        return weighted ? kernel_ptr<1, 8, true>(queued) : kernel_ptr<1, 8, false>(queued);
    }
    if (fb == 16) return weighted ? kernel_ptr<2, 16, true>(queued) : kernel_ptr<2, 16, false>(queued);
    return weighted ? kernel_ptr<2, 8, true>(queued) : kernel_ptr<2, 8, false>(queued);
}

}  // namespace

size_t sweep_smem_bytes(const GraphDev &g, int G, int field_bits, int threads) {
    if (field_bits == 1 || field_bits == 2)   // multi-spin coded: 32 replicas per word (2: CTA pairs)
        return ((size_t)g.np + msc_reserved_words(g.mmax) + ((g.ncol + 1 + 3) & ~3)) * 4;
    if (field_bits == 7)
        return (size_t)(g.np + 32) * 4 + 256 * 4 + (size_t)((g.ncol + 1 + 3) & ~3) * 4 + 16 * 4 +
               (size_t)((((g.np + 31) / 32) + 3) & ~3) * 4 + (size_t)(threads / 32) * PK_QCAP * 8;
    const int HW = field_bits == 16 ? 2 : 1;
    return (size_t)g.np * G * 4 * (1 + HW) + (size_t)((g.mmax + 1 + 3) & ~3) * 4 +
           (size_t)((g.ncol + 1 + 3) & ~3) * 4 + (size_t)(8 * G + 8) * 4;
}

static size_t msc_fixed_bytes(const GraphDev &g) {
    return ((size_t)g.np + msc_table_words(g.mmax) + 72 + ((g.ncol + 1 + 3) & ~3)) * 4;
}

// Threads of an MSC block: 512 where an SM would otherwise hold too few warps, 256
// elsewhere and where a class has no more slices than eight warps. That is where
// the launch has at most one CTA for an SM (us per step of 4 sweeps with 256 / 512
// threads, 140 words of one CTA: G63-shaped 168 / 139, 100 x 100 torus 138 / 111,
// n = 2000 83 / 74; 32 words in clusters of four: 112 / 100, 99 / 58 (the torus
// with 8 slices per CTA 64 / 58), 18,000-vertex planar 137 / 120; five slices per
// class, n = 3000 and degree 48, 140 words: 213 / 216) and where shared memory
// holds at most two CTAs (140 x 140 torus, 18,000-vertex planar and n = 16,272 at
// 64 to 512 words: 1.03 to 1.34 times faster; one CTA, n = 30,000: 1.28). With
// three or four of 256 resident those win, the barrier after a class holds up
// fewer warps (G63-shaped 500 words 376 / 427, 2048 words 1264 / 1475).
static int msc_threads(const GraphDev &g, int ctas, int sms, int per_sm, int limit, bool clusters) {
    const size_t fixed = msc_fixed_bytes(g), entry = (size_t)msc_entry_words(g.mmax) * 4;
    auto fit = [&](int threads) { return (int)std::min<size_t>(1024 / threads, (size_t)per_sm / (fixed + 40 * entry * (threads / 32) + 1024)); };
    if (g.maxcls <= 256 || fixed + 40 * entry * 16 > (size_t)limit) return 256;
    const bool few = ctas <= sms || fit(256) <= (clusters ? 1 : 2);
    return few && fit(512) >= std::min(fit(256), (ctas + sms - 1) / sms) ? 512 : 256;
}

// CTAs per word of the cluster kernel: as many as the largest class keeps busy
// (eight warps each, rounded up) while each has an SM of its own. us per step of 4
// sweeps with 1 / 2 / 4 / 8 CTAs of 512 threads: G63-shaped (largest class 47
// slices) 14 words 138 / 120 / 99 / 98, 25 words 139 / 121 / 100 / 113, 70 words
// 139 / 121 / 126 / 220; torus N = 10000 (157) 14 words 110 / 79 / 57 / 48, 32
// words 111 / 79 / 58 / 72, 98 words 111 / 129 / 131 / -; 18,000-vertex planar
// (139) 14 words 223 / 160 / 119 / 101, 98 words 224 / 255 / 269 / -. One CTA is
// better where a class fits it: n = 2000, degree 12 (14), 14 words 74 / 85 / 87 /
// 92. With a word and more for each SM, pairs of 256 threads still even out the
// last wave where four fit an SM: torus N = 10000 170 words 207 / 183, G63-shaped
// 220 / 203.
int msc_cluster(const GraphDev &g, int words, int sms) {
    int dev = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const int resident = (int)std::min<size_t>(4, (size_t)per_sm / (sweep_smem_bytes(g, 8, 2, 256) + 1024));
    const int busy = (g.maxcls + 31) / 32 / 8;
    const int limit = words > sms && busy >= 5 ? std::min(13 * sms / 5, resident * sms) : sms;
    int c = 1;
    while (c < 8 && c < busy && 2 * c * words <= limit) c *= 2;
    return c;
}

// The int8/int16 kernels: blocks of the launch for each SM, and blocks of t threads
// and smem bytes that an SM holds (at least one).
static int int_blocks_per_sm(int R, int G, int sms) { return ((R + 4 * G - 1) / (4 * G) + sms - 1) / sms; }
static int int_resident(int t, size_t smem, int per_sm) {
    return std::max(1, std::min(1024 / t, (int)((size_t)per_sm / (smem + 1024))));
}

// Whether the int8/int16 kernels queue their accepted items: the block's lanes for
// each position of a class, times the neighbours of a row, from 96. Below that a
// thread is done with its own rows before the queue's barrier pays. us per step of 4
// sweeps without / with the queue (512 threads; that figure in brackets): 18,001-
// vertex planar 259 / 340 (5), n = 7000, degree 12 140 / 169 (8), n = 2000, degree 12
// 69 / 75 (28), n = 7000, degree 48 271 / 279 (70), n = 2000, degree 24 104 / 101 (80),
// n = 2000, degree 48 192 / 157 (233), n = 7000, degree 100 574 / 466 (234), n = 500,
// degree 250 874 / 375 (19,200); groups of 8 replicas, n = 2000, degree 48 189 / 189
// (117), n = 7000, degree 100 750 / 654 (117).
static bool row_queue_pays(const GraphDev &g, int G, int threads) {
    return (double)g.m2 * threads * g.ncol >= 96.0 * g.n * g.n * G;
}

cudaError_t sweep_configure(const GraphDev &g, int R, int G, int field_bits, int threads,
                            bool weighted, SweepConfig *cfg, int cluster, int whole_threads) {
    int dev = 0, sms = 0, occ = 0, limit = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const bool msc = field_bits == 1 || field_bits == 2, automatic = threads == 0;
    bool small = false;
    if (msc) {
        G = 8;
        if (field_bits == 2) {
            if (!cluster) cluster = msc_cluster(g, (R + 31) / 32, sms);
            if (cluster == 1) field_bits = 1;
        }
        threads = whole_threads ? whole_threads
                                : msc_threads(g, (R + 31) / 32 * (field_bits == 2 ? cluster : 1), sms, per_sm, limit, field_bits == 2);
    } else if (field_bits == 7) {
        G = 1;
        // Few blocks: more threads each, so that an SM has about 1024 whatever the
        // number of blocks (G63-shaped, us per step of 4 sweeps with 128 / 256 /
        // 512 / 1024 threads: 128 blocks 214 / 137 / 107 / 98, 256 blocks 214 /
        // 151 / 142 / 188, 475 blocks 269 / 230 / 274 / 363, 1024 blocks 376 / 448
        // / 456 / 632), and no more than the largest class can use.
        if (automatic) {
            const int per = ((R + 3) / 4 + sms - 1) / sms;
            threads = per <= 1 ? 1024 : per == 2 ? 512 : per <= 4 ? 256 : 128;
            while (threads > 128 && threads / 2 >= g.maxcls) threads /= 2;
        }
    } else if (automatic) {
        // 512 threads, and half as many as long as that saves a wave of blocks (an
        // SM holds 1024 threads of these kernels, and what its shared memory has
        // room for) and the classes leave many of the threads idle. us per step of 4
        // sweeps with 512 / 256 / 128 threads: int16, n = 300, degree 24, R = 5000
        // (9 blocks per SM) 334 / 205 / 146; int8, n = 2000, degree 6, 4 blocks per SM
        // 119 / 93 / 112, 9 blocks 251 / 206 / 179. Large classes and few blocks in
        // shared memory keep 512: int8, 18,001-vertex planar 265 / 444 / 808, int16,
        // N = 4900 torus (three fit, 4 per SM) 181 / 261 / 449.
        const int per = int_blocks_per_sm(R, G, sms);
        const size_t block = sweep_smem_bytes(g, G, field_bits, 0);
        auto waves = [&](int t) {
            const int res = int_resident(t, block, per_sm);
            return (per + res - 1) / res;
        };
        threads = 512;
        while (threads > 128 && waves(threads / 2) < waves(threads) && (size_t)g.n * G < (size_t)2 * threads * g.ncol) threads /= 2;
    }
    size_t smem = sweep_smem_bytes(g, G, field_bits, threads);
    if (msc) {
        // Tie queues: 64 entries per warp, 40 where 64 would cost a resident
        // block, and what the reserved words leave when the graph fills shared
        // memory.
        const size_t fixed = msc_fixed_bytes(g);
        const size_t per_entry = (size_t)(threads / 32) * msc_entry_words(g.mmax) * 4;
        auto resident = [&](int cap) { return std::min<size_t>(1024 / threads, (size_t)per_sm / (fixed + cap * per_entry + 1024)); };
        cfg->qcap = resident(64) < resident(40) ? 40 : 64;
        if (fixed + cfg->qcap * per_entry > (size_t)limit) cfg->qcap = (int)((smem - fixed) / per_entry);
        if (cfg->qcap < 1) return cudaErrorInvalidConfiguration;
        smem = fixed + cfg->qcap * per_entry;
    }
    cfg->small = false;
    if (!msc) {
        cfg->qcap = 0;
        // Every class within one round of the block, and blocks few enough: the
        // small-graph kernel.
        const int per = ((R + 3) / 4 + sms - 1) / sms, half = per <= 2 ? 256 : 128;
        const size_t need = 4 * (field_bits == 7 ? small_smem_words<7>(g.np, g.ncol, g.mmax, half)
                                                 : small_smem_words<16>(g.np, g.ncol, g.mmax, half));
        small = automatic && G == 1 && field_bits != 8 && g.packed_ok && per <= (field_bits == 7 ? 5 : 16) && g.maxcls <= half &&
                std::min(per, 2) * (need + 1024) <= (size_t)per_sm;
        if (small) {
            cfg->small = true;
            threads = 2 * half;
            smem = need;
        } else if (field_bits != 7 && row_queue_pays(g, G, threads)) {
            // int8/int16: the block's queue of accepted items, where shared memory
            // has room for it without costing a resident block (without it each
            // thread walks its own rows).
            const size_t with = smem + sweep_queue_bytes(threads);
            const int all = int_blocks_per_sm(R, G, sms);
            if (with <= (size_t)limit &&
                std::min(all, int_resident(threads, with, per_sm)) == std::min(all, int_resident(threads, smem, per_sm))) {
                smem = with;
                cfg->qcap = threads;
            }
        }
    }
    void *fn = select_kernel(G, field_bits, weighted, threads, g.mmax, g.mbig != 0, small, cfg->qcap != 0);
    if (cudaError_t e = raise_smem(fn, smem)) return e;
    const int nblk = (R + 4 * G - 1) / (4 * G);
    if (field_bits == 2) {
        // One cluster per word; the hardware schedules them as slots free up.
        cfg->cluster = cluster;
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(cfg->cluster * nblk);
        lc.blockDim = dim3(threads);
        lc.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cfg->cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        lc.attrs = at;
        lc.numAttrs = 1;
        int ncl = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&ncl, fn, &lc);
        if (e != cudaSuccess) return e;
        if (ncl < 1) return cudaErrorInvalidConfiguration;
        cfg->G = G;
        cfg->field_bits = field_bits;
        cfg->threads = threads;
        cfg->smem = smem;
        cfg->grid = cfg->cluster * nblk;
        return cudaSuccess;
    }
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    cfg->G = G;
    cfg->field_bits = field_bits;
    cfg->threads = threads;
    cfg->smem = smem;
    cfg->grid = nblk < occ * sms ? nblk : occ * sms;
    cfg->occ = occ;
    return cudaSuccess;
}

cudaError_t launch_sweep(const SweepConfig &cfg, const SweepArgs &a, cudaStream_t st, bool early) {
    void *fn = select_kernel(cfg.G, cfg.field_bits, a.g.wt != nullptr, cfg.threads, a.g.mmax, a.g.mbig != 0, cfg.small, cfg.qcap != 0);
    SweepArgs b = a;
    b.qcap = cfg.qcap;
    void *args[] = {&b};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cfg.grid);
    lc.blockDim = dim3(cfg.threads);
    lc.dynamicSmemBytes = cfg.smem;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    early_attribute(at[0]);
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cfg.cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    lc.attrs = early ? at : at + 1;
    lc.numAttrs = (early ? 1 : 0) + (cfg.field_bits == 2 ? 1 : 0);
    return cudaLaunchKernelExC(&lc, fn, args);
}

// SMs that hold a CTA of the resampling get none of the sweep's while others have
// room, so a sweep of at most q blocks per SM is spread as evenly as ever if the other
// SMs take it with q each, or have no room for more. Otherwise some SM runs q + 1
// (us per step of 2 sweeps on 152 SMs beside 8 CTAs, early / not: torus N = 4900 144
// words 42.9 / 44.8, 146 words 65.0 / 44.6, 288 words 71.2 / 72.8, 296 words 91.4 /
// 72.9, 430 words 94.0 / 96.1, 440 words 115.7 / 96.7, 608 words, all slots, 124.8 /
// 126.7; packed, 720 blocks 112.5 / 114.3, 740 blocks 127.4 / 114.2). Clusters need
// free SMs side by side (of four CTAs: 34 words 29.3 / 30.9, 36 words 37.7 / 31.0).
bool sweep_spreads_beside(const SweepConfig &cfg, int beside, int sms) {
    const bool clusters = cfg.field_bits == 2;
    const int q = (cfg.grid + sms - 1) / sms, taken = beside + (clusters ? 2 * cfg.cluster : 0);
    return (!clusters && cfg.occ == q) || cfg.grid <= q * (sms - taken);
}

bool word_energy_fits(const GraphDev &g) {
    int dev = 0, limit = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return g.mcol && word_energy_smem(g) <= (size_t)limit;
}

cudaError_t launch_init_words(const GraphDev &g, int8_t *spins, int32_t *E, int32_t Rpad, uint32_t key0, uint32_t key1,
                              cudaStream_t st) {
    return launch_word_energy(WORDS_INIT, g, nullptr, nullptr, spins, E, Rpad, Rpad / 32, key0, key1, nullptr, st);
}

cudaError_t launch_energy_words(const GraphDev &g, const int8_t *spins, int32_t *E, int32_t Rpad, cudaStream_t st) {
    return launch_word_energy(WORDS_POP, g, nullptr, nullptr, const_cast<int8_t *>(spins), E, Rpad, Rpad / 32, 0u, 0u, nullptr, st);
}

cudaError_t launch_energy_raw(const GraphDev &g, const int8_t *raw, const int32_t *pos, int32_t *E, int32_t R,
                              int32_t *bad, cudaStream_t st) {
    return launch_word_energy(WORDS_RAW, g, raw, pos, nullptr, E, R, (R + 31) / 32, 0u, 0u, bad, st);
}

}  // namespace pa
