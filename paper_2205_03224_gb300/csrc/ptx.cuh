// Device primitives shared by the kernels: warp reductions, deterministic
// column reductions of per-CTA partial sums, and the mbarrier / bulk-copy (TMA,
// non-tensor) PTX of the staged substitution kernels with the chunk ring of the
// batched ones.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "zcomplex.cuh"

namespace gemslr {
namespace {

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
    return v;
}


// Sum over the first `live` lanes (the others hold zeros), in the order of
// warp_sum without the stages that would add zeros: an FP64 addition holds its SM
// quarter for 64 cycles.  Valid in lane 0; live is uniform.
template <typename T>
__device__ __forceinline__ T warp_sum_of(T v, int live) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (live > o) v += shfl_xor(v, o);
    return v;
}

// Column sums of per-CTA partials (column-major: partial c of CTA p at
// c * nparts + p, so a warp's loads of one column are contiguous) into
// out[0..ncols1) (shared memory), by all warps of the finishing CTA.  Warp w
// takes columns w, w+nw, w+2nw, w+3nw together; its lanes load up to eight
// partials each for all four columns before any addition (one memory round
// trip per pass of 256 CTAs), add them in a fixed pairwise tree and finish
// with a warp reduction.  The summation order is fixed (deterministic); additions
// of absent partials are left out (one FP64 add takes on the order of a hundred
// cycles on this part when nothing else is in flight).
template <typename T>
__device__ void reduce_columns(const T *partial, int nparts, int ncols1, T *out) {
    constexpr int RP = 8, CW = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int cb = warp; cb < ncols1; cb += CW * nw) {
        T acc[CW];
#pragma unroll
        for (int u = 0; u < CW; ++u) acc[u] = 0;
        for (int p0 = 0; p0 < nparts; p0 += 32 * RP) {
            T v[CW][RP];
#pragma unroll
            for (int u = 0; u < CW; ++u) {
                const int c = cb + u * nw;
#pragma unroll
                for (int q = 0; q < RP; ++q) {
                    const int p = p0 + q * 32 + lane;
                    v[u][q] = (c < ncols1 && p < nparts) ? ldcg(partial + (int64_t)c * nparts + p) : (T)0;
                }
            }
            if (nparts <= 32) {
#pragma unroll
                for (int u = 0; u < CW; ++u) acc[u] = v[u][0];
            } else if (nparts <= 64) {
#pragma unroll
                for (int u = 0; u < CW; ++u) acc[u] = v[u][0] + v[u][1];
            } else if (nparts <= 128) {
#pragma unroll
                for (int u = 0; u < CW; ++u) acc[u] = (v[u][0] + v[u][1]) + (v[u][2] + v[u][3]);
            } else {
#pragma unroll
                for (int u = 0; u < CW; ++u)
                    acc[u] += ((v[u][0] + v[u][1]) + (v[u][2] + v[u][3])) + ((v[u][4] + v[u][5]) + (v[u][6] + v[u][7]));
            }
        }
#pragma unroll
        for (int u = 0; u < CW; ++u) {
            const int c = cb + u * nw;          // uniform over the warp
            if (c < ncols1) {
                const T t = warp_sum_of(acc[u], nparts);
                if (lane == 0) out[c] = t;
            }
        }
    }
    __syncthreads();
}

// ---- mbarrier / bulk-copy primitives (sm_90+ PTX) ------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Every wait is bounded: about 2 s of clock cycles (or `limit`), or until
// another warp of the CTA has raised `abort`.
constexpr long long kSpinCycles = 4000000000ll;

// Polling wait (no suspension) for the consumers' critical path, bounded like wait_bounded.
__device__ __forceinline__ bool poll_bounded(uint64_t *bar, unsigned parity, volatile int *abort_flag,
                                             long long limit = kSpinCycles) {
    if (mbar_test_wait(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned spins = 0;
    while (!mbar_test_wait(bar, parity)) {
        if ((++spins & 63u) == 0u) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit) return false;
        }
    }
    return true;
}
// The same for a whole warp, with one outcome for all of its lanes: each lane has
// its own clock and reads the abort flag at its own time, and lanes that went
// different ways would wait for each other in the next shuffle, __syncwarp or
// barrier for ever.
__device__ __forceinline__ bool poll_warp(uint64_t *bar, unsigned parity, volatile int *abort_flag,
                                          long long limit = kSpinCycles) {
    return __all_sync(0xffffffffu, poll_bounded(bar, parity, abort_flag, limit));
}
// One bulk copy global -> shared (16-byte aligned addresses, size a multiple of
// 16).  A sweep reads its factors once, and only a Schur level's up sweep, after all
// the levels below, reads the same ones again, so the copy marks them evict-first in
// L2: the vectors that the substitutions gather from (in global memory for blocks
// too large for shared memory) keep their L2 lines.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

__device__ __forceinline__ bool wait_bounded(uint64_t *bar, unsigned parity, volatile int *abort_flag,
                                             long long limit = kSpinCycles) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (abort_flag && *abort_flag) return false;
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

// Producer warp of the batched substitutions: streams the chunks [c0, c1)
// (byte ranges off[c] .. off[c+1] of data) into the ring: chunk c0 + g goes to
// slot g % kMaxSlots and completes on full[slot]; a slot is reused once its
// consumers have arrived on empty[slot].  The offsets are read 32 at a time by
// the whole warp (the next batch while the current one is issued), so that no
// copy waits on a global load of its own size; lane 0 issues the copies.  On an
// expired wait the CTA's abort flag and the device error word are set.
// Before returning, lane 0 waits for the copies still in flight.
__device__ __forceinline__ void produce_chunks(const unsigned char *data, const int64_t *off, int c0, int c1,
                                               unsigned char *ring, uint64_t *full, uint64_t *empty,
                                               volatile int *abort_flag, int32_t *err, int lane) {
    const int nchunk = c1 - c0;
    int issued = 0;
    int64_t o0 = 0, o1 = 0;
    if (lane < nchunk) {
        o0 = off[c0 + lane];
        o1 = off[c0 + lane + 1];
    }
    for (int base = 0; base < nchunk; base += 32) {
        int64_t n0 = 0, n1 = 0;
        if (base + 32 + lane < nchunk) {
            n0 = off[c0 + base + 32 + lane];
            n1 = off[c0 + base + 33 + lane];
        }
        const int cnt = min(32, nchunk - base);
        bool ok = true;
        for (int t = 0; t < cnt; ++t) {
            const int64_t s0 = __shfl_sync(0xffffffffu, o0, t), s1 = __shfl_sync(0xffffffffu, o1, t);
            const int g = base + t, slot = g % kMaxSlots;
            if (g >= kMaxSlots) {
                const bool got = lane == 0 ? wait_bounded(&empty[slot], ((g / kMaxSlots) - 1) & 1, abort_flag) : true;
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) {
                        *abort_flag = 1;
                        atomicExch(err, 1);
                    }
                    ok = false;
                    break;
                }
            }
            if (lane == 0) {
                const unsigned bytes = (unsigned)(s1 - s0);
                mbar_expect_tx(&full[slot], bytes);
                bulk_load(ring + (size_t)slot * kStageBytes, data + s0, bytes, &full[slot]);
            }
            issued = g + 1;
        }
        if (!ok) break;
        o0 = n0;
        o1 = n1;
    }
    if (lane == 0)
        for (int g = issued > kMaxSlots ? issued - kMaxSlots : 0; g < issued; ++g)
            wait_bounded(&full[g % kMaxSlots], (g / kMaxSlots) & 1, nullptr);
}

// Whether chunk k (block-relative) is in shared memory, by this lane's look.
__device__ __forceinline__ bool chunk_ready(uint64_t *full, int k) {
    return mbar_test_wait(&full[k % kMaxSlots], (k / kMaxSlots) & 1);
}
// Wait until chunk k is in shared memory, unless it is known to be (ready: every lane
// has seen it), and return it (nullptr, in every lane: the wait expired).
__device__ __forceinline__ const unsigned char *wait_chunk(const unsigned char *ring, uint64_t *full,
                                                           volatile int *abort_flag, int k, bool ready) {
    const int slot = k % kMaxSlots;
    return ready || poll_warp(&full[slot], (k / kMaxSlots) & 1, abort_flag) ? ring + (size_t)slot * kStageBytes : nullptr;
}

}  // namespace
}  // namespace gemslr
