// The factor stream of the single-system substitutions: one bulk copy per item
// into a ring of slots in shared memory (layout in kernels.cuh).
#pragma once

#include "ptx.cuh"

namespace gemslr {
namespace {

// Named barrier 1 over the NC compute threads of a substitution CTA.
template <int NC>
__device__ __forceinline__ void compute_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(NC) : "memory");
}

// Producer warp: items [i0, i1) into the ring, item i0 + g to slot g % slots,
// completing on full[slot]; a slot is reused once its reader has arrived on
// empty[slot].  The offsets are read 32 at a time by the whole warp (the next
// batch while the current one is issued), so that no copy waits on a global load
// of its own size; lane 0 issues the copies.  On an expired wait the CTA's abort
// flag and the device error word are set.  Returns when no copy is in flight.
__device__ __forceinline__ void produce_items(const StreamView &S, int i0, int i1, StreamHead *H, unsigned char *ring,
                                              int32_t *err, int lane) {
    const int n = i1 - i0;
    volatile int *abort_flag = &H->abort_flag;
    int64_t o0 = 0, o1 = 0;
    if (lane < n) {
        o0 = S.off[i0 + lane];
        o1 = S.off[i0 + lane + 1];
    }
    int g = 0, slot = 0, round = 0;
    bool ok = true;
    for (int base = 0; ok && base < n; base += 32) {
        int64_t n0 = 0, n1 = 0;
        if (base + 32 + lane < n) {
            n0 = S.off[i0 + base + 32 + lane];
            n1 = S.off[i0 + base + 33 + lane];
        }
        const int cnt = min(32, n - base);
        for (int t = 0; t < cnt; ++t) {
            const int64_t s0 = __shfl_sync(0xffffffffu, o0, t), s1 = __shfl_sync(0xffffffffu, o1, t);
            if (round > 0) {
                const bool got = lane == 0 ? wait_bounded(&H->empty[slot], (unsigned)(round - 1) & 1u, abort_flag) : true;
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
                mbar_expect_tx(&H->full[slot], (unsigned)(s1 - s0));
                bulk_load(ring + (size_t)slot * S.slot_bytes, S.data + s0, (unsigned)(s1 - s0), &H->full[slot]);
            }
            ++g;
            if (++slot == S.slots) {
                slot = 0;
                ++round;
            }
        }
        o0 = n0;
        o1 = n1;
    }
    if (lane == 0)
        for (int q = g > S.slots ? g - S.slots : 0; q < g; ++q)
            wait_bounded(&H->full[q % S.slots], (unsigned)(q / S.slots) & 1u, nullptr);
}

// Loads from the ring by 32-bit shared-memory address.
template <typename T> __device__ __forceinline__ T lds(uint32_t a);
template <> __device__ __forceinline__ int lds<int>(uint32_t a) {
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ double lds<double>(uint32_t a) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ zc lds<zc>(uint32_t a) {
    zc v;
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ int2 lds<int2>(uint32_t a) {
    int2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ int4 lds<int4>(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
// The block's vector by the places of the stream: in shared memory (byte offsets;
// right behind the StreamHead: a constant address, so that a gather needs no
// addition) or in global memory (FP64 and complex: row numbers, multiplied by the
// element size in the address's 64-bit sum, so that a block may have any number of
// rows; FP32: byte offsets, which reach 2^29 rows and are 3 to 4% faster there).
// Places kNoRow and kNoEntry: words of the StreamHead.
template <typename VT, bool SMEM>
struct BlockVec;
template <typename VT>
struct BlockVec<VT, true> {
    __device__ explicit BlockVec(VT *) {}
    static __device__ __forceinline__ VT *vec() {
        extern __shared__ __align__(128) unsigned char smem[];
        return reinterpret_cast<VT *>(smem + sizeof(StreamHead));
    }
    static __device__ __forceinline__ int place(int row) { return row * (int)sizeof(VT); }
    __device__ __forceinline__ VT load(int at) const {
        return *reinterpret_cast<const VT *>(reinterpret_cast<const unsigned char *>(vec()) + at);
    }
    __device__ __forceinline__ VT load_entry(int at) const { return load(at); }
    __device__ __forceinline__ void store(int at, VT v) const {
        *reinterpret_cast<VT *>(reinterpret_cast<unsigned char *>(vec()) + at) = v;
    }
    // component `part` of an FP64 or complex entry
    __device__ __forceinline__ double part(int at, int part) const {
        return *reinterpret_cast<const double *>(reinterpret_cast<const unsigned char *>(vec()) + at + 8 * part);
    }
    __device__ __forceinline__ void store_part(int at, int part, double v) const {
        *reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(vec()) + at + 8 * part) = v;
    }
};
template <typename VT>
struct BlockVec<VT, false> {
    VT *base;
    __device__ explicit BlockVec(VT *x) : base(x) {}
    static __device__ __forceinline__ int place(int row) { return row * (int)place_unit<VT>(false); }
    __device__ __forceinline__ VT *address(int at) const {
        if constexpr (place_unit<VT>(false) == 1) return base + at;
        else return reinterpret_cast<VT *>(reinterpret_cast<unsigned char *>(base) + at);
    }
    __device__ __forceinline__ VT load(int at) const { return *address(max(at, 0)); }
    // x at an entry's column, 0 at kNoEntry
    __device__ __forceinline__ VT load_entry(int at) const { return at >= 0 ? *address(at) : (VT)0; }
    __device__ __forceinline__ void store(int at, VT v) const {
        if (at >= 0) *address(at) = v;
    }
    __device__ __forceinline__ double part(int at, int part) const {
        return reinterpret_cast<const double *>(address(at))[part];
    }
    __device__ __forceinline__ void store_part(int at, int part, double v) const {
        reinterpret_cast<double *>(address(at))[part] = v;
    }
};

// A consumer warp's walk over items c, c + consumers, ... of a block.
struct ItemWalk {
    StreamHead *H;
    uint32_t ring;
    int slots, slot_bytes, step, slot;
    unsigned parity = 0;

    __device__ ItemWalk(const StreamView &S, StreamHead *h, const unsigned char *r, int consumer)
        : H(h), ring(smem_u32(r)), slots(S.slots), slot_bytes(S.slot_bytes), step(S.consumers), slot(consumer) {}
    // Shared address of the current item, once it has arrived (0, in every lane: the bounded wait expired).
    __device__ __forceinline__ uint32_t item() {
        if (!poll_warp(&H->full[slot], parity, &H->abort_flag)) {
            *(volatile int *)&H->abort_flag = 1;
            return 0;
        }
        return ring + slot * slot_bytes;
    }
    // Every lane has finished with the item: its slot is free; on to the next.
    __device__ __forceinline__ void next(int lane) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&H->empty[slot]);
        slot += step;
        if (slot >= slots) {
            slot -= slots;
            parity ^= 1u;
        }
    }
};
}  // namespace
}  // namespace gemslr
