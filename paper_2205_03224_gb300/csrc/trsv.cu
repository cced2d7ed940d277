// Block substitutions of the single-system application for sm_103a (Alg. 2
// steps 2 and 10): x = U^-1 L^-1 b for every diagonal block of a level, one CTA
// per block, the block's vector in shared memory (in global memory for blocks
// that do not fit) and its factors streamed by bulk copies through a ring.
//
// What bounds these kernels is the chain of wavefronts, not bandwidth: a 64^3
// level-0 block has about 430 dependent wavefronts of about 17 rows per sweep.
// Measured on this part (cycles): shared-memory load 29, shared store to a
// load by another lane and one FMA 34, named barrier of 8 warps 28, an
// mbarrier test that succeeds 57, a flag in shared memory 150 one way; an FP64
// add, multiply or FMA holds its SM quarter for 64 whatever the active lanes.
// A warp issues one instruction every 2.5 to 3 cycles, so the chain also pays
// for every instruction on it: whatever does not depend on the wavefront before
// (headers, rows, entries, older x) is read ahead by other warps.
// The order of every row's sum is fixed by the layout (kernels.cuh).
#include <type_traits>

#include "device.h"
#include "lowrank.cuh"
#include "stream.cuh"

namespace gemslr {
namespace {

// The sum of a row's two chains, never contracted with a product in front of it:
// with few entries a compiler would, and the result would depend on the variant.
__device__ __forceinline__ float sum_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double sum_rn(double a, double b) { return __dadd_rn(a, b); }

// A product in the rounding of LaneMath.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ zc mul_rn(zc a, zc b) {
    return zc(__fma_rn(a.re, b.re, -__dmul_rn(a.im, b.im)), __fma_rn(a.im, b.re, __dmul_rn(a.re, b.im)));
}

// ---- FP32 rows -----------------------------------------------------------------------
// A row in registers: place of x_i, d_i, and NP pairs of entries (place of x_j,
// value).
template <int NP>
struct RowF32 {
    int row;
    float dinv;
    int4 e[NP];
};

// Row slot t of the slice of last + 1 rows at p; slots past the last repeat it
// (same sums, same store).
template <int NP>
__device__ __forceinline__ void fetch_f32(uint32_t p, int last, int t, RowF32<NP> &R) {
    t = min(t, last);
    const int2 ri = lds<int2>(p + 8 * t);
    const uint32_t q = p + ((8 * last + 23) & ~15) + row_bytes(NP) * t;
#pragma unroll
    for (int i = 0; i < NP; ++i) R.e[i] = lds<int4>(q + 16 * i);
    R.row = ri.x;
    R.dinv = __int_as_float(ri.y);
}

template <int P0, int P1, int NP, typename X>
__device__ __forceinline__ void gather_f32(const RowF32<NP> &R, const X &x, float *xv) {
#pragma unroll
    for (int i = P0; i < P1; ++i) {
        xv[2 * i] = x.load(R.e[i].x);
        xv[2 * i + 1] = x.load(R.e[i].z);
    }
}

// The row's sum over its pairs in order (DOWN: the record holds them in reverse);
// rest: what follows them in the sum of the even ones.
template <int NP, bool DOWN, typename Rest>
__device__ __forceinline__ float row_f32(const RowF32<NP> &R, const float *xv, float self, Rest rest) {
    float a0 = 0, a1 = 0;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const int i = DOWN ? NP - 1 - q : q;
        a0 += __int_as_float(R.e[i].y) * xv[2 * i];
        a1 += __int_as_float(R.e[i].w) * xv[2 * i + 1];
    }
    return fmaf(self, R.dinv, sum_rn(rest(a0), a1));
}

// A row's entries from 16 on (desc: see kernels.cuh), read from the staged item four
// at a time: while four are added the next four x are gathered and the four entries
// after them read; e: the first four, read ahead.  Bound by instructions, so absent
// entries are added like the others.
struct RestF32 {
    int4 e[2];
    uint32_t q;
    __device__ __forceinline__ void fetch(uint32_t item, int desc, int t) {
        q = item + (desc & ((1 << kRestQuads) - 1)) + rest_bytes(desc >> kRestQuads) * t;
        e[0] = lds<int4>(q);
        e[1] = lds<int4>(q + 16);
    }
    template <typename X>
    __device__ __forceinline__ float add(int desc, const X &x, float a) {
        int left = desc >> kRestQuads;
        if (left == 0) return a;
        const uint32_t end = q + 32 * (left - 1);
        float v[4], xv[4];
        auto gather = [&] {                         // x of the four in e, then the four after them
            v[0] = __int_as_float(e[0].y), v[1] = __int_as_float(e[0].w);
            v[2] = __int_as_float(e[1].y), v[3] = __int_as_float(e[1].w);
            xv[0] = x.load_entry(e[0].x), xv[1] = x.load_entry(e[0].z);
            xv[2] = x.load_entry(e[1].x), xv[3] = x.load_entry(e[1].z);
            q = min(q + 32, end);
            e[0] = lds<int4>(q);
            e[1] = lds<int4>(q + 16);
        };
        gather();
        for (; left > 1; --left) {
            const float v0[4] = {v[0], v[1], v[2], v[3]}, x0[4] = {xv[0], xv[1], xv[2], xv[3]};
            gather();
#pragma unroll
            for (int u = 0; u < 4; ++u) a = __fmaf_rn(v0[u], x0[u], a);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) a = __fmaf_rn(v[u], xv[u], a);
        return a;
    }
};

// Named barriers that pass the sweep from the warp of one group to the warp of
// the next (64 threads: one warp arrives, the other waits): kEarly + w tells
// warp w that everything but the last slice of the group before is stored,
// kFinal + w that the last one is too.
enum { kEarly = 2, kFinal = 6 };
__device__ __forceinline__ void await_turn(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void give_turn(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// Groups g, g + 4, ... below end of one factor, by one of four warps that take
// the groups in turn.  A warp holds its next group in registers before the sweep
// reaches it, so the chain of wavefronts waits for gathers, sums and stores only.
// Entries that come from the slice just before sit in the last kLatePairs pairs of
// a record; the others are gathered while that slice is still being summed, and
// for the group's first slice while the warp of the group before works on its
// last.  Nothing in a group's chain is conditional (a branch there costs as much
// as a gather): every group has four slices.  Every warp goes through the same
// sequence of turns whatever happens (an expired wait only skips the
// arithmetic), so that the sweep always comes to its end.
// LONG: rows of more than 16 entries.  What they have beyond their record stays in the
// ring until the group is done and is read there, after the slice before is stored;
// three records are held instead of four, so that nothing spills.  us per application,
// 64^3 mixed: 20 entries 283, 30 entries 611 (one warp walking such levels slice by
// slice 701 and 1178; chunks taken by four warps in turn, before the streams, 487 and
// 900); 80^3 in 8 blocks (vectors in global memory), 20 entries 4.30 ms (5.89, 4.65).
template <int NP, bool LONG, bool DOWN, typename X>
__device__ __forceinline__ void consume_groups(ItemWalk &W, const X &x, int warp, int lane, int &g, int end, bool &ok) {
    constexpr int LP = NP < kLatePairs ? NP : kLatePairs;
    const int nw = (warp + 1) % 4;
    for (; g < end; g += 4) {
        const uint32_t p = ok ? W.item() : 0;
        ok = p != 0;
        if (!ok) {
            await_turn(kEarly + warp);
            await_turn(kFinal + warp);
            give_turn(kEarly + nw);
            give_turn(kFinal + nw);
            continue;
        }
        constexpr int kHeld = LONG ? 3 : 4;     // records in registers
        RowF32<NP> R[kHeld];
        const int4 dx = lds<int4>(p);           // rows - 1 and (high half) place of every slice
        const int d[4] = {dx.x, dx.y, dx.z, dx.w};
#pragma unroll
        for (int s = 0; s < (LONG ? 2 : 4); ++s) fetch_f32(p + (d[s] >> 16), d[s] & 0xffff, lane, R[s]);
        int4 rx = make_int4(0, 0, 0, 0);        // LONG: where the rests are
        RestF32 rest[2];
        if constexpr (LONG) {
            rx = lds<int4>(p + kItemHeader);
            rest[0].fetch(p, rx.x, min(lane, d[0] & 0xffff));
        } else {
            W.next(lane);
        }
        float xv[2][2 * NP], self[2];
        await_turn(kEarly + warp);
        gather_f32<0, NP - LP>(R[0], x, xv[0]);
        self[0] = x.load(R[0].row);
        await_turn(kFinal + warp);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const RowF32<NP> &now = R[s % kHeld], &next = R[(s + 1) % kHeld];
            gather_f32<NP - LP, NP>(now, x, xv[s & 1]);
            if (s < 3) {
                gather_f32<0, NP - LP>(next, x, xv[(s + 1) & 1]);
                self[(s + 1) & 1] = x.load(next.row);
            }
            const int desc[4] = {rx.x, rx.y, rx.z, rx.w};
            if constexpr (LONG) {
                if (s < 2) fetch_f32(p + (d[s + 2] >> 16), d[s + 2] & 0xffff, lane, R[(s + 2) % kHeld]);
                if (s < 3) rest[(s + 1) & 1].fetch(p, desc[s + 1], min(lane, d[s + 1] & 0xffff));
            }
            x.store(now.row, row_f32<NP, DOWN>(now, xv[s & 1], self[s & 1], [&](float a) {
                        if constexpr (LONG) return rest[s & 1].add(desc[s], x, a);
                        else return a;
                    }));
            __syncwarp();
            if (s == 2) give_turn(kEarly + nw);
        }
        give_turn(kFinal + nw);
        if constexpr (LONG) W.next(lane);
    }
}

// ---- FP64 and complex: four lanes per row ----------------------------------------------
// A lane's share of a row in registers: its first KQ entries and the place of x_i.
template <typename VT, int KQ>
struct RowF64 {
    static constexpr int kV = (int)sizeof(VT) / 4, kUsed = (KQ * ((int)sizeof(VT) + 4) + 4 + 15) / 16;
    int w[4 * kUsed];
    __device__ __forceinline__ int col(int k) const { return w[kV * KQ + k]; }
    __device__ __forceinline__ int row() const { return w[(kV + 1) * KQ]; }
    __device__ __forceinline__ double val(int k) const { return __hiloint2double(w[kV * k + 1], w[kV * k]); }
    __device__ __forceinline__ double imag(int k) const { return __hiloint2double(w[kV * k + 3], w[kV * k + 2]); }
};

template <typename VT, int KQ>
__device__ __forceinline__ void fetch_f64(uint32_t p, int t, int sub, RowF64<VT, KQ> &R) {
    const uint32_t q = p + kItemHeader + lane_bytes<VT>(KQ) * (4 * t + sub);
#pragma unroll
    for (int i = 0; i < RowF64<VT, KQ>::kUsed; ++i) {
        const int4 v = lds<int4>(q + 16 * i);
        R.w[4 * i] = v.x;
        R.w[4 * i + 1] = v.y;
        R.w[4 * i + 2] = v.z;
        R.w[4 * i + 3] = v.w;
    }
}

// The barrier of all sets at the end of a wavefront, taken when on != 0 (a
// predicate, not a branch).
template <int NT>
__device__ __forceinline__ void wavefront_end(int on) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %0, 0;\n\t@p bar.sync 2, %1;\n\t}" ::"r"(on), "n"(NT) : "memory");
}

// One lane's arithmetic.  FP64: v x by one FMA into the sum.  Complex: a lane
// holds one component (im: the imaginary one) of its chain, v x rounded as
// fma(v_re, x_re, -(v_im x_im)) and fma(v_im, x_re, v_re x_im), then added, so
// that an entry costs a lane three FP64 instructions instead of six.
template <typename VT, int KQ>
struct LaneMath {
    const RowF64<VT, KQ> &R;
    bool im;
    __device__ __forceinline__ double product(double re, double imag, VT x) const {
        if constexpr (IsComplex<VT>::value) {
            const double m = __dmul_rn(im ? re : imag, x.im);
            return __fma_rn(im ? imag : re, x.re, im ? m : -m);
        } else {
            return __dmul_rn(re, x);
        }
    }
    __device__ __forceinline__ double mul(int k, VT x) const { return product(R.val(k), R.imag(k), x); }
    __device__ __forceinline__ double add(double a, double re, double imag, VT x) const {
        if constexpr (IsComplex<VT>::value) return __dadd_rn(a, product(re, imag, x));
        else return __fma_rn(re, x, a);
    }
    __device__ __forceinline__ double add(double a, int k, VT x) const { return add(a, R.val(k), R.imag(k), x); }
};

// The slices of one item, all of class C (see kernels.cuh), by the four warps of
// a set: four lanes per row, eight in complex arithmetic (two per chain lane).
// Nothing but the loop itself is conditional: row slots past the last repeat it
// without storing.
template <int C, int KQ, int NS, typename VT, typename X>
__device__ __forceinline__ void lane_slices(uint32_t p, const X &x, int warp, int lane, int &nsync) {
    constexpr int NT = 128 * NS, kParts = IsComplex<VT>::value ? 2 : 1;      // lanes per chain lane
    const int slot = (8 * (warp % 4) + (lane >> 2)) / kParts, sub = (lane / kParts) & 3, part = lane & (kParts - 1);
    RowF64<VT, KQ> A, B;
    int4 h = lds<int4>(p);
    fetch_f64(p, min(slot, h.x), sub, A);
    auto step = [&](const RowF64<VT, KQ> &R, RowF64<VT, KQ> &next) {
        const int t = min(slot, h.x), before = h.w >> 24, after = h.w & kSync;
        const uint32_t pn = p + h.y;
        const int4 hn = lds<int4>(pn);
#pragma unroll
        for (int k = 0; k < NS - 1; ++k) wavefront_end<NT>(before > k);
        nsync -= before + after;
        constexpr int kUse = C < kLaneFull ? 1 : KQ;
        VT xq[kUse];
#pragma unroll
        for (int k = 0; k < kUse; ++k) xq[k] = x.load(R.col(k));
        const double self = x.part(R.row(), part);
        const LaneMath<VT, KQ> M{R, part != 0};
        double a0 = M.add(sub == 0 ? self : 0.0, 0, xq[0]);
        if constexpr (C < kLaneFull) {
            if constexpr (C >= kLane2) a0 += shfl_xor(a0, kParts);
            if constexpr (C >= kLane4) a0 += shfl_xor(a0, 2 * kParts);
        } else {
            double a1 = M.mul(1, xq[1]);
            if constexpr (KQ > 3) a1 = M.add(a1, 3, xq[3]);
            if constexpr (KQ > 2) a0 = M.add(a0, 2, xq[2]);
            if constexpr (C == kLaneLong) {     // the rest of long rows, from the staged slice
                constexpr int kRest = ((int)sizeof(VT) + 4 + 15) / 16 * 16;
                const int n4 = 4 * (h.x + 1);
                uint32_t r = p + kItemHeader + lane_bytes<VT>(KQ) * n4 + kRest * (4 * t + sub);
                for (int k = 4; k < (h.z + 3) >> 2; ++k, r += kRest * n4)
                    a0 = M.add(a0, lds<double>(r), kParts > 1 ? lds<double>(r + 8) : 0.0, x.load(lds<int>(r + (uint32_t)sizeof(VT))));
            }
            a0 = sum_rn(a0, a1);
            a0 += shfl_xor(a0, kParts);
            a0 += shfl_xor(a0, 2 * kParts);
        }
        if (sub == 0 && slot == t) x.store_part(R.row(), part, a0);
        const bool more = h.y != 0;
        p = pn;
        h = hn;
        fetch_f64(p, min(slot, h.x), sub, next);    // before the barrier: in flight while the others come to it
        wavefront_end<NT>(after);
        return more;
    };
    while (step(A, B) && step(B, A)) {
    }
}

// NS sets of four warps take the slices in turn, so that a set has its next
// rows in registers when their wavefront is due and slices of one wavefront run
// side by side; a barrier of all sets ends every wavefront.  An FP64 instruction
// holds its SM quarter for 64 cycles whatever the active lanes, so a slice's
// rows are spread over one warp of each quarter and its instructions are fitted
// to its longest row (the slice's class; the parts of the sum that are empty are
// left out).  A warp whose wait expired executes the rest of the barriers (nsync in all).
template <int KQ, int NS, typename VT, typename X>
__device__ __forceinline__ void consume_lanes(ItemWalk &W, const X &x, int warp, int lane, int nitem, int nsync) {
    constexpr int NT = 128 * NS;
    for (int g = warp / 4; g < nitem; g += NS) {
        const uint32_t p = W.item();
        if (!p) break;
        const int4 h = lds<int4>(p);
        switch (h.w >> kLaneShift & 7) {
            case kLane1: lane_slices<kLane1, KQ, NS, VT>(p, x, warp, lane, nsync); break;
            case kLane2: lane_slices<kLane2, KQ, NS, VT>(p, x, warp, lane, nsync); break;
            case kLane4: lane_slices<kLane4, KQ, NS, VT>(p, x, warp, lane, nsync); break;
            case kLaneFull: if constexpr (KQ > 1) lane_slices<kLaneFull, KQ, NS, VT>(p, x, warp, lane, nsync); break;
            case kLaneLong: if constexpr (KQ > 3) lane_slices<kLaneLong, KQ, NS, VT>(p, x, warp, lane, nsync); break;
            default: {
                // rows z .. z + h.x of x times their 1 / u_ii: dense, every lane busy
                for (int k = h.w >> 24; k > 0; --k, --nsync) wavefront_end<NT>(1);
                for (int i = 32 * (warp % 4) + lane; i <= h.x; i += 128) {
                    const int a = x.place(h.z + i);
                    x.store(a, mul_rn(x.load(a), lds<VT>(p + kItemHeader + i * (int)sizeof(VT))));
                }
                wavefront_end<NT>(h.w & kSync);
                nsync -= h.w & kSync;
            }
        }
        W.next(lane);
    }
    for (; nsync > 0; --nsync) wavefront_end<NT>(1);
}

// Warps that form the right-hand side and store the result: those that walk the
// stream and, when they are few, others that only help with this (FP32: NS is their
// number, 8 or the four that walk).
template <typename VT>
__host__ __device__ constexpr int compute_warps(int ns) {
    return OneLaneRows<VT>::value ? ns : ns < 4 ? 8 : 4 * ns;
}

// MODE 0: right-hand side from `in` (FP64 user vector) or `work`; result in work.
// MODE 1: right-hand side F y2 (gathered from work's tail); work[rows] -= result.
// The last warp is the producer; the others form the right-hand side and store
// the result together, the first four (FP32) or the NS sets of four of them walk
// the stream.
template <typename VT, typename WT, int MODE, bool SMEM, int NP, int NS>
__global__ void __launch_bounds__(32 * (compute_warps<VT>(NS) + 1))
k_trsv(const LevelView<VT, WT> lv, const IoT<VT> *__restrict__ in, VT *__restrict__ work,
       IoT<VT> *__restrict__ out_final, VT *__restrict__ scratch, const PendingLowRank<VT, WT> pl, int ring_offset) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kWarps = compute_warps<VT>(NS), NC = 32 * kWarps;
    constexpr int kWalkers = OneLaneRows<VT>::value ? 4 : 4 * NS;
    StreamHead *H = reinterpret_cast<StreamHead *>(smem);
    constexpr int kHead = sizeof(StreamHead);
    VT *xs_smem = reinterpret_cast<VT *>(smem + kHead);

    const int b = blockIdx.x;
    const int64_t r0 = lv.blk_row[b];
    const int nr = (int)(lv.blk_row[b + 1] - r0);
    if (nr == 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *ring = smem + kHead + (SMEM ? ring_offset : 0);
    const int i0 = lv.S.blk_item[b], i1 = lv.S.blk_item[b + 1];
    if ((int)threadIdx.x < lv.S.slots) {        // a thread per slot: one after another, 64 slots take a microsecond
        mbar_init(&H->full[threadIdx.x], 1);
        mbar_init(&H->empty[threadIdx.x], OneLaneRows<VT>::value ? 1 : 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        H->abort_flag = 0;
        H->no_entry = 0.f;
    }
    __syncthreads();
    if (warp == kWarps) {                       // producer
        produce_items(lv.S, i0, i1, H, ring, lv.err, lane);
        return;
    }
    const int ct = threadIdx.x;
    VT *mine = work + lv.s + r0;
    VT *xs = SMEM ? xs_smem : (MODE == 1 ? scratch + r0 : mine);
    if (MODE == 1) {
        // right-hand side F y2: zero, then the (few) block rows with F entries,
        // one thread per row so that their index and value loads overlap
        for (int i = ct; i < nr; i += NC) xs[i] = (VT)0;
        compute_barrier<NC>();
        // four rows per thread at a time, each step's loads for all of them in
        // flight together (row ids, row extents, the first two entries, x)
        const int f1 = lv.F_blk[b + 1];
        for (int t0 = lv.F_blk[b] + ct; t0 < f1; t0 += 4 * NC) {
            int64_t g[4], pa[4], pb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = t0 + u * NC < f1 ? lv.F_rows[t0 + u * NC] : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                pa[u] = g[u] >= 0 ? lv.F_rp[g[u]] : 0;
                pb[u] = g[u] >= 0 ? lv.F_rp[g[u] + 1] : 0;
            }
            int32_t cc[4][2];
            VT vv[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const bool on = pa[u] + q < pb[u];
                    const int64_t pq = on ? pa[u] + q : pa[u];
                    cc[u][q] = g[u] >= 0 ? lv.F_ci[pq] : 0;
                    vv[u][q] = on ? lv.F_v[pq] : (VT)0;
                }
            VT xv[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < 2; ++q) xv[u][q] = g[u] >= 0 ? work[cc[u][q]] : (VT)0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (g[u] < 0) continue;
                VT acc = vv[u][0] * xv[u][0] + vv[u][1] * xv[u][1];
                for (int64_t p = pa[u] + 2; p < pb[u]; ++p) acc += lv.F_v[p] * work[lv.F_ci[p]];
                xs[g[u] - r0] = acc;
            }
        }
    } else if (pl.W) {
        // right-hand side z2 + W u of the previous level (MODE 0, never the first level)
        for (int i = ct; i < nr; i += NC) xs[i] = mine[i] + pending_row<VT, WT>(pl, lv.s + r0 + i);
    } else if (in || SMEM) {
        // eight independent loads in flight per thread
        const IoT<VT> *src_d = in ? in + lv.s + r0 : nullptr;
        for (int i0 = ct; i0 < nr; i0 += 8 * NC) {
            VT v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * NC;
                v[u] = i < nr ? (src_d ? (VT)src_d[i] : mine[i]) : (VT)0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (i0 + u * NC < nr) xs[i0 + u * NC] = v[u];
        }
    }
    compute_barrier<NC>();
    if (warp < kWalkers) {
        const BlockVec<VT, SMEM> x(xs);
        ItemWalk W(lv.S, H, ring, OneLaneRows<VT>::value ? warp : warp / 4);
        if constexpr (!OneLaneRows<VT>::value) consume_lanes<NP, NS, VT>(W, x, warp, lane, i1 - i0, lv.S.split[b]);
        else if (i1 > i0) {
            constexpr bool kLong = NP == kLongRows;
            constexpr int kPairs = kLong ? 8 : NP;
            const int ng = i1 - i0, nl = lv.S.split[b];
            int g = warp;
            bool ok = true;
            if (warp == 3) {                    // the first group's turn
                give_turn(kEarly);
                give_turn(kFinal);
            }
            consume_groups<kPairs, kLong, false>(W, x, warp, lane, g, nl, ok);
            consume_groups<kPairs, kLong, true>(W, x, warp, lane, g, ng, ok);
            if (warp == ng % 4) {               // and the last group's
                await_turn(kEarly + warp);
                await_turn(kFinal + warp);
            }
        }
    }
    compute_barrier<NC>();
    if (*(volatile int *)&H->abort_flag) {
        if (ct == 0) atomicExch(lv.err, 1);
        return;
    }
    for (int i = ct; i < nr; i += NC) {
        VT y = xs[i];
        if (MODE == 1) y = mine[i] - y;
        if (SMEM || MODE == 1) mine[i] = y;
        if (out_final) out_final[lv.s + r0 + i] = (IoT<VT>)y;
    }
}

// Calls f with the kernel instantiation of a level's variant (StreamView::np, variant).
template <typename VT, typename WT, int MODE, bool SMEM, typename Fn>
void with_trsv(int np, int ns, Fn f) {
    auto call = [&](auto n, auto c) {
        f(k_trsv<VT, WT, MODE, SMEM, decltype(n)::value, decltype(c)::value>, compute_warps<VT>(decltype(c)::value));
    };
    constexpr std::integral_constant<int, 1> i1;
    constexpr std::integral_constant<int, 2> i2;
    constexpr std::integral_constant<int, 3> i3;
    constexpr std::integral_constant<int, 4> i4;
    constexpr std::integral_constant<int, 5> i5;
    constexpr std::integral_constant<int, 8> i8;
    constexpr std::integral_constant<int, kLongRows> il;
    if constexpr (OneLaneRows<VT>::value) {
        auto either = [&](auto n) {
            if constexpr (SMEM) {
                if (ns == 4) return call(n, i4);
            }
            call(n, i8);
        };
        switch (np) {
            case 1: return either(i1);
            case 3: return either(i3);
            case 5: return either(i5);
            case 8: return either(i8);
            default: return either(il);
        }
    } else {
        auto either = [&](auto n) {
            if (ns == 4) call(n, i4);
            else call(n, i2);
        };
        switch (np) {
            case 1: return either(i1);
            case 2: return either(i2);
            case 3: return either(i3);
            default: return either(i4);
        }
    }
}

}  // namespace

// Entries per record (FP32: pairs of entries, FP64: entries of each of four lanes) by
// the level's longest row: every entry of a record is gathered and summed, so the
// sizes step with the chains' lengths; rows past the largest record read their rest
// from the staged item, at 283 us per 64^3 mixed application with 20 entries against
// 222 with 16.
int trsv_record(bool one_lane, int longest) {
    if (one_lane) return longest <= 2 ? 1 : longest <= 6 ? 3 : longest <= 10 ? 5 : longest <= 16 ? 8 : kLongRows;
    return longest <= 4 ? 1 : longest <= 8 ? 2 : longest <= 12 ? 3 : 4;
}
// Sets of four warps by the slices per wavefront: two where most wavefronts are one
// slice (every barrier is among fewer warps), four where slices of a wavefront can run
// side by side.  us per sweep with two / four sets: 240 x 240 563 / 668, 45 x 38 x 29
// level 0 87 / 97, 32 x 32 15.8 / 16.8; complex 48^3 level 1 73 / 67; 64^3 FP64 level
// 0 136 / 136 (the FP64 pipe).
int trsv_sets(double slices) { return slices > 1.5 ? 4 : 2; }

template <typename VT, typename WT>
void launch_trsv(const LevelView<VT, WT> &lv, int mode, int smem_rows, const IoT<VT> *in, VT *work,
                 IoT<VT> *out_final, VT *scratch, cudaStream_t st, const PendingLowRank<VT, WT> &pl) {
    if (lv.nblk == 0) return;
    const int ring_offset = (smem_rows * (int)sizeof(VT) + 15) & ~15;
    const size_t bytes = sizeof(StreamHead) + (size_t)ring_offset + (size_t)lv.S.slots * lv.S.slot_bytes;
    auto go = [&](auto kernel, int warps) {
        kernel<<<lv.nblk, 32 * (warps + 1), bytes, st>>>(lv, in, work, out_final, scratch, pl, ring_offset);
    };
    if (smem_rows > 0) {
        if (mode == 0) with_trsv<VT, WT, 0, true>(lv.S.np, lv.S.variant, go);
        else with_trsv<VT, WT, 1, true>(lv.S.np, lv.S.variant, go);
    } else {
        if (mode == 0) with_trsv<VT, WT, 0, false>(lv.S.np, lv.S.variant, go);
        else with_trsv<VT, WT, 1, false>(lv.S.np, lv.S.variant, go);
    }
    count_launch();
}

template <typename VT, typename WT>
void set_trsv_smem_limit(int bytes) {
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    auto in_smem = [&](auto k, int) { cudaFuncSetAttribute(k, attr, bytes); };
    // vectors in global memory: the rest of the SM's 228 KB is L1 for their gathers
    auto in_global = [&](auto k, int) {
        cudaFuncSetAttribute(k, attr, kRingBytes);
        cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100 * (kRingBytes + 1024) / (228 * 1024) + 1);
    };
    constexpr bool one = OneLaneRows<VT>::value;
    for (int longest : {1, 5, 9, 16, 17})
        for (bool first : {true, false}) {
            const int np = trsv_record(one, longest);
            const int ns = one ? (first ? 4 : 8) : trsv_sets(first ? 0.0 : 1e9);
            with_trsv<VT, WT, 0, true>(np, ns, in_smem);
            with_trsv<VT, WT, 1, true>(np, ns, in_smem);
            with_trsv<VT, WT, 0, false>(np, ns, in_global);
            with_trsv<VT, WT, 1, false>(np, ns, in_global);
        }
}

template void launch_trsv<double, double>(const LevelView<double, double> &, int, int, const double *, double *,
                                          double *, double *, cudaStream_t, const PendingLowRank<double, double> &);
template void launch_trsv<float, __nv_bfloat16>(const LevelView<float, __nv_bfloat16> &, int, int, const double *,
                                                float *, double *, float *, cudaStream_t,
                                                const PendingLowRank<float, __nv_bfloat16> &);
template void launch_trsv<zc, zc>(const LevelView<zc, zc> &, int, int, const zc *, zc *, zc *, zc *, cudaStream_t,
                                  const PendingLowRank<zc, zc> &);
template void set_trsv_smem_limit<double, double>(int);
template void set_trsv_smem_limit<zc, zc>(int);
template void set_trsv_smem_limit<float, __nv_bfloat16>(int);

}  // namespace gemslr
