// Device-side views of the GeMSLR hierarchy and the kernel entry points.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "zcomplex.cuh"

namespace gemslr {

constexpr int kCoupleRows = 256;    // tail rows per CTA in the E / W^T kernel
constexpr int kMaxRank = 160;       // k_eff upper bound in the correction kernels
constexpr int kReduceThreads = 256;
constexpr int kMaxCols = 160;     // Krylov columns per Gram-Schmidt pass (m + 1 <= kMaxCols)

// ---- factor stream of the single-system substitutions ------------------------------
// Every block's factors as a sequence of slices in wavefront (level-set) order,
// those of L before those of U; a slice holds independent rows of one wavefront,
// longest first.  Slices are packed into items; item g of a block is one bulk
// copy into ring slot g % slots, and is read by consumer g % consumers (slots is a
// multiple of consumers, so that a slot has one reader).
// Values are -t_ij (L) and -u_ij/u_ii (U), formed in FP64 and rounded once, so
// that a row is x_i = x_i d_i + sum_j v_ij x_j with d_i = 1 (L) or 1/u_ii (U);
// rows and columns are places in the block's vector, place_unit per row: byte offsets,
// or row numbers (FP64 and complex vectors in global memory).
//
// FP32: x_i = fma(x_i, d_i, a0 + a1), a0 the sum of the even entries and of
// those from 16 on, a1 that of the odd ones below 16, in order; one lane per row,
// slices of at most 32 rows.  {row, d}[rows], padded to 16 bytes, then
// row_bytes(np) per row: np pairs of entries (column, value), absent ones (0, 0).
// An item is a group of four slices of
// one factor, four int32 {rows - 1, offset in the high half}, then the slices; four
// consumer warps.  L's records end with the row's last pair; U's hold the pairs in
// reverse.  So the entries of the slice just before, the nearest columns, sit in
// the last kLatePairs pairs: a slice of one row at kNoRow separates slices that
// need more, and L from U, and fills a factor's last group.
// Levels with rows of more than 16 entries (np = kLongRows): records of 8 pairs for the
// first 16, four more int32 in the item's header {offset of the slice's rests, fours
// of entries in the longest << kRestQuads} (0: none) and, behind each slice's records,
// rest_bytes(quads) per row for its entries from 16 on, absent ones (kNoEntry, 0).
// They may come from the slice just before.
//
// FP64 and complex: four chains per row, a row's entry e in chain e % 4 (a lane;
// two in complex arithmetic); chain
// sums start from x_i in lane 0 and use two chains (entries 0, 2, 4, ... and 1,
// 3 of the lane); the row is (s0 + s1) + (s2 + s3).  A consumer is a set of four
// warps, a slice at most kLaneRows rows; slice k of the block belongs to consumer k %
// consumers, an item holds several slices of one consumer.  Slice header int32
// {rows - 1, distance to the next slice of the item (0: none), z, flags}; z =
// entries of the longest row.  Per lane (lane_bytes): VT v[np], int32 c[np], int32
// row (absent: 0, 0); then {VT v, int32 c, pad}[.][4 rows] for the lanes' entries
// from 4 on.  The products x_i / u_ii are formed for the whole block between L
// and U by kLaneScale slices (VT d[rows], z: first row; an item of its own).  The
// slices of an item have the same class.  kSync: the slice ends its wavefront;
// bits 24 and up: number of wavefronts that end in the other consumers' slices
// since this consumer's last one.
// Records are an odd number of 16-byte words, so that 16-byte shared loads of
// consecutive records touch every bank once.
constexpr int kStageBytes = 4096;               // batched substitutions: largest chunk
constexpr int kRingData = 64 * 1024;
constexpr int kMaxSlots = kRingData / kStageBytes;
constexpr int kRingBytes = kRingData + 2 * kMaxSlots * 8 + 64;   // ring + mbarriers + flags
constexpr int kItemHeader = 16;
template <typename VT> constexpr int kLaneRows = sizeof(VT) == 8 ? 32 : 16;   // rows per slice, FP64 and complex
constexpr int kMaxItemBytes = 16192;            // head and a slot for each of four consumers within kRingBytes
constexpr int kItemDepth = 16;                  // most slots per consumer
constexpr int kLatePairs = 3;
constexpr int kNoRow = -4, kNoEntry = -8;      // byte offsets of words of the StreamHead
constexpr int kLaneItemBytes = 8192;            // FP64: slices of a consumer are joined into items of about this size
constexpr int kLongRows = 16;
constexpr int kRestQuads = 16;
enum { kSync = 1 };
// class of a slice (flags >> kLaneShift & 7): longest row 1, 2, up to 4 entries, more, more than 16; scaling
enum { kLaneShift = 4, kLane1 = 0, kLane2, kLane4, kLaneFull, kLaneLong, kLaneScale };
template <typename VT> struct OneLaneRows { static constexpr bool value = false; };
template <> struct OneLaneRows<float> { static constexpr bool value = true; };
template <typename VT>
__host__ __device__ constexpr int64_t place_unit(bool smem) { return smem || OneLaneRows<VT>::value ? sizeof(VT) : 1; }
__host__ __device__ constexpr int odd16(int bytes) { return (((bytes + 15) / 16) | 1) * 16; }
__host__ __device__ constexpr int row_bytes(int np) { return odd16(16 * np); }
__host__ __device__ constexpr int rest_bytes(int quads) { return odd16(32 * quads); }
template <typename VT>
__host__ __device__ constexpr int lane_bytes(int kq) { return odd16(kq * ((int)sizeof(VT) + 4) + 4); }

// Start of a substitution CTA's shared memory: the ring's barriers and the flag
// that ends every wait of the CTA; the block's vector and the ring follow.
struct StreamHead {
    uint64_t full[4 * kItemDepth], empty[4 * kItemDepth];
    int abort_flag, pad;
    float no_entry, no_row;    // FP32: zero, for absent entries; the slot of slices without rows
};
static_assert(sizeof(StreamHead) % 16 == 0 && (int)sizeof(StreamHead) + 4 * kMaxItemBytes <= kRingBytes, "smallest ring");

struct StreamView {
    const unsigned char *data;
    const int64_t *off;        // items + 1 byte offsets into data
    const int32_t *blk_item;   // nblk + 1 item range of every block
    const int32_t *split;      // nblk: items of L (FP32), slices with kSync (FP64)
    int32_t np;                // pairs per row record (FP32), entries per lane record (FP64)
    int32_t consumers;         // FP32: 4; FP64: 2 or 4
    int32_t slots, slot_bytes; // the ring
    int32_t variant;           // FP32: compute warps of a CTA, 8 or 4; FP64: consumers
};

// ---- chunks of the batched substitutions --------------------------------------------
// Per block the L chunks in wavefront order, then the U chunks.  A chunk holds
// independent rows of one wavefront and is one contiguous, 16-byte aligned byte
// range of at most kStageBytes bytes:
//   int32 {nrows, S, upper, 0}        S = entry slots per row
//   int32 rows[pad4(nrows)]           block-local row of every slot
//   int32 lens[pad4(nrows)]           entries of every slot
//   int32 cols[pad4(S*nrows)]         block-local columns, entry q of slot t at q*nrows + t
//   float vals[pad4(S*nrows)]         as in the stream above
//   float dinv[pad4(nrows)]           U chunks: 1/u_ii
// Chunk k of a block is one bulk copy into ring slot k % kMaxSlots.
struct ChunkView {
    const unsigned char *data;
    const int64_t *off;        // nchunk + 1 byte offsets into data
    const int32_t *blk_chunk;  // nblk + 1 chunk range of every block
};

// Everything one Schur level (or the last level) needs on the device.
template <typename VT, typename WT>
struct LevelView {
    int64_t s, e;              // rows [s, e) of the multilevel order
    int64_t stail;             // n - e
    int32_t nblk;
    const int64_t *blk_row;    // nblk + 1, level-local
    StreamView S;              // L and U of every block (see above)
    int32_t *err;              // device error word (1: a bounded wait expired)
    const int64_t *F_rp;       // d rows
    const int32_t *F_ci;       // global column (>= e)
    const VT *F_v;
    const int32_t *F_rows;     // level-local rows with F entries, ascending (so grouped by block)
    const int32_t *F_blk;      // nblk + 1 ranges of every block's rows in F_rows
    const int64_t *E_rp;       // stail rows
    const int32_t *E_ci;       // level-local column
    const VT *E_v;
    int32_t k;
    const WT *W;               // stail x k, column-major
    const VT *H;               // k x k, column-major
};

// The low-rank term W u of the previous level (Alg. 2 step 7: the right-hand
// side of level l+1 is z2 + W u), applied by the kernels that first read each
// row of that level's tail instead of by a separate pass: row g of the
// multilevel order takes sum_c W[g - row0 + c*ld] u[c].  W == nullptr: none.
template <typename VT, typename WT>
struct PendingLowRank {
    const WT *W = nullptr;
    const VT *u = nullptr;
    int64_t ld = 0, row0 = 0;
    int32_t k = 0;
};

// Control block of one FGMRES / Arnoldi step sequence (device memory).
struct KrylovCtl {
    int32_t j;            // current column
    int32_t m;            // restart length
    int32_t stop;         // cycle must end after this step
    int32_t reorth;       // current step needs the second Gram-Schmidt pass
    int32_t breakdown;
    int32_t nonfinite;
    int32_t nreorth;      // count of reorthogonalised steps
    int32_t givens;       // 1: FGMRES (update rotations), 0: Arnoldi
    int32_t force_reorth; // 1: always two passes (Arnoldi)
    int32_t iters;        // total inner iterations
    int32_t maxit;
    int32_t jdone;        // columns of the finished cycle
    double wnorm2;        // ||A z_j||^2 before orthogonalisation
    double beta;          // h_{j+1,j}
    double resid;         // |g_{j+1}|
    double tol_abs;       // rtol * ||b||
    double rnorm2;        // ||r||^2 (restart)
    int32_t restarts;     // completed cycles that did not converge
    int32_t converged;    // true residual met tol_abs
    double rnorm;         // ||b - A x|| after the last cycle
    double nu;            // delayed CGS2: norm of the reorthogonalised direction of this step
    double btil;          // delayed CGS2: lagged norm of the next direction
    double btil_prev;     // delayed CGS2: btil of the step before (row j of column j-1)
    double gam_pre;       // delayed CGS2: vt.vt of the current direction (formed beside M^{-1})
};

// Device buffers of FGMRES with delayed reorthogonalisation (one reduction
// per step): the unrotated Hessenberg matrix, the rotated one with its
// rotations and right-hand side, the triangular R relating the stored
// directions' preconditioned vectors to those of the final basis, and the
// per-step coefficient vectors.
struct DgsBufs {
    double *Hraw;          // (m+1) x m, column-major
    double *Hrot;          // (m+1) x m, column-major (least-squares factor)
    double *cs, *sn, *g;   // rotations and rotated right-hand side
    double *R;             // (m+1) x (m+1), column-major, upper triangular
    double *a;             // kMaxCols: V^T (direction) of this step
    double *apre;          // kMaxCols: the same, formed beside M^{-1} (k_dgs_fix_adots)
    double *coef;          // kMaxCols: projection coefficients of the next direction
    double *hprev;         // kMaxCols: first-pass column of the previous step
};

// Inner GMRES at the root level (Alg. 2 step 9): up to kMaxInner steps of
// right-preconditioned GMRES on S_hat_0 y2 = z2, S_hat_0 = C_0 - E_0 U^-1 L^-1 F_0
// (Sec. 2.4), preconditioned by the level-0 correction and the levels below.
constexpr int kMaxInner = 8;

struct InnerCtl {
    int32_t steps;         // Arnoldi steps taken (columns of H in use)
    int32_t done;          // 1: z2 = 0 or a happy breakdown ended the steps
    double beta;           // ||z2||
    double wn0;            // ||S_hat z_j|| before orthogonalisation (breakdown test)
    double h2[kMaxInner + 1];  // second-pass coefficients of the current step
    double c[kMaxInner];   // least-squares coefficients of y2 = sum_j c_j z_j
};

// Device state of the inner GMRES.  Vectors have the tail length m = n - e0
// (rows [e0, n) of the multilevel order).
template <typename VT>
struct InnerView {
    int64_t m;                 // n - e0
    int64_t e0;                // first tail row
    int32_t k;                 // steps per application (<= kMaxInner)
    const int64_t *rp;         // rows [e0, n) of A_hat: m + 1 offsets
    const int32_t *ci;         // global columns
    const VT *v;
    VT *V;                     // m x (k + 1), column-major: Arnoldi basis
    VT *Z;                     // m x k: preconditioned basis (M_S^-1 v_j)
    VT *w;                     // m
    double *H;                 // (kMaxInner + 1) x kMaxInner, column-major
    double *partial;           // grid x (kMaxInner + 2), column-major
    unsigned *counter;
    InnerCtl *ctl;
    int grid;                  // CTAs of the reduction kernels
};

}  // namespace gemslr
