// Device layout of the GeMSLR hierarchy and the application of M^{-1} (Alg. 2).
#include <algorithm>
#include <complex>
#include <atomic>
#include <cstring>
#include <mutex>

#include "device.h"

namespace gemslr {

void cuda_check(cudaError_t e, const char *what) {
    if (e != cudaSuccess) fail(GEMSLR_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// ---- instrumentation ---------------------------------------------------------
namespace {
struct ProfEntry { std::string name; cudaEvent_t a, b; };
struct ProfStat { double ms = 0.0; int64_t count = 0; };
std::atomic<uint64_t> g_launches{0};
std::mutex g_prof_mu;
bool g_prof_on = false;
std::vector<ProfEntry> g_prof_pending;
std::vector<std::pair<cudaEvent_t, cudaEvent_t>> g_prof_pool;
std::vector<std::pair<std::string, ProfStat>> g_prof_stats;
}  // namespace

void count_launch(int n) { g_launches += (uint64_t)n; }

bool profile_enabled() { return g_prof_on; }

ProfScope::ProfScope(const char *name, cudaStream_t s) : slot(-1), st(s) {
    if (!g_prof_on) return;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return;
    std::lock_guard<std::mutex> lk(g_prof_mu);
    std::pair<cudaEvent_t, cudaEvent_t> ev;
    if (!g_prof_pool.empty()) { ev = g_prof_pool.back(); g_prof_pool.pop_back(); }
    else { cudaEventCreate(&ev.first); cudaEventCreate(&ev.second); }
    cudaEventRecord(ev.first, st);
    g_prof_pending.push_back({name, ev.first, ev.second});
    slot = (int)g_prof_pending.size() - 1;
}

ProfScope::~ProfScope() {
    if (slot < 0) return;
    std::lock_guard<std::mutex> lk(g_prof_mu);
    cudaEventRecord(g_prof_pending[slot].b, st);
}

void profile_enable(bool on) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof_on = on;
}

// Synchronise the recorded events and fold them into the per-name totals.
void profile_collect() {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    for (auto &e : g_prof_pending) {
        cudaEventSynchronize(e.b);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e.a, e.b);
        auto it = std::find_if(g_prof_stats.begin(), g_prof_stats.end(),
                               [&](const std::pair<std::string, ProfStat> &p) { return p.first == e.name; });
        if (it == g_prof_stats.end()) { g_prof_stats.push_back({e.name, ProfStat()}); it = g_prof_stats.end() - 1; }
        it->second.ms += ms;
        it->second.count += 1;
        g_prof_pool.push_back({e.a, e.b});
    }
    g_prof_pending.clear();
}

void profile_reset() {
    profile_collect();
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof_stats.clear();
}

int profile_read(char *names, size_t len, double *ms, int64_t *counts, int maxn) {
    profile_collect();
    std::lock_guard<std::mutex> lk(g_prof_mu);
    std::string all;
    int k = 0;
    for (auto &p : g_prof_stats) {
        if (k < maxn) {
            if (ms) ms[k] = p.second.ms;
            if (counts) counts[k] = p.second.count;
        }
        all += p.first;
        all += '\n';
        ++k;
    }
    if (names && len) {
        const size_t c = std::min(len - 1, all.size());
        std::memcpy(names, all.data(), c);
        names[c] = 0;
    }
    return k;
}

uint64_t launches_total() { return g_launches.load(); }

Arena::~Arena() {
    // cudaFree waits for the device; a caller's allocator may hand the memory
    // out again at once, so the handle's work must be finished first
    if (free_fn_ && !ptrs_.empty()) cudaDeviceSynchronize();
    for (void *p : ptrs_) {
        if (free_fn_) free_fn_(p, ctx_);
        else cudaFree(p);
    }
}

void *Arena::alloc(size_t bytes) {
    void *p = nullptr;
    const size_t b = bytes ? (bytes + 255) & ~size_t(255) : 256;
    if (alloc_fn_) {
        p = alloc_fn_(b, ctx_);
        if (!p) fail(GEMSLR_ERR_NOMEM, "device allocation of " + std::to_string(b) + " bytes failed (caller's allocator)");
        if (reinterpret_cast<uintptr_t>(p) % 256 != 0) {
            free_fn_(p, ctx_);
            fail(GEMSLR_ERR_ARG, "caller's allocator returned a pointer not aligned to 256 bytes");
        }
    } else if (cudaMalloc(&p, b) != cudaSuccess) {
        cudaGetLastError();
        fail(GEMSLR_ERR_NOMEM, "device allocation of " + std::to_string(b) + " bytes failed");
    }
    ptrs_.push_back(p);
    total_ += b;
    return p;
}

namespace {


// Every entry must lie in its row's diagonal block, strictly below (L) or on
// and above (U) the diagonal, and U needs a nonzero diagonal: the kernels
// index the block's shared-memory vector with these columns.
void validate_tri(const Csr &T, const std::vector<int64_t> &bp, bool upper) {
    if (T.nrows != bp.back()) fail(GEMSLR_ERR_ARG, "factor rows do not match the level");
    for (size_t b = 0; b + 1 < bp.size(); ++b)
        for (int64_t i = bp[b]; i < bp[b + 1]; ++i) {
            bool diag = false;
            for (int64_t p = T.rp[i]; p < T.rp[i + 1]; ++p) {
                const int64_t c = T.ci[p];
                if (c < bp[b] || c >= bp[b + 1]) fail(GEMSLR_ERR_ARG, "factor entry outside its diagonal block");
                if (!upper && c >= i) fail(GEMSLR_ERR_ARG, "L must be strictly lower triangular");
                if (upper && c < i) fail(GEMSLR_ERR_ARG, "U must be upper triangular");
                if (upper && c == i) diag = T.v[p] != 0.0 || (!T.vi.empty() && T.vi[p] != 0.0);
            }
            if (upper && !diag) fail(GEMSLR_ERR_ARG, "U needs a nonzero diagonal");
        }
}

size_t pad16(size_t x) { return (x + 15) & ~size_t(15); }

// Entry p of a factor (and the reciprocal of a diagonal entry) in the value
// type of the substitution; complex factors keep their imaginary parts in vi.
template <typename VT> VT entry_at(const Csr &T, int64_t p) { return cast_to<VT>(T.v[p]); }
template <> zc entry_at<zc>(const Csr &T, int64_t p) { return zc(T.v[p], T.vi.empty() ? 0.0 : T.vi[p]); }
template <typename VT> VT inv_entry(const Csr &T, int64_t p) { return cast_to<VT>(1.0 / T.v[p]); }
template <> zc inv_entry<zc>(const Csr &T, int64_t p) {
    const std::complex<double> r = 1.0 / std::complex<double>(T.v[p], T.vi.empty() ? 0.0 : T.vi[p]);
    return zc(r.real(), r.imag());
}
// The stored value of an off-diagonal entry: -t_ij (L, pdiag < 0) or
// -u_ij / u_ii (U, u_ii at pdiag), formed in FP64 and rounded once.
template <typename VT> VT stored_entry(const Csr &T, int64_t p, int64_t pdiag) {
    return cast_to<VT>(pdiag < 0 ? -T.v[p] : -(T.v[p] * (1.0 / T.v[pdiag])));
}
template <> zc stored_entry<zc>(const Csr &T, int64_t p, int64_t pdiag) {
    const zc v = entry_at<zc>(T, p);
    return pdiag < 0 ? -v : -(v * inv_entry<zc>(T, pdiag));
}

}  // namespace

namespace {

// Rows [r0, r1) of one triangular factor in wavefront order: row ids, longest
// first inside a wavefront (equal lengths in order), the wavefronts' ranges,
// and every row's entries off the diagonal.
struct Waves {
    std::vector<int64_t> rows, ptr;
    std::vector<int32_t> len;          // by block-local row
};

Waves order_rows(const Csr &T, int64_t r0, int64_t r1, bool upper) {
    const std::vector<int32_t> lev = upper ? wavefronts_upper(T, r0, r1) : wavefronts_lower(T, r0, r1);
    Waves w;
    int32_t nw = 0;
    for (int32_t x : lev) nw = std::max(nw, x + 1);
    w.ptr.assign(nw + 1, 0);
    for (int32_t x : lev) ++w.ptr[x + 1];
    for (int32_t q = 0; q < nw; ++q) w.ptr[q + 1] += w.ptr[q];
    w.rows.resize(r1 - r0);
    w.len.resize(r1 - r0);
    std::vector<int64_t> at(w.ptr.begin(), w.ptr.end() - 1);
    for (int64_t i = r0; i < r1; ++i) {
        int32_t c = 0;
        for (int64_t p = T.rp[i]; p < T.rp[i + 1]; ++p) c += (T.ci[p] != i);
        w.len[i - r0] = c;
        w.rows[at[lev[i - r0]]++] = i;
    }
    for (int32_t q = 0; q < nw; ++q)
        std::stable_sort(w.rows.begin() + w.ptr[q], w.rows.begin() + w.ptr[q + 1],
                         [&](int64_t x, int64_t y) { return w.len[x - r0] > w.len[y - r0]; });
    return w;
}

int64_t diagonal(const Csr &T, int64_t i) {
    int64_t pd = -1;
    for (int64_t p = T.rp[i]; p < T.rp[i + 1]; ++p)
        if (T.ci[p] == i) pd = p;
    return pd;
}

size_t chunk_bytes(int64_t nrows, int64_t maxlen, bool upper) {
    const size_t pr = (size_t)((nrows + 3) & ~int64_t(3)), ne = (size_t)(maxlen * nrows);
    return 16 + 8 * pr + 2 * pad16(ne * 4) + (upper ? pad16((size_t)nrows * 4) : 0);
}

// Append the chunks of one triangular factor of block [r0, r1) (see kernels.cuh).
void append_factor_chunks(const Csr &T, int64_t r0, int64_t r1, bool upper, ChunkHost &out, int max_rows) {
    const Waves W = order_rows(T, r0, r1, upper);
    for (size_t w = 0; w + 1 < W.ptr.size(); ++w) {
        const int64_t *R = W.rows.data() + W.ptr[w];
        const int64_t nR = W.ptr[w + 1] - W.ptr[w];
        if (!upper && W.len[R[0] - r0] == 0) continue;          // rows without L entries: x_i unchanged
        int64_t start = 0;
        while (start < nR) {
            const int64_t S = W.len[R[start] - r0];
            int64_t n = 0;
            while (start + n < nR && n < max_rows && chunk_bytes(n + 1, S, upper) <= (size_t)kStageBytes) ++n;
            if (n == 0) fail(GEMSLR_ERR_UNSUPPORTED, "a factor row has too many entries for the staged substitution");
            const size_t bytes = chunk_bytes(n, S, upper);
            const size_t base = out.data.size();
            out.data.resize(base + bytes, 0);
            int32_t *hdr = reinterpret_cast<int32_t *>(out.data.data() + base);
            hdr[0] = (int32_t)n;
            hdr[1] = (int32_t)S;
            hdr[2] = upper ? 1 : 0;
            const int64_t pr = (n + 3) & ~int64_t(3);
            int32_t *rr = hdr + 4, *ll = rr + pr, *cc = ll + pr;
            float *vv = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(cc) + pad16((size_t)(S * n) * 4));
            float *dd = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(vv) + pad16((size_t)(S * n) * 4));
            for (int64_t t = 0; t < n; ++t) {
                const int64_t i = R[start + t];
                rr[t] = (int32_t)(i - r0);
                ll[t] = W.len[i - r0];
                const int64_t pdiag = upper ? diagonal(T, i) : -1;
                if (upper) dd[t] = inv_entry<float>(T, pdiag);
                int64_t q = 0;
                for (int64_t pp = T.rp[i]; pp < T.rp[i + 1]; ++pp) {
                    if (T.ci[pp] == i) continue;
                    cc[q * n + t] = (int32_t)(T.ci[pp] - r0);
                    vv[q * n + t] = stored_entry<float>(T, pp, pdiag);
                    ++q;
                }
            }
            out.off.push_back((int64_t)out.data.size());
            start += n;
        }
    }
}

// ---- factor stream (layout in kernels.cuh) ---------------------------------------------
// A row with more entries than this is refused (the bound of a 4 KB stage for
// FP64 values, of 8 KB for FP32 and complex ones).
template <typename VT>
bool row_too_long(int64_t len, bool upper) {
    const int64_t slots = OneLaneRows<VT>::value ? len : 4 * ((len + 3) / 4);
    const size_t limit = sizeof(VT) == 8 ? 4096 : 8192;
    return 16 + 32 + pad16((size_t)slots * 4) + pad16((size_t)slots * sizeof(VT)) + (upper ? pad16(sizeof(VT)) : 0) >
           limit;
}

// A zeroed item of `bytes` bytes, appended; returns its offset in out.data.
size_t add_item(StreamHost &out, size_t bytes) {
    const size_t at = out.data.size();
    bytes = pad16(bytes);
    if (bytes > (size_t)kMaxItemBytes) fail(GEMSLR_ERR_ARG, "factor stream item too large");
    out.data.resize(at + bytes, 0);
    out.off.push_back((int64_t)out.data.size());
    out.slot_bytes = std::max(out.slot_bytes, (int)bytes);
    return at;
}

// Slices of one factor in wavefront order, longest rows first, of at most max_rows rows.
struct SliceRows {
    const int64_t *rows;
    int64_t n, longest;
    bool sync;                         // ends its wavefront
};

template <typename VT>
std::vector<SliceRows> cut_slices(const Waves &W, int64_t r0, bool upper, int64_t max_rows) {
    std::vector<SliceRows> out;
    for (size_t q = 0; q + 1 < W.ptr.size(); ++q) {
        const int64_t *R = W.rows.data() + W.ptr[q];
        int64_t nR = W.ptr[q + 1] - W.ptr[q];
        // rows with nothing off the diagonal: x_i unchanged (L), or only multiplied
        // by 1/u_ii (U: by the scaling items, in FP32 by the row itself)
        if (!(OneLaneRows<VT>::value && upper))
            while (nR > 0 && W.len[R[nR - 1] - r0] == 0) --nR;
        for (int64_t at = 0; at < nR; at += max_rows) {
            const int64_t longest = W.len[R[at] - r0];
            if (row_too_long<VT>(longest, upper))
                fail(GEMSLR_ERR_UNSUPPORTED, "a factor row has too many entries for the staged substitution");
            out.push_back({R + at, std::min(max_rows, nR - at), longest, at + max_rows >= nR});
        }
    }
    return out;
}

struct EntryF32 { int32_t col; float v; };

// FP32 row i into its record of np pairs: pair p at slot(p), entries from 16 on to rest.
template <typename Slot>
void put_row_f32(const Csr &T, int64_t r0, int64_t i, bool upper, int64_t unit, EntryF32 *rec, Slot slot, EntryF32 *rest) {
    const int64_t pdiag = upper ? diagonal(T, i) : -1;
    int64_t e = 0;
    for (int64_t p = T.rp[i]; p < T.rp[i + 1]; ++p) {
        if (T.ci[p] == i) continue;
        const EntryF32 en{vector_place(T.ci[p] - r0, unit), stored_entry<float>(T, p, pdiag)};
        if (e < 16) rec[2 * slot(e / 2) + e % 2] = en;
        else rest[e - 16] = en;
        ++e;
    }
}
EntryF32 row_head_f32(const Csr &T, int64_t r0, int64_t i, bool upper, int64_t unit) {
    return {vector_place(i - r0, unit), upper ? inv_entry<float>(T, diagonal(T, i)) : 1.f};
}

// FP32: rows to their heads and records of np pairs, entries from 16 on to their rests.
void put_rows_f32(const Csr &T, int64_t r0, const Waves &W, bool upper, const int64_t *rows, int64_t n, int np,
                  int64_t unit, unsigned char *p, unsigned char *rest, size_t rest_bytes) {
    EntryF32 *head = reinterpret_cast<EntryF32 *>(p);
    unsigned char *recs = p + pad16((size_t)(8 * n));
    for (int64_t t = 0; t < n; ++t) {
        const int64_t i = rows[t], shift = np - (std::min<int64_t>(16, W.len[i - r0]) + 1) / 2;
        head[t] = row_head_f32(T, r0, i, upper, unit);
        put_row_f32(T, r0, i, upper, unit, reinterpret_cast<EntryF32 *>(recs + row_bytes(np) * t),
                    [&](int64_t pr) { return upper ? np - 1 - pr : pr + shift; },
                    reinterpret_cast<EntryF32 *>(rest + rest_bytes * t));
    }
}

// Slices of FP32 rows, cut further where their entries from 16 on would fill more than a
// third of an item.
struct SliceF32 {
    const int64_t *rows;
    int64_t n, quads = 0;              // rows; fours of entries from 16 on
    size_t bytes(int np) const { return pad16((size_t)(8 * n)) + (size_t)(row_bytes(np) * n); }
    size_t rests() const { return quads ? (size_t)(rest_bytes((int)quads) * n) : 0; }
};
std::vector<SliceF32> cut_f32(const Waves &W, int64_t r0, bool upper, int np, bool longer) {
    std::vector<SliceF32> out;
    for (const SliceRows &s : cut_slices<float>(W, r0, upper, np == 8 ? 24 : 32))      // four fit kMaxItemBytes
        for (int64_t at = 0; at < s.n; at += out.back().n) {
            SliceF32 c{s.rows + at, s.n - at};
            if (longer) {
                const int64_t longest = W.len[s.rows[at] - r0];
                c.quads = std::max<int64_t>(0, longest - 16 + 3) / 4;
                while (c.n > 1 && c.bytes(np) + c.rests() > (size_t)kMaxItemBytes / 3 - 64) --c.n;
            }
            out.push_back(c);
        }
    return out;
}

// FP32: groups of four slices of one factor (see kernels.cuh).
void append_groups(const Csr &T, int64_t r0, const Waves &W, bool upper, StreamHost &out) {
    const bool longer = out.np == kLongRows;
    const int np = longer ? 8 : out.np, header = longer ? 2 * kItemHeader : kItemHeader;
    const std::vector<SliceF32> sl = cut_f32(W, r0, upper, np, longer);
    // the sequence of slices; -1: without rows
    std::vector<int64_t> seq;
    std::vector<int32_t> slice_of(W.len.size(), -1);
    auto bytes = [&](int64_t k) { return k < 0 ? SliceF32{nullptr, 1}.bytes(np) : sl[k].bytes(np) + sl[k].rests(); };
    size_t total = header;             // of the last group
    auto push = [&](int64_t k) {
        if (seq.size() % 4 == 0) total = header;
        // a long row's slice that does not fit beside the others starts a group
        while (total + bytes(k) + (3 - seq.size() % 4) * bytes(-1) > (size_t)kMaxItemBytes && seq.size() % 4) {
            seq.push_back(-1);
            total = seq.size() % 4 ? total + bytes(-1) : header;
        }
        seq.push_back(k);
        total += bytes(k);
    };
    for (size_t k = 0; k < sl.size(); ++k) {
        int64_t late = 0;
        for (int64_t t = 0; k > 0 && t < sl[k].n; ++t) {
            const int64_t i = sl[k].rows[t], len = std::min<int64_t>(16, W.len[i - r0]);
            int64_t e = 0;
            for (int64_t p = T.rp[i]; p < T.rp[i + 1] && e < 16; ++p) {
                if (T.ci[p] == i) continue;
                if (slice_of[T.ci[p] - r0] == (int32_t)k - 1)
                    late = std::max(late, upper ? e / 2 + 1 : (len + 1) / 2 - e / 2);
                ++e;
            }
        }
        for (int64_t t = 0; t < sl[k].n; ++t) slice_of[sl[k].rows[t] - r0] = (int32_t)k;
        if (late > kLatePairs || (upper && k == 0)) push(-1);
        push((int64_t)k);
    }
    while (seq.size() % 4) seq.push_back(-1);
    for (size_t g = 0; g < seq.size(); g += 4) {
        size_t all = header;
        for (size_t q = g; q < g + 4; ++q) all += bytes(seq[q]);
        const size_t item = add_item(out, all);
        unsigned char *p = out.data.data() + item;
        int32_t *h = reinterpret_cast<int32_t *>(p);
        size_t off = header;
        for (size_t q = g; q < g + 4; ++q) {
            const int64_t k = seq[q];
            const SliceF32 c = k < 0 ? SliceF32{nullptr, 1} : sl[k];
            h[q - g] = (int32_t)(off << 16) | (int32_t)(c.n - 1);
            unsigned char *rest = p + off + c.bytes(np);
            if (c.quads) {
                h[4 + q - g] = (int32_t)(off + c.bytes(np)) | (int32_t)(c.quads << kRestQuads);
                for (size_t e = 0; e < c.rests() / sizeof(EntryF32); ++e) reinterpret_cast<EntryF32 *>(rest)[e] = {kNoEntry, 0.f};
            }
            if (k < 0) *reinterpret_cast<EntryF32 *>(p + off) = {kNoRow, 1.f};
            else put_rows_f32(T, r0, W, upper, c.rows, c.n, np, out.unit, p + off, rest, rest_bytes((int)c.quads));
            off += bytes(k);
        }
    }
}

// FP64 and complex slices of one block, back to back, before they are packed.
struct LaneSlices {
    std::vector<unsigned char> data;
    std::vector<size_t> off{0};
    unsigned char *add(size_t bytes, int64_t n, int64_t z, int flags) {
        const size_t at = data.size();
        data.resize(at + pad16(bytes), 0);
        off.push_back(data.size());
        int32_t *h = reinterpret_cast<int32_t *>(data.data() + at);
        h[0] = (int32_t)n - 1;
        h[2] = (int32_t)z;
        h[3] = flags;
        return data.data() + at + kItemHeader;
    }
};

template <typename VT>
void append_lanes(const Csr &T, int64_t r0, const Waves &W, bool upper, int np, int64_t unit, LaneSlices &out) {
    const size_t lb = lane_bytes<VT>(np), tb = pad16(sizeof(VT) + 4);
    auto bytes = [&](int64_t n, int64_t m) {
        return kItemHeader + (size_t)(4 * n) * (lb + (size_t)std::max<int64_t>(0, (m + 3) / 4 - 4) * tb);
    };
    for (const SliceRows &s : cut_slices<VT>(W, r0, upper, kLaneRows<VT>)) {
        for (int64_t at = 0; at < s.n;) {
            int64_t n = 1;
            while (at + n < s.n && bytes(n + 1, s.longest) <= (size_t)kMaxItemBytes) ++n;
            const int cls = s.longest <= 1 ? kLane1 : s.longest <= 2 ? kLane2 : s.longest <= 4 ? kLane4 : s.longest <= 16 ? kLaneFull : kLaneLong;
            unsigned char *p = out.add(bytes(n, s.longest), n, s.longest,
                                       cls << kLaneShift | (s.sync && at + n == s.n ? kSync : 0));
            for (int64_t t = 0; t < n; ++t) {
                const int64_t i = s.rows[at + t], pdiag = upper ? diagonal(T, i) : -1;
                auto put = [&](unsigned char *rv, unsigned char *rc, int64_t col, VT v) {
                    *reinterpret_cast<VT *>(rv) = v;
                    *reinterpret_cast<int32_t *>(rc) = vector_place(col - r0, unit);
                };
                for (int64_t q = 0; q < 4; ++q)
                    *reinterpret_cast<int32_t *>(p + lb * (4 * t + q) + np * (sizeof(VT) + 4)) =
                        vector_place(i - r0, unit);
                int64_t e = 0;
                for (int64_t pp = T.rp[i]; pp < T.rp[i + 1]; ++pp) {
                    if (T.ci[pp] == i) continue;
                    const int64_t k = e >> 2, lane = 4 * t + (e & 3);
                    unsigned char *rec = p + lb * lane, *rest = p + lb * 4 * n + tb * ((k - 4) * 4 * n + lane);
                    const VT v = stored_entry<VT>(T, pp, pdiag);
                    if (k < 4) put(rec + k * sizeof(VT), rec + np * sizeof(VT) + 4 * k, T.ci[pp], v);
                    else put(rest, rest + sizeof(VT), T.ci[pp], v);
                    ++e;
                }
            }
            at += n;
        }
    }
}

// The x_i / u_ii products of a block between L and U.
template <typename VT>
void append_scaling(const Csr &U, int64_t r0, int64_t nr, LaneSlices &out) {
    const int64_t step = 4096 / (int64_t)sizeof(VT);
    for (int64_t i0 = 0; i0 < nr; i0 += step) {
        const int64_t n = std::min(step, nr - i0);
        VT *d = reinterpret_cast<VT *>(out.add(kItemHeader + (size_t)n * sizeof(VT), n, i0,
                                                  kLaneScale << kLaneShift | (i0 + n == nr ? kSync : 0)));
        for (int64_t i = 0; i < n; ++i) d[i] = inv_entry<VT>(U, diagonal(U, r0 + i0 + i));
    }
}

// Slices to items: consecutive rounds of one slice per consumer are joined while
// every consumer's share keeps its class and stays within item_bytes.  Returns the slices with kSync.
int32_t pack_lanes(LaneSlices &s, size_t item_bytes, StreamHost &out) {
    const size_t nc = out.consumers, ns = s.off.size() - 1;
    auto header = [&](size_t k) { return reinterpret_cast<int32_t *>(s.data.data() + s.off[k]); };
    auto bytes = [&](size_t k) { return s.off[k + 1] - s.off[k]; };
    auto cls = [&](size_t k) { return header(k)[3] >> kLaneShift & 7; };
    int32_t nsync = 0;
    for (size_t k = 0; k < ns; ++k) {
        int between = 0;                              // wavefronts that end in the other consumers' slices
        for (size_t j = k; j-- > 0 && j + nc > k;) between += header(j)[3] & kSync ? 1 : 0;
        nsync += header(k)[3] & kSync ? 1 : 0;
        header(k)[3] |= between << 24;
    }
    for (size_t k0 = 0; k0 < ns;) {
        std::vector<size_t> share(nc, 0);
        size_t k1 = k0;
        while (k1 < ns) {
            bool fits = true;
            for (size_t c = 0; c < nc && k1 + c < ns; ++c)
                fits = fits && (k1 == k0 || (cls(k1 + c) == cls(k0 + c) && cls(k0 + c) != kLaneScale &&
                                             share[c] + bytes(k1 + c) <= item_bytes));
            if (!fits) break;
            for (size_t c = 0; c < nc && k1 + c < ns; ++c) share[c] += bytes(k1 + c);
            k1 = std::min(ns, k1 + nc);
        }
        for (size_t c = 0; c < nc && k0 + c < k1; ++c) {
            size_t at = add_item(out, share[c]);
            for (size_t k = k0 + c; k < k1; k += nc) {
                header(k)[1] = k + nc < k1 ? (int32_t)bytes(k) : 0;
                std::memcpy(out.data.data() + at, s.data.data() + s.off[k], bytes(k));
                at += bytes(k);
            }
        }
        k0 = k1;
    }
    return nsync;
}

// Slices of one factor in the batched layout (batch.cuh).
void append_batch_rows(const Csr &T, int64_t r0, const Waves &W, bool upper, int np, int max_rows, LaneSlices &out) {
    auto place = [&](int64_t i) { return vector_place(i - r0 + 1, 16); };
    for (const SliceRows &s : cut_slices<float>(W, r0, upper, max_rows)) {
        unsigned char *p = out.add(kItemHeader + pad16((size_t)(8 * s.n)) + (size_t)(row_bytes(np) * s.n), s.n, 0,
                                   s.sync ? kSync : 0);
        EntryF32 *head = reinterpret_cast<EntryF32 *>(p);
        unsigned char *recs = p + pad16((size_t)(8 * s.n));
        for (int64_t t = 0; t < s.n; ++t) {
            const int64_t i = s.rows[t], pdiag = upper ? diagonal(T, i) : -1;
            head[t] = {place(i), upper ? inv_entry<float>(T, pdiag) : 1.f};
            EntryF32 *rec = reinterpret_cast<EntryF32 *>(recs + row_bytes(np) * t);
            for (int64_t q = T.rp[i]; q < T.rp[i + 1]; ++q)
                if (T.ci[q] != i) *rec++ = {place(T.ci[q]), stored_entry<float>(T, q, pdiag)};
        }
    }
}

}  // namespace

void build_chunks(const Csr &L, const Csr &U, const std::vector<int64_t> &bp, ChunkHost &out, int max_rows) {
    validate_tri(L, bp, false);
    validate_tri(U, bp, true);
    for (size_t b = 0; b + 1 < bp.size(); ++b) {
        append_factor_chunks(L, bp[b], bp[b + 1], false, out, max_rows);
        append_factor_chunks(U, bp[b], bp[b + 1], true, out, max_rows);
        out.blk_chunk.push_back((int32_t)(out.off.size() - 1));
    }
}

void append_batch_stream(const Csr &L, const Csr &U, const std::vector<int64_t> &bp, int max_rows, size_t item_bytes,
                         StreamHost &out, int64_t &l_bytes, int64_t &u_bytes) {
    validate_tri(L, bp, false);
    validate_tri(U, bp, true);
    for (size_t b = 0; b + 1 < bp.size(); ++b) {
        LaneSlices s;
        append_batch_rows(L, bp[b], order_rows(L, bp[b], bp[b + 1], false), false, out.np, max_rows, s);
        const size_t lower = s.data.size();
        append_batch_rows(U, bp[b], order_rows(U, bp[b], bp[b + 1], true), true, out.np, max_rows, s);
        l_bytes += (int64_t)lower;
        u_bytes += (int64_t)(s.data.size() - lower);
        out.split.push_back(pack_lanes(s, item_bytes, out));
        out.blk_item.push_back((int32_t)(out.off.size() - 1));
    }
}

template <typename VT>
void build_stream(const Csr &L, const Csr &U, const std::vector<int64_t> &bp, StreamHost &out) {
    validate_tri(L, bp, false);
    validate_tri(U, bp, true);
    const size_t nb = bp.size() - 1;
    std::vector<Waves> wl(nb), wu(nb);
    int32_t longest = 0;
    for (size_t b = 0; b < nb; ++b) {
        wl[b] = order_rows(L, bp[b], bp[b + 1], false);
        wu[b] = order_rows(U, bp[b], bp[b + 1], true);
        for (int32_t x : wl[b].len) longest = std::max(longest, x);
        for (int32_t x : wu[b].len) longest = std::max(longest, x);
        out.maxwf_L = std::max(out.maxwf_L, (int)wl[b].ptr.size() - 1);
        out.maxwf_U = std::max(out.maxwf_U, (int)wu[b].ptr.size() - 1);
    }
    constexpr bool one = OneLaneRows<VT>::value;
    out.np = trsv_record(one, longest);
    int64_t nwave = 1;
    for (size_t b = 0; b < nb; ++b) nwave += (int64_t)(wl[b].ptr.size() + wu[b].ptr.size());
    out.consumers = !one ? trsv_sets((double)(2 * bp.back()) / (double)(nwave * kLaneRows<VT>)) : 4;
    for (size_t b = 0; b < nb; ++b) {
        const int64_t r0 = bp[b];
        if constexpr (one) {
            const size_t first = out.off.size();
            append_groups(L, r0, wl[b], false, out);
            out.split.push_back((int32_t)(out.off.size() - first));
            append_groups(U, r0, wu[b], true, out);
        } else {
            LaneSlices s;
            append_lanes<VT>(L, r0, wl[b], false, out.np, out.unit, s);
            append_scaling<VT>(U, r0, bp[b + 1] - r0, s);
            append_lanes<VT>(U, r0, wu[b], true, out.np, out.unit, s);
            out.split.push_back(pack_lanes(s, kLaneItemBytes, out));
        }
        out.blk_item.push_back((int32_t)(out.off.size() - 1));
        wl[b] = Waves();
        wu[b] = Waves();
    }
    if (out.data.empty()) out.data.resize(16, 0);
}

template void build_stream<float>(const Csr &, const Csr &, const std::vector<int64_t> &, StreamHost &);
template void build_stream<double>(const Csr &, const Csr &, const std::vector<int64_t> &, StreamHost &);
template void build_stream<zc>(const Csr &, const Csr &, const std::vector<int64_t> &, StreamHost &);

namespace {


template <typename VT, typename WT>
void upload_level(const HostLevel &hl, int64_t n, bool schur, Arena &a, DevLevel<VT, WT> &d, int smem_limit) {
    LevelView<VT, WT> &v = d.view;
    v.s = hl.s;
    v.e = hl.e;
    v.stail = schur ? n - hl.e : 0;
    v.nblk = (int32_t)hl.bp.size() - 1;
    v.blk_row = a.upload(hl.bp);
    int64_t maxrows = 0;
    for (size_t b = 0; b + 1 < hl.bp.size(); ++b) maxrows = std::max(maxrows, hl.bp[b + 1] - hl.bp[b]);
    d.smem_rows = (kRingBytes + maxrows * (int64_t)sizeof(VT) <= smem_limit) ? (int)maxrows : 0;
    StreamHost sh;
    sh.unit = place_unit<VT>(d.smem_rows > 0);
    build_stream<VT>(hl.L, hl.U, hl.bp, sh);
    v.S.data = a.upload(sh.data);
    v.S.off = a.upload(sh.off);
    v.S.blk_item = a.upload(sh.blk_item);
    v.S.split = a.upload(sh.split);
    v.S.np = sh.np;
    v.S.consumers = sh.consumers;
    // More blocks than SMs: a ring that leaves room for up to three CTAs on an SM, in FP32
    // without the four warps that only help (their registers are another CTA's).  us per
    // application with a CTA per SM / now: 96^3 in 1,024 blocks mixed 370 / 210, FP64 1315 /
    // 1148; 64^3 in 256 mixed 142 / 92, FP64 483 / 392, complex 975 / 911.
    int dev = 0, sms = 1, per_sm = 0;
    GEMSLR_CUDA(cudaGetDevice(&dev));
    GEMSLR_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    GEMSLR_CUDA(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    const int64_t share = d.smem_rows ? std::min<int64_t>(3, (v.nblk + sms - 1) / sms) : 1;
    v.S.variant = !OneLaneRows<VT>::value ? sh.consumers : share > 1 ? 4 : 8;
    // the ring: up to kItemDepth slots per consumer, in twice kRingData where the
    // vector leaves that much (more bytes in flight), at least one
    const int64_t limit = std::min<int64_t>(smem_limit, per_sm / std::max<int64_t>(1, share) - 1024);
    const int64_t room = (d.smem_rows ? limit - (int64_t)pad16(d.smem_rows * sizeof(VT)) : (int64_t)kRingBytes) -
                         (int64_t)sizeof(StreamHead);
    v.S.slot_bytes = std::max(sh.slot_bytes, 128);
    const int64_t depth = std::min<int64_t>(room, 2 * kRingData) / ((int64_t)v.S.slot_bytes * sh.consumers);
    v.S.slots = sh.consumers * (int)std::max<int64_t>(1, std::min<int64_t>(depth, kItemDepth));
    d.nwf_L = sh.maxwf_L;
    d.nwf_U = sh.maxwf_U;
    if (schur) {
        std::vector<int32_t> fci(hl.F.ci.size());
        for (size_t p = 0; p < fci.size(); ++p) fci[p] = (int32_t)(hl.F.ci[p] + hl.e);
        v.F_rp = a.upload(hl.F.rp);
        v.F_ci = a.upload(fci);
        v.F_v = a.upload(convert<VT>(hl.F.v));
        std::vector<int32_t> frows, fblk(1, 0);
        for (size_t b = 0; b + 1 < hl.bp.size(); ++b) {
            for (int64_t i = hl.bp[b]; i < hl.bp[b + 1]; ++i)
                if (hl.F.rp[i + 1] > hl.F.rp[i]) frows.push_back((int32_t)i);
            fblk.push_back((int32_t)frows.size());
        }
        if (frows.empty()) frows.push_back(0);
        v.F_rows = a.upload(frows);
        v.F_blk = a.upload(fblk);
        v.E_rp = a.upload(hl.E.rp);
        v.E_ci = a.upload(hl.E.ci);
        v.E_v = a.upload(convert<VT>(hl.E.v));
    }
    if (!schur) {
        v.F_rp = nullptr;
        v.F_ci = nullptr;
        v.F_v = nullptr;
        v.F_rows = nullptr;
        v.F_blk = nullptr;
    }
    v.k = 0;
    v.W = nullptr;
    v.H = nullptr;
}

}  // namespace

template <typename VT, typename WT>
void set_lowrank(DevLevel<VT, WT> &d, const HostLevel &hl, Arena &a) {
    d.view.k = hl.k;
    if (hl.k > 0) {
        d.view.W = a.upload(convert<WT>(hl.W));
        d.view.H = a.upload(convert<VT>(hl.H));
    }
}

// complex W, H: real parts in W, H and imaginary parts in Wi, Hi (empty: real)
template <>
void set_lowrank<zc, zc>(DevLevel<zc, zc> &d, const HostLevel &hl, Arena &a) {
    d.view.k = hl.k;
    if (hl.k > 0) {
        auto pack = [](const std::vector<double> &re, const std::vector<double> &im) {
            std::vector<zc> z(re.size());
            for (size_t i = 0; i < re.size(); ++i) z[i] = zc(re[i], im.empty() ? 0.0 : im[i]);
            return z;
        };
        d.view.W = a.upload(pack(hl.W, hl.Wi));
        d.view.H = a.upload(pack(hl.H, hl.Hi));
    }
}

template <typename VT, typename WT>
void upload_hierarchy(const Hierarchy &h, Arena &a, DevHierarchy<VT, WT> &d, int smem_limit) {
    set_trsv_smem_limit<VT, WT>(smem_limit);
    d.err = (int32_t *)a.alloc(sizeof(int32_t) * 4);
    GEMSLR_CUDA(cudaMemset(d.err, 0, sizeof(int32_t) * 4));
    d.lev.resize(h.lev.size());
    int64_t maxd = 1;
    for (size_t l = 0; l < h.lev.size(); ++l) {
        upload_level<VT, WT>(h.lev[l], h.n, true, a, d.lev[l], smem_limit);
        d.lev[l].view.err = d.err;
        set_lowrank<VT, WT>(d.lev[l], h.lev[l], a);
        maxd = std::max(maxd, h.lev[l].e - h.lev[l].s);
    }
    upload_level<VT, WT>(h.last, h.n, false, a, d.last, smem_limit);
    d.last.view.err = d.err;
    maxd = std::max(maxd, h.n - h.last.s);
    d.work = (VT *)a.alloc(sizeof(VT) * std::max<int64_t>(h.n, 1));
    d.scratch = (VT *)a.alloc(sizeof(VT) * maxd);
    int64_t maxgrid = 1;
    for (auto &l : h.lev) maxgrid = std::max(maxgrid, (h.n - l.e + kCoupleRows - 1) / kCoupleRows);
    d.partial = (VT *)a.alloc(sizeof(VT) * maxgrid * kMaxRank);
    d.counter = (unsigned *)a.alloc(sizeof(unsigned) * 4);
    GEMSLR_CUDA(cudaMemset(d.counter, 0, sizeof(unsigned) * 4));
    d.u = (VT *)a.alloc(sizeof(VT) * kMaxRank);
}

template <typename VT, typename WT>
void setup_inner(const Hierarchy &h, Arena &a, DevHierarchy<VT, WT> &d, int k, int sms) {
    DevInner<VT> &I = d.inner;
    if (k > 0 && !I.work2) {
        const int64_t e0 = h.lev[0].e, n = h.n, m = n - e0;
        // rows [e0, n) of A_hat with global columns, values in the application's precision
        const Csr &A = h.Ahat;
        std::vector<int64_t> rp(m + 1);
        for (int64_t i = 0; i <= m; ++i) rp[i] = A.rp[e0 + i] - A.rp[e0];
        std::vector<int32_t> ci(A.ci.begin() + A.rp[e0], A.ci.begin() + A.rp[n]);
        std::vector<double> v(A.v.begin() + A.rp[e0], A.v.begin() + A.rp[n]);
        InnerView<VT> &iv = I.iv;
        iv.m = m;
        iv.e0 = e0;
        iv.rp = a.upload(rp);
        iv.ci = a.upload(ci);
        iv.v = a.upload(convert<VT>(v));
        const size_t mm = (size_t)std::max<int64_t>(m, 1);
        iv.V = (VT *)a.alloc(sizeof(VT) * mm * (kMaxInner + 1));
        iv.Z = (VT *)a.alloc(sizeof(VT) * mm * kMaxInner);
        iv.w = (VT *)a.alloc(sizeof(VT) * mm);
        iv.H = (double *)a.alloc(sizeof(double) * (kMaxInner + 1) * kMaxInner);
        GEMSLR_CUDA(cudaMemset(iv.H, 0, sizeof(double) * (kMaxInner + 1) * kMaxInner));
        iv.grid = (int)std::max<int64_t>(1, std::min<int64_t>((m + kReduceThreads - 1) / kReduceThreads, 2 * sms));
        iv.partial = (double *)a.alloc(sizeof(double) * iv.grid * (kMaxInner + 2));
        iv.counter = (unsigned *)a.alloc(16);
        GEMSLR_CUDA(cudaMemset(iv.counter, 0, 16));
        iv.ctl = (InnerCtl *)a.alloc(sizeof(InnerCtl));
        GEMSLR_CUDA(cudaMemset(iv.ctl, 0, sizeof(InnerCtl)));
        I.work2 = (VT *)a.alloc(sizeof(VT) * std::max<int64_t>(n, 1));
        GEMSLR_CUDA(cudaMemset(I.work2, 0, sizeof(VT) * std::max<int64_t>(n, 1)));
        I.zero_rp = (int64_t *)a.alloc(sizeof(int64_t) * (mm + 1));
        GEMSLR_CUDA(cudaMemset(I.zero_rp, 0, sizeof(int64_t) * (mm + 1)));
    }
    I.k = k;
    I.iv.k = k;
}

// Alg. 2 at the root level with step 9: z1 = U^-1 L^-1 b1, z2 = b2 - E z1,
// k GMRES steps on S_hat_0 y2 = z2 (inner.cu) whose preconditioner is the
// level-0 correction plus the levels below, y1 = z1 - U^-1 L^-1 F y2.
template <typename VT, typename WT>
void apply_root_inner(DevHierarchy<VT, WT> &d, const IoT<VT> *in, VT *work, IoT<VT> *out_final, cudaStream_t st) {
    DevLevel<VT, WT> &L0 = d.lev[0];
    DevInner<VT> &I = d.inner;
    const InnerView<VT> &iv = I.iv;
    VT *work2 = I.work2;
    {
        ProfScope ps("trsv_down_L0", st);
        launch_trsv<VT, WT>(L0.view, 0, L0.smem_rows, in, work, nullptr, d.scratch, st);
    }
    LevelView<VT, WT> v0 = L0.view;
    v0.k = 0;                                       // z2 only: the correction acts inside the preconditioner
    {
        ProfScope ps("couple_EWt_L0", st);
        launch_couple<VT, WT>(v0, in, work, d.partial, d.counter, d.u, st);
    }
    {
        ProfScope ps("inner_start", st);
        launch_inner_norm<VT>(iv, work + iv.e0, st);
        launch_inner_start<VT>(iv, work + iv.e0, work2, st);
    }
    LevelView<VT, WT> vz = L0.view;
    vz.E_rp = I.zero_rp;                            // E_0 empty: z2 = v_j unchanged, u = H_0 W_0^T v_j
    PendingLowRank<VT, WT> pend;
    if (L0.view.k > 0 && L0.view.stail > 0) {
        pend.W = L0.view.W;
        pend.u = d.u;
        pend.ld = L0.view.stail;
        pend.row0 = L0.view.e;
        pend.k = L0.view.k;
    }
    for (int j = 0; j < I.k; ++j) {
        if (pend.W) {
            ProfScope ps("couple_EWt_L0", st);
            launch_couple<VT, WT>(vz, nullptr, work2, d.partial, d.counter, d.u, st);
        }
        apply_levels<VT, WT>(d, 1, nullptr, work2, nullptr, st, pend);   // z_j = M_S^-1 v_j in the tail
        {
            ProfScope ps("inner_trsv_L0", st);                              // level part: -U^-1 L^-1 F z_j
            launch_trsv<VT, WT>(L0.view, 1, L0.smem_rows, nullptr, work2, nullptr, d.scratch, st);
        }
        {
            ProfScope ps("inner_spmv_gs", st);
            launch_inner_spmv_dots<VT>(iv, j, work2, st);
            launch_inner_sub_dots<VT>(iv, j, st);
            launch_inner_scale<VT>(iv, j, work2, st);
        }
    }
    {
        ProfScope ps("inner_finish", st);
        launch_inner_lsq<VT>(iv, st);
        launch_inner_combine<VT>(iv, work, out_final, st);
    }
    {
        ProfScope ps("trsv_up_L0", st);
        launch_trsv<VT, WT>(L0.view, 1, L0.smem_rows, nullptr, work, out_final, d.scratch, st);
    }
}

template <typename VT, typename WT>
void apply_levels(DevHierarchy<VT, WT> &d, int from, const IoT<VT> *in, VT *work, IoT<VT> *out_final,
                  cudaStream_t st, const PendingLowRank<VT, WT> &pend0) {
    const int nl = (int)d.lev.size();
    constexpr bool kReal = !IsComplex<VT>::value;   // the complex hierarchy has neither inner steps nor a learned stage
    if constexpr (kReal) {
        if (from == 0 && nl >= 1 && d.inner.k > 0) {
            apply_root_inner<VT, WT>(d, in, work, out_final, st);
            return;
        }
    }
    static const char *kDown[] = {"trsv_down_L0", "trsv_down_L1", "trsv_down_L2", "trsv_down_L3", "trsv_down_L4+"};
    static const char *kUp[] = {"trsv_up_L0", "trsv_up_L1", "trsv_up_L2", "trsv_up_L3", "trsv_up_L4+"};
    static const char *kCouple[] = {"couple_EWt_L0", "couple_EWt_L1", "couple_EWt_L2", "couple_EWt_L3", "couple_EWt_L4+"};
    // learned correction at the deepest Schur level (active only when that level is part of this application)
    const bool learn = kReal && d.learned && d.learned->enabled && nl >= 1 && from <= nl - 1;
    // W_l u_l of the level before is added where its tail rows are first read
    PendingLowRank<VT, WT> pend = pend0;
    for (int l = from; l < nl; ++l) {
        DevLevel<VT, WT> &L = d.lev[l];
        const IoT<VT> *src = (l == from) ? in : nullptr;
        {
            ProfScope ps(kDown[std::min(l, 4)], st);
            launch_trsv<VT, WT>(L.view, 0, L.smem_rows, src, work, nullptr, d.scratch, st, pend);
        }
        {
            ProfScope ps(kCouple[std::min(l, 4)], st);
            launch_couple<VT, WT>(L.view, src, work, d.partial, d.counter, d.u, st, pend);
        }
        if constexpr (kReal)
            if (learn && l == nl - 1) learned_save<VT>(*d.learned, L.view.e, work, st);   // z2 of level l*
        pend = PendingLowRank<VT, WT>();
        if (L.view.k > 0 && L.view.stail > 0) {
            pend.W = L.view.W;
            pend.u = d.u;
            pend.ld = L.view.stail;
            pend.row0 = L.view.e;
            pend.k = L.view.k;
        }
    }
    {
        ProfScope ps("trsv_last", st);
        launch_trsv<VT, WT>(d.last.view, 0, d.last.smem_rows, from == nl ? in : nullptr, work,
                            learn ? nullptr : out_final, d.scratch, st, pend);
    }
    if constexpr (kReal) if (learn) {
        // S_hat y2 = C y2 - E (LU)^{-1} F y2 on a scratch vector, then y2 += N(rho)
        ProfScope ps("learned_stage", st);
        DevLevel<VT, WT> &L = d.lev[nl - 1];
        LearnedStage<VT> &Ls = *d.learned;
        const int64_t e = L.view.e, s0 = L.view.s, ntail = L.view.stail;
        GEMSLR_CUDA(cudaMemcpyAsync(Ls.work2 + e, work + e, sizeof(VT) * ntail, cudaMemcpyDeviceToDevice, st));
        GEMSLR_CUDA(cudaMemsetAsync(Ls.work2 + s0, 0, sizeof(VT) * (e - s0), st));
        launch_trsv<VT, WT>(L.view, 1, L.smem_rows, nullptr, Ls.work2, nullptr, d.scratch, st);
        LevelView<VT, WT> v0 = L.view;
        v0.k = 0;
        launch_couple<VT, WT>(v0, Ls.zeros, Ls.work2, d.partial, d.counter, d.u, st);
        learned_rho_and_update<VT>(Ls, e, work, st);
        if (out_final) launch_cast_out<VT>(ntail, work + e, out_final + e, st);
    }
    for (int l = nl - 1; l >= from; --l) {
        ProfScope ps(kUp[std::min(l, 4)], st);
        launch_trsv<VT, WT>(d.lev[l].view, 1, d.lev[l].smem_rows, nullptr, work, out_final, d.scratch, st);
    }
}

template <>
void apply_hierarchy<double, double>(DevHierarchy<double, double> &d, int64_t, const double *in, double *out,
                                     cudaStream_t st) {
    apply_levels<double, double>(d, 0, in, out, nullptr, st);
}

template <>
void apply_hierarchy<float, __nv_bfloat16>(DevHierarchy<float, __nv_bfloat16> &d, int64_t, const double *in,
                                           double *out, cudaStream_t st) {
    apply_levels<float, __nv_bfloat16>(d, 0, in, d.work, out, st);
}

template void upload_hierarchy<double, double>(const Hierarchy &, Arena &, DevHierarchy<double, double> &, int);
template void upload_hierarchy<float, __nv_bfloat16>(const Hierarchy &, Arena &,
                                                     DevHierarchy<float, __nv_bfloat16> &, int);
template void upload_hierarchy<zc, zc>(const Hierarchy &, Arena &, DevHierarchy<zc, zc> &, int);
template void apply_levels<zc, zc>(DevHierarchy<zc, zc> &, int, const zc *, zc *, zc *, cudaStream_t,
                                   const PendingLowRank<zc, zc> &);
template void set_lowrank<double, double>(DevLevel<double, double> &, const HostLevel &, Arena &);
template void apply_levels<double, double>(DevHierarchy<double, double> &, int, const double *, double *, double *,
                                           cudaStream_t, const PendingLowRank<double, double> &);
template void setup_inner<double, double>(const Hierarchy &, Arena &, DevHierarchy<double, double> &, int, int);
template void setup_inner<float, __nv_bfloat16>(const Hierarchy &, Arena &, DevHierarchy<float, __nv_bfloat16> &,
                                                int, int);

}  // namespace gemslr
