// C ABI of the library (include/spmv.h): handle management, validation, the
// row-length-histogram autotuner and tile planning, the split plan, the reverse
// pass, the batched graph launch and the CG solvers.
#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <new>
#include <utility>
#include <vector>

#include "spmv.h"
#include "internal.h"
#include "cg.h"
#include "warp_kernel.cuh"
#include "slot_kernel.cuh"
#include "sell_kernel.cuh"

namespace spmv {
int64_t transpose_work_len(int32_t n_cols);

bool tile_ops(int vk, int xk, int yk, int acc, int R, int E, bool indirect, bool batched,
              TileOps *ops) {
    if (vk == kF64) {
        if (xk != kF64 || yk != kF64) return false;
        return tile_ops_f64(R, E, indirect, batched, ops);
    }
    return tile_ops_f32(xk, yk, acc, R, E, indirect, batched, ops);
}

bool warp_ops(int vk, int xk, int yk, int acc, int E, bool indirect, bool batched, WarpOps *ops) {
    if (vk == kF64) {
        if (xk != kF64 || yk != kF64) return false;
        return warp_ops_f64(E, indirect, batched, ops);
    }
    if (xk != kF32) return false;
    return warp_ops_f32(yk, acc, E, indirect, batched, ops);
}
}  // namespace spmv

using namespace spmv;

namespace {

struct TileTable {
    TileDesc *d = nullptr;
    int32_t n = 0;
    int32_t n_long = 0;
    std::vector<TileDesc> host;
};

std::vector<TileDesc> make_tiles(const int32_t *rp, int32_t n_rows, int cap, int rowcap, int mat,
                                 int32_t *n_long) {
    std::vector<TileDesc> t;
    int32_t nl = 0;
    int32_t r = 0;
    while (r < n_rows) {
        const int32_t k0 = rp[r];
        if (static_cast<int64_t>(rp[r + 1]) - k0 > cap) {
            TileDesc d{r, r + 1, k0, rp[r + 1], mat, 0, 0, 0};
            t.push_back(d);
            ++nl;
            ++r;
            continue;
        }
        const int32_t lim = static_cast<int32_t>(std::min<int64_t>(n_rows, static_cast<int64_t>(r) + rowcap));
        const int64_t target = static_cast<int64_t>(k0) + cap;
        const int32_t *it = std::upper_bound(rp + r + 1, rp + lim + 1, target,
                                             [](int64_t v, int32_t e) { return v < e; });
        const int32_t r1 = static_cast<int32_t>(it - rp) - 1;
        TileDesc d{r, r1, k0, rp[r1], mat, 0, 0, 0};
        t.push_back(d);
        r = r1;
    }
    if (n_long) *n_long = nl;
    return t;
}

#define CK(call)                                             \
    do {                                                     \
        cudaError_t e__ = (call);                            \
        if (e__ != cudaSuccess) return SPMV_ERR_CUDA;        \
    } while (0)

template <typename T>
cudaError_t dmalloc(T **p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
}

// The capture that records what is enqueued on s (0: work on s runs).
unsigned long long capture_id(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(s, &st, &id) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return st == cudaStreamCaptureStatusActive ? id : 0;
}

// Whether a derived copy holds the current values.  A layout recorded while a stream
// is captured runs with the graph, so it counts for the rest of that capture only: a
// call outside the graph lays the values out itself.
struct Laid {
    bool now = false;
    unsigned long long in_capture = 0;  // the capture that lays them out
    bool on(cudaStream_t s) const { return now || (in_capture != 0 && in_capture == capture_id(s)); }
    void set(cudaStream_t s) {
        const unsigned long long id = capture_id(s);
        if (id) in_capture = id;
        else now = true;
    }
};

// Slot-major copy of a matrix for plan family 4 (per entries-per-lane E).
struct SlotTable {
    void *block = nullptr;      // one allocation that holds the four arrays (a handle's own copy)
    ChunkDesc *d = nullptr;
    uint32_t *lmask = nullptr;  // 32 words per chunk
    void *vals = nullptr;       // n * 32E values, slot-major
    int32_t *cols = nullptr;    // n * 32E column indices, slot-major
    int32_t n = 0;
    int32_t n_long = 0, n_empty = 0;
    Laid laid;
};

// Sorted row-slice copy of a matrix for plan family 5 (per window sigma).
struct SellTable {
    void *meta = nullptr;       // one allocation: the tables d, srows, cstart, dtmp, dorder
    int2 *d = nullptr;          // per slice: first slot row and width (width < 0: long row)
    int32_t *srows = nullptr;   // kSellC rows per slice (-1: none)
    int32_t *cstart = nullptr;  // n_ctas + 1: first slice of each CTA of a launch
    int32_t n_ctas = 0;
    void *vals = nullptr;       // slot_rows * 32 values
    int32_t *cols = nullptr;    // slot_rows * 32 column indices
    int32_t n = 0;
    int32_t n_long = 0;
    int64_t slot_rows = 0;
    Laid laid;
    bool read = false;          // something has read the values since the last new ones
    // diagonal slices: descriptors with each slice's place in diag (in slice order
    // and in launch order), and the diagonals of the slot rows, padded to 4 per slice
    // (behind cols)
    int4 *dtmp = nullptr, *dorder = nullptr;
    int4 *diag = nullptr;
    bool diagonal = false;      // enough slices are diagonal for k_sell_diag
    // A^T: position of each slot's value in A's copy for a window (built on first use;
    // held for each window of A that reverse passes ran on: captured ones read them)
    std::map<int32_t, int32_t *> vpos;
};

struct ChunkTable {
    ChunkDesc *d = nullptr;
    uint32_t *masks = nullptr;
    int32_t *cmat = nullptr;
    int32_t n = 0;
    int32_t n_long = 0;
    int32_t n_empty = 0;
};

// Cut rows into warp chunks: whole rows whose entries fit in 32*E slots from the
// 16-byte aligned start below the first entry, at most kWarpRowCap rows; one bit
// per slot marks the row starts.  Rows that do not fit alone become long chunks.
void make_chunks(const int32_t *rp, int32_t n_rows, int E, int32_t mat, std::vector<ChunkDesc> &out,
                 std::vector<uint32_t> &masks, std::vector<int32_t> *cmat, int32_t *n_long,
                 int32_t *n_empty) {
    const int64_t SL = 32LL * E;
    const int MW = ((E + 3) / 4) * 4;  // mask words per chunk, rows of 16 bytes
    if (out.empty() && n_rows > 0) {
        const size_t guess = static_cast<size_t>((rp[n_rows] - rp[0]) / SL + n_rows / kWarpRowCap);
        out.reserve(guess + guess / 8 + 8);
        masks.reserve(MW * (guess + guess / 8 + 8));
    }
    int32_t r = 0;
    while (r < n_rows) {
        const int32_t k0 = rp[r];
        const int32_t base = k0 & ~3;
        const size_t mo = masks.size();
        masks.resize(mo + MW, 0u);
        if (cmat) cmat->push_back(mat);
        if (static_cast<int64_t>(rp[r + 1]) - base > SL) {
            out.push_back(ChunkDesc{k0, rp[r + 1], r, (r + 1) | kChunkLong});
            ++*n_long;
            ++r;
            continue;
        }
        bool empty = (rp[r + 1] == rp[r]);
        int32_t r1 = r + 1;
        while (r1 < n_rows && r1 - r < kWarpRowCap && static_cast<int64_t>(rp[r1 + 1]) - base <= SL) {
            empty = empty || (rp[r1 + 1] == rp[r1]);
            ++r1;
        }
        out.push_back(ChunkDesc{k0, rp[r1], r, r1 | (empty ? kChunkEmpty : 0)});
        if (empty) ++*n_empty;
        for (int32_t q = r; q < r1; ++q)
            if (rp[q + 1] > rp[q]) {
                const int32_t sl = rp[q] - base;
                masks[mo + (sl >> 5)] |= 1u << (sl & 31);
            }
        r = r1;
    }
}

spmv_status upload_chunks(ChunkTable *ct, const std::vector<ChunkDesc> &d, const std::vector<uint32_t> &m,
                          const std::vector<int32_t> *cmat) {
    ct->n = static_cast<int32_t>(d.size());
    if (dmalloc(&ct->d, d.size()) != cudaSuccess || dmalloc(&ct->masks, m.size()) != cudaSuccess)
        return SPMV_ERR_ALLOC;
    if (cmat && dmalloc(&ct->cmat, cmat->size()) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (!d.empty() && cudaMemcpy(ct->d, d.data(), sizeof(ChunkDesc) * d.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return SPMV_ERR_CUDA;
    if (!m.empty() && cudaMemcpy(ct->masks, m.data(), 4 * m.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return SPMV_ERR_CUDA;
    if (cmat && !cmat->empty() &&
        cudaMemcpy(ct->cmat, cmat->data(), 4 * cmat->size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return SPMV_ERR_CUDA;
    return SPMV_OK;
}

void free_chunks(ChunkTable &ct) {
    cudaFree(ct.d);
    cudaFree(ct.masks);
    cudaFree(ct.cmat);
    ct = ChunkTable();
}

// Chunks for the slot-major layout: the same row packing as make_chunks, from
// the chunk's first entry itself (no alignment), with one word per lane: the row
// starts in its E slots (bits 0..E-1), the rows starting before them (bits
// kSlotPreShift..) and whether its last slot ends a row or the chunk (kSlotEnds).
template <int E>
void make_slot_chunks_of(const int32_t *rp, int32_t n_rows, std::vector<ChunkDesc> &out, std::vector<uint32_t> &lmask,
                         int32_t *n_long, int32_t *n_empty) {
    constexpr int64_t SL = 32LL * E;
    if (out.empty() && n_rows > 0) {
        const size_t guess = static_cast<size_t>((rp[n_rows] - rp[0]) / SL + n_rows / kWarpRowCap);
        out.reserve(guess + guess / 8 + 8);
        lmask.reserve(32 * (guess + guess / 8 + 8));
    }
    int32_t r = 0;
    while (r < n_rows) {
        const int32_t k0 = rp[r];
        uint32_t w[32] = {0};
        if (static_cast<int64_t>(rp[r + 1]) - k0 > SL) {
            out.push_back(ChunkDesc{k0, rp[r + 1], r, (r + 1) | kChunkLong});
            lmask.insert(lmask.end(), w, w + 32);
            ++*n_long;
            ++r;
            continue;
        }
        // a row's start is marked as it joins the chunk (not that of an empty row)
        bool empty = false;
        int32_t r1 = r, start = k0;
        while (r1 < n_rows && r1 - r < kWarpRowCap) {
            const int32_t end = rp[r1 + 1];
            if (static_cast<int64_t>(end) - k0 > SL) break;
            const uint32_t sl = static_cast<uint32_t>(start - k0);
            if (end > start) w[sl / E] |= 1u << (sl % E);
            else empty = true;
            start = end;
            ++r1;
        }
        out.push_back(ChunkDesc{k0, start, r, r1 | (empty ? kChunkEmpty : 0)});
        if (empty) ++*n_empty;
        if (!empty) {
            const int n_used = start - k0;
            uint32_t pre = 0;
            int through_run = 0;  // lanes just before this one that lie inside one row
            for (int lane = 0; lane < 32; ++lane) {
                const uint32_t bits = w[lane];
                const bool active = lane * E < n_used;
                const bool ends = (lane + 1) * E >= n_used || (lane < 31 && (w[lane + 1] & 1u));
                const bool started = bits != 0u;
                // a piece of a row begun in an earlier lane ends in this lane
                const bool pending = active && !(bits & 1u) && (started || ends);
                const uint32_t chain = pending ? static_cast<uint32_t>(1 + through_run) : 0u;
                through_run = (active && !ends && !started) ? through_run + 1 : 0;
                w[lane] = bits | (pre << kSlotPreShift) | (ends ? kSlotEnds : 0u) | (chain << kSlotChainShift);
                pre += static_cast<uint32_t>(__builtin_popcount(bits));
            }
        }
        lmask.insert(lmask.end(), w, w + 32);
        r = r1;
    }
}

void make_slot_chunks(const int32_t *rp, int32_t n_rows, int E, std::vector<ChunkDesc> &out,
                      std::vector<uint32_t> &lmask, int32_t *n_long, int32_t *n_empty) {
    switch (E) {  // the entries per lane that the kernels are compiled for
        case 7: return make_slot_chunks_of<7>(rp, n_rows, out, lmask, n_long, n_empty);
        case 9: return make_slot_chunks_of<9>(rp, n_rows, out, lmask, n_long, n_empty);
        case 11: return make_slot_chunks_of<11>(rp, n_rows, out, lmask, n_long, n_empty);
        default: return make_slot_chunks_of<15>(rp, n_rows, out, lmask, n_long, n_empty);
    }
}

// Rows longer than this are summed by a whole warp from the CRS arrays instead
// of by one lane of a slice.
constexpr int32_t kSellLongRow = 128;
// Share of the slots that diagonal slices must cover for k_sell_diag to run (the
// others read column indices there too, without k_sell's loads a block ahead).
// The 27-point pattern on 24^3 (0.73) runs in 4.7 us (FP64; 3.5 FP32) against
// 9.4 (7.0) on k_sell; on 13^3 to 22^3 none is slower than there.
constexpr double kDiagMinShare = 0.5;

// Slices of the sorted row-slice layout: in each window of sigma rows, the rows
// of at most kSellLongRow entries ordered by length (longest first, ties in row
// order) and cut into slices of kSellC; each longer row is a slice of its own
// (width -1, x = the row).  Slot rows are numbered consecutively over the slices
// after kSellU rows of padding (a short block loads the slot rows before it).
// Returns false when the slot rows do not fit in int32.
bool make_sell_slices(const int32_t *rp, int32_t n_rows, int32_t sigma, std::vector<int2> &out,
                      std::vector<int32_t> &srows, int32_t *n_long, int64_t *slot_rows) {
    int64_t off = kSellU;
    std::vector<int32_t> idx, sorted;
    for (int64_t w0 = 0; w0 < n_rows; w0 += sigma) {
        const int32_t w1 = static_cast<int32_t>(std::min<int64_t>(n_rows, w0 + sigma));
        idx.clear();
        for (int32_t r = static_cast<int32_t>(w0); r < w1; ++r) {
            if (rp[r + 1] - rp[r] > kSellLongRow) {
                out.push_back(make_int2(r, -1));
                srows.insert(srows.end(), kSellC, -1);
                ++*n_long;
            } else {
                idx.push_back(r);
            }
        }
        // longest first, ties in row order: a counting sort
        int32_t at[kSellLongRow + 2] = {0};  // place of the next row of length kSellLongRow - q
        for (int32_t r : idx) ++at[kSellLongRow - (rp[r + 1] - rp[r]) + 1];
        for (int q = 1; q <= kSellLongRow + 1; ++q) at[q] += at[q - 1];
        sorted.resize(idx.size());
        for (int32_t r : idx) sorted[static_cast<size_t>(at[kSellLongRow - (rp[r + 1] - rp[r])]++)] = r;
        idx.swap(sorted);
        for (size_t i = 0; i < idx.size(); i += kSellC) {
            const int32_t w = rp[idx[i] + 1] - rp[idx[i]];
            if (off > INT32_MAX) return false;
            out.push_back(make_int2(static_cast<int32_t>(off), w));
            const size_t real = std::min<size_t>(kSellC, idx.size() - i);
            srows.insert(srows.end(), idx.begin() + i, idx.begin() + i + real);
            srows.insert(srows.end(), kSellC - real, -1);
            off += w;
        }
    }
    *slot_rows = off;
    return off <= INT32_MAX;
}

// Padding of the sorted row-slice layout (stored slots / entries - 1) from the
// row lengths alone: per window, a histogram of lengths gives every slice's width.
double sell_padding(const int32_t *rp, int32_t n_rows, int32_t sigma) {
    int64_t slots = 0, used = 0;
    std::vector<int32_t> hist(kSellLongRow + 1);
    for (int64_t w0 = 0; w0 < n_rows; w0 += sigma) {
        const int32_t w1 = static_cast<int32_t>(std::min<int64_t>(n_rows, w0 + sigma));
        std::fill(hist.begin(), hist.end(), 0);
        for (int32_t r = static_cast<int32_t>(w0); r < w1; ++r) {
            const int32_t len = rp[r + 1] - rp[r];
            if (len > kSellLongRow) continue;
            ++hist[len];
            used += len;
        }
        // walk the lengths from the longest: every kSellC-th row opens a slice of its width
        int64_t seen = 0;
        for (int32_t len = kSellLongRow; len >= 0; --len) {
            const int64_t c = hist[len];
            if (c == 0) continue;
            const int64_t opened = (seen + c + kSellC - 1) / kSellC - (seen + kSellC - 1) / kSellC;
            slots += opened * kSellC * len;
            seen += c;
        }
    }
    return used ? static_cast<double>(slots) / used - 1.0 : 0.0;
}

// Contiguous slice ranges of equal work for G CTAs: ws[g] is the first slice
// of CTA g.  A slice's work is its slots plus one slot row for its descriptor,
// rows and stores; a long row's is its entries plus the same.
void sell_ranges(const std::vector<int2> &d, const int32_t *rp, int G, std::vector<int32_t> &ws) {
    std::vector<int64_t> pre(d.size() + 1, 0);
    for (size_t i = 0; i < d.size(); ++i) {
        const int64_t wk = d[i].y >= 0 ? (static_cast<int64_t>(d[i].y) + 1) * kSellC
                                       : static_cast<int64_t>(rp[d[i].x + 1] - rp[d[i].x]) + kSellC;
        pre[i + 1] = pre[i] + wk;
    }
    const int64_t total = pre.back();
    ws.assign(static_cast<size_t>(G) + 1, 0);
    size_t i = 0;
    for (int g = 1; g < G; ++g) {
        const int64_t target = total * g / G;
        while (i < d.size() && pre[i] < target) ++i;
        ws[g] = static_cast<int32_t>(i);
    }
    ws[G] = static_cast<int32_t>(d.size());
}

void free_sell(SellTable &t) {
    cudaFree(t.meta);
    for (auto &kv : t.vpos) cudaFree(kv.second);
    cudaFree(t.vals);
    cudaFree(t.cols);
    t = SellTable();
}

void free_slots(SlotTable &t) {
    cudaFree(t.block);
    if (!t.block) {
        cudaFree(t.d);
        cudaFree(t.lmask);
        cudaFree(t.vals);
        cudaFree(t.cols);
    }
    t = SlotTable();
}

// Several arrays in one allocation: add() each, alloc(), then take() them in the same
// order.  (An allocation of a megabyte or more takes some 40 to 80 us, a smaller one 4.)
// Large arrays start where allocations of their own would, on 2 MB: on 256 bytes the
// symmetric product of 1 M rows took 42.1 to 42.6 us instead of 42.0, the split 63.0 to
// 63.9 instead of 62.8.
struct Block {
    std::vector<size_t> at;
    size_t bytes = 0, next = 0;
    char *base = nullptr;
    void add(size_t b) {
        const size_t unit = b >= (size_t(1) << 20) ? size_t(2) << 20 : 256;
        bytes = (bytes + unit - 1) / unit * unit;
        at.push_back(bytes);
        bytes += b;
    }
    bool alloc() {
        if (cudaMalloc(&base, std::max<size_t>(bytes, 256)) != cudaSuccess) base = nullptr;
        return base != nullptr;
    }
    template <typename T> void take(T **p) { *p = reinterpret_cast<T *>(base + at[next++]); }
    void take(void **p) { *p = base + at[next++]; }
};

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

}  // namespace

constexpr int32_t kCheckEvery = kCgCheckEvery;  // CG iterations between residual read-backs

struct CgWork {
    int64_t n = 0;
    double *r64 = nullptr, *p64 = nullptr, *q64 = nullptr;
    float *r32 = nullptr, *d32 = nullptr, *p32 = nullptr, *q32 = nullptr;
    double *sc = nullptr, *partials = nullptr;
    double *host = nullptr;  // pinned scalars
    // the one-kernel solve: the barrier marks of one_ctas CTAs, results
    double *one = nullptr;
    int32_t one_ctas = 0;
    // kCheckEvery CG iterations captured once and replayed (host launch overhead
    // paid once per block); re-captured when the operands or the plan change
    cudaGraphExec_t inner32 = nullptr;  // FP32 inner CG of the IR solver
    int64_t inner32_key = -1;
    cudaGraphExec_t cg64 = nullptr;     // FP64 CG (x is the caller's pointer)
    const void *cg64_x = nullptr;
    int64_t cg64_key = -1;
};

struct spmv_matrix {
    int32_t n_rows = 0, n_cols = 0;
    int64_t nnz = 0;
    // symmetric CRS: the CRS arrays hold the upper triangle with the diagonal,
    // and the transposed slots (d_rowT, d_colT, d_perm, h_rowT) the transposed
    // structure of its strictly upper part (perm: positions in the values)
    bool sym = false;
    int vk = kF64;
    int device = 0;
    bool owns_structure = true;
    void *block = nullptr;      // holds the arrays below in one allocation (a symmetric handle's full matrix)
    // values of the CRS arrays as val_of[map_of[k]] (an FP32 full matrix: U's), for rows
    // that the slot-major kernel sums again
    const int32_t *map_of = nullptr;
    const void *val_of = nullptr;
    int32_t *d_rp = nullptr;
    int32_t *d_col = nullptr;
    void *d_val = nullptr;
    int32_t *d_err = nullptr;
    uint64_t values_version = 0;  // incremented by spmv_set_values (batches copy values)
    std::vector<int32_t> h_rp;
    // plan
    double col_random = 0.0;  // column_randomness() of the pattern
    double col_diag = 0.0;    // diagonal_rows() of the pattern
    int32_t max_row = 0x7fffffff;  // longest row (set by the tuner)
    int family = 0;  // 0 warp chunks, 1 row-vector, 2 staged tiles, 3 three-stage chunks
    int E = 16;      // entries per lane (family 0) or per thread segment (family 2)
    int T = 8;
    int acc32 = kAccFF;
    std::map<std::pair<int, int>, TileTable> tables;  // (cap, rowcap) -> tiles
    std::map<int, ChunkTable> chunks;                   // E -> warp chunks
    std::map<int, ChunkTable> chunksT;                  // E -> warp chunks of A^T
    std::map<int, SlotTable> slots;                     // E -> slot-major copy (family 4)
    std::map<int, SlotTable> slotsT;                    // E -> slot-major copy of A^T (reverse pass)
    std::map<int, SellTable> sells;                     // sigma -> sorted row-slice copy (family 5)
    std::map<int, SellTable> sellsT;                    // sigma -> sorted row-slice copy of A^T (reverse pass)
    double sell_padT = -1.0;                            // padding of A^T's slices (computed on first use)
    int32_t sigma = 4096;                               // family 5: rows per sorting window
    bool planned = false;                               // the caller chose the plan
    bool sell_if_diag = false;                          // family 5 by the tuner for its diagonal slices only
    double sell_pad = 1.0;                              // padding of sorted slices of 4096-row windows
    int32_t *d_rmap = nullptr;                          // output row of each stored row
    // transposed structure (built on first use)
    bool has_T = false;
    int32_t *d_rowT = nullptr, *d_colT = nullptr, *d_perm = nullptr;
    // values of A^T in its row order (val[perm]): laid out by the second reverse
    // pass on the same values (valT_requested records the first one) and
    // invalidated by spmv_set_values
    void *d_valT = nullptr;
    Laid valT;
    bool valT_requested = false;
    std::vector<int32_t> h_rowT;
    std::map<std::pair<int, int>, TileTable> tablesT;
    // symmetric CRS: the full matrix laid out once (get_full) and the position of
    // each of its values among U's; full_off: two passes for good
    spmv_matrix *full = nullptr;
    int32_t *d_fullmap = nullptr;  // in full's block
    int32_t *d_slotmap = nullptr;  // the map in the order of the slots that full's products read
    bool slotmap_inside = false;   // it lies in full's CRS values, which nothing reads then
    bool crs_in_graph = false;     // a captured graph writes full's CRS values
    Laid full_laid;             // U's current values in full
    bool full_off = false;
    // FP32 mirror for IR-CG
    spmv_matrix *mirror32 = nullptr;
    CgWork cg;
};

struct spmv_split {
    spmv_handle A = nullptr;
    int32_t nblocks = 0;
    std::vector<int32_t> block_start, halo_count;
    std::vector<int64_t> nnz_local, nnz_nonlocal;
    std::vector<int32_t> h_halo_map;
    int64_t total_halo = 0;
    int32_t *d_halo_map = nullptr;
    double *d_halo = nullptr;
    spmv_handle Aloc = nullptr, Anl = nullptr;
    cudaEvent_t ev_x = nullptr, ev_halo = nullptr;
    // vector mode: the whole matrix with each nonlocal column renumbered to
    // n + (its position in the concatenated halo), applied to xe = [x | halo]
    spmv_handle Avec = nullptr;
    double *d_xe = nullptr;
};

struct spmv_batch {
    int32_t count = 0;
    int vk = kF64;
    int device = 0;
    std::vector<spmv_handle> mats;
    TileTable tiles;
    ChunkTable chunks;
    int E = 16;
    int grid = 0;
    MatRef *d_mats = nullptr;
    std::vector<MatRef> h_mats;
    int32_t *d_err = nullptr;
    std::vector<const void *> cur_x;
    std::vector<void *> cur_y;
    double cur_alpha = 0.0, cur_beta = 0.0;
    bool graph_valid = false;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    // slot-major path: one copy of all matrices (chunks of matrix m start at
    // slot_off[m]), the matrix of each chunk, and the member values versions the
    // copy was laid out from
    bool use_slots = false;
    SlotTable slots;
    int32_t *d_scmat = nullptr;
    std::vector<int32_t> slot_off;
    std::vector<uint64_t> vals_ver;
    // members tuned apart: member m runs with member_E[m] entries per lane; when
    // both 7 and 9 occur, `slots` holds the E = 7 members and `slots9` the E = 9
    // ones (slot_off[m]: the member's first chunk in its group's copy)
    bool mixed = false;
    std::vector<int32_t> member_E;
    std::vector<int32_t> slot_cnt;  // chunks of each member (mixed batches)
    SlotTable slots9;
    int32_t *d_scmat9 = nullptr;
    // members on diagonal row slices (member_E 0): the slices in launch order, the
    // members' tables (structure from the handles' copies, values in d_dvals, member
    // m's from byte dval_off[m])
    int2 *d_dlist = nullptr;
    SellMember *d_dmembers = nullptr;
    char *d_dvals = nullptr;
    std::vector<int64_t> dval_off;
    int32_t n_dlist = 0;
};

namespace {

TileTable *get_table(spmv_matrix *h, int cap, int rowcap, bool transposed) {
    auto &tabs = transposed ? h->tablesT : h->tables;
    auto key = std::make_pair(cap, rowcap);
    auto it = tabs.find(key);
    if (it != tabs.end()) return &it->second;
    TileTable tt;
    const std::vector<int32_t> &rp = transposed ? h->h_rowT : h->h_rp;
    const int32_t nr = transposed ? h->n_cols : h->n_rows;
    tt.host = make_tiles(rp.data(), nr, cap, rowcap, 0, &tt.n_long);
    tt.n = static_cast<int32_t>(tt.host.size());
    if (dmalloc(&tt.d, tt.host.size()) != cudaSuccess) return nullptr;
    if (!tt.host.empty() &&
        cudaMemcpy(tt.d, tt.host.data(), sizeof(TileDesc) * tt.host.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(tt.d);
        return nullptr;
    }
    auto res = tabs.emplace(key, std::move(tt));
    return &res.first->second;
}

void free_tables(std::map<std::pair<int, int>, TileTable> &tabs) {
    for (auto &kv : tabs) cudaFree(kv.second.d);
    tabs.clear();
}

// E values compiled for a (value, x, y, accumulator) combination, largest first.
int pick_E(int vk, int xk, int yk, int acc, int want) {
    const int cands[3] = {31, 15, 7};
    TileOps ops;
    int best = -1;
    for (int c : cands)
        if (tile_ops(vk, xk, yk, acc, 1, c, false, false, &ops)) {
            if (c == want) return c;
            if (best < 0 || std::abs(c - want) < std::abs(best - want)) best = c;
        }
    return best;
}

// Autotuner: from the row-length histogram and the column scatter choose the
// kernel and its work per lane.
//   Columns near the previous row's (stencils, banded matrices) and at least
//   12 entries per row: the sorted row-slice kernel (family 5, windows of 4096
//   rows), when its padding is at most 10 % (27-point 128^3: 113.0 against
//   139.1 us in FP64, 89.6 against 102.9 us with FP32 storage, against the best
//   chunk kernels).  With short rows it takes stencils on a grid, whose slices
//   need no column indices (k_sell_diag, kDiagMinRows); the others keep the
//   chunk kernels, which read as many bytes.
//   Scattered columns: one row per lane gathers x from as many places as the
//   slice has rows, so the slot-major chunk kernel (family 4) stays ahead
//   (Hamiltonian-like 150.4 against 167.3 us): FP64 with E = 7 entries per lane
//   for mean row lengths below 8 and E = 9 above (against the staged chunk
//   kernels 150.6 vs 196.6 us; E = 11, 13, 15 lose to 9; at 8.7 per row, the
//   split's local part, E = 9 takes the one-stream split from 245.9 to 237.1 us;
//   the 7-point matrix, 7 per row, keeps E = 7), FP32 storage with
//   E = 9 (130.2 us; E = 7 133.5, E = 11 135.9, E = 15 138.1, the staged
//   kernel 152 us).
//   Otherwise: family 4 as above for FP64, the two-stage staged chunk kernel
//   with E = 15 for FP32 storage.
// The row-vector kernel's lanes per row T (family 1) is the power of two
// nearest half the mean row length, used when chosen explicitly.
constexpr int32_t kSellSigma = 4096;
constexpr double kSellMaxPadding = 0.10;
constexpr double kSellMinRowLength = 12.0;
// FP64 matrices with shorter rows take the row slices when at least this share
// of the rows lies on the previous row's diagonals, so that nearly all slices
// are diagonal (k_sell_diag), and they are large enough to fill the GPU's warps:
// 5-point 128^2 2.4 against 2.5 us on the slot-major kernel, 256^2 3.1 against
// 3.4, 2000^2 42 against 50; 7-point 64^3 6.2 against 6.8, 160^3 55 against 68.
constexpr double kDiagMinRows = 0.9;
constexpr int32_t kDiagMinSize = 16384;
// Batched slot-major launch: each member's entries per lane from its own mean
// row length, E = 7 below this many entries per row, else 9.  The threshold is
// lower than a single matrix's (8): on the 256-matrix batch of 5-point
// Laplacians (4.9 per row) and Hamiltonian-like patterns (13 per row), giving
// the Laplacians their own E = 7 group took 0.836 ms against 0.803 ms with every
// member at E = 9 (FP32 storage: 0.660 against 0.631 ms); the whole batch at
// E = 7: 0.90 ms.  Members with shorter rows still get a group of their own.
constexpr double kBatchSlotMeanE9 = 4.0;
// Members of at least this many rows whose slices are diagonal run on them instead
// (64 5-point members of 182^2 rows: 25.5 us, 181^2 on the chunks 35.6).
constexpr int32_t kBatchDiagMinSize = 32768;

// Share of far entries (column_randomness) above which columns count as scattered.
constexpr double kScattered = 0.25;
// Entries from which a reverse pass reads A's slices: grad_x through their positions
// (rows of up to 8 entries), grad_val (spmv_backward).
constexpr int64_t kPosMinEntries = 400000, kGradValMinEntries = 2000000;
// Rows from which 2 or 3 right-hand sides run on the row slices (spmm_apply).
constexpr int32_t kRhsFew = 65536, kRhsFewScattered = 262144;

// slices = false: the row slices are not considered (their padding is not counted).
void autotune(spmv_matrix *h, bool slices = true) {
    const double mean = h->n_rows ? static_cast<double>(h->nnz) / h->n_rows : 0.0;
    const int32_t *rp = h->h_rp.data();
    int32_t longest = 0;
    for (int32_t i = 0; i < h->n_rows; ++i) longest = std::max(longest, rp[i + 1] - rp[i]);
    h->max_row = longest;
    int T = 1;
    while (T < 32 && T < mean * 0.5) T <<= 1;
    h->T = T;
    const bool scattered = h->col_random > kScattered;
    h->sigma = kSellSigma;
    h->sell_pad = slices && h->n_rows > 0 ? sell_padding(h->h_rp.data(), h->n_rows, kSellSigma) : 1.0;
    if (h->vk == kF32) {
        h->family = scattered ? 4 : 0;
        h->E = scattered ? 9 : 15;
    } else {
        h->family = 4;
        h->E = (mean < 8.0) ? 7 : 9;
    }
    const bool diagonal = h->col_diag >= kDiagMinRows && h->n_rows >= kDiagMinSize;
    const bool sells = h->vk == kF32 || mean >= kSellMinRowLength;
    if (!scattered && h->sell_pad <= kSellMaxPadding && (sells || diagonal)) {
        h->family = 5;
        h->sell_if_diag = !sells;
    }
}

// Share of entries (sampled rows) whose column is more than 8 away from every
// column of the previous row: near 0 for stencils and banded matrices, large for
// scattered patterns whose x gathers find nothing in L1.
double column_randomness(const int32_t *rp, const int32_t *col, int32_t n_rows) {
    if (!col || n_rows < 2) return 0.0;
    const int32_t step = std::max<int32_t>(1, n_rows / 32768);
    int64_t far = 0, total = 0;
    std::vector<int32_t> prev;
    for (int32_t i = 1; i < n_rows; i += step) {
        prev.assign(col + rp[i - 1], col + rp[i]);
        std::sort(prev.begin(), prev.end());
        for (int32_t k = rp[i]; k < rp[i + 1]; ++k) {
            const int32_t c = col[k];
            auto it = std::lower_bound(prev.begin(), prev.end(), c);
            int64_t best = INT64_MAX;
            if (it != prev.end()) best = static_cast<int64_t>(*it) - c;
            if (it != prev.begin()) best = std::min<int64_t>(best, static_cast<int64_t>(c) - *(it - 1));
            far += (best > 8) ? 1 : 0;
            ++total;
        }
    }
    return total ? static_cast<double>(far) / total : 0.0;
}

// Share of (sampled) rows whose entries lie on the same diagonals, in the same
// order, as the previous row's: near 1 for stencils on a grid, where a slice of
// 64 rows of one length then needs one diagonal per slot row instead of column
// indices.
double diagonal_rows(const int32_t *rp, const int32_t *col, int32_t n_rows) {
    if (!col || n_rows < 2) return 0.0;
    // (8,192 rows: with 32,768 the statistic took 9 % of spmv_create on the 27-point
    // 64^3 pattern)
    const int32_t step = std::max<int32_t>(1, n_rows / 8192) | 1;  // odd: no grid line is sampled alone
    int64_t same = 0, total = 0;
    for (int32_t i = 1; i < n_rows; i += step) {
        const int32_t len = rp[i + 1] - rp[i];
        bool eq = len > 0 && len == rp[i] - rp[i - 1];
        for (int32_t k = 0; eq && k < len; ++k) eq = col[rp[i] + k] - col[rp[i - 1] + k] == 1;
        same += eq ? 1 : 0;
        ++total;
    }
    return total ? static_cast<double>(same) / total : 0.0;
}

ChunkTable *get_chunks(spmv_matrix *h, int E, bool transposed) {
    auto &tabs = transposed ? h->chunksT : h->chunks;
    auto it = tabs.find(E);
    if (it != tabs.end()) return &it->second;
    std::vector<ChunkDesc> d;
    std::vector<uint32_t> m;
    ChunkTable ct;
    const std::vector<int32_t> &rp = transposed ? h->h_rowT : h->h_rp;
    const int32_t nr = transposed ? h->n_cols : h->n_rows;
    make_chunks(rp.data(), nr, E, 0, d, m, nullptr, &ct.n_long, &ct.n_empty);
    if (upload_chunks(&ct, d, m, nullptr) != SPMV_OK) {
        free_chunks(ct);
        return nullptr;
    }
    return &tabs.emplace(E, ct).first->second;
}

// The slot-major copy for E (built on first use; its values are laid out again
// on the stream after spmv_set_values).  transposed: the copy of A^T, from the
// transposed structure and the values laid out in A^T order (d_valT).
SlotTable *get_slots(spmv_matrix *h, int E, cudaStream_t s, bool transposed = false) {
    auto &tabs = transposed ? h->slotsT : h->slots;
    const int32_t *d_col = transposed ? h->d_colT : h->d_col;
    const void *d_val = transposed ? h->d_valT : h->d_val;
    auto it = tabs.find(E);
    if (it == tabs.end()) {
        if (capture_id(s)) return nullptr;  // its columns would be laid out by the graph
        std::vector<ChunkDesc> d;
        std::vector<uint32_t> lm;
        SlotTable t;
        if (transposed)
            make_slot_chunks(h->h_rowT.data(), h->n_cols, E, d, lm, &t.n_long, &t.n_empty);
        else
            make_slot_chunks(h->h_rp.data(), h->n_rows, E, d, lm, &t.n_long, &t.n_empty);
        t.n = static_cast<int32_t>(d.size());
        const size_t nslots = static_cast<size_t>(t.n) * 32 * E;
        const size_t vb = (h->vk == kF64) ? 8 : 4;
        bool ok;
        if (nslots * vb + 16 < (size_t(1) << 20)) {
            ok = dmalloc(&t.d, d.size()) == cudaSuccess && dmalloc(&t.lmask, lm.size()) == cudaSuccess &&
                 cudaMalloc(&t.vals, nslots * vb + 16) == cudaSuccess && dmalloc(&t.cols, nslots + 4) == cudaSuccess;
        } else {
            Block b;
            b.add(sizeof(ChunkDesc) * d.size());
            b.add(4 * lm.size());
            b.add(nslots * vb + 16);
            b.add(4 * (nslots + 4));
            ok = b.alloc();
            if (ok) {
                t.block = b.base;
                b.take(&t.d);
                b.take(&t.lmask);
                b.take(&t.vals);
                b.take(&t.cols);
            }
        }
        ok = ok && (d.empty() || cudaMemcpy(t.d, d.data(), sizeof(ChunkDesc) * d.size(), cudaMemcpyHostToDevice) ==
                                     cudaSuccess);
        ok = ok && (lm.empty() || cudaMemcpy(t.lmask, lm.data(), 4 * lm.size(), cudaMemcpyHostToDevice) == cudaSuccess);
        // (waited for: the next product may run on another stream)
        ok = ok && launch_slot_relayout(t.d, E, static_cast<int64_t>(nslots), h->vk, d_val, d_col, t.vals, t.cols,
                                        s) == cudaSuccess &&
             cudaStreamSynchronize(s) == cudaSuccess;
        if (!ok) {
            free_slots(t);
            (void)cudaGetLastError();  // a failed allocation must not surface at a later launch check
            return nullptr;
        }
        t.laid.now = true;
        it = tabs.emplace(E, t).first;
    }
    SlotTable &t = it->second;
    if (!t.laid.on(s)) {
        if (launch_slot_relayout(t.d, E, static_cast<int64_t>(t.n) * 32 * E, h->vk, d_val, nullptr, t.vals,
                                 nullptr, s) != cudaSuccess)
            return nullptr;
        t.laid.set(s);
    }
    return &t;
}

// Fewer rows than this: the host sorts them faster than six launches and a read-back take
// (27-point 12^3, first product: 102 against 131 us).
constexpr int32_t kSellHostRows = 8192;

// The tables of a row-slice copy built on the device, in one allocation, when the
// window is the default and no row is long; *done tells whether they were.  Waits for
// s.  (The 2.1 M-row scattered matrix: first block product 12.6 -> 1.4 ms; first
// training step on the 27-point 128^3 pattern 37 -> 5.3 ms.)
bool build_sell(SellTable &t, const int32_t *d_rp, int32_t n_rows, int32_t sigma, bool *done, cudaStream_t s) {
    static_assert(kSellBuildSigma == kSellSigma && kSellBuildMaxRow == kSellLongRow, "the device's tables");
    *done = false;
    if (sigma != kSellBuildSigma) return true;
    const size_t n = static_cast<size_t>(t.n);
    // dtmp, dorder, d, srows, cstart + counts, width, off, sums, flag
    const size_t o_out = sizeof(int4) * n, o_d = 2 * o_out, o_sr = o_d + sizeof(int2) * n,
                 o_ws = o_sr + 4 * n * kSellC, o_wd = o_ws + 4 * (static_cast<size_t>(t.n_ctas) + 3), o_off = o_wd + 4 * n,
                 o_sum = o_off + 4 * (n + 1), o_flag = o_sum + 4 * static_cast<size_t>(scan_sums_len(t.n));
    if (cudaMalloc(&t.meta, o_flag + 4) != cudaSuccess) {
        t.meta = nullptr;
        return false;
    }
    char *m = static_cast<char *>(t.meta);
    t.dtmp = reinterpret_cast<int4 *>(m);
    t.dorder = reinterpret_cast<int4 *>(m + o_out);
    t.d = reinterpret_cast<int2 *>(m + o_d);
    t.srows = reinterpret_cast<int32_t *>(m + o_sr);
    t.cstart = reinterpret_cast<int32_t *>(m + o_ws);
    int32_t *off = reinterpret_cast<int32_t *>(m + o_off);
    uint32_t *flag = reinterpret_cast<uint32_t *>(m + o_flag);
    uint32_t too_long = 0;
    int32_t rows = 0;
    if (cudaMemsetAsync(m + o_ws, 0, 4 * (static_cast<size_t>(t.n_ctas) + 3), s) != cudaSuccess ||
        cudaMemsetAsync(flag, 0, 4, s) != cudaSuccess ||
        launch_sell_build(d_rp, n_rows, t.n, t.n_ctas, t.srows, reinterpret_cast<int32_t *>(m + o_wd), off,
                          reinterpret_cast<int32_t *>(m + o_sum), flag, t.d, t.dtmp, t.cstart, s) != cudaSuccess ||
        cudaMemcpyAsync(&too_long, flag, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&rows, off + n, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return false;
    if (too_long) {
        cudaFree(t.meta);
        t.meta = nullptr;
        return true;
    }
    t.slot_rows = static_cast<int64_t>(rows) + kSellU;
    *done = true;
    return true;
}

// The tables of a row-slice copy from the host (descriptors, rows, CTA ranges, places
// of the diagonals) in one allocation and one copy on s.
bool upload_sell(SellTable &t, const std::vector<int2> &d, const std::vector<int32_t> &sr,
                 const std::vector<int32_t> &ws, cudaStream_t s) {
    std::vector<int4> order(d.size());
    int packed = 0;
    for (size_t i = 0; i < d.size(); ++i) {
        order[i] = make_int4(d[i].x, d[i].y, static_cast<int>(i), packed);
        packed += d[i].y > 0 ? (d[i].y + 3) / 4 : 0;
    }
    const size_t o_order = 0, o_d = o_order + sizeof(int4) * order.size(), o_sr = o_d + sizeof(int2) * d.size(),
                 o_ws = o_sr + 4 * sr.size(), host_end = o_ws + 4 * ws.size() + 8, o_out = (host_end + 15) / 16 * 16;
    std::vector<char> host(host_end, 0);  // the last two words: the marking's counts
    if (!d.empty()) {
        std::memcpy(host.data() + o_order, order.data(), sizeof(int4) * order.size());
        std::memcpy(host.data() + o_d, d.data(), sizeof(int2) * d.size());
        std::memcpy(host.data() + o_sr, sr.data(), 4 * sr.size());
    }
    std::memcpy(host.data() + o_ws, ws.data(), 4 * ws.size());
    if (cudaMalloc(&t.meta, o_out + sizeof(int4) * order.size()) != cudaSuccess) {
        t.meta = nullptr;
        return false;
    }
    char *m = static_cast<char *>(t.meta);
    t.dtmp = reinterpret_cast<int4 *>(m + o_order);
    t.dorder = reinterpret_cast<int4 *>(m + o_out);
    t.d = reinterpret_cast<int2 *>(m + o_d);
    t.srows = reinterpret_cast<int32_t *>(m + o_sr);
    t.cstart = reinterpret_cast<int32_t *>(m + o_ws);
    return cudaMemcpyAsync(m, host.data(), host.size(), cudaMemcpyHostToDevice, s) == cudaSuccess;
}

// Marks the diagonal slices of a row-slice copy whose columns are laid out on s:
// the diagonals into diag, the descriptors in launch order into dorder.  Waits
// for s; false on an error.
bool mark_diagonals(SellTable &t, cudaStream_t s) {
    if (t.n == 0) return true;
    uint32_t *count = reinterpret_cast<uint32_t *>(t.cstart + t.n_ctas + 1);  // [0]: slot rows of diagonal slices
    uint32_t in = 0;
    if (launch_sell_mark_diag(t.dtmp, t.n, t.srows, t.cols, t.diag, count, t.dorder, s) != cudaSuccess ||
        cudaMemcpyAsync(&in, count, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return false;
    const double all = static_cast<double>(t.slot_rows - kSellU) + static_cast<double>(t.n_long) * kSellLongRow;
    t.diagonal = in > 0 && static_cast<double>(in) >= kDiagMinShare * all;
    return true;
}

// The sorted row-slice copy for window sigma (built on first use; its values are
// laid out again on the stream after spmv_set_values).  transposed: the copy of
// A^T, from the transposed structure and the values laid out in A^T order.
// need_vals: false for a copy whose own values are not used (yet).
SellTable *get_sell(spmv_matrix *h, int32_t sigma, cudaStream_t s, bool transposed = false, bool need_vals = true) {
    auto &tabs = transposed ? h->sellsT : h->sells;
    const int32_t *h_rp = transposed ? h->h_rowT.data() : h->h_rp.data();
    const int32_t nr = transposed ? h->n_cols : h->n_rows;
    const int32_t *d_rp = transposed ? h->d_rowT : h->d_rp;
    const int32_t *d_col = transposed ? h->d_colT : h->d_col;
    const void *d_val = transposed ? h->d_valT : h->d_val;
    const size_t vb = (h->vk == kF64) ? 8 : 4;
    auto alloc_vals = [&](SellTable &t) {
        const size_t nslots = static_cast<size_t>(t.slot_rows) * kSellC;
        if (cudaMalloc(&t.vals, nslots * vb + 16) != cudaSuccess) {
            t.vals = nullptr;
            return false;
        }
        return cudaMemsetAsync(t.vals, 0, static_cast<size_t>(kSellU) * kSellC * vb, s) == cudaSuccess;
    };
    auto it = tabs.find(sigma);
    if ((it == tabs.end() || (need_vals && !it->second.vals)) && capture_id(s)) return nullptr;  // nothing is built
    if (it == tabs.end()) {
        SellTable t;
        SellOps o;
        const int acc = (h->vk == kF32) ? kAccFF : kAccF64;
        if (!sell_ops(h->vk, h->vk, h->vk, acc, &o, transposed ? 0x7fffffff : h->max_row)) return nullptr;
        // on the device (slices of a window without long rows), else on the host
        t.n = static_cast<int32_t>((static_cast<int64_t>(nr) + kSellC - 1) / kSellC);
        t.n_ctas = o.ctas_for(t.n);
        if (t.n_ctas <= 0) return nullptr;
        bool done = false;
        bool ok = nr < kSellHostRows || (!transposed && h->max_row > kSellLongRow) ||
                  build_sell(t, d_rp, nr, sigma, &done, s);
        if (ok && !done) {
            std::vector<int2> d;
            std::vector<int32_t> sr, ws;
            if (!make_sell_slices(h_rp, nr, sigma, d, sr, &t.n_long, &t.slot_rows)) return nullptr;
            t.n = static_cast<int32_t>(d.size());
            t.n_ctas = o.ctas_for(t.n);
            sell_ranges(d, h_rp, t.n_ctas, ws);
            ok = t.n_ctas > 0 && upload_sell(t, d, sr, ws, s);
        }
        // the diagonals (places up to slot_rows / 4 + n on either path) follow the columns
        const size_t nslots = static_cast<size_t>(t.slot_rows) * kSellC;
        const size_t ndiag = static_cast<size_t>(t.slot_rows) / 4 + static_cast<size_t>(t.n) + 2;
        ok = ok && dmalloc(&t.cols, (nslots + 4) + 4 * ndiag) == cudaSuccess;
        if (ok) t.diag = reinterpret_cast<int4 *>(t.cols + nslots + 4);
        ok = ok && cudaMemsetAsync(t.diag, 0, sizeof(int4) * ndiag, s) == cudaSuccess;
        ok = ok && (!need_vals || alloc_vals(t));
        // the leading padding rows: column -1 (and value 0)
        ok = ok && cudaMemsetAsync(t.cols, 0xff, static_cast<size_t>(kSellU) * kSellC * 4, s) == cudaSuccess;
        ok = ok && launch_sell_relayout(t.d, t.srows, t.n, d_rp, h->vk, d_val, d_col, t.vals, t.cols, s) == cudaSuccess;
        ok = ok && mark_diagonals(t, s);
        if (!ok) {
            free_sell(t);
            (void)cudaGetLastError();  // a failed allocation must not surface at a later launch check
            return nullptr;
        }
        t.laid.now = need_vals;
        it = tabs.emplace(sigma, t).first;
    }
    SellTable &t = it->second;
    if (need_vals && !t.laid.on(s)) {
        if (!t.vals && !alloc_vals(t)) {
            (void)cudaGetLastError();
            return nullptr;
        }
        if (launch_sell_relayout(t.d, t.srows, t.n, d_rp, h->vk, d_val, nullptr, t.vals, nullptr, s) != cudaSuccess)
            return nullptr;
        t.laid.set(s);
    }
    t.read = t.read || need_vals;
    return &t;
}

// The slices of A^T with the positions of their values in A's row-slice copy (null
// when A does not run on diagonal slices, its copy is not there, or A has rows
// outside the slices): what a reverse pass on new values reads.
SellTable *get_sell_positions(spmv_matrix *h, cudaStream_t s) {
    auto f = h->sells.find(h->sigma);
    if (h->family != 5 || f == h->sells.end()) return nullptr;
    const SellTable &a = f->second;
    if (!a.diagonal || a.n_long > 0 || a.slot_rows * kSellC > INT32_MAX) return nullptr;
    SellTable *t = get_sell(h, kSellSigma, s, true, false);
    if (!t || !t->diagonal) return nullptr;
    if (t->vpos.count(h->sigma)) return t;
    if (capture_id(s)) return nullptr;  // nothing is built
    const size_t nslots = (static_cast<size_t>(t->slot_rows) * kSellC + 7) / 4 * 4;
    int32_t *vpos = nullptr;  // and behind it a work array, kept: freeing it would wait once more
    bool ok = dmalloc(&vpos, nslots + static_cast<size_t>(h->n_rows)) == cudaSuccess;
    int32_t *rowpos = ok ? vpos + nslots : nullptr;
    ok = ok && cudaMemsetAsync(vpos, 0xff, static_cast<size_t>(kSellU) * kSellC * 4, s) == cudaSuccess &&
         launch_sell_vpos(a.d, a.srows, a.n, t->d, t->srows, t->n, h->d_rp, h->d_rowT, h->d_colT, h->d_perm, rowpos,
                          vpos, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
    if (!ok) {
        cudaFree(vpos);
        (void)cudaGetLastError();
        return nullptr;
    }
    t->vpos[h->sigma] = vpos;
    return t;
}

// Whether every row fits the tile kernels (k_sell_set_values, k_sell_grad_val).
bool sell_tile_fits(const spmv_matrix *h) { return h->max_row <= sell_tile_max_row() && h->nnz < INT32_MAX - 64; }

// The launch parameters of a row-slice copy of the matrix m.
SellParams sell_params(const SellTable &t, const MatRef &m, double alpha, double beta) {
    SellParams p{};
    p.slices = t.d;
    p.srows = t.srows;
    p.cstart = t.cstart;
    p.n_ctas = t.n_ctas;
    p.vals = t.vals;
    p.cols = t.cols;
    p.m = m;
    p.n_slices = t.n;
    p.alpha = alpha;
    p.beta = beta;
    p.ff = epi_ff(alpha, beta);
    p.dorder = t.diagonal ? t.dorder : nullptr;
    p.diag = t.diag;
    p.dshort = t.slot_rows <= 8LL * t.n;
    return p;
}

void free_chunk_map(std::map<int, ChunkTable> &tabs) {
    for (auto &kv : tabs) free_chunks(kv.second);
    tabs.clear();
}

spmv_status upload_matrix(spmv_matrix *h, const int32_t *row_ptr, const int32_t *col_idx,
                          const void *val, int val_t, bool dev_ptrs, cudaStream_t s) {
    const size_t vsz = (h->vk == kF64) ? 8 : 4;
    const size_t nrp = static_cast<size_t>(h->n_rows) + 1 + kRowPad;
    const size_t nent = static_cast<size_t>(h->nnz) + kEntryPad;
    if (dmalloc(&h->d_rp, nrp) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (dmalloc(&h->d_col, nent) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (cudaMalloc(&h->d_val, nent * vsz) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (dmalloc(&h->d_err, 1) != cudaSuccess) return SPMV_ERR_ALLOC;
    CK(cudaMemsetAsync(h->d_err, 0, sizeof(int32_t), s));
    CK(cudaMemsetAsync(h->d_rp, 0, nrp * 4, s));
    CK(cudaMemsetAsync(h->d_col, 0, nent * 4, s));
    CK(cudaMemsetAsync(h->d_val, 0, nent * vsz, s));
    CK(cudaMemcpyAsync(h->d_rp, h->h_rp.data(), (static_cast<size_t>(h->n_rows) + 1) * 4,
                       cudaMemcpyHostToDevice, s));
    const cudaMemcpyKind kind = dev_ptrs ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    if (h->nnz > 0) {
        CK(cudaMemcpyAsync(h->d_col, col_idx, static_cast<size_t>(h->nnz) * 4, kind, s));
        if (val_t == h->vk) {
            CK(cudaMemcpyAsync(h->d_val, val, static_cast<size_t>(h->nnz) * vsz, kind, s));
        } else {
            // convert on the device through a staging buffer
            void *tmp = nullptr;
            const size_t tsz = static_cast<size_t>(h->nnz) * (val_t == kF64 ? 8 : 4);
            if (cudaMalloc(&tmp, tsz) != cudaSuccess) return SPMV_ERR_ALLOC;
            cudaError_t e = cudaMemcpyAsync(tmp, val, tsz, kind, s);
            if (e == cudaSuccess) e = launch_convert(tmp, val_t, h->d_val, h->vk, h->nnz, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            cudaFree(tmp);
            if (e != cudaSuccess) return SPMV_ERR_CUDA;
        }
    }
    (void)row_ptr;
    CK(cudaStreamSynchronize(s));
    return SPMV_OK;
}

void destroy_cg(CgWork &w) {
    if (w.inner32) cudaGraphExecDestroy(w.inner32);
    if (w.cg64) cudaGraphExecDestroy(w.cg64);
    cudaFree(w.r64); cudaFree(w.p64); cudaFree(w.q64);
    cudaFree(w.r32); cudaFree(w.d32); cudaFree(w.p32); cudaFree(w.q32);
    cudaFree(w.sc); cudaFree(w.partials); cudaFree(w.one);
    if (w.host) cudaFreeHost(w.host);
    w = CgWork();
}

void destroy_matrix(spmv_matrix *h) {
    if (!h) return;
    DeviceGuard g(h->device);
    cudaDeviceSynchronize();
    if (h->block) {
        cudaFree(h->block);
    } else {
        if (h->owns_structure) {
            cudaFree(h->d_rp);
            cudaFree(h->d_col);
        }
        cudaFree(h->d_val);
        cudaFree(h->d_err);
    }
    cudaFree(h->d_rowT);
    cudaFree(h->d_colT);
    cudaFree(h->d_perm);
    cudaFree(h->d_valT);
    free_tables(h->tables);
    free_tables(h->tablesT);
    free_chunk_map(h->chunks);
    free_chunk_map(h->chunksT);
    for (auto &kv : h->slots) free_slots(kv.second);
    for (auto &kv : h->slotsT) free_slots(kv.second);
    for (auto &kv : h->sells) free_sell(kv.second);
    for (auto &kv : h->sellsT) free_sell(kv.second);
    cudaFree(h->d_rmap);
    destroy_cg(h->cg);
    if (h->mirror32) destroy_matrix(h->mirror32);
    if (h->full) destroy_matrix(h->full);
    if (!h->slotmap_inside) cudaFree(h->d_slotmap);
    delete h;
}

spmv_status create_from_host(spmv_handle *out, int32_t n_rows, int32_t n_cols, int64_t nnz,
                             std::vector<int32_t> &&h_rp, const int32_t *col_idx, const void *val,
                             int val_t, int store_t, bool dev_ptrs, cudaStream_t s,
                             const int32_t *host_col) {
    spmv_matrix *h = new (std::nothrow) spmv_matrix();
    if (!h) return SPMV_ERR_ALLOC;
    cudaGetDevice(&h->device);
    h->n_rows = n_rows;
    h->n_cols = n_cols;
    h->nnz = nnz;
    h->vk = store_t;
    h->h_rp = std::move(h_rp);
    h->col_random = column_randomness(h->h_rp.data(), host_col, n_rows);
    h->col_diag = diagonal_rows(h->h_rp.data(), host_col, n_rows);
    spmv_status st = upload_matrix(h, nullptr, col_idx, val, val_t, dev_ptrs, s);
    if (st != SPMV_OK) {
        destroy_matrix(h);
        return st;
    }
    autotune(h);
    *out = h;
    return SPMV_OK;
}

spmv_status validate_host(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t *rp,
                          const int32_t *col) {
    if (rp[0] != 0) return SPMV_ERR_INVALID_INDEX;
    for (int32_t i = 0; i < n_rows; ++i)
        if (rp[i + 1] < rp[i]) return SPMV_ERR_INVALID_INDEX;
    if (rp[n_rows] != nnz) return SPMV_ERR_INVALID_INDEX;
    for (int64_t k = 0; k < nnz; ++k)
        if (col[k] < 0 || col[k] >= n_cols) return SPMV_ERR_INVALID_INDEX;
    return SPMV_OK;
}

struct TileRun {
    TileOps ops;
    TileTable *tt;
    int grid;
};

// Select the compiled kernel and tile table for an apply of h with group width R.
spmv_status prepare_run(spmv_matrix *h, int xk, int yk, int R, int E, bool transposed, TileRun *run) {
    const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
    if (!tile_ops(h->vk, xk, yk, acc, R, E, transposed, false, &run->ops)) return SPMV_ERR_UNSUPPORTED;
    const TileCfg c = run->ops.cfg();
    run->tt = get_table(h, c.cap, c.rowcap, transposed);
    if (!run->tt) return SPMV_ERR_ALLOC;
    const int lim = run->ops.grid_limit();
    if (lim <= 0) return SPMV_ERR_CUDA;
    run->grid = std::min<int>(run->tt->n, lim);
    return SPMV_OK;
}

// A plan taken for its diagonal slices only (sell_if_diag), from a sample of the rows,
// is settled when the slices are known: too few diagonal ones, and the handle runs on
// the slot-major kernel and gives the copy back, unless other calls had built it.
void settle_plan(spmv_matrix *h, cudaStream_t s) {
    if (!h->sell_if_diag) return;
    const bool had = h->sells.count(h->sigma) != 0;
    const SellTable *t = get_sell(h, h->sigma, s, false, false);
    if (!t) return;  // not built now: asked again by the next call
    h->sell_if_diag = false;
    if (t->diagonal) return;
    h->family = 4;  // E as the tuner chose it
    if (had) return;
    free_sell(h->sells[h->sigma]);
    h->sells.erase(h->sigma);
}

// The row-slice launch of h for these operands (plan family 5, no row map):
// its compiled configuration and parameters, with the slice copy built on first
// use; false when h does not run on the row slices here.
bool sell_launch_of(spmv_matrix *h, double alpha, const void *x, int xk, double beta, void *y, int yk,
                    cudaStream_t s, SellOps *ops, SellParams *lp) {
    if (h->family != 5 || h->d_rmap) return false;
    settle_plan(h, s);
    if (h->family != 5 || h->sell_if_diag) return false;
    const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
    SellTable *lt = nullptr;
    if (!sell_ops(h->vk, xk, yk, acc, ops, h->max_row) || (lt = get_sell(h, h->sigma, s)) == nullptr) return false;
    *lp = sell_params(*lt, MatRef{h->d_rp, h->d_col, h->d_val, nullptr, x, y, nullptr}, alpha, beta);
    return true;
}

spmv_status apply_impl(spmv_matrix *h, double alpha, const void *x, int xk, double beta, void *y,
                       int yk, cudaStream_t s) {
    if (h->n_rows == 0) return SPMV_OK;
    const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
    {
        SellOps lops;
        SellParams lp;
        if (sell_launch_of(h, alpha, x, xk, beta, y, yk, s, &lops, &lp))
            return lops.launch(lp, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    }
    if (h->family == 6 && !h->d_rmap) {
        SlotOps tops;
        SlotTable *tt = nullptr;
        if (slot_ops_tv(h->vk, xk, yk, acc, h->E, &tops) && (tt = get_slots(h, h->E, s)) != nullptr) {
            SlotParams sp{};
            sp.chunks = tt->d;
            sp.lmask = tt->lmask;
            sp.vals = tt->vals;
            sp.cols = tt->cols;
            sp.m = MatRef{h->d_rp, h->d_col, h->d_val, nullptr, x, y, nullptr};
            sp.n_chunks = tt->n;
            sp.alpha = alpha;
            sp.beta = beta;
            sp.ff = epi_ff(alpha, beta);
            sp.err = h->d_err;
            return tops.launch(sp, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
        }
    }
    SlotOps sops;
    SlotTable *t = nullptr;
    if ((h->family == 4 || h->family == 5 || h->family == 6) &&
        (!h->d_rmap || beta == 1.0) &&  // the row-mapped form adds to y
        slot_ops(h->vk, xk, yk, acc, h->E, h->d_rmap != nullptr, &sops) &&
        (t = get_slots(h, h->E, s)) != nullptr) {
        SlotParams sp{};
        sp.chunks = t->d;
        sp.lmask = t->lmask;
        sp.vals = t->vals;
        sp.cols = t->cols;
        sp.m = MatRef{h->d_rp, h->d_col, h->d_val, nullptr, x, y, h->d_rmap};
        if (h->map_of && t->n_long == 0 && t->n_empty == 0) {
            sp.m.vs = h->map_of;
            sp.m.vind = h->val_of;
        }
        sp.n_chunks = t->n;
        sp.alpha = alpha;
        sp.beta = beta;
        sp.ff = epi_ff(alpha, beta);
        sp.err = h->d_err;
        return sops.launch(sp, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    }
    // the staged chunk kernels (also families 4 and 5 in the vector and
    // accumulator combinations their kernels are not compiled for, FP32 storage
    // with an FP64 result or FP64 accumulation, and when their copies could not
    // be allocated)
    if (h->family == 0 || h->family == 3 || h->family == 4 || h->family == 5 || h->family == 6 || h->d_rmap) {
        int E = h->E;
        if ((h->family == 4 || h->family == 5 || h->family == 6) && E != 7 && E != 15) E = 15;
        WarpOps ops;
        // family 3 selects the three-stage kernel of the same chunking
        const bool ok3 = h->family == 3 && warp_ops(h->vk, xk, yk, acc, E + 100, false, false, &ops);
        if (!ok3 && !warp_ops(h->vk, xk, yk, acc, E, false, false, &ops)) {
            E = 16;
            if (!warp_ops(h->vk, xk, yk, acc, E, false, false, &ops)) return SPMV_ERR_UNSUPPORTED;
        }
        ChunkTable *ct = get_chunks(h, E, false);
        if (!ct) return SPMV_ERR_ALLOC;
        WarpParams wp{};
        wp.m = MatRef{h->d_rp, h->d_col, h->d_val, nullptr, x, y, h->d_rmap};
        wp.chunks = ct->d;
        wp.masks = ct->masks;
        wp.n_chunks = ct->n;
        wp.alpha = alpha;
        wp.beta = beta;
        wp.err = h->d_err;
        return ops.launch(wp, ct->n, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    }
    KParams p{};
    p.m = MatRef{h->d_rp, h->d_col, h->d_val, nullptr, x, y, nullptr};
    p.rhs_count = 1;
    p.ldx = 1;
    p.ldy = 1;
    p.alpha = alpha;
    p.beta = beta;
    p.err = h->d_err;
    if (h->family == 1) {
        return launch_rowvec(p, h->n_rows, h->vk, xk, yk, acc, h->T, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    }
    int E = pick_E(h->vk, xk, yk, acc, h->E);
    if (E < 0) return SPMV_ERR_UNSUPPORTED;
    TileRun run;
    spmv_status st = prepare_run(h, xk, yk, 1, E, false, &run);
    if (st != SPMV_OK) return st;
    p.tiles = run.tt->d;
    p.n_tiles = run.tt->n;
    return run.ops.launch(p, run.grid, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
}

spmv_status ensure_transpose(spmv_matrix *h, cudaStream_t s) {
    if (h->has_T) return SPMV_OK;
    const size_t nT = static_cast<size_t>(h->n_cols) + 1 + kRowPad;
    const size_t nent = static_cast<size_t>(h->nnz) + kEntryPad;
    if (dmalloc(&h->d_rowT, nT) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (dmalloc(&h->d_colT, nent) != cudaSuccess) return SPMV_ERR_ALLOC;
    if (dmalloc(&h->d_perm, nent) != cudaSuccess) return SPMV_ERR_ALLOC;
    int32_t *work = nullptr;
    if (dmalloc(&work, static_cast<size_t>(transpose_work_len(h->n_cols))) != cudaSuccess) return SPMV_ERR_ALLOC;
    cudaError_t e = cudaMemsetAsync(h->d_rowT, 0, nT * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_colT, 0, nent * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_perm, 0, nent * 4, s);
    if (e == cudaSuccess)
        e = launch_transpose(h->n_rows, h->n_cols, h->nnz, h->d_rp, h->d_col, h->d_rowT, h->d_colT,
                             h->d_perm, work, s);
    h->h_rowT.assign(static_cast<size_t>(h->n_cols) + 1, 0);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h->h_rowT.data(), h->d_rowT, h->h_rowT.size() * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(work);
    if (e != cudaSuccess) return SPMV_ERR_CUDA;
    h->has_T = true;
    return SPMV_OK;
}

spmv_status ensure_cg(spmv_matrix *h, bool mixed) {
    CgWork &w = h->cg;
    const int64_t n = h->n_rows;
    if (w.sc == nullptr) {
        w.n = n;
        if (dmalloc(&w.sc, kScCount) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.partials, static_cast<size_t>(cg_partials_len())) != cudaSuccess) return SPMV_ERR_ALLOC;
        // the reductions' ticket word (after the partials) starts at zero
        if (cudaMemset(w.partials, 0, static_cast<size_t>(cg_partials_len()) * 8) != cudaSuccess) return SPMV_ERR_CUDA;
        if (cudaMallocHost(reinterpret_cast<void **>(&w.host), 8 * sizeof(double)) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.r64, n) != cudaSuccess) return SPMV_ERR_ALLOC;
        CK(cudaDeviceGetAttribute(&w.one_ctas, cudaDevAttrMultiProcessorCount, h->device));
        if (dmalloc(&w.one, 4 * static_cast<size_t>(w.one_ctas) + 4) != cudaSuccess) return SPMV_ERR_ALLOC;
    }
    if (!mixed && w.p64 == nullptr) {
        if (dmalloc(&w.p64, n) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.q64, n) != cudaSuccess) return SPMV_ERR_ALLOC;
    }
    if (mixed && w.r32 == nullptr) {
        if (dmalloc(&w.r32, n) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.d32, n) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.p32, n) != cudaSuccess) return SPMV_ERR_ALLOC;
        if (dmalloc(&w.q32, n) != cudaSuccess) return SPMV_ERR_ALLOC;
    }
    return SPMV_OK;
}

spmv_status ensure_mirror32(spmv_matrix *h, cudaStream_t s) {
    if (h->vk == kF32) return SPMV_OK;
    if (h->mirror32) return SPMV_OK;
    spmv_matrix *m = new (std::nothrow) spmv_matrix();
    if (!m) return SPMV_ERR_ALLOC;
    m->device = h->device;
    m->n_rows = h->n_rows;
    m->n_cols = h->n_cols;
    m->nnz = h->nnz;
    m->vk = kF32;
    m->owns_structure = false;
    m->d_rp = h->d_rp;
    m->d_col = h->d_col;
    m->h_rp = h->h_rp;
    m->col_random = h->col_random;
    m->col_diag = h->col_diag;
    const size_t nent = static_cast<size_t>(h->nnz) + kEntryPad;
    if (cudaMalloc(&m->d_val, nent * 4) != cudaSuccess || dmalloc(&m->d_err, 1) != cudaSuccess) {
        destroy_matrix(m);
        return SPMV_ERR_ALLOC;
    }
    cudaError_t e = cudaMemsetAsync(m->d_val, 0, nent * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->d_err, 0, 4, s);
    if (e == cudaSuccess) e = launch_convert(h->d_val, kF64, m->d_val, kF32, h->nnz, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        destroy_matrix(m);
        return SPMV_ERR_CUDA;
    }
    autotune(m);
    h->mirror32 = m;
    return SPMV_OK;
}

}  // namespace

// CG on h as one cooperative kernel (launch_cg), when h runs on diagonal row slices
// (by the tuner, whatever its size) and the vectors of a CTA's rows fit in shared
// memory.  res: rho, iterations, b.b.  SPMV_ERR_UNSUPPORTED: not this matrix.
// SPMV_ERR_TIMEOUT: a grid barrier gave up (the GPU taken away for a second between two
// barriers), and x, dir, dir2 and r are void; the callers solve on the other path then.
// work: the CG work array of the handle that runs the solve (its partials).
static spmv_status cg_in_one_kernel(spmv_matrix *h, CgWork &w, const void *b, void *x, void *dir, void *dir2, void *r,
                                    double tol, int32_t max_iter, double *res, cudaStream_t s) {
    const bool grid_like = h->col_diag >= kDiagMinShare && h->sell_pad <= kSellMaxPadding && h->acc32 == kAccFF;
    if (h->n_rows == 0 || h->max_row > kSellLongRow || h->d_rmap ||
        !(h->planned ? h->family == 5 && h->sigma == kSellSigma : grid_like))
        return SPMV_ERR_UNSUPPORTED;
    const int32_t few = (h->n_rows + kSellC - 1) / kSellC;  // at least this many slices
    if (!cg_kernel_fits(h->vk, few, h->max_row)) return SPMV_ERR_UNSUPPORTED;
    SellTable *t = get_sell(h, kSellSigma, s, false, false);
    if (!t || !t->diagonal || t->n_long > 0 || !cg_kernel_fits(h->vk, t->n, h->max_row) ||
        !(t = get_sell(h, kSellSigma, s)))
        return SPMV_ERR_UNSUPPORTED;
    const SellParams p =
        sell_params(*t, MatRef{h->d_rp, h->d_col, h->d_val, nullptr, nullptr, nullptr, nullptr}, 1.0, 0.0);
    double *out = w.one + 4 * static_cast<int64_t>(w.one_ctas);
    if (launch_cg(p, t->dtmp, h->vk, h->max_row, b, x, dir, dir2, r, tol, max_iter, w.one, out, s) != cudaSuccess) {
        (void)cudaGetLastError();  // not launched: the kernel-by-kernel path runs
        return SPMV_ERR_UNSUPPORTED;
    }
    CK(cudaMemcpyAsync(w.host, out, 4 * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (w.host[3] != 0.0) return SPMV_ERR_TIMEOUT;
    for (int i = 0; i < 3; ++i) res[i] = w.host[i];
    return SPMV_OK;
}

// Everything an apply needs (chunk tables) is built before a capture, so no
// allocation happens while a stream is being captured.
static spmv_status ready_for_capture(spmv_matrix *h, int xk, int yk) {
    const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
    SellOps lops;
    SellParams lp;
    if (sell_launch_of(h, 1.0, nullptr, xk, 0.0, nullptr, yk, nullptr, &lops, &lp))
        return cudaDeviceSynchronize() == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    SlotOps sops;
    if ((h->family == 4 || h->family == 5 || h->family == 6) &&
        (slot_ops(h->vk, xk, yk, acc, h->E, h->d_rmap != nullptr, &sops) ||
         (h->family == 6 && !h->d_rmap && slot_ops_tv(h->vk, xk, yk, acc, h->E, &sops))) &&
        get_slots(h, h->E, nullptr))
        return cudaDeviceSynchronize() == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
    if (h->family == 0 || h->family == 3 || h->family == 4 || h->family == 5 || h->family == 6 || h->d_rmap) {
        int E = h->E;
        if ((h->family == 4 || h->family == 5 || h->family == 6) && E != 7 && E != 15) E = 15;
        WarpOps ops;
        const bool ok3 = h->family == 3 && warp_ops(h->vk, xk, yk, acc, E + 100, false, false, &ops);
        if (!ok3 && !warp_ops(h->vk, xk, yk, acc, E, false, false, &ops)) E = 16;
        return get_chunks(h, E, false) ? SPMV_OK : SPMV_ERR_ALLOC;
    }
    if (h->family == 2) {
        const int E = pick_E(h->vk, xk, yk, acc, h->E);
        TileRun run;
        return prepare_run(h, xk, yk, 1, E, false, &run);
    }
    return SPMV_OK;
}

// Capture `body` (which enqueues kernels on the given stream) into a graph.
template <typename F>
static spmv_status capture_graph(F body, cudaGraphExec_t *exec) {
    cudaStream_t cap;
    CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    spmv_status st = SPMV_OK;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        st = body(cap);
        e = cudaStreamEndCapture(cap, &g);
    }
    if (e == cudaSuccess && st == SPMV_OK) e = cudaGraphInstantiate(exec, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    if (st != SPMV_OK) return st;
    return e == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
}

// Symmetric CRS (Sect. 1.3.1): the handle holds U, the upper triangle with the
// diagonal.  The product y = alpha*(U + U_s^T)*x + beta*y runs on the full matrix,
// expanded on the device once (get_full): reading an entry twice in order costs far
// less than finding it through its position (Hamiltonian-like, 4.2 M rows: FP64 148
// against 429 us, FP32 storage 139 against 372; 1.05 M rows 41 against 87, 41 / 66).
// With a plan chosen by the caller, or without the full matrix, it runs in two passes
// with a fixed summation order: the row sums of U on the autotuned kernel (with beta),
// then the row sums of U_s^T (the strictly upper part, transposed) added onto y by the
// warp-chunk kernel that reads each value through its position in U.
static spmv_status create_symmetric_index(spmv_matrix *h, const int32_t *col_host, cudaStream_t s) {
    const int32_t n = h->n_rows;
    std::vector<int32_t> rowS(static_cast<size_t>(n) + 1, 0);
    for (int32_t i = 0; i < n; ++i)
        for (int32_t k = h->h_rp[i]; k < h->h_rp[i + 1]; ++k)
            if (col_host[k] != i) rowS[static_cast<size_t>(col_host[k]) + 1] += 1;
    for (int32_t j = 0; j < n; ++j) rowS[j + 1] += rowS[j];
    const int64_t ns = rowS[n];
    std::vector<int32_t> colS(static_cast<size_t>(ns)), permS(static_cast<size_t>(ns));
    std::vector<int32_t> next(rowS.begin(), rowS.end() - 1);
    for (int32_t i = 0; i < n; ++i)  // rows of U_s^T list their entries by increasing position in U
        for (int32_t k = h->h_rp[i]; k < h->h_rp[i + 1]; ++k)
            if (col_host[k] != i) {
                const int32_t p = next[col_host[k]]++;
                colS[p] = i;
                permS[p] = k;
            }
    const size_t nT = static_cast<size_t>(n) + 1 + kRowPad;
    const size_t nent = static_cast<size_t>(ns) + kEntryPad;
    if (dmalloc(&h->d_rowT, nT) != cudaSuccess || dmalloc(&h->d_colT, nent) != cudaSuccess ||
        dmalloc(&h->d_perm, nent) != cudaSuccess)
        return SPMV_ERR_ALLOC;
    CK(cudaMemsetAsync(h->d_rowT, 0, nT * 4, s));
    CK(cudaMemsetAsync(h->d_colT, 0, nent * 4, s));
    CK(cudaMemsetAsync(h->d_perm, 0, nent * 4, s));
    CK(cudaMemcpyAsync(h->d_rowT, rowS.data(), rowS.size() * 4, cudaMemcpyHostToDevice, s));
    if (ns) {
        CK(cudaMemcpyAsync(h->d_colT, colS.data(), static_cast<size_t>(ns) * 4, cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(h->d_perm, permS.data(), static_cast<size_t>(ns) * 4, cudaMemcpyHostToDevice, s));
    }
    CK(cudaStreamSynchronize(s));
    h->h_rowT = std::move(rowS);
    h->has_T = true;
    return SPMV_OK;
}

// The slots that full's products read, when every entry has one (no chunks or rows
// summed from the CRS arrays): their values, how many there are, and their part of the
// map laid out like them (built on first use; null while a stream is captured, or
// without room).  Products then never read full's CRS values, whose array takes the map
// in FP64 (FP32 sums out of range read U's, through the map).
struct FullSlots {
    void *vals = nullptr;
    int64_t n = 0;
    Laid *laid = nullptr;
};
static FullSlots full_slots(spmv_matrix *h, cudaStream_t s) {
    spmv_matrix *f = h->full;
    FullSlots r;
    const auto c = f->slots.find(f->E);
    const auto l = f->sells.find(f->sigma);
    const bool chunks = f->family == 4 && c != f->slots.end() && c->second.n_long == 0 && c->second.n_empty == 0;
    const bool slices = f->family == 5 && l != f->sells.end() && l->second.vals && l->second.n_long == 0;
    if (chunks) r = FullSlots{c->second.vals, static_cast<int64_t>(c->second.n) * 32 * f->E, &c->second.laid};
    if (slices) r = FullSlots{l->second.vals, l->second.slot_rows * kSellC, &l->second.laid};
    if (!r.vals || h->d_slotmap) return r;
    const bool inside = f->vk == kF64 && 4 * r.n <= 8 * f->nnz && !h->crs_in_graph;
    if (capture_id(s) || (!inside && cudaMalloc(&h->d_slotmap, 4 * static_cast<size_t>(r.n) + 16) != cudaSuccess)) {
        h->d_slotmap = nullptr;
        (void)cudaGetLastError();
        return FullSlots();
    }
    if (inside) h->d_slotmap = static_cast<int32_t *>(f->d_val);
    h->slotmap_inside = inside;
    cudaError_t e = chunks ? launch_slot_map(c->second.d, f->E, r.n, h->d_fullmap, h->d_slotmap, s)
                           : cudaMemsetAsync(h->d_slotmap, 0xff, 4 * static_cast<size_t>(kSellU) * kSellC, s);
    if (e == cudaSuccess && slices)
        e = launch_sell_relayout(l->second.d, l->second.srows, l->second.n, f->d_rp, f->vk, nullptr, h->d_fullmap,
                                 nullptr, h->d_slotmap, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the next values may come on another stream
    if (e == cudaSuccess) return r;
    if (!inside) cudaFree(h->d_slotmap);
    h->d_slotmap = nullptr;
    h->slotmap_inside = false;
    return FullSlots();
}

// U's values in the full matrix: in the slots that the products read, through their map,
// else in the CRS arrays (1.05 M rows, new values and one apply: FP64 124 us, two passes
// 143; FP32 87, 110; 27-point 64^3 FP64 65, 59, where the gathers' cache lines bound it).
static cudaError_t fill_full(spmv_matrix *h, cudaStream_t s) {
    spmv_matrix *f = h->full;
    for (auto &kv : f->slots) kv.second.laid = Laid();
    for (auto &kv : f->sells) kv.second.laid = Laid();
    const FullSlots t = full_slots(h, s);
    cudaError_t e = cudaSuccess;
    if (!t.vals) {
        e = launch_permute(h->d_val, h->d_fullmap, f->d_val, f->nnz, f->vk, s);
        h->crs_in_graph = h->crs_in_graph || capture_id(s) != 0;
    }
    if (e == cudaSuccess && t.vals) {
        e = launch_fill_slots(h->d_val, h->d_slotmap, t.vals, t.n, f->vk, s);
        if (e == cudaSuccess) t.laid->set(s);
    }
    return e;
}

// The full matrix A = U + U_s^T of a symmetric handle, built by the first apply from U and
// the transposed index, with U's current values; null when it does not fit (in memory or
// in int32 entry numbers) or the first apply is captured, where nothing is allocated: the
// handle then keeps to the two passes, so that all its applies sum in one order.
static spmv_matrix *get_full(spmv_matrix *h, cudaStream_t s) {
    if (h->full_off) return nullptr;
    if (!h->full) {
        const int32_t n = h->n_rows;
        const int64_t ns = h->h_rowT[n], nnz = h->nnz + ns;
        spmv_matrix *f = nnz < (int64_t(1) << 31) && !capture_id(s) ? new (std::nothrow) spmv_matrix() : nullptr;
        bool ok = f != nullptr;
        if (ok) {
            f->device = h->device;
            f->n_rows = f->n_cols = n;
            f->nnz = nnz;
            f->vk = h->vk;
            f->acc32 = h->acc32;
            f->col_random = h->col_random;
            f->col_diag = h->col_diag;
            f->h_rp.resize(static_cast<size_t>(n) + 1);
            const int32_t *ru = h->h_rp.data(), *rs = h->h_rowT.data();
            int32_t *rf = f->h_rp.data();
            for (int32_t i = 0; i <= n; ++i) rf[i] = ru[i] + rs[i];
            const size_t nrp = static_cast<size_t>(n) + 1 + kRowPad, nent = static_cast<size_t>(nnz) + kEntryPad;
            const size_t vb = h->vk == kF64 ? 8 : 4;
            Block b;
            b.add(4 * nrp);
            b.add(4 * nent);
            b.add(vb * nent);
            b.add(4);
            b.add(4 * nent);
            ok = b.alloc();
            if (ok) {
                f->block = b.base;
                b.take(&f->d_rp);
                b.take(&f->d_col);
                b.take(&f->d_val);
                b.take(&f->d_err);
                b.take(&h->d_fullmap);
            }
            ok = ok && cudaMemsetAsync(f->d_err, 0, 4, s) == cudaSuccess &&
                 cudaMemsetAsync(f->d_rp + n + 1, 0, kRowPad * 4, s) == cudaSuccess &&
                 cudaMemsetAsync(f->d_col + nnz, 0, kEntryPad * 4, s) == cudaSuccess &&
                 cudaMemsetAsync(static_cast<char *>(f->d_val) + nnz * vb, 0, kEntryPad * vb, s) == cudaSuccess &&
                 launch_expand_sym(n, h->d_rp, h->d_col, h->d_rowT, h->d_colT, h->d_perm, f->d_rp, f->d_col,
                                   h->d_fullmap, s) == cudaSuccess &&
                 launch_permute(h->d_val, h->d_fullmap, f->d_val, nnz, h->vk, s) == cudaSuccess &&
                 cudaStreamSynchronize(s) == cudaSuccess;  // the next apply may run on another stream
        }
        if (!ok) {
            if (f) destroy_matrix(f);
            h->d_fullmap = nullptr;
            (void)cudaGetLastError();  // a failed allocation must not surface at a later launch check
            h->full_off = true;
            return nullptr;
        }
        autotune(f, f->vk == kF64 && f->col_random <= kScattered);
        if (f->vk == kF32) {
            // float-float sums: the two passes round y twice, but sum half of each row
            // in float-float, so FP32 runs over all of it would be less exact (1.05 M
            // rows: relative error 5.7e-8 against 4.5e-8)
            f->family = 4;
            f->E = 15;
            f->sell_if_diag = false;
            f->map_of = h->d_fullmap;
            f->val_of = h->d_val;
        }
        h->full = f;
        h->full_laid.now = true;
    }
    if (!h->full_laid.on(s)) {
        if (fill_full(h, s) != cudaSuccess) return nullptr;
        h->full_laid.set(s);
    }
    return h->full;
}

static spmv_status apply_sym(spmv_matrix *h, double alpha, const void *x, int xk, double beta, void *y, int yk,
                      cudaStream_t s) {
    const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
    const int32_t n = h->n_rows;
    const int64_t ns = h->h_rowT.empty() ? 0 : h->h_rowT[n];
    WarpOps ops;
    const double meanT = n ? static_cast<double>(ns) / n : 0.0;
    int ET = (meanT < 20.0) ? 7 : 15;
    if (!warp_ops(h->vk, xk, yk, acc, ET, true, false, &ops)) ET = (ET == 7) ? 15 : 7;
    if (ns > 0 && !warp_ops(h->vk, xk, yk, acc, ET, true, false, &ops)) return SPMV_ERR_UNSUPPORTED;
    if (ns > 0 && !h->planned) {
        if (spmv_matrix *f = get_full(h, s)) return apply_impl(f, alpha, x, xk, beta, y, yk, s);
    }
    spmv_status st = apply_impl(h, alpha, x, xk, beta, y, yk, s);
    if (st != SPMV_OK || ns == 0 || n == 0) return st;
    ChunkTable *ct = get_chunks(h, ET, true);
    if (!ct) return SPMV_ERR_ALLOC;
    WarpParams wp{};
    wp.m = MatRef{h->d_rowT, h->d_colT, h->d_perm, h->d_val, x, y, nullptr};
    wp.chunks = ct->d;
    wp.masks = ct->masks;
    wp.n_chunks = ct->n;
    wp.alpha = alpha;
    wp.beta = 1.0;
    wp.err = h->d_err;
    return ops.launch(wp, ct->n, s) == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
}

// Member m's values laid out again in the batch's own slices, on s.
static bool batch_diag_values(spmv_batch *b, int32_t m, cudaStream_t s) {
    spmv_matrix *h = b->mats[m];
    const SellTable &t = h->sells.at(kSellSigma);
    if (launch_sell_relayout(t.d, t.srows, t.n, h->d_rp, h->vk, h->d_val, nullptr, b->d_dvals + b->dval_off[m], nullptr,
                             s) != cudaSuccess)
        return false;
    if (!capture_id(s)) b->vals_ver[m] = h->values_version;
    return true;
}

// The batch's members on diagonal slices (member_E 0): large grid stencils, whose
// chunks spend more on their rows than on their entries (32 5-point members of 110,000
// rows on average: 46 against 59 us).
// False when something failed; members whose slices are not diagonal stay with the
// chunks.
static bool batch_diagonals(spmv_batch *b) {
    const int32_t count = b->count;
    b->vals_ver.assign(static_cast<size_t>(count), 0);
    b->dval_off.assign(static_cast<size_t>(count), 0);
    const size_t vb = b->vk == kF64 ? 8 : 4;
    std::vector<SellMember> members;
    std::vector<int2> list;
    std::vector<int32_t> which;
    int64_t bytes = 0;
    for (int32_t m = 0; m < count; ++m) {
        spmv_matrix *h = b->mats[m];
        if (h->col_diag < kDiagMinRows || h->sell_pad > kSellMaxPadding || h->n_rows < kBatchDiagMinSize ||
            h->max_row > (b->vk == kF64 ? kSellLongRow : kFRMaxRun))
            continue;
        const SellTable *t = get_sell(h, kSellSigma, nullptr, false, false);
        if (!t || !t->diagonal || t->n_long > 0) continue;
        b->member_E[m] = 0;
        b->dval_off[m] = bytes;
        for (int32_t k = 0; k < t->n; ++k) list.push_back(make_int2(static_cast<int>(members.size()), k));
        members.push_back(SellMember{t->dorder, t->srows, t->diag, nullptr, t->cols, m});
        which.push_back(m);
        bytes += (t->slot_rows * kSellC * static_cast<int64_t>(vb) + 255) / 256 * 256;
    }
    if (members.empty()) return true;
    if (cudaMalloc(&b->d_dvals, static_cast<size_t>(bytes)) != cudaSuccess) {
        b->d_dvals = nullptr;
        return false;
    }
    for (size_t i = 0; i < members.size(); ++i) {
        members[i].vals = b->d_dvals + b->dval_off[which[i]];
        if (!batch_diag_values(b, which[i], nullptr)) return false;
    }
    b->n_dlist = static_cast<int32_t>(list.size());
    return dmalloc(&b->d_dlist, list.size()) == cudaSuccess && dmalloc(&b->d_dmembers, members.size()) == cudaSuccess &&
           cudaMemcpy(b->d_dlist, list.data(), sizeof(int2) * list.size(), cudaMemcpyHostToDevice) == cudaSuccess &&
           cudaMemcpy(b->d_dmembers, members.data(), sizeof(SellMember) * members.size(), cudaMemcpyHostToDevice) ==
               cudaSuccess;
}

extern "C" {

const char *spmv_status_string(spmv_status s) {
    switch (s) {
    case SPMV_OK: return "SPMV_OK";
    case SPMV_ERR_INVALID_ARG: return "SPMV_ERR_INVALID_ARG: invalid argument";
    case SPMV_ERR_INVALID_INDEX: return "SPMV_ERR_INVALID_INDEX: invalid row_ptr or column index";
    case SPMV_ERR_CUDA: return "SPMV_ERR_CUDA: CUDA runtime or kernel error";
    case SPMV_ERR_ALLOC: return "SPMV_ERR_ALLOC: allocation failed";
    case SPMV_ERR_UNSUPPORTED: return "SPMV_ERR_UNSUPPORTED: combination not provided";
    case SPMV_ERR_TIMEOUT: return "SPMV_ERR_TIMEOUT: bounded device wait gave up";
    case SPMV_ERR_NOT_CONVERGED: return "SPMV_ERR_NOT_CONVERGED: iteration cap reached";
    }
    return "unknown status";
}

int32_t spmv_version(void) { return 100; }

spmv_status spmv_create(spmv_handle *out, int32_t n_rows, int32_t n_cols, int64_t nnz,
                        const int32_t *row_ptr, const int32_t *col_idx, const void *val,
                        spmv_dtype val_t, int is_device_ptr, void *stream) {
    if (!out) return SPMV_ERR_INVALID_ARG;
    *out = nullptr;
    if (n_rows < 0 || n_cols < 0 || nnz < 0 || nnz >= (int64_t(1) << 31)) return SPMV_ERR_INVALID_ARG;
    if (val_t != SPMV_F64 && val_t != SPMV_F32) return SPMV_ERR_INVALID_ARG;
    if (!row_ptr || (nnz > 0 && (!col_idx || !val))) return SPMV_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    std::vector<int32_t> h_rp(static_cast<size_t>(n_rows) + 1);
    std::vector<int32_t> h_col;
    const int32_t *col_host = col_idx;
    if (is_device_ptr) {
        CK(cudaMemcpyAsync(h_rp.data(), row_ptr, h_rp.size() * 4, cudaMemcpyDeviceToHost, s));
        h_col.resize(static_cast<size_t>(nnz));
        if (nnz) CK(cudaMemcpyAsync(h_col.data(), col_idx, static_cast<size_t>(nnz) * 4, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        col_host = h_col.data();
    } else {
        std::memcpy(h_rp.data(), row_ptr, h_rp.size() * 4);
    }
    spmv_status st = validate_host(n_rows, n_cols, nnz, h_rp.data(), col_host);
    if (st != SPMV_OK) return st;
    return create_from_host(out, n_rows, n_cols, nnz, std::move(h_rp), col_idx, val, val_t, val_t,
                            is_device_ptr != 0, s, col_host);
}

void spmv_destroy(spmv_handle h) { destroy_matrix(h); }

// New values for h; y not null: also y = alpha*A*x with them in the same pass where
// it can be done (*applied).  The vectors have h's value type.
static spmv_status set_values_impl(spmv_matrix *h, const void *val, spmv_dtype t, double alpha, const void *x, void *y,
                                   bool *applied, cudaStream_t s) {
    if (h->nnz == 0) return SPMV_OK;
    // a row-slice copy that served the last values, or serves this product, gets the new
    // ones in the same pass (27-point 128^3: 226 us where the CRS copy alone takes 136);
    // other copies are laid out again when they are used.  Small grids of short rows get
    // only product and values in one pass: the tile's chain of loads takes longer than
    // the copy and the layout one after the other (new values and a product, 5-point
    // 140^2 FP64 8.3 against 6.2 us, 200^2 8.8 / 7.2, 300^2 9.2 / 10.2; 7-point 25^3 FP32
    // 9.3 / 7.7, 40^3 8.9 / 9.0; 27-point 12^3 11.0 / 12.7)
    auto f = h->sells.find(h->sigma);
    const bool slices = h->family == 5 && f != h->sells.end() && f->second.laid.on(s) && f->second.diagonal &&
                        sell_tile_fits(h);
    const bool prod = slices && y && static_cast<int>(t) == h->vk && !h->sym && !h->d_rmap &&
                      (h->vk == kF64 || h->acc32 == kAccFF);
    const bool fused = slices && (prod || (f->second.read && (h->nnz > 8LL * h->n_rows || h->nnz >= kPosMinEntries)));
    if (fused) {
        const SellParams p = sell_params(
            f->second, MatRef{h->d_rp, h->d_col, prod ? val : nullptr, nullptr, prod ? x : nullptr, prod ? y : nullptr, nullptr},
            alpha, 0.0);
        CK(launch_sell_set_values(p, val, t, h->d_val, h->vk, h->max_row, s));
        f->second.read = prod;
        if (applied) *applied = prod;
    } else {
        CK(launch_convert(val, t, h->d_val, h->vk, h->nnz, s));
    }
    if (h->mirror32) {
        CK(launch_convert(val, t, h->mirror32->d_val, kF32, h->nnz, s));
        for (auto &kv : h->mirror32->slots) kv.second.laid = Laid();
        for (auto &kv : h->mirror32->sells) kv.second.laid = Laid();
    }
    // captured CG iterations read the copies laid out from the old values: the next
    // solve runs its first iterations plainly, which lays them out again
    h->cg.cg64_key = h->cg.inner32_key = -1;
    h->valT = h->full_laid = Laid();
    h->valT_requested = false;
    ++h->values_version;
    const Laid with = fused ? f->second.laid : Laid();
    for (auto &kv : h->slots) kv.second.laid = Laid();
    for (auto &kv : h->sells) kv.second.laid = Laid();
    if (fused) f->second.laid = with;  // it holds what the CRS copy holds, before and after this call's work
    return SPMV_OK;
}

spmv_status spmv_set_values(spmv_handle h, const void *val, spmv_dtype t, void *stream) {
    if (!h || (h->nnz > 0 && !val)) return SPMV_ERR_INVALID_ARG;
    if (t != SPMV_F64 && t != SPMV_F32) return SPMV_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    return set_values_impl(h, val, t, 1.0, nullptr, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

spmv_status spmv_set_values_apply(spmv_handle h, const void *val, spmv_dtype t, double alpha, const void *x,
                                  spmv_dtype xt, void *y, spmv_dtype yt, void *stream) {
    if (!h || (h->nnz > 0 && !val)) return SPMV_ERR_INVALID_ARG;
    if (t != SPMV_F64 && t != SPMV_F32) return SPMV_ERR_INVALID_ARG;
    if ((h->n_rows > 0 && !y) || (h->n_cols > 0 && h->n_rows > 0 && !x)) return SPMV_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    const bool same = static_cast<int>(xt) == h->vk && static_cast<int>(yt) == h->vk;
    bool applied = false;
    const spmv_status st =
        set_values_impl(h, val, t, alpha, x, same ? y : nullptr, &applied, static_cast<cudaStream_t>(stream));
    if (st != SPMV_OK || applied) return st;
    return spmv_apply(h, alpha, x, xt, 0.0, y, yt, stream);
}

spmv_status spmv_get_info(spmv_handle h, int32_t *n_rows, int32_t *n_cols, int64_t *nnz, int32_t *plan) {
    if (!h) return SPMV_ERR_INVALID_ARG;
    if (n_rows) *n_rows = h->n_rows;
    if (n_cols) *n_cols = h->n_cols;
    if (nnz) *nnz = h->nnz;
    if (plan) {
        DeviceGuard g(h->device);
        settle_plan(h, nullptr);
        const int acc = (h->vk == kF32) ? h->acc32 : kAccF64;
        int32_t E = h->E, nunits = 0, rowcap = 0, nlong = 0, threads = 256;
        if (h->family == 2) {
            E = pick_E(h->vk, h->vk, h->vk, acc, h->E);
            TileOps ops;
            if (E > 0 && tile_ops(h->vk, h->vk, h->vk, acc, 1, E, false, false, &ops)) {
                const TileCfg c = ops.cfg();
                TileTable *tt = get_table(h, c.cap, c.rowcap, false);
                if (tt) {
                    nunits = tt->n;
                    nlong = tt->n_long;
                }
                rowcap = c.rowcap;
                threads = c.threads;
            }
        } else if (h->family == 5) {
            SellTable *t = get_sell(h, h->sigma, nullptr);
            if (t) {
                nunits = t->n;
                nlong = t->n_long;
            }
            E = h->sigma;
            rowcap = kSellC;
            if (cudaDeviceSynchronize() != cudaSuccess) return SPMV_ERR_CUDA;
        } else if (h->family == 4 || h->family == 6) {
            SlotTable *t = get_slots(h, E, nullptr);
            if (t) {
                nunits = t->n;
                nlong = t->n_long;
            }
            rowcap = kWarpRowCap;
            if (cudaDeviceSynchronize() != cudaSuccess) return SPMV_ERR_CUDA;
        } else {
            WarpOps ops;
            const bool ok3 = h->family == 3 && warp_ops(h->vk, h->vk, h->vk, acc, E + 100, false, false, &ops);
            if (!ok3 && !warp_ops(h->vk, h->vk, h->vk, acc, E, false, false, &ops)) E = 16;
            ChunkTable *ct = get_chunks(h, E, false);
            if (ct) {
                nunits = ct->n;
                nlong = ct->n_long;
            }
            rowcap = kWarpRowCap;
        }
        plan[0] = h->family;
        plan[1] = E;
        plan[2] = threads;
        plan[3] = nunits;
        plan[4] = rowcap;
        plan[5] = h->T;
        plan[6] = nlong;
        plan[7] = h->vk;
    }
    return SPMV_OK;
}

spmv_status spmv_row_histogram(spmv_handle h, int32_t nbins, int64_t *counts) {
    if (!h || nbins < 1 || !counts) return SPMV_ERR_INVALID_ARG;
    for (int32_t b = 0; b < nbins; ++b) counts[b] = 0;
    for (int32_t i = 0; i < h->n_rows; ++i) {
        const int32_t len = h->h_rp[i + 1] - h->h_rp[i];
        counts[len < nbins - 1 ? len : nbins - 1] += 1;
    }
    return SPMV_OK;
}

spmv_status spmv_set_plan(spmv_handle h, int32_t family, int32_t param) {
    if (!h || family < 0 || family > 6) return SPMV_ERR_INVALID_ARG;
    // a refused parameter leaves the handle as it was
    const bool f64 = h->vk == kF64;
    bool ok = param == 0;
    switch (family) {
        case 0: ok = ok || param == 7 || param == 8 || param == 15 || param == 16; break;
        case 1: ok = ok || (param >= 1 && param <= 32 && !(param & (param - 1))); break;
        case 2: ok = ok || (param >= 3 && param <= 31 && param % 2 != 0); break;
        case 3: ok = ok || param == 7 || param == 11 || param == 15; break;
        case 4: ok = ok || param == 7 || param == 9 || param == 11 || param == 15; break;
        case 5: ok = ok || (param >= 32 && param <= (1 << 20) && !(param & (param - 1))); break;
        default: ok = ok || param == 9 || param == (f64 ? 7 : 15); break;
    }
    if (!ok) return SPMV_ERR_INVALID_ARG;
    constexpr int kDefaultE[7] = {16, 0, 15, 7, 9, 0, 9};
    h->family = family;
    h->planned = true;
    h->sell_if_diag = false;
    if (family == 5) h->sigma = param ? param : 4096;
    else if (family == 1) h->T = param ? param : h->T;
    else h->E = param ? param : (family == 4 && !f64 ? 15 : kDefaultE[family]);
    return SPMV_OK;
}

spmv_status spmv_set_accumulator(spmv_handle h, int32_t acc) {
    if (!h || (acc != 0 && acc != 1)) return SPMV_ERR_INVALID_ARG;
    h->acc32 = (acc == 0) ? kAccF64 : kAccFF;
    if (h->full) h->full->acc32 = h->acc32;
    return SPMV_OK;
}

spmv_status spmv_apply(spmv_handle h, double alpha, const void *x, spmv_dtype xt, double beta,
                       void *y, spmv_dtype yt, void *stream) {
    if (!h) return SPMV_ERR_INVALID_ARG;
    if ((h->n_rows > 0 && !y) || (h->n_cols > 0 && h->n_rows > 0 && !x)) return SPMV_ERR_INVALID_ARG;
    if (h->vk == kF64 && (xt != SPMV_F64 || yt != SPMV_F64)) return SPMV_ERR_UNSUPPORTED;
    if (h->vk == kF32 && xt != SPMV_F32) return SPMV_ERR_UNSUPPORTED;
    if (yt != SPMV_F64 && yt != SPMV_F32) return SPMV_ERR_INVALID_ARG;
    DeviceGuard g(h->device);
    if (h->sym) return apply_sym(h, alpha, x, xt, beta, y, yt, static_cast<cudaStream_t>(stream));
    return apply_impl(h, alpha, x, xt, beta, y, yt, static_cast<cudaStream_t>(stream));
}

spmv_status spmv_create_symmetric(spmv_handle *out, int32_t n, int64_t nnz, const int32_t *row_ptr,
                                  const int32_t *col_idx, const void *val, spmv_dtype val_t, int is_device_ptr,
                                  void *stream) {
    if (!out) return SPMV_ERR_INVALID_ARG;
    *out = nullptr;
    if (n < 0 || nnz < 0 || nnz >= (int64_t(1) << 31)) return SPMV_ERR_INVALID_ARG;
    if (val_t != SPMV_F64 && val_t != SPMV_F32) return SPMV_ERR_INVALID_ARG;
    if (!row_ptr || (nnz > 0 && (!col_idx || !val))) return SPMV_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    std::vector<int32_t> h_rp(static_cast<size_t>(n) + 1);
    std::vector<int32_t> h_col(static_cast<size_t>(nnz));
    if (is_device_ptr) {
        CK(cudaMemcpyAsync(h_rp.data(), row_ptr, h_rp.size() * 4, cudaMemcpyDeviceToHost, s));
        if (nnz) CK(cudaMemcpyAsync(h_col.data(), col_idx, static_cast<size_t>(nnz) * 4, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
    } else {
        std::memcpy(h_rp.data(), row_ptr, h_rp.size() * 4);
        if (nnz) std::memcpy(h_col.data(), col_idx, static_cast<size_t>(nnz) * 4);
    }
    spmv_status st = validate_host(n, n, nnz, h_rp.data(), h_col.data());
    if (st != SPMV_OK) return st;
    for (int32_t i = 0; i < n; ++i)  // the upper triangle: no entry left of the diagonal
        for (int32_t k = h_rp[i]; k < h_rp[i + 1]; ++k)
            if (h_col[k] < i) return SPMV_ERR_INVALID_INDEX;
    spmv_handle h = nullptr;
    st = create_from_host(&h, n, n, nnz, std::move(h_rp), col_idx, val, val_t, val_t, is_device_ptr != 0, s,
                          h_col.data());
    if (st != SPMV_OK) return st;
    DeviceGuard g(h->device);
    h->sym = true;
    st = create_symmetric_index(h, h_col.data(), s);
    if (st != SPMV_OK) {
        destroy_matrix(h);
        return st;
    }
    *out = h;
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// Split form
// ---------------------------------------------------------------------------

spmv_status spmv_split_create(spmv_split_handle *out, spmv_handle h, int32_t nblocks,
                              const int32_t *block_row_start, int32_t *halo_count_out) {
    if (!out || !h || nblocks < 1) return SPMV_ERR_INVALID_ARG;
    *out = nullptr;
    if (h->n_rows != h->n_cols) return SPMV_ERR_INVALID_ARG;
    if (h->vk != kF64 || h->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard g(h->device);
    const int32_t n = h->n_rows;
    const int64_t nnz = h->nnz;
    std::vector<int32_t> bs(static_cast<size_t>(nblocks) + 1);
    if (block_row_start) {
        for (int b = 0; b <= nblocks; ++b) bs[b] = block_row_start[b];
        if (bs[0] != 0 || bs[nblocks] != n) return SPMV_ERR_INVALID_ARG;
        for (int b = 0; b < nblocks; ++b)
            if (bs[b + 1] < bs[b]) return SPMV_ERR_INVALID_ARG;
    } else {
        // Sect. 3.2: balanced nonzeros; block b starts at the first row whose
        // offset is at least ceil(b*nnz/nblocks)
        bs[0] = 0;
        for (int b = 1; b < nblocks; ++b) {
            const int64_t target = (static_cast<int64_t>(b) * nnz + nblocks - 1) / nblocks;
            const int32_t *it = std::lower_bound(h->h_rp.data(), h->h_rp.data() + n, target,
                                                 [](int32_t e, int64_t v) { return e < v; });
            bs[b] = static_cast<int32_t>(it - h->h_rp.data());
        }
        bs[nblocks] = n;
    }
    // bring the column indices to the host for the one-time bookkeeping
    std::vector<int32_t> col(static_cast<size_t>(nnz));
    if (nnz) CK(cudaMemcpy(col.data(), h->d_col, static_cast<size_t>(nnz) * 4, cudaMemcpyDeviceToHost));
    std::vector<double> val(static_cast<size_t>(nnz));
    if (nnz) CK(cudaMemcpy(val.data(), h->d_val, static_cast<size_t>(nnz) * 8, cudaMemcpyDeviceToHost));

    spmv_split *sp = new (std::nothrow) spmv_split();
    if (!sp) return SPMV_ERR_ALLOC;
    sp->A = h;
    sp->nblocks = nblocks;
    sp->block_start = bs;
    sp->halo_count.assign(nblocks, 0);
    sp->nnz_local.assign(nblocks, 0);
    sp->nnz_nonlocal.assign(nblocks, 0);

    std::vector<int32_t> pos(static_cast<size_t>(n) + 1, -1);
    std::vector<int32_t> rp_loc(static_cast<size_t>(n) + 1, 0), rp_nl(static_cast<size_t>(n) + 1, 0);
    std::vector<int32_t> col_loc, col_nl;
    std::vector<double> val_loc, val_nl;
    std::vector<int32_t> col_vec(static_cast<size_t>(nnz));
    col_loc.reserve(static_cast<size_t>(nnz));
    val_loc.reserve(static_cast<size_t>(nnz));
    for (int b = 0; b < nblocks; ++b) {
        const int32_t lo = bs[b], hi = bs[b + 1];
        // mark the nonlocal columns of this block, then number them in order
        std::vector<char> used;
        used.assign(static_cast<size_t>(n), 0);
        for (int32_t i = lo; i < hi; ++i)
            for (int32_t k = h->h_rp[i]; k < h->h_rp[i + 1]; ++k) {
                const int32_t c = col[k];
                if (c < lo || c >= hi) used[c] = 1;
            }
        const int64_t off = sp->total_halo;
        int32_t cnt = 0;
        for (int32_t c = 0; c < n; ++c)
            if (used[c]) {
                pos[c] = static_cast<int32_t>(off + cnt);
                sp->h_halo_map.push_back(c);
                ++cnt;
            }
        sp->halo_count[b] = cnt;
        sp->total_halo += cnt;
        for (int32_t i = lo; i < hi; ++i) {
            for (int32_t k = h->h_rp[i]; k < h->h_rp[i + 1]; ++k) {
                const int32_t c = col[k];
                if (c >= lo && c < hi) {
                    col_loc.push_back(c);
                    val_loc.push_back(val[k]);
                    col_vec[k] = c;
                } else {
                    col_nl.push_back(pos[c]);
                    val_nl.push_back(val[k]);
                    col_vec[k] = n + pos[c];
                }
            }
            rp_loc[i + 1] = static_cast<int32_t>(col_loc.size());
            rp_nl[i + 1] = static_cast<int32_t>(col_nl.size());
        }
        sp->nnz_local[b] = rp_loc[hi] - rp_loc[lo];
        sp->nnz_nonlocal[b] = rp_nl[hi] - rp_nl[lo];
    }
    if (sp->total_halo + n >= (int64_t(1) << 31)) {
        delete sp;
        return SPMV_ERR_UNSUPPORTED;
    }
    cudaStream_t s = nullptr;
    spmv_status st = create_from_host(&sp->Aloc, n, n, static_cast<int64_t>(col_loc.size()),
                                      std::vector<int32_t>(rp_loc), col_loc.data(), val_loc.data(),
                                      kF64, kF64, false, s, col_loc.data());
    // the nonlocal part keeps only rows with nonlocal entries; each stored row
    // carries the output row it updates
    std::vector<int32_t> nl_rows, rp_c(1, 0);
    for (int32_t i = 0; i < n; ++i)
        if (rp_nl[i + 1] > rp_nl[i]) {
            nl_rows.push_back(i);
            rp_c.push_back(rp_nl[i + 1]);
        }
    if (st == SPMV_OK)
        st = create_from_host(&sp->Anl, static_cast<int32_t>(nl_rows.size()), static_cast<int32_t>(sp->total_halo),
                              static_cast<int64_t>(col_nl.size()), std::move(rp_c),
                              col_nl.data(), val_nl.data(), kF64, kF64, false, s, nullptr);
    if (st == SPMV_OK) {
        if (dmalloc(&sp->Anl->d_rmap, nl_rows.size()) != cudaSuccess) st = SPMV_ERR_ALLOC;
        else if (!nl_rows.empty() && cudaMemcpy(sp->Anl->d_rmap, nl_rows.data(), 4 * nl_rows.size(),
                                                cudaMemcpyHostToDevice) != cudaSuccess)
            st = SPMV_ERR_CUDA;
    }
    if (st == SPMV_OK) {
        if (dmalloc(&sp->d_halo_map, static_cast<size_t>(sp->total_halo)) != cudaSuccess ||
            dmalloc(&sp->d_halo, static_cast<size_t>(sp->total_halo)) != cudaSuccess)
            st = SPMV_ERR_ALLOC;
    }
    if (st == SPMV_OK && sp->total_halo > 0 &&
        cudaMemcpy(sp->d_halo_map, sp->h_halo_map.data(), static_cast<size_t>(sp->total_halo) * 4,
                   cudaMemcpyHostToDevice) != cudaSuccess)
        st = SPMV_ERR_CUDA;
    if (st == SPMV_OK)
        st = create_from_host(&sp->Avec, n, static_cast<int32_t>(n + sp->total_halo), nnz,
                              std::vector<int32_t>(h->h_rp), col_vec.data(), val.data(), kF64, kF64, false, s,
                              col_vec.data());
    if (st == SPMV_OK && dmalloc(&sp->d_xe, static_cast<size_t>(n + sp->total_halo)) != cudaSuccess)
        st = SPMV_ERR_ALLOC;
    if (st == SPMV_OK && (cudaEventCreateWithFlags(&sp->ev_x, cudaEventDisableTiming) != cudaSuccess ||
                          cudaEventCreateWithFlags(&sp->ev_halo, cudaEventDisableTiming) != cudaSuccess))
        st = SPMV_ERR_CUDA;
    if (st != SPMV_OK) {
        spmv_split_destroy(sp);
        return st;
    }
    // Plans of the parts (measured on the Hamiltonian-like matrix, 8 blocks): the
    // local part takes the autotuned plan (slot-major); the nonlocal part runs
    // the slot-major kernel with 7 entries per lane and its row epilogue (row
    // map, old y) loaded ahead of the FMA chains (split 283 -> 267 us against the
    // staged three-stage kernel).
    if (sp->Aloc->family == 3) {
        const double mean = n ? static_cast<double>(sp->Aloc->nnz) / n : 0.0;
        sp->Aloc->family = 0;
        sp->Aloc->E = (mean < 20.0) ? 7 : 15;
    }
    sp->Anl->family = 4;
    sp->Anl->E = 7;
    if (halo_count_out)
        for (int b = 0; b < nblocks; ++b) halo_count_out[b] = sp->halo_count[b];
    *out = sp;
    return SPMV_OK;
}

void spmv_split_destroy(spmv_split_handle hs) {
    if (!hs) return;
    DeviceGuard g(hs->A ? hs->A->device : 0);
    cudaDeviceSynchronize();
    destroy_matrix(hs->Aloc);
    destroy_matrix(hs->Anl);
    destroy_matrix(hs->Avec);
    cudaFree(hs->d_xe);
    cudaFree(hs->d_halo_map);
    cudaFree(hs->d_halo);
    if (hs->ev_x) cudaEventDestroy(hs->ev_x);
    if (hs->ev_halo) cudaEventDestroy(hs->ev_halo);
    delete hs;
}

spmv_status spmv_split_get_plan(spmv_split_handle hs, int32_t *nblocks, int32_t *block_start,
                                int32_t *halo_count, int64_t *total_halo, int32_t *halo_map,
                                int64_t *nnz_local, int64_t *nnz_nonlocal) {
    if (!hs) return SPMV_ERR_INVALID_ARG;
    if (nblocks) *nblocks = hs->nblocks;
    if (block_start) std::copy(hs->block_start.begin(), hs->block_start.end(), block_start);
    if (halo_count) std::copy(hs->halo_count.begin(), hs->halo_count.end(), halo_count);
    if (total_halo) *total_halo = hs->total_halo;
    if (halo_map) std::copy(hs->h_halo_map.begin(), hs->h_halo_map.end(), halo_map);
    if (nnz_local) std::copy(hs->nnz_local.begin(), hs->nnz_local.end(), nnz_local);
    if (nnz_nonlocal) std::copy(hs->nnz_nonlocal.begin(), hs->nnz_nonlocal.end(), nnz_nonlocal);
    return SPMV_OK;
}

spmv_status spmv_apply_split(spmv_split_handle hs, double alpha, const double *x, double beta,
                             double *y, void *s_compute, void *s_comm) {
    if (!hs) return SPMV_ERR_INVALID_ARG;
    spmv_matrix *A = hs->A;
    if (A->n_rows > 0 && (!x || !y)) return SPMV_ERR_INVALID_ARG;
    DeviceGuard g(A->device);
    cudaStream_t sc = static_cast<cudaStream_t>(s_compute);
    cudaStream_t sm = static_cast<cudaStream_t>(s_comm);
    // stream 2 ("communication"): wait until x is ready, gather the halo
    if (sm != sc) {
        CK(cudaEventRecord(hs->ev_x, sc));
        CK(cudaStreamWaitEvent(sm, hs->ev_x, 0));
    }
    CK(launch_gather(x, hs->d_halo_map, hs->d_halo, hs->total_halo, sm));
    if (sm != sc) CK(cudaEventRecord(hs->ev_halo, sm));
    // stream 1: local part (overlaps the gather), then the nonlocal part
    spmv_status st = apply_impl(hs->Aloc, alpha, x, kF64, beta, y, kF64, sc);
    if (st != SPMV_OK) return st;
    if (sm != sc) CK(cudaStreamWaitEvent(sc, hs->ev_halo, 0));
    if (hs->Anl->nnz > 0) st = apply_impl(hs->Anl, alpha, hs->d_halo, kF64, 1.0, y, kF64, sc);
    return st;
}

// Vector mode (Sect. 3.4, Fig. kernel_schemes (a)): the whole halo is gathered
// first, then one pass over the full matrix reads local columns from x and
// nonlocal ones from the halo (both in xe), writing y once.
spmv_status spmv_apply_split_vector(spmv_split_handle hs, double alpha, const double *x, double beta,
                                    double *y, void *stream) {
    if (!hs) return SPMV_ERR_INVALID_ARG;
    spmv_matrix *A = hs->A;
    if (A->n_rows > 0 && (!x || !y)) return SPMV_ERR_INVALID_ARG;
    if (!hs->Avec) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard g(A->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t n = A->n_rows;
    if (n > 0) CK(cudaMemcpyAsync(hs->d_xe, x, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToDevice, s));
    CK(launch_gather(x, hs->d_halo_map, hs->d_xe + n, hs->total_halo, s));
    return apply_impl(hs->Avec, alpha, hs->d_xe, kF64, beta, y, kF64, s);
}

spmv_status spmv_split_get_halo(spmv_split_handle hs, double *halo_out, void *stream) {
    if (!hs || (!halo_out && hs->total_halo > 0)) return SPMV_ERR_INVALID_ARG;
    DeviceGuard g(hs->A->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (hs->total_halo > 0)
        CK(cudaMemcpyAsync(halo_out, hs->d_halo, static_cast<size_t>(hs->total_halo) * 8, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// Block vectors
// ---------------------------------------------------------------------------

spmv_status spmm_apply(spmv_handle h, int32_t nrhs, double alpha, const void *X, double beta,
                       void *Y, spmv_dtype vt, void *stream) {
    if (!h || nrhs < 1 || nrhs > 64) return SPMV_ERR_INVALID_ARG;
    if (h->n_rows > 0 && (!X || !Y)) return SPMV_ERR_INVALID_ARG;
    if (vt != SPMV_F64 || h->vk != kF64 || h->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard g(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (h->n_rows == 0) return SPMV_OK;
    if (nrhs == 1) return apply_impl(h, alpha, X, kF64, beta, Y, kF64, s);
    int32_t c0 = 0;
    // On the sorted row slices when they pad little: lanes across the right-hand
    // sides, up to 32 per pass; exactly 4 with a lane per two rows (k_sell_mr) when
    // neighbouring rows share x in L1, or when X is too large for L2 to keep the
    // rows of X between its reads either way (Hamiltonian-like: 4.2 M rows, X 134
    // MB, 461 against 478 us; 1.9 M rows, 61 MB, 201 against 196; 300,000 rows 50 against
    // 36; 27-point 101^3 192 against 194, 5-point 1400^2 74 against 80).
    // Not for 2 or 3 right-hand sides on few rows: a warp then walks 16 or 32 whole rows
    // at the latency of its loads, where the tile kernel cuts the entries evenly (3:
    // 27-point 25^3 15.7 against 7.9 us, 32^3 17.6 / 13.9, 40^3 17.6 / 21.3; scattered
    // 30,000 rows 13.1 / 8.2, 130,000 23.0 / 22.1, 260,000 30.7 / 39.7).
    // Nor with rows outside the slices (long_row): one warp and its lane groups walk
    // such a row, which the tile kernel gives a CTA (3,000 rows, 3 of them of 1,500
    // entries: 3 right-hand sides 47 against 10 us, 32 468 against 164).  Groups of 4
    // stay on k_sell_mr there, whose 32 lanes share the row, while X fits in L2.
    int l2 = 0;
    cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, h->device);
    const bool scattered = h->col_random > kScattered;
    const bool long_rows = h->max_row > kSellLongRow;
    const double x_bytes = static_cast<double>(h->n_cols) * nrhs * 8.0;
    const bool slices = nrhs < kSellR ? !long_rows && h->n_rows >= (scattered ? kRhsFewScattered : kRhsFew)
                                      : !long_rows || !scattered || x_bytes <= 1.25 * l2;
    SellTable *t = nullptr;
    if (slices && h->sell_pad <= kSellMaxPadding && (t = get_sell(h, kSellSigma, s)) != nullptr) {
        const bool vec = (nrhs % 2 == 0) && (reinterpret_cast<uintptr_t>(X) % 16 == 0) &&
                         (reinterpret_cast<uintptr_t>(Y) % 16 == 0);
        const SellParams b =
            sell_params(*t, MatRef{h->d_rp, h->d_col, h->d_val, nullptr, nullptr, nullptr, nullptr}, alpha, beta);
        const double *Xd = static_cast<const double *>(X);
        double *Yd = static_cast<double *>(Y);
        if (long_rows || (nrhs == kSellR && (!scattered || x_bytes > 0.5 * l2))) {
            for (; c0 + kSellR <= nrhs; c0 += kSellR) CK(launch_sell_mr(b, Xd + c0, Yd + c0, nrhs, nrhs, vec, s));
        } else {
            for (; c0 < nrhs; c0 += kSellMaxRhs)
                CK(launch_sell_rhs(b, Xd + c0, Yd + c0, nrhs, nrhs, std::min(kSellMaxRhs, nrhs - c0), vec, scattered, s));
        }
    }
    // what is left (all of it without the slices): the tile kernel, up to 32 per launch
    for (; c0 < nrhs; c0 += 32) {
        const int cnt = std::min(32, nrhs - c0);
        int R = 2;
        while (R < cnt) R <<= 1;
        TileRun run;
        spmv_status st = prepare_run(h, kF64, kF64, R, 15, false, &run);
        if (st != SPMV_OK) return st;
        KParams p{};
        p.m = MatRef{h->d_rp, h->d_col, h->d_val, nullptr, static_cast<const double *>(X) + c0,
                     static_cast<double *>(Y) + c0};
        p.tiles = run.tt->d;
        p.n_tiles = run.tt->n;
        p.rhs_count = cnt;
        p.ldx = nrhs;
        p.ldy = nrhs;
        p.alpha = alpha;
        p.beta = beta;
        p.err = h->d_err;
        if (run.ops.launch(p, run.grid, s) != cudaSuccess) return SPMV_ERR_CUDA;
    }
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// Reverse pass
// ---------------------------------------------------------------------------

// Entries per lane of the staged chunk kernel over A^T (ind: values through the permutation).
static int ind_chunk_E(const spmv_matrix *h, bool ind = true) {
    const double meanT = h->n_cols ? static_cast<double>(h->nnz) / h->n_cols : 0.0;
    WarpOps ops;
    return meanT < 20.0 && warp_ops(h->vk, h->vk, h->vk, h->vk == kF32 ? kAccFF : kAccF64, 7, ind, false, &ops) ? 7 : 15;
}

spmv_status spmv_backward(spmv_handle h, double alpha, const void *g, const void *x, void *grad_x,
                          void *grad_val, void *stream) {
    if (!h) return SPMV_ERR_INVALID_ARG;
    if (h->sym) return SPMV_ERR_UNSUPPORTED;
    if (grad_x && h->n_rows > 0 && !g) return SPMV_ERR_INVALID_ARG;
    if (grad_val && h->nnz > 0 && (!g || !x)) return SPMV_ERR_INVALID_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool again = h->valT_requested;  // not the first reverse pass on these values
    if (grad_x && h->n_cols > 0) {
        spmv_status st = ensure_transpose(h, s);
        if (st != SPMV_OK) return st;
        // grad_x = alpha * A^T g: warp chunks over the rows of A^T.  The first
        // reverse pass on a set of values reads them through the permutation
        // (val[perm], inside the staged chunk kernel); a second one on the same
        // values lays them out in the order of A^T once (a streaming permutation
        // pass), and from then on the product runs like a forward product on a
        // slot-major copy of A^T.
        const size_t vb = (h->vk == kF64) ? 8 : 4;
        if (h->valT_requested && h->nnz > 0 && !h->valT.on(s)) {
            if (!h->d_valT && cudaMalloc(&h->d_valT, static_cast<size_t>(h->nnz) * vb) != cudaSuccess) {
                h->d_valT = nullptr;
                return SPMV_ERR_ALLOC;
            }
            CK(launch_permute(h->d_val, h->d_perm, h->d_valT, h->nnz, h->vk, s));
            h->valT.set(s);
            for (auto &kv : h->slotsT) kv.second.laid = Laid();
            for (auto &kv : h->sellsT) kv.second.laid = Laid();
        }
        const bool ind = !h->valT.on(s);
        h->valT_requested = true;
        bool done = false;
        if (ind) {
            // new values on diagonal slices: the slices of A^T read them where A's
            // slices hold them.  With rows of up to 8 entries on average only when a
            // product has laid them out there: doing it for this pass alone costs what
            // the pass then saves (new values and a reverse pass: 7-point 160^3 290
            // against 257 us through the permutation, 5-point 2000^2 210 / 195; 27-point
            // 128^3 500 against 606).  Such rows also need kPosMinEntries entries: a
            // smaller grid's pass is one chain of loads, which the positions lengthen
            // (new values, product and reverse pass, FP32: 5-point 100^2 12.7 against
            // 11.4 us, 200^2 13.3 / 12.2, 300^2 13.8 / 15.0; 27-point 12^3 14.2 / 16.1
            // for grad_x).
            SellOps lops;
            const int acc = (h->vk == kF32) ? kAccFF : kAccF64;
            const SellTable *t = nullptr, *a = nullptr;
            const bool longer = h->nnz > 8LL * h->n_rows;
            if ((longer || h->nnz >= kPosMinEntries) && sell_ops(h->vk, h->vk, h->vk, acc, &lops) &&
                (t = get_sell_positions(h, s)) != nullptr) {
                // (also where the capture of the other path would have to build its chunks)
                const SellTable &own = h->sells.at(h->sigma);
                const bool laid = own.vals && own.laid.on(s);
                a = longer || (!h->chunksT.count(ind_chunk_E(h)) && capture_id(s) != 0) ? get_sell(h, h->sigma, s)
                    : laid                                                              ? &own
                                                                                        : nullptr;
            }
            if (a) {
                SellParams lp =
                    sell_params(*t, MatRef{h->d_rowT, h->d_colT, h->d_perm, h->d_val, g, grad_x, nullptr}, alpha, 0.0);
                lp.vals = a->vals;
                lp.vpos = t->vpos.at(h->sigma);
                if (lops.launch_ind(lp, s) != cudaSuccess) return SPMV_ERR_CUDA;
                done = true;
            }
        }
        const double meanT = h->n_cols ? static_cast<double>(h->nnz) / h->n_cols : 0.0;
        if (!ind && h->col_random <= kScattered && meanT >= kSellMinRowLength) {
            // A^T of a stencil-like matrix with long rows: the sorted row-slice
            // kernel on a row-slice copy of A^T (as the tuner picks for a forward
            // product of such a matrix)
            if (h->sell_padT < 0.0) h->sell_padT = sell_padding(h->h_rowT.data(), h->n_cols, kSellSigma);
            SellOps lops;
            const int acc = (h->vk == kF32) ? kAccFF : kAccF64;
            SellTable *t = nullptr;
            // without its copy (allocation failed) the slot-major path below runs
            if (h->sell_padT <= kSellMaxPadding && sell_ops(h->vk, h->vk, h->vk, acc, &lops) &&
                (t = get_sell(h, kSellSigma, s, true)) != nullptr) {
                const SellParams lp = sell_params(
                    *t, MatRef{h->d_rowT, h->d_colT, h->d_valT, nullptr, g, grad_x, nullptr}, alpha, 0.0);
                if (lops.launch(lp, s) != cudaSuccess) return SPMV_ERR_CUDA;
                done = true;
            }
        }
        if (!ind && !done) {
            // A^T's values in its own order: the slot-major kernel on a slot-major
            // copy of A^T (E by A^T's mean row length, as for a forward product)
            const int ES = (h->vk == kF32) ? 15 : ((meanT < 8.0) ? 7 : 9);
            SlotOps sops;
            const int acc = (h->vk == kF32) ? kAccFF : kAccF64;
            if (slot_ops(h->vk, h->vk, h->vk, acc, ES, false, &sops)) {
                SlotTable *t = get_slots(h, ES, s, true);
                if (!t) return SPMV_ERR_ALLOC;
                SlotParams sp{};
                sp.chunks = t->d;
                sp.lmask = t->lmask;
                sp.vals = t->vals;
                sp.cols = t->cols;
                sp.m = MatRef{h->d_rowT, h->d_colT, h->d_valT, nullptr, g, grad_x, nullptr};
                sp.n_chunks = t->n;
                sp.alpha = alpha;
                sp.beta = 0.0;
                sp.ff = epi_ff(alpha, 0.0);
                sp.err = h->d_err;
                if (sops.launch(sp, s) != cudaSuccess) return SPMV_ERR_CUDA;
                done = true;
            }
        }
        if (!done) {
            WarpOps ops;
            const int acc = (h->vk == kF32) ? kAccFF : kAccF64;
            const int ET = ind_chunk_E(h, ind);
            if (!warp_ops(h->vk, h->vk, h->vk, acc, ET, ind, false, &ops)) return SPMV_ERR_UNSUPPORTED;
            ChunkTable *ct = get_chunks(h, ET, true);
            if (!ct) return SPMV_ERR_ALLOC;
            WarpParams wp{};
            wp.m = ind ? MatRef{h->d_rowT, h->d_colT, h->d_perm, h->d_val, g, grad_x, nullptr}
                       : MatRef{h->d_rowT, h->d_colT, h->d_valT, nullptr, g, grad_x, nullptr};
            wp.chunks = ct->d;
            wp.masks = ct->masks;
            wp.n_chunks = ct->n;
            wp.alpha = alpha;
            wp.beta = 0.0;
            wp.err = h->d_err;
            if (ops.launch(wp, ct->n, s) != cudaSuccess) return SPMV_ERR_CUDA;
        }
    }
    if (grad_val && h->nnz > 0) {
        // Rows of more than 8 entries on average: on A's diagonal slices, when a
        // forward product or a second reverse pass has built them (27-point 128^3:
        // FP64 138 against 162 us, FP32 63 against 112), from kGradValMinEntries
        // entries on (a half slice is one long chain: 24^3 FP64 6.2 against 3.8 us, FP32
        // 4.9 / 2.4; 32^3 6.6 / 5.6, 5.0 / 4.5; 48^3 13.0 / 14.1, 6.3 / 8.0).  Else warp
        // chunks of kGradValE entries per lane, rows from the row-start bitmasks
        // (7-point 160^3 FP64 88 us on either, 5-point 2000^2 FP32 45 against 54-65 on
        // the slices, whose work per half slice no longer covers its set-up).
        const SellTable *f = nullptr;
        if (h->family == 5 && h->nnz > 8LL * h->n_rows && h->nnz >= kGradValMinEntries &&
            (again || h->sells.count(h->sigma)) && sell_tile_fits(h))
            f = get_sell(h, h->sigma, s, false, false);
        if (f && f->diagonal && (reinterpret_cast<uintptr_t>(grad_val) & 15u) == 0) {
            const SellParams p = sell_params(
                *f, MatRef{h->d_rp, h->d_col, nullptr, nullptr, x, nullptr, nullptr}, alpha, 0.0);
            CK(launch_sell_grad_val(p, h->vk, g, grad_val, h->max_row, s));
            return SPMV_OK;
        }
        ChunkTable *ct = get_chunks(h, kGradValE, false);
        if (!ct) return SPMV_ERR_ALLOC;
        const int mwp = ((kGradValE + 3) / 4) * 4;
        if (launch_grad_val_chunks(h->d_rp, h->d_col, ct->d, ct->masks, mwp, ct->n, h->vk, g, x, alpha,
                                   grad_val, s) != cudaSuccess)
            return SPMV_ERR_CUDA;
    }
    return SPMV_OK;
}

spmv_status spmv_get_transpose(spmv_handle h, int32_t *rowT_ptr, int32_t *colT_idx, int32_t *perm,
                               void *stream) {
    if (!h) return SPMV_ERR_INVALID_ARG;
    if (h->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    spmv_status st = ensure_transpose(h, s);
    if (st != SPMV_OK) return st;
    if (rowT_ptr) std::copy(h->h_rowT.begin(), h->h_rowT.end(), rowT_ptr);
    if (colT_idx && h->nnz) CK(cudaMemcpyAsync(colT_idx, h->d_colT, static_cast<size_t>(h->nnz) * 4, cudaMemcpyDeviceToHost, s));
    if (perm && h->nnz) CK(cudaMemcpyAsync(perm, h->d_perm, static_cast<size_t>(h->nnz) * 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    return SPMV_OK;
}

spmv_status spmv_transpose_noalloc(int32_t n_rows, int32_t n_cols, int64_t nnz,
                                   const int32_t *row_ptr, const int32_t *col_idx,
                                   int32_t *rowT_ptr, int32_t *colT_idx, int32_t *perm,
                                   void *stream) {
    if (n_rows < 0 || n_cols < 0 || nnz < 0 || nnz >= (int64_t(1) << 31)) return SPMV_ERR_INVALID_ARG;
    if (n_cols > transpose_noalloc_max_cols()) return SPMV_ERR_UNSUPPORTED;
    if (!row_ptr || !rowT_ptr || (nnz > 0 && (!col_idx || !colT_idx || !perm))) return SPMV_ERR_INVALID_ARG;
    cudaError_t e = launch_transpose_noalloc(n_rows, n_cols, nnz, row_ptr, col_idx, rowT_ptr, colT_idx,
                                             perm, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? SPMV_OK : SPMV_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// Batched persistent launch
// ---------------------------------------------------------------------------

spmv_status spmv_batched_create(spmv_batch_handle *out, int32_t count, const spmv_handle *mats) {
    if (!out || count < 1 || !mats) return SPMV_ERR_INVALID_ARG;
    *out = nullptr;
    const int vk = mats[0] ? mats[0]->vk : -1;
    for (int32_t m = 0; m < count; ++m)
        if (!mats[m] || mats[m]->vk != vk) return SPMV_ERR_INVALID_ARG;
    for (int32_t m = 0; m < count; ++m)
        if (mats[m]->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard dg(mats[0]->device);
    spmv_batch *b = new (std::nothrow) spmv_batch();
    if (!b) return SPMV_ERR_ALLOC;
    b->count = count;
    b->vk = vk;
    b->device = mats[0]->device;
    b->mats.assign(mats, mats + count);
    const int acc = (vk == kF32) ? kAccFF : kAccF64;
    WarpOps ops;
    // entries per lane from the batch's combined row-length histogram (mean row
    // length); 16 is compiled for both storage types
    int64_t nnz = 0, rows = 0;
    for (int32_t m = 0; m < count; ++m) {
        nnz += mats[m]->nnz;
        rows += mats[m]->n_rows;
    }
    b->E = (rows && static_cast<double>(nnz) / rows < 20.0) ? 7 : 15;
    // slot-major entries per lane from each member's own row-length histogram
    // (its mean row length): 7 below kBatchSlotMeanE9 entries per row, else 9
    b->member_E.resize(static_cast<size_t>(count));
    bool any7 = false, any9 = false;
    for (int32_t m = 0; m < count; ++m) {
        const double mean = mats[m]->n_rows ? static_cast<double>(mats[m]->nnz) / mats[m]->n_rows : 0.0;
        b->member_E[m] = (mean < kBatchSlotMeanE9) ? 7 : 9;
        (b->member_E[m] == 7 ? any7 : any9) = true;
    }
    SlotOps sops;
    if (slot_ops_batched(vk, acc, any7 ? 7 : 9, &sops) && !batch_diagonals(b)) {
        spmv_batched_destroy(b);
        return SPMV_ERR_ALLOC;
    }
    any7 = any9 = false;
    for (int32_t m = 0; m < count; ++m) {
        any7 = any7 || b->member_E[m] == 7;
        any9 = any9 || b->member_E[m] == 9;
    }
    if (any7 && any9 && slot_ops_batched(vk, acc, 7, &sops) && slot_ops_batched(vk, acc, 9, &sops)) {
        // two groups, one copy each, one launch over both
        b->mixed = true;
        b->use_slots = true;
        b->E = 7;
        b->slot_off.assign(static_cast<size_t>(count) + 1, 0);
        b->slot_cnt.assign(static_cast<size_t>(count), 0);
        const size_t vb = (vk == kF64) ? 8 : 4;
        bool ok = true;
        for (int g = 0; g < 2 && ok; ++g) {
            const int EG = g == 0 ? 7 : 9;
            SlotTable &t = g == 0 ? b->slots : b->slots9;
            int32_t *&dcm = g == 0 ? b->d_scmat : b->d_scmat9;
            std::vector<ChunkDesc> d;
            std::vector<uint32_t> lm;
            std::vector<int32_t> cm;
            for (int32_t m = 0; m < count; ++m) {
                if (b->member_E[m] != EG) continue;
                b->slot_off[m] = static_cast<int32_t>(d.size());
                make_slot_chunks(mats[m]->h_rp.data(), mats[m]->n_rows, EG, d, lm, &t.n_long, &t.n_empty);
                b->slot_cnt[m] = static_cast<int32_t>(d.size()) - b->slot_off[m];
                cm.resize(d.size(), m);
            }
            t.n = static_cast<int32_t>(d.size());
            const size_t nslots = d.size() * 32 * EG;
            ok = dmalloc(&t.d, d.size()) == cudaSuccess && dmalloc(&t.lmask, lm.size()) == cudaSuccess &&
                 dmalloc(&dcm, cm.size()) == cudaSuccess && cudaMalloc(&t.vals, nslots * vb + 16) == cudaSuccess &&
                 dmalloc(&t.cols, nslots + 4) == cudaSuccess;
            ok = ok && (d.empty() || cudaMemcpy(t.d, d.data(), sizeof(ChunkDesc) * d.size(), cudaMemcpyHostToDevice) ==
                                         cudaSuccess);
            ok = ok && (lm.empty() || cudaMemcpy(t.lmask, lm.data(), 4 * lm.size(), cudaMemcpyHostToDevice) == cudaSuccess);
            ok = ok && (cm.empty() || cudaMemcpy(dcm, cm.data(), 4 * cm.size(), cudaMemcpyHostToDevice) == cudaSuccess);
            for (int32_t m = 0; ok && m < count; ++m) {
                if (b->member_E[m] != EG) continue;
                const int64_t off = b->slot_off[m];
                const int64_t nch = b->slot_cnt[m];
                ok = launch_slot_relayout(t.d + off, EG, nch * 32 * EG, vk, mats[m]->d_val, mats[m]->d_col,
                                          static_cast<char *>(t.vals) + off * 32 * EG * vb, t.cols + off * 32 * EG,
                                          nullptr) == cudaSuccess;
                b->vals_ver[m] = mats[m]->values_version;
            }
            t.laid.now = true;
        }
        ok = ok && cudaDeviceSynchronize() == cudaSuccess;
        b->h_mats.resize(static_cast<size_t>(count));
        for (int32_t m = 0; m < count; ++m)
            b->h_mats[m] = MatRef{mats[m]->d_rp, mats[m]->d_col, mats[m]->d_val, nullptr, nullptr, nullptr, nullptr};
        b->cur_x.assign(static_cast<size_t>(count), nullptr);
        b->cur_y.assign(static_cast<size_t>(count), nullptr);
        if (ok && (dmalloc(&b->d_mats, b->h_mats.size()) != cudaSuccess || dmalloc(&b->d_err, 1) != cudaSuccess))
            ok = false;
        if (ok && cudaMemset(b->d_err, 0, 4) != cudaSuccess) ok = false;
        if (!ok) {
            spmv_batched_destroy(b);
            return SPMV_ERR_ALLOC;
        }
        *out = b;
        return SPMV_OK;
    }
    const int ES = any7 ? 7 : 9;
    if (slot_ops_batched(vk, acc, ES, &sops)) {
        // the slot-major chunk kernel over one concatenated copy of all matrices
        b->E = ES;
        b->use_slots = true;
        b->slot_off.assign(static_cast<size_t>(count) + 1, 0);
        std::vector<ChunkDesc> d;
        std::vector<uint32_t> lm;
        std::vector<int32_t> cm;
        for (int32_t m = 0; m < count; ++m) {
            b->slot_off[m] = static_cast<int32_t>(d.size());
            if (b->member_E[m] == 0) continue;  // on diagonal slices
            make_slot_chunks(mats[m]->h_rp.data(), mats[m]->n_rows, ES, d, lm, &b->slots.n_long, &b->slots.n_empty);
            cm.resize(d.size(), m);
        }
        b->slot_off[count] = static_cast<int32_t>(d.size());
        b->slots.n = static_cast<int32_t>(d.size());
        const size_t nslots = d.size() * 32 * ES;
        const size_t vb = (vk == kF64) ? 8 : 4;
        bool ok = dmalloc(&b->slots.d, d.size()) == cudaSuccess && dmalloc(&b->slots.lmask, lm.size()) == cudaSuccess &&
                  dmalloc(&b->d_scmat, cm.size()) == cudaSuccess &&
                  cudaMalloc(&b->slots.vals, nslots * vb + 16) == cudaSuccess &&
                  dmalloc(&b->slots.cols, nslots + 4) == cudaSuccess;
        ok = ok && (d.empty() || cudaMemcpy(b->slots.d, d.data(), sizeof(ChunkDesc) * d.size(),
                                            cudaMemcpyHostToDevice) == cudaSuccess);
        ok = ok && (lm.empty() || cudaMemcpy(b->slots.lmask, lm.data(), 4 * lm.size(), cudaMemcpyHostToDevice) ==
                                      cudaSuccess);
        ok = ok && (cm.empty() || cudaMemcpy(b->d_scmat, cm.data(), 4 * cm.size(), cudaMemcpyHostToDevice) ==
                                      cudaSuccess);
        for (int32_t m = 0; ok && m < count; ++m) {
            const int64_t off = b->slot_off[m], nch = b->slot_off[m + 1] - off;
            b->vals_ver[m] = mats[m]->values_version;
            if (nch == 0) continue;
            ok = launch_slot_relayout(b->slots.d + off, ES, nch * 32 * ES, vk, mats[m]->d_val, mats[m]->d_col,
                                      static_cast<char *>(b->slots.vals) + off * 32 * ES * vb,
                                      b->slots.cols + off * 32 * ES, nullptr) == cudaSuccess;
        }
        ok = ok && cudaDeviceSynchronize() == cudaSuccess;
        b->slots.laid.now = true;
        b->h_mats.resize(static_cast<size_t>(count));
        for (int32_t m = 0; m < count; ++m)
            b->h_mats[m] = MatRef{mats[m]->d_rp, mats[m]->d_col, mats[m]->d_val, nullptr, nullptr, nullptr, nullptr};
        b->cur_x.assign(static_cast<size_t>(count), nullptr);
        b->cur_y.assign(static_cast<size_t>(count), nullptr);
        if (ok && (dmalloc(&b->d_mats, b->h_mats.size()) != cudaSuccess || dmalloc(&b->d_err, 1) != cudaSuccess))
            ok = false;
        if (ok && cudaMemset(b->d_err, 0, 4) != cudaSuccess) ok = false;
        b->grid = 0;
        if (!ok) {
            spmv_batched_destroy(b);
            return SPMV_ERR_ALLOC;
        }
        *out = b;
        return SPMV_OK;
    }
    if (!warp_ops(vk, vk, vk, acc, b->E, false, true, &ops)) b->E = 15;
    if (!warp_ops(vk, vk, vk, acc, b->E, false, true, &ops)) {
        delete b;
        return SPMV_ERR_UNSUPPORTED;
    }
    std::vector<ChunkDesc> d;
    std::vector<uint32_t> mk;
    std::vector<int32_t> cm;
    for (int32_t m = 0; m < count; ++m)
        make_chunks(mats[m]->h_rp.data(), mats[m]->n_rows, b->E, m, d, mk, &cm, &b->chunks.n_long,
                    &b->chunks.n_empty);
    b->h_mats.resize(static_cast<size_t>(count));
    for (int32_t m = 0; m < count; ++m)
        b->h_mats[m] = MatRef{mats[m]->d_rp, mats[m]->d_col, mats[m]->d_val, nullptr, nullptr, nullptr, nullptr};
    b->cur_x.assign(static_cast<size_t>(count), nullptr);
    b->cur_y.assign(static_cast<size_t>(count), nullptr);
    spmv_status st = upload_chunks(&b->chunks, d, mk, &cm);
    if (st == SPMV_OK && (dmalloc(&b->d_mats, b->h_mats.size()) != cudaSuccess || dmalloc(&b->d_err, 1) != cudaSuccess))
        st = SPMV_ERR_ALLOC;
    if (st == SPMV_OK && cudaMemset(b->d_err, 0, 4) != cudaSuccess) st = SPMV_ERR_CUDA;
    b->grid = (b->chunks.n + 7) / 8;
    if (st != SPMV_OK) {
        spmv_batched_destroy(b);
        return st;
    }
    *out = b;
    return SPMV_OK;
}

void spmv_batched_destroy(spmv_batch_handle b) {
    if (!b) return;
    DeviceGuard dg(b->device);
    cudaDeviceSynchronize();
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    free_chunks(b->chunks);
    free_slots(b->slots);
    free_slots(b->slots9);
    cudaFree(b->d_scmat);
    cudaFree(b->d_scmat9);
    cudaFree(b->d_dlist);
    cudaFree(b->d_dmembers);
    cudaFree(b->d_dvals);
    cudaFree(b->d_mats);
    cudaFree(b->d_err);
    delete b;
}

spmv_status spmv_batched_apply(spmv_batch_handle b, double alpha, const void *const *x, double beta,
                               void *const *y, void *stream) {
    if (!b || !x || !y) return SPMV_ERR_INVALID_ARG;
    DeviceGuard dg(b->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool recapture = (alpha != b->cur_alpha || beta != b->cur_beta || !b->graph_valid);
    bool ptrs_changed = false;
    for (int32_t m = 0; m < b->count; ++m) {
        if (b->mats[m]->n_rows > 0 && (!x[m] || !y[m])) return SPMV_ERR_INVALID_ARG;
        if (x[m] != b->cur_x[m] || y[m] != b->cur_y[m]) ptrs_changed = true;
    }
    if (ptrs_changed) {
        for (int32_t m = 0; m < b->count; ++m) {
            b->cur_x[m] = x[m];
            b->cur_y[m] = y[m];
            b->h_mats[m].x = x[m];
            b->h_mats[m].y = y[m];
        }
        // the table is read by the kernel when the graph runs; copy it in stream order
        CK(cudaMemcpyAsync(b->d_mats, b->h_mats.data(), sizeof(MatRef) * b->h_mats.size(), cudaMemcpyHostToDevice, s));
        CK(cudaStreamSynchronize(s));
    }
    const int acc = (b->vk == kF32) ? kAccFF : kAccF64;
    if (b->use_slots) {
        if (b->slots.n == 0 && b->slots9.n == 0 && b->n_dlist == 0) return SPMV_OK;
        // members given new values since the copy: lay their values out again
        const size_t vb = (b->vk == kF64) ? 8 : 4;
        for (int32_t m = 0; m < b->count; ++m)
            if (b->mats[m]->values_version != b->vals_ver[m]) {
                if (b->member_E[m] == 0) {
                    if (!batch_diag_values(b, m, s)) return SPMV_ERR_CUDA;
                    continue;
                }
                const int EG = b->mixed ? b->member_E[m] : b->E;
                const SlotTable &t = (b->mixed && EG == 9) ? b->slots9 : b->slots;
                const int64_t off = b->slot_off[m];
                const int64_t nch = b->mixed ? b->slot_cnt[m] : b->slot_off[m + 1] - off;
                CK(launch_slot_relayout(t.d + off, EG, nch * 32 * EG, b->vk, b->mats[m]->d_val, nullptr,
                                        static_cast<char *>(t.vals) + off * 32 * EG * vb, nullptr, s));
                if (!capture_id(s)) b->vals_ver[m] = b->mats[m]->values_version;
            }
        SlotOps sops;
        if (!b->mixed && !slot_ops_batched(b->vk, acc, b->E, &sops)) return SPMV_ERR_UNSUPPORTED;
        if (recapture) {
            if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
            if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
            b->graph_valid = false;
            SlotParams p{};
            p.chunks = b->slots.d;
            p.lmask = b->slots.lmask;
            p.vals = b->slots.vals;
            p.cols = b->slots.cols;
            p.mats = b->d_mats;
            p.cmat = b->d_scmat;
            p.n_chunks = b->slots.n;
            p.alpha = alpha;
            p.beta = beta;
            p.ff = epi_ff(alpha, beta);
            SlotParams p9 = p;
            if (b->mixed) {
                p9.chunks = b->slots9.d;
                p9.lmask = b->slots9.lmask;
                p9.vals = b->slots9.vals;
                p9.cols = b->slots9.cols;
                p9.cmat = b->d_scmat9;
                p9.n_chunks = b->slots9.n;
            }
            // the members on diagonal slices as a second branch of the graph: it fills
            // the SMs that the chunks' last warps leave idle
            cudaStream_t cap, side = nullptr;
            cudaEvent_t join = nullptr;
            const bool fork = b->n_dlist > 0;
            CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
            cudaError_t e = cudaSuccess;
            if (fork) {
                e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
                if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
            }
            if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                cudaError_t le = cudaSuccess;
                if (fork) {
                    le = cudaEventRecord(join, cap);
                    if (le == cudaSuccess) le = cudaStreamWaitEvent(side, join, 0);
                }
                if (le == cudaSuccess && b->mixed) {
                    // the two groups as two kernel nodes of the one graph
                    SlotOps s7, s9;
                    if (!slot_ops_batched(b->vk, acc, 7, &s7) || !slot_ops_batched(b->vk, acc, 9, &s9)) {
                        le = cudaErrorInvalidValue;
                    } else {
                        le = s7.launch(p, cap);
                        if (le == cudaSuccess) le = s9.launch(p9, cap);
                    }
                } else if (le == cudaSuccess) {
                    le = sops.launch(p, cap);
                }
                if (le == cudaSuccess && fork)
                    le = launch_sell_diag_batch(SellBatchParams{b->d_dlist, b->d_dmembers, b->d_mats, b->n_dlist, alpha,
                                                                beta, epi_ff(alpha, beta)}, b->vk, side);
                if (fork) {  // join, also after an error: the capture must end on `cap`
                    if (le == cudaSuccess) le = cudaEventRecord(join, side);
                    const cudaError_t we = cudaStreamWaitEvent(cap, join, 0);
                    if (le == cudaSuccess) le = we;
                }
                e = cudaStreamEndCapture(cap, &b->graph);
                if (le != cudaSuccess) e = le;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
            cudaStreamDestroy(cap);
            if (side) cudaStreamDestroy(side);
            if (join) cudaEventDestroy(join);
            if (e != cudaSuccess) return SPMV_ERR_CUDA;
            b->graph_valid = true;
            b->cur_alpha = alpha;
            b->cur_beta = beta;
        }
        CK(cudaGraphLaunch(b->exec, s));
        return SPMV_OK;
    }
    if (b->chunks.n == 0) return SPMV_OK;
    WarpOps ops;
    if (!warp_ops(b->vk, b->vk, b->vk, acc, b->E, false, true, &ops)) return SPMV_ERR_UNSUPPORTED;
    if (recapture) {
        if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
        if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
        b->graph_valid = false;
        WarpParams p{};
        p.mats = b->d_mats;
        p.chunks = b->chunks.d;
        p.masks = b->chunks.masks;
        p.cmat = b->chunks.cmat;
        p.n_chunks = b->chunks.n;
        p.alpha = alpha;
        p.beta = beta;
        p.err = b->d_err;
        cudaStream_t cap;
        CK(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaError_t le = ops.launch(p, b->chunks.n, cap);
            e = cudaStreamEndCapture(cap, &b->graph);
            if (le != cudaSuccess) e = le;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        cudaStreamDestroy(cap);
        if (e != cudaSuccess) return SPMV_ERR_CUDA;
        b->graph_valid = true;
        b->cur_alpha = alpha;
        b->cur_beta = beta;
    }
    CK(cudaGraphLaunch(b->exec, s));
    return SPMV_OK;
}

spmv_status spmv_batched_get_info(spmv_batch_handle b, int32_t *plan) {
    if (!b || !plan) return SPMV_ERR_INVALID_ARG;
    plan[0] = b->mixed ? 0 : b->E;
    plan[1] = 256;
    plan[2] = b->use_slots ? b->slots.n + b->slots9.n : b->chunks.n;
    plan[3] = b->grid;
    return SPMV_OK;
}

spmv_status spmv_batched_get_member_plan(spmv_batch_handle b, int32_t *entries_per_lane) {
    if (!b || !entries_per_lane) return SPMV_ERR_INVALID_ARG;
    for (int32_t m = 0; m < b->count; ++m)
        entries_per_lane[m] = b->use_slots ? (b->mixed || b->member_E[m] == 0 ? b->member_E[m] : b->E) : b->E;
    return SPMV_OK;
}

// ---------------------------------------------------------------------------
// CG solvers
// ---------------------------------------------------------------------------

spmv_status spmv_cg(spmv_handle h, const double *b, double *x, double tol, int32_t max_iter,
                    double *stats, void *stream) {
    if (!h || !b || !x || h->n_rows != h->n_cols || h->vk != kF64 || max_iter < 0) return SPMV_ERR_INVALID_ARG;
    if (h->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const auto t0 = std::chrono::steady_clock::now();
    spmv_status st = ensure_cg(h, false);
    if (st != SPMV_OK) return st;
    CgWork &w = h->cg;
    const int64_t n = h->n_rows;
    double bb = 0.0, rho = 0.0;
    int32_t it = 0;
    double one[3];
    st = cg_in_one_kernel(h, w, b, x, w.p64, w.q64, w.r64, tol, max_iter, one, s);
    if (st != SPMV_OK && st != SPMV_ERR_UNSUPPORTED && st != SPMV_ERR_TIMEOUT) return st;
    const bool solved = st == SPMV_OK;
    if (solved) {
        rho = one[0];
        it = static_cast<int32_t>(one[1]);
        bb = one[2];
    } else {
    // x = 0, r = b, p = b, rho = b.b
    CK(cudaMemsetAsync(x, 0, static_cast<size_t>(n) * 8, s));
    CK(cudaMemcpyAsync(w.r64, b, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToDevice, s));
    CK(cudaMemcpyAsync(w.p64, b, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToDevice, s));
    CK(cg_dot(b, kF64, b, kF64, n, w.partials, w.sc, kOpStore, kScRho, s));
    CK(cudaMemcpyAsync(w.host, w.sc + kScRho, 8, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    bb = rho = w.host[0];
    // the residual is read back every kCheckEvery iterations (one host round trip
    // per check, not per iteration); CG may run up to kCheckEvery-1 extra steps
    auto iter = [&](cudaStream_t cs) -> spmv_status {
        spmv_status s2 = apply_impl(h, 1.0, w.p64, kF64, 0.0, w.q64, kF64, cs);
        if (s2 != SPMV_OK) return s2;
        if (cg_dot(w.p64, kF64, w.q64, kF64, n, w.partials, w.sc, kOpAlpha, 0, cs) != cudaSuccess ||
            cg_update64(x, w.r64, w.p64, w.q64, n, w.partials, w.sc, cs) != cudaSuccess ||
            cg_direction(w.p64, w.r64, kF64, w.sc, n, cs) != cudaSuccess)
            return SPMV_ERR_CUDA;
        return SPMV_OK;
    };
    const int64_t key = static_cast<int64_t>(h->family) * 1000 + h->E;
    while (it < max_iter && std::sqrt(rho) > tol * std::sqrt(bb)) {
        if (max_iter - it >= kCheckEvery && w.cg64 && w.cg64_key == key && w.cg64_x == x) {
            CK(cudaGraphLaunch(w.cg64, s));
            it += kCheckEvery;
        } else {
            const int blk = std::min<int32_t>(kCheckEvery, max_iter - it);
            for (int j = 0; j < blk; ++j) {
                st = iter(s);
                if (st != SPMV_OK) return st;
            }
            it += blk;
            if (blk == kCheckEvery && (!w.cg64 || w.cg64_key != key || w.cg64_x != x)) {
                if (w.cg64) { cudaGraphExecDestroy(w.cg64); w.cg64 = nullptr; }
                st = ready_for_capture(h, kF64, kF64);
                if (st == SPMV_OK)
                    st = capture_graph([&](cudaStream_t cs) -> spmv_status {
                        for (int j = 0; j < kCheckEvery; ++j) {
                            const spmv_status s3 = iter(cs);
                            if (s3 != SPMV_OK) return s3;
                        }
                        return SPMV_OK;
                    }, &w.cg64);
                if (st != SPMV_OK) return st;
                w.cg64_key = key;
                w.cg64_x = x;
            }
        }
        CK(cudaMemcpyAsync(w.host, w.sc + kScRho, 8, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        rho = w.host[0];
    }
    }
    // true residual in FP64
    CK(cudaMemcpyAsync(w.r64, b, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToDevice, s));
    st = apply_impl(h, -1.0, x, kF64, 1.0, w.r64, kF64, s);
    if (st != SPMV_OK) return st;
    CK(cg_dot(w.r64, kF64, w.r64, kF64, n, w.partials, w.sc, kOpStore, kScNorm, s));
    CK(cudaMemcpyAsync(w.host, w.sc + kScNorm, 8, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    const double relres = bb > 0 ? std::sqrt(w.host[0] / bb) : 0.0;
    if (stats) {
        stats[0] = 1;
        stats[1] = it;
        stats[2] = relres;
        stats[3] = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    return (std::sqrt(rho) > tol * std::sqrt(bb)) ? SPMV_ERR_NOT_CONVERGED : SPMV_OK;
}

spmv_status spmv_ir_cg(spmv_handle h, const double *b, double *x, double outer_tol,
                       int32_t max_outer, double inner_tol, int32_t max_inner, double *stats,
                       void *stream) {
    if (!h || !b || !x || h->n_rows != h->n_cols || h->vk != kF64 || max_outer < 0 || max_inner < 1)
        return SPMV_ERR_INVALID_ARG;
    if (h->sym) return SPMV_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const auto t0 = std::chrono::steady_clock::now();
    spmv_status st = ensure_cg(h, true);
    if (st != SPMV_OK) return st;
    st = ensure_mirror32(h, s);
    if (st != SPMV_OK) return st;
    spmv_matrix *A32 = h->mirror32;
    CgWork &w = h->cg;
    const int64_t n = h->n_rows;
    CK(cudaMemsetAsync(x, 0, static_cast<size_t>(n) * 8, s));
    CK(cg_dot(b, kF64, b, kF64, n, w.partials, w.sc, kOpStore, kScNorm, s));
    CK(cudaMemcpyAsync(w.host, w.sc + kScNorm, 8, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    const double bnorm = std::sqrt(w.host[0]);
    int32_t outer = 0;
    int64_t inner_total = 0;
    double relres = 0.0;
    bool converged = false, one_kernel = true;
    for (;;) {
        // outer (FP64): r = b - A x, ||r||
        CK(cudaMemcpyAsync(w.r64, b, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToDevice, s));
        st = apply_impl(h, -1.0, x, kF64, 1.0, w.r64, kF64, s);
        if (st != SPMV_OK) return st;
        CK(cg_dot(w.r64, kF64, w.r64, kF64, n, w.partials, w.sc, kOpStore, kScNorm, s));
        CK(cudaMemcpyAsync(w.host, w.sc + kScNorm, 8, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        const double rnorm = std::sqrt(w.host[0]);
        relres = bnorm > 0 ? rnorm / bnorm : 0.0;
        if (relres <= outer_tol) { converged = true; break; }
        if (outer >= max_outer) break;
        // inner (FP32 storage): CG on A d = r / ||r||
        CK(cg_scale_to32(w.r64, w.r32, 1.0 / rnorm, n, s));
        double one[3];
        st = one_kernel ? cg_in_one_kernel(A32, w, w.r32, w.d32, w.p32, w.q32, w.r32, inner_tol, max_inner, one, s)
                        : SPMV_ERR_UNSUPPORTED;
        if (st == SPMV_OK) {
            inner_total += static_cast<int32_t>(one[1]);
            CK(cg_axpy_64_32(x, w.d32, rnorm, n, s));
            ++outer;
            continue;
        }
        if (st == SPMV_ERR_TIMEOUT) {  // no second wait in this call
            one_kernel = false;
            CK(cg_scale_to32(w.r64, w.r32, 1.0 / rnorm, n, s));
        } else if (st != SPMV_ERR_UNSUPPORTED) {
            return st;
        }
        CK(cudaMemsetAsync(w.d32, 0, static_cast<size_t>(n) * 4, s));
        CK(cudaMemcpyAsync(w.p32, w.r32, static_cast<size_t>(n) * 4, cudaMemcpyDeviceToDevice, s));
        CK(cg_dot(w.r32, kF32, w.r32, kF32, n, w.partials, w.sc, kOpStore, kScRho, s));
        CK(cudaMemcpyAsync(w.host, w.sc + kScRho, 8, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        const double rho0 = w.host[0];
        double rho = rho0;
        int32_t it = 0;
        auto inner_iter = [&](cudaStream_t cs) -> spmv_status {
            // q = A p with p.q (and the step alpha) reduced by the product itself
            // on the row slices; elsewhere the product, then the dot
            SellOps lo;
            SellParams lp;
            if (sell_launch_of(A32, 1.0, w.p32, kF32, 0.0, w.q32, kF32, cs, &lo, &lp) && lo.launch_dot &&
                lp.n_slices > 0 && lp.n_ctas <= cg_partials_cap()) {
                if (lo.launch_dot(lp, cg_red_out(w.partials, w.sc, kOpAlpha, 0), cs) != cudaSuccess)
                    return SPMV_ERR_CUDA;
            } else {
                spmv_status s2 = apply_impl(A32, 1.0, w.p32, kF32, 0.0, w.q32, kF32, cs);
                if (s2 != SPMV_OK) return s2;
                if (cg_dot(w.p32, kF32, w.q32, kF32, n, w.partials, w.sc, kOpAlpha, 0, cs) != cudaSuccess)
                    return SPMV_ERR_CUDA;
            }
            if (cg_update32(w.d32, w.r32, w.p32, w.q32, n, w.partials, w.sc, cs) != cudaSuccess ||
                cg_direction(w.p32, w.r32, kF32, w.sc, n, cs) != cudaSuccess)
                return SPMV_ERR_CUDA;
            return SPMV_OK;
        };
        const int64_t key = static_cast<int64_t>(A32->family) * 1000 + A32->E;
        while (it < max_inner && std::sqrt(rho) > inner_tol * std::sqrt(rho0)) {
            if (max_inner - it >= kCheckEvery && w.inner32 && w.inner32_key == key) {
                CK(cudaGraphLaunch(w.inner32, s));
                it += kCheckEvery;
            } else {
                // plain launches (also the first block, which prepares every
                // kernel before the block is captured)
                const int blk = std::min<int32_t>(kCheckEvery, max_inner - it);
                for (int j = 0; j < blk; ++j) {
                    st = inner_iter(s);
                    if (st != SPMV_OK) return st;
                }
                it += blk;
                if (blk == kCheckEvery && (!w.inner32 || w.inner32_key != key)) {
                    if (w.inner32) { cudaGraphExecDestroy(w.inner32); w.inner32 = nullptr; }
                    st = ready_for_capture(A32, kF32, kF32);
                    if (st == SPMV_OK)
                        st = capture_graph([&](cudaStream_t cs) -> spmv_status {
                            for (int j = 0; j < kCheckEvery; ++j) {
                                const spmv_status s3 = inner_iter(cs);
                                if (s3 != SPMV_OK) return s3;
                            }
                            return SPMV_OK;
                        }, &w.inner32);
                    if (st != SPMV_OK) return st;
                    w.inner32_key = key;
                }
            }
            CK(cudaMemcpyAsync(w.host, w.sc + kScRho, 8, cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            rho = w.host[0];
        }
        inner_total += it;
        // update (FP64): x += ||r|| d
        CK(cg_axpy_64_32(x, w.d32, rnorm, n, s));
        ++outer;
    }
    if (stats) {
        stats[0] = outer;
        stats[1] = static_cast<double>(inner_total);
        stats[2] = relres;
        stats[3] = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    return converged ? SPMV_OK : SPMV_ERR_NOT_CONVERGED;
}

spmv_status spmv_validate_device(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t *row_ptr,
                                 const int32_t *col_idx, void *stream) {
    if (n_rows < 0 || n_cols < 0 || nnz < 0 || nnz >= (int64_t(1) << 31)) return SPMV_ERR_INVALID_ARG;
    if (!row_ptr || (nnz > 0 && !col_idx)) return SPMV_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int32_t *bad = nullptr;
    if (dmalloc(&bad, 1) != cudaSuccess) return SPMV_ERR_ALLOC;
    int32_t v = 0;
    cudaError_t e = cudaMemsetAsync(bad, 0, 4, s);
    if (e == cudaSuccess) e = launch_validate(n_rows, n_cols, nnz, row_ptr, col_idx, bad, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&v, bad, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(bad);
    if (e != cudaSuccess) return SPMV_ERR_CUDA;
    return v ? SPMV_ERR_INVALID_INDEX : SPMV_OK;
}

spmv_status spmv_selftest_wait_timeout(spmv_handle h, int64_t limit_ns, void *stream) {
    if (!h || limit_ns < 1000 || limit_ns > static_cast<int64_t>(kWaitLimitNs)) return SPMV_ERR_INVALID_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CK(launch_wait_timeout(static_cast<uint64_t>(limit_ns), h->d_err, s));
    return spmv_check_device_error(h, stream);
}

spmv_status spmv_check_device_error(spmv_handle h, void *stream) {
    if (!h) return SPMV_ERR_INVALID_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int32_t v = 0;
    CK(cudaMemcpyAsync(&v, h->d_err, 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (v != 0) {
        CK(cudaMemsetAsync(h->d_err, 0, 4, s));
        CK(cudaStreamSynchronize(s));
        return SPMV_ERR_TIMEOUT;
    }
    return SPMV_OK;
}

}  // extern "C"
