// Compiled configurations of the sorted row-slice kernel (plan family 5) and its
// relayout kernel: FP64 values and vectors, and FP32 storage with FP32 runs
// (every row at most 11 entries, so a lane's chain over a row is a run) or FP32
// runs of one block (4 slot rows) each folded into float-float.
#include <algorithm>
#include <map>
#include <mutex>

#include "internal.h"
#include "sell_kernel.cuh"

namespace spmv {

bool sell_ops(int vk, int xk, int yk, int acc, SellOps *ops, int32_t max_row) {
    if (vk == kF64 && xk == kF64 && yk == kF64 && acc == kAccF64) {
        ops->launch = &SellKernel<double, double, double, AccF64>::launch;
        ops->ctas_for = &SellKernel<double, double, double, AccF64>::ctas_for;
        ops->launch_ind = &SellKernel<double, double, double, AccF64>::launch_ind;
        ops->launch_dot = nullptr;
        return true;
    }
    if (vk == kF32 && xk == kF32 && yk == kF32 && acc == kAccFF && max_row <= kFRMaxRun) {
        ops->launch = &SellKernel<float, float, float, AccFR>::launch;
        ops->ctas_for = &SellKernel<float, float, float, AccFR>::ctas_for;
        ops->launch_ind = &SellKernel<float, float, float, AccFF>::launch_ind;
        ops->launch_dot = &SellKernel<float, float, float, AccFR>::launch_dot;
        return true;
    }
    if (vk == kF32 && xk == kF32 && yk == kF32 && acc == kAccFF) {
        ops->launch = &SellKernel<float, float, float, AccFRF>::launch;
        ops->ctas_for = &SellKernel<float, float, float, AccFRF>::ctas_for;
        ops->launch_ind = &SellKernel<float, float, float, AccFF>::launch_ind;
        ops->launch_dot = &SellKernel<float, float, float, AccFRF>::launch_dot;
        return true;
    }
    return false;
}

cudaError_t launch_sell_mr(const SellParams &b, const double *X, double *Y, int64_t ldx, int64_t ldy, bool vec,
                           cudaStream_t s) {
    if (b.n_slices <= 0 || b.n_ctas <= 0) return cudaSuccess;
    const SellMrParams q{b, X, Y, ldx, ldy};
    if (vec) k_sell_mr<true><<<b.n_ctas, 256, 0, s>>>(q);
    else k_sell_mr<false><<<b.n_ctas, 256, 0, s>>>(q);
    return cudaGetLastError();
}

// Resident CTAs of 256 threads of KERNEL on the device with smem bytes of shared memory
// (up to `most`), asked once per amount: the queries cost a few us, as much as a small
// launch.  0: an error.
template <auto KERNEL>
static int resident(size_t smem, size_t most) {
    static int dev_of = -1;
    static std::map<size_t, int> known;
    static std::mutex m;
    std::lock_guard<std::mutex> lock(m);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    if (dev != dev_of) {
        known.clear();
        if (most > 0 && cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(most)) != cudaSuccess)
            return 0;
        dev_of = dev;
    }
    const auto it = known.find(smem);
    if (it != known.end()) return it->second;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, KERNEL, 256, smem) != cudaSuccess) return 0;
    return known[smem] = per_sm * sms;
}

template <typename VT, typename ACC>
static cudaError_t diag_batch_as(const SellBatchParams &p, cudaStream_t s) {
    const int64_t want = (2 * static_cast<int64_t>(p.n_list) + 7) / 8, lim = resident<k_sell_diag_batch<VT, ACC>>(0, 0);
    if (lim <= 0) return cudaErrorInvalidConfiguration;
    k_sell_diag_batch<VT, ACC><<<static_cast<int>(want < lim ? want : lim), 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_sell_diag_batch(const SellBatchParams &p, int vk, cudaStream_t s) {
    if (p.n_list <= 0) return cudaSuccess;
    return vk == kF64 ? diag_batch_as<double, AccF64>(p, s) : diag_batch_as<float, AccFRF>(p, s);
}

// How a pass of R right-hand sides runs: V per lane, L = ceil(R/V) lanes per row, G =
// 32/L rows at a time.  The FP64 pipe needs V warp FMAs (17 cycles each) per G rows
// and slot; with scattered columns L1 also looks up a line per row for each of the
// pass's load instructions; 6 stand for the rest of a slot's work (16 right-hand
// sides on the 5-point matrix: V = 4 280 us, V = 2 350).  V odd, or rows not 16-byte aligned: one load per
// right-hand side, else one per two.
static void rhs_plan(int R, bool vec, bool scattered, int *V_out, bool *vec_out) {
    double best = 1e30;
    for (int V = 2; V <= 7; ++V) {
        const bool pv = vec && V % 2 == 0 && R % V == 0;
        if (V == 6 && !pv) continue;
        const int L = (R + V - 1) / V;
        if (L > 16) continue;
        const int G = 32 / L;
        const double fma = 17.0 * V, lines = scattered ? (pv ? V / 2 : V) * G + 4.0 : 0.0;
        const double cost = ((fma > lines ? fma : lines) + 6.0) / G * (pv ? 1.0 : 1.02);
        if (cost < best) {
            best = cost;
            *V_out = V;
            *vec_out = pv;
        }
    }
}

cudaError_t launch_sell_rhs(const SellParams &b, const double *X, double *Y, int64_t ldx, int64_t ldy, int R, bool vec,
                            bool scattered, cudaStream_t s) {
    if (b.n_slices <= 0 || b.n_ctas <= 0) return cudaSuccess;
    if (R < 1 || R > kSellMaxRhs) return cudaErrorInvalidValue;
    int V = 2;
    bool pv = false;
    rhs_plan(R, vec, scattered, &V, &pv);
    const int L = (R + V - 1) / V;
    const SellRhsParams q{SellMrParams{b, X, Y, ldx, ldy}, R, L, 32 / L};
    switch (V) {
        case 2:
            if (pv) k_sell_rhs<2, true><<<b.n_ctas, 512, 0, s>>>(q);
            else k_sell_rhs<2, false><<<b.n_ctas, 512, 0, s>>>(q);
            break;
        case 3: k_sell_rhs<3, false><<<b.n_ctas, 512, 0, s>>>(q); break;
        case 4:
            if (pv) k_sell_rhs<4, true><<<b.n_ctas, 512, 0, s>>>(q);
            else k_sell_rhs<4, false><<<b.n_ctas, 512, 0, s>>>(q);
            break;
        case 5: k_sell_rhs<5, false><<<b.n_ctas, 512, 0, s>>>(q); break;
        case 6: k_sell_rhs<6, true><<<b.n_ctas, 512, 0, s>>>(q); break;
        default: k_sell_rhs<7, false><<<b.n_ctas, 512, 0, s>>>(q); break;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The row-slice tables on the device (windows of kSellBuildSigma rows, no row of more
// than kSellBuildMaxRow entries), the same as the host builds for any window: one CTA
// sorts a window's rows by length, longest first, ties in row order (a stable counting
// sort: ranks of equal lengths from a match in each warp, warps and rounds of 256 rows
// in order); the widths' exclusive scan gives the first slot rows.
// ---------------------------------------------------------------------------
constexpr int kBuildBins = kSellBuildMaxRow + 1;

__global__ void __launch_bounds__(256) k_sell_sort(const int32_t *__restrict__ rp, int32_t n_rows,
                                                   int32_t *__restrict__ srows, int32_t *__restrict__ width,
                                                   uint32_t *__restrict__ too_long) {
    constexpr int NW = 8;
    __shared__ int32_t s_base[kBuildBins];      // next place of each length, longest first
    __shared__ int32_t s_wc[NW][kBuildBins];    // a round's counts per warp, then its offsets
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kSellBuildSigma;
    const int nr = static_cast<int>(min(static_cast<int64_t>(kSellBuildSigma), n_rows - r0));
    // bin of a row: kSellBuildMaxRow - length (a longer row only sets the flag)
    auto bin_of = [&](int i) {
        const int32_t len = __ldg(rp + r0 + i + 1) - __ldg(rp + r0 + i);
        return max(0, kSellBuildMaxRow - len);
    };
    for (int b = t; b < kBuildBins; b += 256) {
        s_base[b] = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) s_wc[q][b] = 0;
    }
    __syncthreads();
    for (int i = t; i < nr; i += 256) {
        atomicAdd(&s_base[bin_of(i)], 1);
        if (__ldg(rp + r0 + i + 1) - __ldg(rp + r0 + i) > kSellBuildMaxRow) atomicOr(too_long, 1u);
    }
    __syncthreads();
    if (w == 0) {  // exclusive scan of the bins
        int32_t run = 0;
        for (int b0 = 0; b0 < kBuildBins; b0 += 32) {
            const int b = b0 + lane;
            const int32_t v = b < kBuildBins ? s_base[b] : 0;
            int32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (b < kBuildBins) s_base[b] = run + inc - v;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
    for (int i0 = 0; i0 < nr; i0 += 256) {
        const int i = i0 + t;
        const bool ok = i < nr;
        const int b = ok ? bin_of(i) : kBuildBins;
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (ok && rank == 0) s_wc[w][b] = __popc(peers);
        __syncthreads();
        for (int q = t; q < kBuildBins; q += 256) {
            int32_t run = s_base[q];
#pragma unroll
            for (int u = 0; u < NW; ++u) {
                const int32_t c = s_wc[u][q];
                s_wc[u][q] = run;
                run += c;
            }
            s_base[q] = run;
        }
        __syncthreads();
        if (ok) {
            const int pos = s_wc[w][b] + rank;
            srows[r0 + pos] = static_cast<int32_t>(r0 + i);
            if (pos % kSellC == 0) width[(r0 + pos) / kSellC] = kSellBuildMaxRow - b;
        }
        __syncthreads();
        for (int q = t; q < kBuildBins; q += 256)
#pragma unroll
            for (int u = 0; u < NW; ++u) s_wc[u][q] = 0;
        __syncthreads();
    }
    // the last slice's missing rows
    for (int i = nr + t; i < (nr + kSellC - 1) / kSellC * kSellC; i += 256) srows[r0 + i] = -1;
}

// Descriptors from the scanned widths (off[n_slices] = their sum); a slice's place
// among the diagonals is off / 4 + slice, which leaves room for its (w + 3) / 4.  The
// first n_ctas + 1 threads also cut the slices into ranges of equal work (w + 1 slot
// rows per slice).
__global__ void __launch_bounds__(256) k_sell_tables(const int32_t *__restrict__ width, const int32_t *__restrict__ off,
                                                     int32_t n_slices, int32_t n_ctas, int2 *__restrict__ d,
                                                     int4 *__restrict__ dtmp, int32_t *__restrict__ cstart) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < n_slices; i += stride) {
        const int32_t o = off[i], w = width[i];
        d[i] = make_int2(o + kSellU, w);
        dtmp[i] = make_int4(o + kSellU, w, static_cast<int>(i), o / 4 + static_cast<int>(i));
    }
    for (int64_t g = i0; g <= n_ctas; g += stride) {
        if (g == n_ctas) {
            cstart[g] = n_slices;
            continue;
        }
        const int64_t target = (static_cast<int64_t>(off[n_slices]) + n_slices) * kSellC * g / n_ctas;
        int32_t lo = 0, hi = n_slices;  // the first slice with as much work before it
        while (lo < hi) {
            const int32_t mid = lo + (hi - lo) / 2;
            if ((static_cast<int64_t>(off[mid]) + mid) * kSellC < target) lo = mid + 1;
            else hi = mid;
        }
        cstart[g] = lo;
    }
}

cudaError_t launch_sell_build(const int32_t *rp, int32_t n_rows, int32_t n_slices, int32_t n_ctas, int32_t *srows,
                              int32_t *width, int32_t *off, int32_t *sums, uint32_t *too_long, void *d, void *dtmp,
                              int32_t *cstart, cudaStream_t s) {
    static_assert(kSellBuildSigma % kSellC == 0, "windows hold whole slices");
    k_sell_sort<<<(n_rows + kSellBuildSigma - 1) / kSellBuildSigma, 256, 0, s>>>(rp, n_rows, srows, width, too_long);
    cudaError_t e = launch_scan(width, n_slices, sums, off, s);
    if (e != cudaSuccess) return e;
    const int want = (std::max(n_slices, n_ctas + 1) + 255) / 256;
    k_sell_tables<<<std::min(want, 2048), 256, 0, s>>>(width, off, n_slices, n_ctas, static_cast<int2 *>(d),
                                                       static_cast<int4 *>(dtmp), cstart);
    return cudaGetLastError();
}

// One warp per slice of dtmp: the diagonals of a diagonal slice into diag from
// the slice's place on; place -1 for a slice that is not diagonal.  count[0], [1]:
// slot rows and number of the diagonal slices.  A row of a diagonal slice has a
// stored row and a column in every slot; a sum row + diagonal is then a stored
// column, so it is in range.
__global__ void __launch_bounds__(256) k_sell_mark_diag(int4 *__restrict__ dtmp, int32_t n_slices,
                                                        const int32_t *__restrict__ srows,
                                                        const int32_t *__restrict__ cols, int32_t *__restrict__ diag,
                                                        uint32_t *__restrict__ count) {
    const int lane = threadIdx.x & 31;
    uint32_t rows = 0, num = 0;
    for (int s = blockIdx.x * 8 + (threadIdx.x >> 5); s < n_slices; s += gridDim.x * 8) {
        const int4 d = dtmp[s];
        bool ok = d.y > 0;
        if (ok) {
            const int32_t *rs = srows + static_cast<int64_t>(d.z) * kSellC + lane;
            const int32_t ra = rs[0], rb = rs[32];
            bool mine = ra >= 0 && rb >= 0;
            for (int j = 0; j < d.y; ++j) {
                const int32_t *c = cols + (static_cast<int64_t>(d.x) + j) * kSellC + lane;
                const int32_t ca = c[0], cb = c[32];
                const int32_t da = ca - ra;  // two numbers in [-1, 2^31): no overflow
                const int32_t d0 = __shfl_sync(0xffffffffu, da, 0);
                mine = mine && ca >= 0 && cb >= 0 && da == d0 && cb - rb == d0;
                if (lane == 0) diag[static_cast<int64_t>(d.w) * 4 + j] = d0;
            }
            ok = __all_sync(0xffffffffu, mine);
        }
        if (ok) {
            rows += static_cast<uint32_t>(d.y);
            ++num;
        } else if (lane == 0) {
            dtmp[s].w = -1;
        }
    }
    if (lane == 0 && num) {
        atomicAdd(count, rows);
        atomicAdd(count + 1, num);
    }
}

// dorder = the slices of dtmp that are not diagonal, then the diagonal ones, each
// in their order (one block; count[1] diagonal slices).  The others come first
// because their chains are the longest, and because left in place they recur with
// a period that divides the number of warps, which would hand them to the same
// warps every time (7-point 160^3 FP32 34.5 against 28.4 us).
__global__ void __launch_bounds__(1024) k_sell_order(const int4 *__restrict__ dtmp, int32_t n_slices,
                                                     const uint32_t *__restrict__ count, int4 *__restrict__ dorder) {
    __shared__ int s_warp[32];
    __shared__ int s_total;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n_rest = n_slices - static_cast<int>(count[1]);
    int before = 0;  // slices that are not diagonal ahead of this round
    for (int s0 = 0; s0 < n_slices; s0 += 1024) {
        const int s = s0 + static_cast<int>(threadIdx.x);
        const int4 d = s < n_slices ? dtmp[s] : make_int4(0, 0, 0, 0);
        const bool rest = s < n_slices && d.w < 0;
        const unsigned m = __ballot_sync(0xffffffffu, rest);
        if (lane == 0) s_warp[w] = __popc(m);
        __syncthreads();
        if (w == 0) {
            const int v = s_warp[lane];
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            s_warp[lane] = inc - v;
            if (lane == 31) s_total = inc;
        }
        __syncthreads();
        const int rank = before + s_warp[w] + __popc(m & ((1u << lane) - 1u));
        if (s < n_slices) dorder[rest ? rank : n_rest + (s - rank)] = d;
        before += s_total;
        __syncthreads();
    }
}

cudaError_t launch_sell_mark_diag(void *dtmp, int32_t n_slices, const int32_t *srows, const int32_t *cols,
                                  void *diag, uint32_t *count, void *dorder, cudaStream_t s) {
    if (n_slices <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int want = (n_slices + 7) / 8;
    k_sell_mark_diag<<<want < 8 * sms ? want : 8 * sms, 256, 0, s>>>(static_cast<int4 *>(dtmp), n_slices, srows,
                                                                     cols, static_cast<int32_t *>(diag), count);
    k_sell_order<<<1, 1024, 0, s>>>(static_cast<const int4 *>(dtmp), n_slices, count, static_cast<int4 *>(dorder));
    return cudaGetLastError();
}

// rowpos[r] = position of row r's first slot in a row-slice copy (-1 before: rows
// outside the slices).
__global__ void __launch_bounds__(256) k_sell_rowpos(const int2 *__restrict__ slices, const int32_t *__restrict__ srows,
                                                     int32_t n_slices, int32_t *__restrict__ rowpos) {
    const int64_t total = static_cast<int64_t>(n_slices) * kSellC;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int32_t r = srows[t];
        if (r >= 0) rowpos[r] = slices[t / kSellC].x * kSellC + static_cast<int32_t>(t % kSellC);
    }
}

// vpos[slot] of the slices of A^T: where the slot's value is in A's slices (rowpos:
// the first slot of each row of A; entry perm[k] of A lies in row colT[k]).
__global__ void __launch_bounds__(256) k_sell_vpos(const int2 *__restrict__ slices, const int32_t *__restrict__ srows,
                                                   int32_t n_slices, const int32_t *__restrict__ rowT,
                                                   const int32_t *__restrict__ colT, const int32_t *__restrict__ perm,
                                                   const int32_t *__restrict__ rp, const int32_t *__restrict__ rowpos,
                                                   int32_t *__restrict__ vpos) {
    const int64_t total = static_cast<int64_t>(n_slices) * kSellC;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int2 d = slices[t / kSellC];
        if (d.y <= 0) continue;
        const int32_t row = srows[t];
        const int32_t k0 = row >= 0 ? rowT[row] : 0;
        const int32_t len = row >= 0 ? rowT[row + 1] - k0 : 0;
        for (int j = 0; j < d.y; ++j) {
            int32_t pos = -1;
            if (j < len) {
                const int32_t i = colT[k0 + j];
                pos = rowpos[i] + (perm[k0 + j] - rp[i]) * kSellC;
            }
            vpos[(static_cast<int64_t>(d.x) + j) * kSellC + t % kSellC] = pos;
        }
    }
}

static int slice_grid(int32_t n_slices) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (static_cast<int64_t>(n_slices) * kSellC + 255) / 256;
    return static_cast<int>(want < 16LL * sms ? want : 16LL * sms);
}

cudaError_t launch_sell_vpos(const void *slicesA, const int32_t *srowsA, int32_t nA, const void *slicesT,
                             const int32_t *srowsT, int32_t nT, const int32_t *rp, const int32_t *rowT,
                             const int32_t *colT, const int32_t *perm, int32_t *rowpos, int32_t *vpos, cudaStream_t s) {
    if (nA <= 0 || nT <= 0) return cudaSuccess;
    k_sell_rowpos<<<slice_grid(nA), 256, 0, s>>>(static_cast<const int2 *>(slicesA), srowsA, nA, rowpos);
    k_sell_vpos<<<slice_grid(nT), 256, 0, s>>>(static_cast<const int2 *>(slicesT), srowsT, nT, rowT, colT, perm, rp,
                                               rowpos, vpos);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// CRS order <-> row slices through shared memory.  A warp takes half a slice (32
// rows of at most kTileMaxW entries, one per lane) and holds its entries in a
// shared-memory tile, packed as they lie in CRS order: rows that follow each other
// there form a segment (on a grid nearly always the whole half slice, two across
// the end of a grid line), and a segment starts at its entries' alignment.  On the
// CRS side a segment is then one contiguous run, and what goes to CRS order leaves
// by one bulk copy (cp.async.bulk) per segment, without passing through registers;
// on the slice side lane l reads or writes row l.  The descriptor, row and row
// pointers of the following half slices are loaded ahead (a chain of three loads).
// ---------------------------------------------------------------------------
constexpr int kTileMaxW = 32;

// The half slices i, i + nw, ... of a warp, each with its descriptor d, the lane's
// row r (-1: none) and the entries [k0, k1) of that row; f(i, d, r, k0, k1).
template <typename F>
__device__ __forceinline__ void each_half_slice(const int4 *__restrict__ dorder, const int32_t *__restrict__ srows,
                                                int32_t n_slices, const int32_t *__restrict__ rp, int lane, F f) {
    const int n = 2 * n_slices, nw = gridDim.x * 8;
    int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    auto desc_of = [&](int k) { return __ldg(dorder + (k < n ? k >> 1 : n_slices - 1)); };
    auto row_of = [&](const int4 &d, int k) {
        return __ldg(srows + static_cast<int64_t>(d.z) * kSellC + (k & 1) * 32 + lane);
    };
    int4 d0 = desc_of(i), d1 = desc_of(i + nw), d2 = desc_of(i + 2 * nw);
    int r0 = row_of(d0, i), r1 = row_of(d1, i + nw);
    int k0 = r0 >= 0 ? __ldg(rp + r0) : 0, k1 = r0 >= 0 ? __ldg(rp + r0 + 1) : 0;
    for (; i < n; i += nw) {
        const int4 d3 = desc_of(i + 3 * nw);
        const int r2 = row_of(d2, i + 2 * nw);
        const int n0 = r1 >= 0 ? __ldg(rp + r1) : 0, n1 = r1 >= 0 ? __ldg(rp + r1 + 1) : 0;
        f(i, d0, r0, k0, k1);
        d0 = d1;
        d1 = d2;
        d2 = d3;
        r0 = r1;
        r1 = r2;
        k0 = n0;
        k1 = n1;
    }
}

// The packing of one half slice's rows into the tile (A entries are 16 bytes).
template <typename VT>
struct TilePack {
    static constexpr int A = 16 / sizeof(VT);
    int pos;         // tile index of the lane's row
    unsigned heads;  // lanes whose row starts a segment
    int kend;        // at a segment's first lane: the end of its entries in CRS order
    static __host__ __device__ constexpr int entries(int max_w) { return 32 * max_w + 33 * A; }
    __device__ __forceinline__ TilePack(int w, int k0, int k1, int lane) {
        const int prev = __shfl_up_sync(0xffffffffu, k1, 1);
        heads = __ballot_sync(0xffffffffu, lane == 0 || k0 != prev);
        const unsigned upto = heads & (0xffffffffu >> (31 - lane));
        const int first = 31 - __clz(upto);  // the segment's first lane
        const int ks = __shfl_sync(0xffffffffu, k0, first);
        const int base = first * w + A * (__popc(upto) - 1);
        pos = base + ((ks - base) & (A - 1)) + (k0 - ks);
        const unsigned after = lane == 31 ? 0u : heads & ~(0xffffffffu >> (31 - lane));
        kend = __shfl_sync(0xffffffffu, k1, after ? __ffs(after) - 2 : 31);
    }
    // The tile's entries to dst in CRS order (16-byte aligned; whole 16-byte units by
    // bulk copy, a segment's ragged ends by its first lane).  Every lane calls it
    // after writing its part; the tile may be written again after drain().
    __device__ __forceinline__ void store(const VT *tile, VT *dst, int k0, int lane) const {
        fence_proxy_async_smem();
        __syncwarp();
        if ((heads >> lane) & 1u) {
            const VT *src = tile + pos - k0;  // src[k]: entry k
            const int a0 = min((k0 + A - 1) & ~(A - 1), kend), a1 = max(a0, kend & ~(A - 1));
            if (a1 > a0) {
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + a0),
                             "r"(smem_u32(src + a0)), "r"(static_cast<uint32_t>((a1 - a0) * sizeof(VT)))
                             : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            for (int k = k0; k < a0; ++k) dst[k] = src[k];
            for (int k = a1; k < kend; ++k) dst[k] = src[k];
        }
    }
    static __device__ __forceinline__ void drain() {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
    }
};

template <typename VT> __device__ __forceinline__ VT value_as(double v) { return narrow<VT>(v); }
template <typename VT> __device__ __forceinline__ VT value_as(float v) {
    if constexpr (std::is_same<VT, float>::value) return v;
    else return widen(v);
}

// CNT slot rows of a half slice, their values from the lane's row of the tile (len
// entries): into the slots and into the sum, in sell_diag_block's order.
template <int CNT, bool DIAG, typename ACC, typename VT>
__device__ __forceinline__ void set_values_block(ACC &acc, VT *out, const VT *row, int len,
                                                 const int32_t *__restrict__ cb, const int4 *__restrict__ dp, int r,
                                                 const VT *__restrict__ x) {
    int32_t c[CNT];
    if constexpr (DIAG) {
        const int4 a = __ldg(dp);
        int4 b = make_int4(0, 0, 0, 0);
        if constexpr (CNT > 4) b = __ldg(dp + 1);
        const int32_t o[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = r + o[u];
    } else {
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = __ldg(cb + u * kSellC);
    }
    VT xv[CNT];
#pragma unroll
    for (int u = 0; u < CNT; ++u) xv[u] = (DIAG || c[u] >= 0) ? __ldg(x + c[u]) : VT(0);
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        const VT v = u < len ? row[u] : VT(0);
        out[u * kSellC] = v;
        acc.fma(v, xv[u]);
        if (u % kSellU == kSellU - 1 || u == CNT - 1) end_run(acc);
    }
}

template <bool DIAG, typename ACC, typename VT>
__device__ __forceinline__ void set_values_row(ACC &acc, int w, VT *out, const VT *row, int len,
                                               const int32_t *__restrict__ cb, const int4 *__restrict__ dp, int r,
                                               const VT *__restrict__ x) {
    for (; w >= 8; w -= 8) {
        set_values_block<8, DIAG>(acc, out, row, len, cb, dp, r, x);
        out += 8 * kSellC;
        row += 8;
        len -= 8;
        if constexpr (DIAG) dp += 2;
        else cb += 8 * kSellC;
    }
    switch (w) {
        case 7: set_values_block<7, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 6: set_values_block<6, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 5: set_values_block<5, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 4: set_values_block<4, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 3: set_values_block<3, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 2: set_values_block<2, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        case 1: set_values_block<1, DIAG>(acc, out, row, len, cb, dp, r, x); break;
        default: break;
    }
}

// New values: from CRS order (type ST) into the handle's CRS copy dval and into
// the slices, one read and two writes (27-point 128^3 FP64, 1.34 GB: 225 us, 5.9
// TB/s; a copy and a layout pass of its own took 314).  Rows of at most kTileMaxW
// entries.  ACC not void: also y = alpha*A*x with them, the sums of k_sell_diag (a
// poisoned FP32 row is summed again from val: dval may still be on its way).  Memory
// bounds the one and the FP64 pipe the other: together 236 us (5.7 TB/s), one after
// the other 327 (FP32 144 against 180; 7-point 160^3 143 and 183).
template <typename ST, typename VT, typename ACC>
__global__ void __launch_bounds__(256) k_sell_set_values(const SellParams p, const ST *__restrict__ val,
                                                         VT *__restrict__ dval, int max_w) {
    extern __shared__ __align__(16) unsigned char smem[];
    VT *__restrict__ vals = static_cast<VT *>(const_cast<void *>(p.vals));
    const VT *__restrict__ x = static_cast<const VT *>(p.m.x);
    VT *__restrict__ y = static_cast<VT *>(p.m.y);
    const double alpha = p.alpha;
    const int emode = epi_mode(alpha, 0.0);
    const int lane = threadIdx.x & 31;
    VT *tile = reinterpret_cast<VT *>(smem) + (threadIdx.x >> 5) * TilePack<VT>::entries(max_w);
    const uint64_t pol = l2_evict_first_policy();
    each_half_slice(p.dorder, p.srows, p.n_slices, p.m.rp, lane, [&](int i, const int4 &d, int r, int k0, int k1) {
        const TilePack<VT> t(d.y, k0, k1, lane);
        bool free = false;  // the tile's last bulk copies have read it
        for (unsigned m = t.heads; m; m &= m - 1) {  // segments, coalesced
            const int h = __ffs(m) - 1;
            const int ks = __shfl_sync(0xffffffffu, k0, h), ke = __shfl_sync(0xffffffffu, t.kend, h);
            VT *out = tile + __shfl_sync(0xffffffffu, t.pos, h) - ks;
            if constexpr (std::is_same<ST, VT>::value) {
                // asynchronous copies: all of the half slice's values in flight at once (8
                // to a lane in registers: 268 us with the product)
                if (!free) TilePack<VT>::drain();
                free = true;
                for (int k = ks + lane; k < ke; k += 32)
                    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;" ::"r"(smem_u32(out + k)),
                                 "l"(val + k), "n"(sizeof(VT)), "l"(pol)
                                 : "memory");
            } else {
                for (int k = ks + lane; __any_sync(0xffffffffu, k < ke); k += 256) {
                    ST v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = k + 32 * u < ke ? ld_stream_p(val + k + 32 * u, pol) : ST(0);
                    if (!free) TilePack<VT>::drain();
                    free = true;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (k + 32 * u < ke) out[k + 32 * u] = value_as<VT>(v[u]);
                }
            }
        }
        if constexpr (std::is_same<ST, VT>::value) asm volatile("cp.async.wait_all;" ::: "memory");
        t.store(tile, dval, k0, lane);
        VT *out = vals + static_cast<int64_t>(d.x) * kSellC + (i & 1) * 32 + lane;
        const VT *row = tile + t.pos;
        const int len = k1 - k0;
        if constexpr (std::is_void<ACC>::value) {
#pragma unroll 8
            for (int j = 0; j < d.y; ++j) out[j * kSellC] = j < len ? row[j] : VT(0);
        } else {
            ACC acc;
            acc.zero();
            if (d.w >= 0)
                set_values_row<true>(acc, d.y, out, row, len, static_cast<const int32_t *>(nullptr), p.diag + d.w, r, x);
            else
                set_values_row<false>(acc, d.y, out, row, len,
                                      p.cols + static_cast<int64_t>(d.x) * kSellC + (i & 1) * 32 + lane,
                                      static_cast<const int4 *>(nullptr), r, x);
            if (r >= 0) {
                if constexpr (std::is_same<ACC, AccF64>::value)
                    y[r] = epi_apply(acc.get(), y + r, alpha, 0.0, emode);
                else
                    sell_store<VT>(p.m, x, y, r, acc, alpha, 0.0, p.ff, emode == kEpiPlain, VT(0));
            }
        }
        __syncwarp();
    });
    TilePack<VT>::drain();
}

// CNT products of a lane's row along its diagonals.  wait: the tile's last bulk
// copies may still read it; their end is waited for with the gathers in flight.
template <int CNT, typename VT>
__device__ __forceinline__ void grad_val_block(VT *row, VT gr, const int4 *__restrict__ dp, const VT *__restrict__ xr,
                                               bool wait) {
    const int4 a = __ldg(dp);
    int4 b = make_int4(0, 0, 0, 0);
    if constexpr (CNT > 4) b = __ldg(dp + 1);
    const int32_t o[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    VT xv[CNT];
#pragma unroll
    for (int q = 0; q < CNT; ++q) xv[q] = __ldg(xr + o[q]);
    if (wait) TilePack<VT>::drain();
#pragma unroll
    for (int q = 0; q < CNT; ++q) row[q] = gr * xv[q];
}

// grad_val[k] = (alpha*g[row]) * x[col[k]] on the row slices: a lane holds its
// row's g, x is gathered along diagonals (no column indices are read for diagonal
// slices), and the products leave through the tile in CRS order (gv 16-byte
// aligned).  Rows of at most kTileMaxW entries.  FP64: the FP64 pipe (one multiply
// per entry, 93 us on the 27-point 128^3 pattern) is 67 % busy at 136 us (162 on
// the chunks of k_grad_val_pipe); FP32 60 against 111 us.  Writing each product
// from the tile by ordinary stores instead of bulk copies: 165 and 76 us.
template <typename VT>
__global__ void __launch_bounds__(256) k_sell_grad_val(const SellParams p, const VT *__restrict__ g, VT *__restrict__ gv,
                                                       int max_w) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    VT *tile = reinterpret_cast<VT *>(smem) + (threadIdx.x >> 5) * TilePack<VT>::entries(max_w);
    const VT *__restrict__ x = static_cast<const VT *>(p.m.x);
    const VT a = static_cast<VT>(p.alpha);
    const bool scaled = p.alpha != 1.0;
    each_half_slice(p.dorder, p.srows, p.n_slices, p.m.rp, lane, [&](int i, const int4 &d, int r, int k0, int k1) {
        VT gr = r >= 0 ? __ldg(g + r) : VT(0);
        const TilePack<VT> t(d.y, k0, k1, lane);
        VT *row = tile + t.pos;
        const int32_t *__restrict__ cb = p.cols + static_cast<int64_t>(d.x) * kSellC + (i & 1) * 32 + lane;
        const int4 *__restrict__ dp = p.diag + d.w;
        if (scaled) gr = static_cast<VT>(a * gr);
        if (d.w >= 0) {
            int w = d.y;
            for (; w >= 8; w -= 8, row += 8, dp += 2) grad_val_block<8>(row, gr, dp, x + r, w == d.y);
            switch (w) {
                case 7: grad_val_block<7>(row, gr, dp, x + r, w == d.y); break;
                case 6: grad_val_block<6>(row, gr, dp, x + r, w == d.y); break;
                case 5: grad_val_block<5>(row, gr, dp, x + r, w == d.y); break;
                case 4: grad_val_block<4>(row, gr, dp, x + r, w == d.y); break;
                case 3: grad_val_block<3>(row, gr, dp, x + r, w == d.y); break;
                case 2: grad_val_block<2>(row, gr, dp, x + r, w == d.y); break;
                case 1: grad_val_block<1>(row, gr, dp, x + r, w == d.y); break;
                default: break;
            }
        } else {
            const int len = k1 - k0;
            TilePack<VT>::drain();
            for (int j0 = 0; j0 < d.y; j0 += 8) {
                VT xv[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) xv[q] = j0 + q < len ? __ldg(x + __ldg(cb + (j0 + q) * kSellC)) : VT(0);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (j0 + q < len) row[j0 + q] = gr * xv[q];
            }
        }
        t.store(tile, gv, k0, lane);
    });
    TilePack<VT>::drain();
}

// Grid of a tile kernel: its resident CTAs, 8 half slices per CTA and turn.
template <auto KERNEL>
static int tile_grid(int32_t n_slices, size_t smem) {
    const int64_t want = (2 * static_cast<int64_t>(n_slices) + 7) / 8;
    return static_cast<int>(std::min<int64_t>(want, resident<KERNEL>(smem, 8 * 8 * TilePack<double>::entries(kTileMaxW))));
}

int sell_tile_max_row() { return kTileMaxW; }

template <typename ST, typename VT, typename ACC = void>
static cudaError_t set_values_as(const SellParams &p, const void *val, void *dval, int max_w, cudaStream_t s) {
    const size_t smem = sizeof(VT) * 8 * TilePack<VT>::entries(max_w);
    const int grid = tile_grid<k_sell_set_values<ST, VT, ACC>>(p.n_slices, smem);
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    k_sell_set_values<ST, VT, ACC>
        <<<grid, 256, smem, s>>>(p, static_cast<const ST *>(val), static_cast<VT *>(dval), max_w);
    return cudaGetLastError();
}

cudaError_t launch_sell_set_values(const SellParams &p, const void *val, int sk, void *dval, int vk, int max_w,
                                   cudaStream_t s) {
    if (p.n_slices <= 0) return cudaSuccess;
    if (p.m.y) {  // with the product: the accumulators of sell_ops
        if (sk != vk) return cudaErrorInvalidValue;
        if (vk == kF64) return set_values_as<double, double, AccF64>(p, val, dval, max_w, s);
        return max_w <= kFRMaxRun ? set_values_as<float, float, AccFR>(p, val, dval, max_w, s)
                                  : set_values_as<float, float, AccFRF>(p, val, dval, max_w, s);
    }
    if (vk == kF64)
        return sk == kF64 ? set_values_as<double, double>(p, val, dval, max_w, s)
                          : set_values_as<float, double>(p, val, dval, max_w, s);
    return sk == kF64 ? set_values_as<double, float>(p, val, dval, max_w, s)
                      : set_values_as<float, float>(p, val, dval, max_w, s);
}

template <typename VT>
static cudaError_t grad_val_as(const SellParams &p, const void *g, void *gv, int max_w, cudaStream_t s) {
    const size_t smem = sizeof(VT) * 8 * TilePack<VT>::entries(max_w);
    const int grid = tile_grid<k_sell_grad_val<VT>>(p.n_slices, smem);
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    k_sell_grad_val<VT><<<grid, 256, smem, s>>>(p, static_cast<const VT *>(g), static_cast<VT *>(gv), max_w);
    return cudaGetLastError();
}

cudaError_t launch_sell_grad_val(const SellParams &p, int vk, const void *g, void *gv, int max_w, cudaStream_t s) {
    if (p.n_slices <= 0) return cudaSuccess;
    return vk == kF64 ? grad_val_as<double>(p, g, gv, max_w, s) : grad_val_as<float>(p, g, gv, max_w, s);
}

cudaError_t launch_sell_relayout(const void *slices, const int32_t *srows, int32_t n_slices, const int32_t *rp,
                                 int vk, const void *val, const int32_t *col, void *vals_out, int32_t *cols_out,
                                 cudaStream_t s) {
    if (n_slices <= 0) return cudaSuccess;
    const int grid = slice_grid(n_slices);
    const int2 *d = static_cast<const int2 *>(slices);
    if (vk == kF64)
        k_sell_relayout<double><<<grid, 256, 0, s>>>(d, srows, n_slices, rp, static_cast<const double *>(val), col,
                                                     static_cast<double *>(vals_out), cols_out);
    else
        k_sell_relayout<float><<<grid, 256, 0, s>>>(d, srows, n_slices, rp, static_cast<const float *>(val), col,
                                                    static_cast<float *>(vals_out), cols_out);
    return cudaGetLastError();
}

}  // namespace spmv
