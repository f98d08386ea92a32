// Sorted row-slice kernel (plan family 5).
//
// The rows of each window of `sigma` consecutive rows are ordered by length
// (longest first) and cut into slices of kSellC = 64 rows; lane l of a warp owns
// rows l and l + 32 of a slice from their first entries to their last, so a row
// sum is one FMA chain in one lane: no row-start bits, no carries between lanes
// and no row buffer, and each lane runs two independent chains (one chain per
// lane leaves the FP64 pipe waiting on its own results).  Entry j of the slice's
// row h*32 + l is stored at slot (off + j)*64 + h*32 + l (the slice's width w is
// its longest row; shorter rows are padded with value 0 and column -1), so every
// load of a warp reads 32 consecutive elements.  Sorting inside windows keeps
// the padding small (equal-length rows share slices) while the rows of a slice
// stay close together in x and y.  This is the SELL-C-sigma layout of Kreutzer,
// Hager, Wellein, Fehske and Bishop (SIAM J. Sci. Comput. 36(5), 2014) with
// C = 64, built as a derived copy of the CRS arrays.
//
// CTA b owns the slices [cstart[b], cstart[b+1]), a contiguous range chosen on
// the host so that every CTA gets the same number of slots (a fixed
// round-robin over windows sorted by length would hand some warps the widest
// slices of every window); its 8 warps take the range's slices in turn, so the
// CTA works on one or two windows at a time and their x entries stay in L1.  A
// warp walks its slices in blocks of kSellU slot rows.  The values and gathers
// of the next block and the column indices of the block after it are in flight
// in registers while the current block's FMAs run (two register sets in turn).
// A block shorter than kSellU holds its entries at the end of the register
// arrays (the loads before it read the preceding slot rows, which exist because
// the arrays start with kSellU rows of padding, and their columns are masked)
// and enters the FMA sequence part-way, so every FMA issued belongs to a stored
// slot.
#pragma once
#include "slot_kernel.cuh"
#include "reduce.cuh"

namespace spmv {

constexpr int kSellK = 2;            // rows per lane
constexpr int kSellC = 32 * kSellK;  // rows per slice
constexpr int kSellU = 4;            // slot rows per block

struct SellParams {
    const int2 *slices;    // per slice: x = first slot row (>= kSellU), y = width w; y < 0: long row x (CRS)
    const int32_t *srows;  // kSellC per slice: the row of each lane and half (-1: none)
    const int32_t *cstart; // n_ctas + 1: the first slice of each CTA
    const void *vals;      // slot-major values (0 in padding)
    const int32_t *cols;   // slot-major column indices (-1 in padding)
    MatRef m;              // the CRS itself (long rows), x, y
    int32_t n_slices;
    int32_t n_ctas;        // CTAs of the launch
    double alpha, beta;
    EpiFF ff;              // alpha and beta for FP32 rows
    // diagonal slices (k_sell_diag below); dorder is null when k_sell runs
    const int4 *dorder;    // n_slices: x, y = the descriptor, z = the slice, w = its place in diag (-1: not diagonal)
    const int4 *diag;      // column minus row of each slot row of the diagonal slices, 4 to an element
    bool dshort;           // at most 8 slot rows per slice on average
    const int32_t *vpos;   // launch_ind: position in vals of each slot's value (-1: padding)
};

// For i = 0 .. cnt-1 and both rows h of the lane, in that order:
// acc[h] += v[U-cnt+i][h] * xv[U-cnt+i][h].  A jump into an unrolled sequence
// (cnt is the same in all lanes), so no FMA is issued for an empty register.
template <typename ACC, typename VT, typename XT>
__device__ __forceinline__ void sell_fma_tail(ACC (&acc)[kSellK], const VT (&v)[kSellU][kSellK],
                                              const XT (&xv)[kSellU][kSellK], int cnt) {
    static_assert(kSellU == 4 && kSellK == 2, "the jump table below is written for 4 slot rows of 2 rows");
    switch (cnt) {
        case 4:
            acc[0].fma(v[0][0], xv[0][0]);
            acc[1].fma(v[0][1], xv[0][1]);
            [[fallthrough]];
        case 3:
            acc[0].fma(v[1][0], xv[1][0]);
            acc[1].fma(v[1][1], xv[1][1]);
            [[fallthrough]];
        case 2:
            acc[0].fma(v[2][0], xv[2][0]);
            acc[1].fma(v[2][1], xv[2][1]);
            [[fallthrough]];
        case 1:
            acc[0].fma(v[3][0], xv[3][0]);
            acc[1].fma(v[3][1], xv[3][1]);
            [[fallthrough]];
        default:
            break;
    }
}

// As ld_stream, but free for the compiler to schedule among other loads.
__device__ __forceinline__ double ld_stream_p(const double *p, uint64_t pol) {
    double v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ int32_t ld_stream_p(const int32_t *p, uint64_t pol) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_stream_p(const float *p, uint64_t pol) {
    float v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}

// Final store of stored row `row` of m; `old` is y[row], loaded ahead
// (read only when beta is nonzero).  A poisoned float-float sum is summed again
// in FP64 from the CRS arrays of m.
template <typename VT, bool INDIRECT = false, typename XT, typename YT, typename ACC>
__device__ __forceinline__ YT sell_store(const MatRef &m, const XT *__restrict__ x, YT *__restrict__ y, int row,
                                         const ACC &a, double alpha, double beta, const EpiFF &ff, bool plain, YT old) {
    if constexpr ((std::is_same<ACC, AccFF>::value || std::is_same<ACC, AccFR>::value ||
                   std::is_same<ACC, AccFRF>::value) &&
                  std::is_same<YT, float>::value) {
        if (plain && !a.poisoned()) {
            const float out = a.h + a.l;
            y[row] = out;
            return out;
        }
        float out;
        if (!plain && epi_ff_row(ff, a, old, out)) {
            y[row] = out;
            return out;
        }
    }
    const double v = acc_value<VT, INDIRECT>(a, m, row, x);
    double out;
    if (plain) out = v;
    else if (beta == 0.0) out = alpha * v;
    else out = fma(alpha, v, beta * widen(old));
    const YT yo = narrow<YT>(out);
    y[row] = yo;
    return yo;
}

// Gather of x through L1, issued where it stands in the source (the compiler may
// not move it next to its use, which would leave no time for its latency).
__device__ __forceinline__ double ld_gather(const double *p) {
    double v;
    asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_gather(const float *p) {
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// The walk of one warp over its CTA's slices.  DOT: also dsum += x[r] * y[r]
// (exact products of the stored values, FP64 sums) for every row r the warp
// stores (the p.q of a CG step, with x = p and y = q).
template <typename VT, typename XT, typename YT, typename ACC, bool DOT>
__device__ __forceinline__ void sell_walk(const SellParams &p, double &dsum) {
    constexpr int U = kSellU, K = kSellK, C = kSellC;
    const int lane = threadIdx.x & 31;
    if (static_cast<int>(blockIdx.x) >= p.n_ctas) return;
    const int s0 = __ldg(p.cstart + blockIdx.x) + (threadIdx.x >> 5);
    const int n = __ldg(p.cstart + blockIdx.x + 1);  // end of this CTA's slices
    if (s0 >= n) return;
    const uint64_t pol = l2_evict_first_policy();
    const VT *__restrict__ vals = static_cast<const VT *>(p.vals);
    const int32_t *__restrict__ cols = p.cols;
    const XT *__restrict__ x = static_cast<const XT *>(p.m.x);
    YT *__restrict__ y = static_cast<YT *>(p.m.y);
    const double alpha = p.alpha, beta = p.beta;
    const bool plain = (alpha == 1.0 && beta == 0.0);
    const bool read_y = !plain && beta != 0.0;

    // block cursor: slice s (descriptor off, w) and the block's first slot row j0
    struct Cur {
        int s, off, w, j0;
    };
    auto slice_of = [&](int s) { return s < n ? __ldg(p.slices + s) : make_int2(0, 0); };
    auto cnt_of = [](const Cur &c) { return max(0, min(U, c.w - c.j0)); };
    auto last_of = [](const Cur &c) { return c.j0 + U >= c.w; };
    // next block of the warp; dnext is the descriptor of slice c.s + 8
    auto advance = [&](Cur &c, int2 &dnext) {
        if (!last_of(c)) {
            c.j0 += U;
            return;
        }
        c.s += 8;
        c.off = dnext.x;
        c.w = dnext.y;
        c.j0 = 0;
        dnext = slice_of(c.s + 8);
    };
    // Element of register row 0 of the block (a block of cnt slot rows starts at
    // register row U - cnt; the slot rows before it exist, see above).  Blocks
    // without slots (long rows, past the end) read the leading padding rows.
    // The loads are unconditional and nothing inspects their results until the
    // block is used (a select on a fresh column index would wait for it).
    auto base_of = [&](const Cur &c) {
        const int cnt = c.s < n ? cnt_of(c) : 0;
        return cnt > 0 ? (static_cast<int64_t>(c.off) + c.j0 - (U - cnt)) * C + lane : static_cast<int64_t>(lane);
    };
    auto load_cols = [&](const Cur &c, int32_t (&cl)[U][K]) {
        const int32_t *b = cols + base_of(c);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int h = 0; h < K; ++h) cl[u][h] = ld_stream(b + u * C + h * 32, pol);
    };
    auto load_vals = [&](const Cur &c, VT (&v)[U][K]) {
        const VT *b = vals + base_of(c);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int h = 0; h < K; ++h) v[u][h] = ld_stream(b + u * C + h * 32, pol);
    };
    // gathers of the block's slots (register rows U - cnt .. U - 1, stored columns)
    auto gather = [&](const Cur &c, const int32_t (&cl)[U][K], XT (&xv)[U][K]) {
        const int cnt = c.s < n ? cnt_of(c) : 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int h = 0; h < K; ++h)
                xv[u][h] = (u >= U - cnt && cl[u][h] >= 0) ? ld_gather(x + cl[u][h]) : XT(0);
    };
    // the output rows of the lane, for the last block of a regular slice
    auto rows_of = [&](const Cur &c, int (&r)[K]) {
        const bool ok = c.s < n && c.w >= 0 && last_of(c);
#pragma unroll
        for (int h = 0; h < K; ++h) r[h] = ok ? __ldg(p.srows + static_cast<int64_t>(c.s) * C + h * 32 + lane) : -1;
    };

    // cursors: a (FMAs now), b (gathers and values in flight), c (columns in flight)
    Cur ca{s0, 0, 0, 0};
    {
        const int2 d = slice_of(s0);
        ca.off = d.x;
        ca.w = d.y;
    }
    int2 dnext = slice_of(s0 + 8);
    Cur cb = ca;
    advance(cb, dnext);
    Cur cc = cb;
    advance(cc, dnext);

    // Two register sets used in turn: set P holds block a (values, gathers,
    // output rows, old y) and receives block c's column indices and rows once
    // block a no longer needs them; set Q holds block b.  Nothing is copied
    // between the sets, so no register still waiting for its load is read
    // before the FMAs that need it.
    struct Set {
        VT v[U][K];
        XT x[U][K];
        int32_t c[U][K];
        int r[K];
        YT y[K];
    };
    Set S0, S1;
    rows_of(ca, S0.r);
    load_cols(ca, S0.c);
    gather(ca, S0.c, S0.x);
    load_vals(ca, S0.v);
#pragma unroll
    for (int h = 0; h < K; ++h) S0.y[h] = YT(0);
    if (read_y) {
#pragma unroll
        for (int h = 0; h < K; ++h)
            if (S0.r[h] >= 0) S0.y[h] = y[S0.r[h]];
    }
    load_cols(cb, S1.c);
    rows_of(cb, S1.r);

    ACC acc[K];
#pragma unroll
    for (int h = 0; h < K; ++h) acc[h].zero();
    auto step = [&](Set &P, Set &Q) {
        // block b: gathers, values, old y (into Q); block c: columns (into P)
        gather(cb, Q.c, Q.x);
        load_vals(cb, Q.v);
        if (read_y) {
#pragma unroll
            for (int h = 0; h < K; ++h) Q.y[h] = (Q.r[h] >= 0) ? y[Q.r[h]] : YT(0);
        }
        load_cols(cc, P.c);
        // ---- block a ----------------------------------------------------------
        if (ca.w < 0) {
            const int row = ca.off;
            const ChunkDesc d{__ldg(p.m.rp + row), __ldg(p.m.rp + row + 1), row, (row + 1) | kChunkLong};
            long_row<VT, XT, YT, ACC, false>(p.m, d, x, y, alpha, beta, plain, lane);
            if constexpr (DOT) {
                if (lane == 0) dsum = fma(widen(x[row]), widen(y[row]), dsum);  // lane 0 stored it
            }
        } else {
            sell_fma_tail(acc, P.v, P.x, cnt_of(ca));
#pragma unroll
            for (int h = 0; h < K; ++h) end_run(acc[h]);
            if (last_of(ca)) {
#pragma unroll
                for (int h = 0; h < K; ++h) {
                    if (P.r[h] >= 0) {
                        const YT q = sell_store<VT>(p.m, x, y, P.r[h], acc[h], alpha, beta, p.ff, plain, P.y[h]);
                        if constexpr (DOT) dsum = fma(widen(x[P.r[h]]), widen(q), dsum);
                    }
                    acc[h].zero();
                }
            }
        }
        rows_of(cc, P.r);
        ca = cb;
        cb = cc;
        advance(cc, dnext);
    };
    while (ca.s < n) {
        step(S0, S1);
        if (ca.s >= n) break;
        step(S1, S0);
    }
}

template <typename VT, typename XT, typename YT, typename ACC, bool DOT = false>
__global__ void __launch_bounds__(256) k_sell(const SellParams p, const RedOut o) {
    double dsum = 0.0;
    sell_walk<VT, XT, YT, ACC, DOT>(p, dsum);
    if constexpr (DOT) {
        __shared__ double s_red[32];
        finish(block_sum(dsum, s_red), o, s_red);
    }
}

// ---------------------------------------------------------------------------
// Diagonal slices.  In a stencil-like matrix nearly every slice has full rows
// whose entries at slot row j all lie on one diagonal: column - row is the same
// number in its 64 rows (k_sell_mark_diag finds these slices once, when the copy
// is built).  Such a slice needs no column indices: 4 bytes per slot row instead
// of 256, a third of the matrix bytes in FP64 and half in FP32, and the address
// of a gather is row + diagonal, known without waiting for a column load.  So
// nothing is staged ahead in registers: a warp takes half a slice (one row per
// lane), issues up to 8 slot rows of values and gathers, then their FMAs, and the
// resident warps hide each other's latency.  The sums run in the same order as
// in k_sell (and the FP32 runs fold at the same places).  Slices that are not
// diagonal (the grid's boundary rows: a few per cent) take the same path with
// their column indices.
// ---------------------------------------------------------------------------

// Where a half slice's values are: in its own slots (v), or, IND, at position
// p[slot] of another copy's values (the reverse pass: the slices of A^T read the
// values of A's slices, so new values need no layout in A^T's order).  On a grid
// the 32 positions of a slot row are nearly consecutive in A's slices, where the
// permutation of the CRS order put them in 32 places: 27-point 128^3, first pass
// after new values, FP64 306 -> 132 us, FP32 684 -> 95.
template <typename VT, bool IND>
struct SellVals {
    const VT *__restrict__ v;       // the slots (IND: the other copy's values)
    const int32_t *__restrict__ p;  // IND: the slots' positions there (-1: padding)
    __device__ __forceinline__ void skip(int rows) {
        if constexpr (IND) p += rows * kSellC;
        else v += rows * kSellC;
    }
};

// CNT slot rows of a half slice (kSellC apart): their columns are row + diagonal
// (DIAG; 8 diagonals at dp) or as stored (cb).  RUN: the longest run of FP32 FMAs.
template <int CNT, bool DIAG, int RUN, bool IND, typename ACC, typename VT, typename XT>
__device__ __forceinline__ void sell_diag_block(ACC &acc, const SellVals<VT, IND> &sv, const int32_t *__restrict__ cb,
                                                const int4 *__restrict__ dp, int row, const XT *__restrict__ x,
                                                uint64_t pol) {
    int32_t pos[CNT];
    if constexpr (IND) {
#pragma unroll
        for (int u = 0; u < CNT; ++u) pos[u] = ld_stream_p(sv.p + u * kSellC, pol);
    }
    int32_t c[CNT];
    if constexpr (DIAG) {
        const int4 a = __ldg(dp);
        int4 b = make_int4(0, 0, 0, 0);
        if constexpr (CNT > 4) b = __ldg(dp + 1);
        const int32_t g[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = row + g[u];
    } else {
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = __ldg(cb + u * kSellC);
    }
    VT v[CNT];
    XT xv[CNT];
    if constexpr (!IND) {
#pragma unroll
        for (int u = 0; u < CNT; ++u) v[u] = ld_stream_p(sv.v + u * kSellC, pol);
    }
#pragma unroll
    for (int u = 0; u < CNT; ++u) xv[u] = (DIAG || c[u] >= 0) ? __ldg(x + c[u]) : XT(0);
    if constexpr (IND) {
#pragma unroll
        for (int u = 0; u < CNT; ++u) v[u] = (DIAG || pos[u] >= 0) ? __ldg(sv.v + pos[u]) : VT(0);
    }
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        acc.fma(v[u], xv[u]);
        if (u % RUN == RUN - 1 || u == CNT - 1) end_run(acc);
    }
}

// All w slot rows of a half slice.
template <bool DIAG, int RUN = kSellU, bool IND, typename ACC, typename VT, typename XT>
__device__ __forceinline__ void sell_diag_row(ACC &acc, int w, SellVals<VT, IND> sv, const int32_t *__restrict__ cb,
                                              const int4 *__restrict__ dp, int row, const XT *__restrict__ x,
                                              uint64_t pol) {
    for (; w >= 8; w -= 8) {
        sell_diag_block<8, DIAG, RUN>(acc, sv, cb, dp, row, x, pol);
        sv.skip(8);
        if constexpr (DIAG) dp += 2;
        else cb += 8 * kSellC;
    }
    switch (w) {
        case 7: sell_diag_block<7, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 6: sell_diag_block<6, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 5: sell_diag_block<5, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 4: sell_diag_block<4, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 3: sell_diag_block<3, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 2: sell_diag_block<2, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        case 1: sell_diag_block<1, DIAG, RUN>(acc, sv, cb, dp, row, x, pol); break;
        default: break;
    }
}

template <typename VT, typename XT, typename YT, typename ACC, bool DOT, bool IND>
__device__ __forceinline__ void sell_diag_walk(const SellParams &p, double &dsum) {
    constexpr int C = kSellC;
    const int lane = threadIdx.x & 31;
    const int n = 2 * p.n_slices;  // half slices
    const int nw = gridDim.x * 8;
    const uint64_t pol = l2_evict_first_policy();
    const XT *__restrict__ x = static_cast<const XT *>(p.m.x);
    YT *__restrict__ y = static_cast<YT *>(p.m.y);
    const VT *__restrict__ vals = static_cast<const VT *>(p.vals);
    const double alpha = p.alpha, beta = p.beta;
    const int emode = epi_mode<true>(alpha, beta);
    int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    auto desc_of = [&](int k) { return __ldg(p.dorder + (k < n ? k >> 1 : p.n_slices - 1)); };
    auto row_of = [&](const int4 &d, int k) {
        return __ldg(p.srows + static_cast<int64_t>(d.z) * C + (k & 1) * 32 + lane);
    };
    int4 d = desc_of(i), dn = desc_of(i + nw);
    int r = row_of(d, i);
    for (; i < n; i += nw) {
        const int4 d2 = desc_of(i + 2 * nw);
        const int rn = row_of(dn, i + nw);
        if (d.y < 0) {
            if ((i & 1) == 0) {
                const int row = d.x;
                const ChunkDesc cd{__ldg(p.m.rp + row), __ldg(p.m.rp + row + 1), row, (row + 1) | kChunkLong};
                long_row<VT, XT, YT, ACC, IND>(p.m, cd, x, y, alpha, beta, emode == kEpiPlain, lane);
                if constexpr (DOT) {
                    if (lane == 0) dsum = fma(widen(x[row]), widen(y[row]), dsum);  // lane 0 stored it
                }
            }
        } else {
            const int64_t base = static_cast<int64_t>(d.x) * C + (i & 1) * 32 + lane;
            ACC acc;
            acc.zero();
            SellVals<VT, IND> sv{IND ? vals : vals + base, IND ? p.vpos + base : nullptr};
            if (d.w >= 0)
                sell_diag_row<true>(acc, d.y, sv, static_cast<const int32_t *>(nullptr), p.diag + d.w, r, x, pol);
            else
                sell_diag_row<false>(acc, d.y, sv, p.cols + base, static_cast<const int4 *>(nullptr), r, x, pol);
            if (r >= 0) {
                YT q;
                if constexpr (std::is_same<ACC, AccF64>::value) {
                    // (y - A*x as one subtraction: 160^3 74 -> 68 us, 2000^2 58 -> 53)
                    // no tests on alpha and beta per row: with 5 and 7 entries per row
                    // they cost 62 and 79 instead of 47 and 60 us (2000^2 and 160^3)
                    q = epi_apply<true>(acc.get(), y + r, alpha, beta, emode);
                    y[r] = q;
                } else {
                    const YT old = emode >= kEpiAdd ? y[r] : YT(0);
                    q = sell_store<VT, IND>(p.m, x, y, r, acc, alpha, beta, p.ff, emode == kEpiPlain, old);
                }
                if constexpr (DOT) dsum = fma(widen(__ldg(x + r)), widen(q), dsum);
            }
        }
        d = dn;
        dn = d2;
        r = rn;
    }
}

// The same over the slices of many matrices in one launch (the batch): half slice i
// is half i & 1 of entry i / 2 of `list`: x = the member, y = the slice in the
// member's launch order.  The list entry, descriptor and rows of the half slices
// that follow are loaded ahead, one step of the chain per turn.
struct SellMember {
    const int4 *dorder;
    const int32_t *srows;
    const int4 *diag;
    const void *vals;
    const int32_t *cols;
    int32_t mat;  // the member's place in the matrix table
};
struct SellBatchParams {
    const int2 *list;
    const SellMember *members;
    const MatRef *mats;
    int32_t n_list;
    double alpha, beta;
    EpiFF ff;
};

// FP32 runs of up to 5 entries, folded into float-float: at most as long as in the chunks
// that sum the other members (7 or 9 entries of a row in a lane), and no less exact on
// average: relative error of members of 5, 7, 9 and 11 entries per row 4.4, 4.9, 4.7 and
// 4.7e-8 (runs over whole rows 4.4, 5.0, 5.6, 6.2; of 4 entries 4.6, 4.7, 4.7, 4.7; the
// chunks 4.4, 5.0, 5.6, 5.6).
constexpr int kBatchRun = 5;

template <typename VT, typename ACC>
__global__ void __launch_bounds__(256, sizeof(VT) == 8 ? 4 : 5) k_sell_diag_batch(const SellBatchParams p) {
    constexpr int C = kSellC;
    const int lane = threadIdx.x & 31;
    const int n = 2 * p.n_list, nw = gridDim.x * 8;
    const uint64_t pol = l2_evict_first_policy();
    const double alpha = p.alpha, beta = p.beta;
    const int emode = epi_mode(alpha, beta);
    int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    auto entry_of = [&](int k) { return __ldg(p.list + (k < n ? k >> 1 : p.n_list - 1)); };
    auto desc_of = [&](const int2 &e) { return __ldg(p.members[e.x].dorder + e.y); };
    auto row_of = [&](const int2 &e, const int4 &d, int k) {
        return __ldg(p.members[e.x].srows + static_cast<int64_t>(d.z) * C + (k & 1) * 32 + lane);
    };
    int2 e0 = entry_of(i), e1 = entry_of(i + nw), e2 = entry_of(i + 2 * nw);
    int4 d0 = desc_of(e0), d1 = desc_of(e1);
    int r = row_of(e0, d0, i);
    for (; i < n; i += nw) {
        const int2 e3 = entry_of(i + 3 * nw);
        const int4 d2 = desc_of(e2);
        const int rn = row_of(e1, d1, i + nw);
        const SellMember &t = p.members[e0.x];
        const MatRef m = p.mats[t.mat];
        const VT *__restrict__ x = static_cast<const VT *>(m.x);
        VT *__restrict__ y = static_cast<VT *>(m.y);
        const int64_t base = static_cast<int64_t>(d0.x) * C + (i & 1) * 32 + lane;
        ACC acc;
        acc.zero();
        const SellVals<VT, false> sv{static_cast<const VT *>(t.vals) + base, nullptr};
        if (d0.w >= 0)
            sell_diag_row<true, kBatchRun>(acc, d0.y, sv, static_cast<const int32_t *>(nullptr), t.diag + d0.w, r, x, pol);
        else
            sell_diag_row<false, kBatchRun>(acc, d0.y, sv, t.cols + base, static_cast<const int4 *>(nullptr), r, x, pol);
        if (r >= 0) {
            if constexpr (std::is_same<ACC, AccF64>::value) {
                y[r] = epi_apply(acc.get(), y + r, alpha, beta, emode);
            } else {
                const VT old = emode >= kEpiAdd ? y[r] : VT(0);
                sell_store<VT>(m, x, y, r, acc, alpha, beta, p.ff, emode == kEpiPlain, old);
            }
        }
        e0 = e1;
        e1 = e2;
        e2 = e3;
        d0 = d1;
        d1 = d2;
        r = rn;
    }
}

// CTAs per SM the registers must allow.  Rows of up to 8 entries (SHORT: one
// block per half slice, so the warps are latency-bound) take one more: 160^3
// Laplacian FP64 55.3 against 60.3 us, FP32 28.9 against 30.2; longer rows lose
// by it (27-point 128^3: FP64 106.6 against 98.6, FP32 46.6 against 44.9 us).
template <typename VT, bool SHORT>
constexpr int kSellDiagCtas = (sizeof(VT) == 8 ? 4 : 5) + (SHORT ? 1 : 0);

template <typename VT, typename XT, typename YT, typename ACC, bool SHORT, bool DOT, bool IND = false>
__global__ void __launch_bounds__(256, (kSellDiagCtas<VT, SHORT>)) k_sell_diag(const SellParams p, const RedOut o) {
    double dsum = 0.0;
    sell_diag_walk<VT, XT, YT, ACC, DOT, IND>(p, dsum);
    if constexpr (DOT) {
        __shared__ double s_red[32];
        finish(block_sum(dsum, s_red), o, s_red);
    }
}

// ---------------------------------------------------------------------------
// Block vectors on the same slices: Y[:, c0:c0+4] = alpha*A*X[:, c0:c0+4] +
// beta*Y[:, c0:c0+4] for row-major X (leading dimension ldx) and Y (ldy).  Each
// lane keeps 2 rows x 4 right-hand sides = 8 independent FMA chains and walks
// its slices one slot row at a time; a slot's four x values are one 32-byte
// sector (two 16-byte loads when VEC).  FP64 only.
// ---------------------------------------------------------------------------
constexpr int kSellR = 4;  // right-hand sides per pass

struct SellMrParams {
    SellParams b;   // slices, rows, copies, CRS (long rows), n_slices, cstart, alpha, beta
    const double *X;
    double *Y;
    int64_t ldx, ldy;
};

__device__ __forceinline__ double2 ld_gather2(const double *p) {
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// A row too long for a slice, for 4 right-hand sides: lanes stride the row, then
// a butterfly reduction of each sum.
template <bool VEC>
__device__ __forceinline__ void long_row_mr(const SellMrParams &q, int row, double alpha, double beta, bool plain,
                                            int lane) {
    const int32_t *__restrict__ col = q.b.m.col;
    const double *__restrict__ val = static_cast<const double *>(q.b.m.vs);
    const int k0 = __ldg(q.b.m.rp + row), k1 = __ldg(q.b.m.rp + row + 1);
    double acc[kSellR];
#pragma unroll
    for (int r = 0; r < kSellR; ++r) acc[r] = 0.0;
    for (int k = k0 + lane; k < k1; k += 32) {
        const double v = __ldg(val + k);
        const double *xp = q.X + static_cast<int64_t>(__ldg(col + k)) * q.ldx;
#pragma unroll
        for (int r = 0; r < kSellR; ++r) acc[r] = fma(v, __ldg(xp + r), acc[r]);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
        for (int r = 0; r < kSellR; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
    if (lane == 0) {
        double *yp = q.Y + static_cast<int64_t>(row) * q.ldy;
#pragma unroll
        for (int r = 0; r < kSellR; ++r)
            yp[r] = plain ? acc[r] : (beta == 0.0 ? alpha * acc[r] : fma(alpha, acc[r], beta * yp[r]));
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256, 2) k_sell_mr(const SellMrParams q) {
    constexpr int K = kSellK, C = kSellC, R = kSellR;
    const SellParams &p = q.b;
    const int lane = threadIdx.x & 31;
    if (static_cast<int>(blockIdx.x) >= p.n_ctas) return;
    const int s0 = __ldg(p.cstart + blockIdx.x) + (threadIdx.x >> 5);
    const int n = __ldg(p.cstart + blockIdx.x + 1);
    if (s0 >= n) return;
    const uint64_t pol = l2_evict_first_policy();
    const double *__restrict__ vals = static_cast<const double *>(p.vals);
    const int32_t *__restrict__ cols = p.cols;
    const double *__restrict__ X = q.X;
    double *__restrict__ Y = q.Y;
    const int64_t ldx = q.ldx, ldy = q.ldy;
    const double alpha = p.alpha, beta = p.beta;
    const bool plain = (alpha == 1.0 && beta == 0.0);

    // cursor: slice s (descriptor off, w) and its slot row j (one per step)
    struct Cur {
        int s, off, w, j;
    };
    auto slice_of = [&](int s) { return s < n ? __ldg(p.slices + s) : make_int2(0, 0); };
    auto has_slot = [&](const Cur &c) { return c.s < n && c.j < c.w; };
    auto last_of = [](const Cur &c) { return c.j + 1 >= c.w; };
    auto advance = [&](Cur &c, int2 &dnext) {
        if (!last_of(c)) {
            c.j += 1;
            return;
        }
        c.s += 8;
        c.off = dnext.x;
        c.w = dnext.y;
        c.j = 0;
        dnext = slice_of(c.s + 8);
    };
    // steps without a slot (long rows, empty slices, past the end) read the
    // leading padding row; nothing inspects the loaded columns before the gather
    auto base_of = [&](const Cur &c) {
        return has_slot(c) ? (static_cast<int64_t>(c.off) + c.j) * C + lane : static_cast<int64_t>(lane);
    };
    struct Set {
        double v[K];
        double x[K][R];
        int32_t c[K];
        int r[K];
    };
    auto load_cols = [&](const Cur &c, Set &S) {
        const int32_t *b = cols + base_of(c);
#pragma unroll
        for (int h = 0; h < K; ++h) S.c[h] = ld_stream(b + h * 32, pol);
    };
    auto load_vals = [&](const Cur &c, Set &S) {
        const double *b = vals + base_of(c);
#pragma unroll
        for (int h = 0; h < K; ++h) S.v[h] = ld_stream(b + h * 32, pol);
    };
    auto gather = [&](const Cur &c, Set &S) {
        const bool ok = has_slot(c);
#pragma unroll
        for (int h = 0; h < K; ++h) {
            if (ok && S.c[h] >= 0) {
                const double *xp = X + static_cast<int64_t>(S.c[h]) * ldx;
                if constexpr (VEC) {
                    const double2 a = ld_gather2(xp), b2 = ld_gather2(xp + 2);
                    S.x[h][0] = a.x;
                    S.x[h][1] = a.y;
                    S.x[h][2] = b2.x;
                    S.x[h][3] = b2.y;
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) S.x[h][r] = ld_gather(xp + r);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) S.x[h][r] = 0.0;
            }
        }
    };
    auto rows_of = [&](const Cur &c, Set &S) {
        const bool ok = c.s < n && c.w >= 0 && last_of(c);
#pragma unroll
        for (int h = 0; h < K; ++h) S.r[h] = ok ? __ldg(p.srows + static_cast<int64_t>(c.s) * C + h * 32 + lane) : -1;
    };

    Cur ca{s0, 0, 0, 0};
    {
        const int2 d = slice_of(s0);
        ca.off = d.x;
        ca.w = d.y;
    }
    int2 dnext = slice_of(s0 + 8);
    Cur cb = ca;
    advance(cb, dnext);
    Cur cc = cb;
    advance(cc, dnext);

    Set S0, S1;
    rows_of(ca, S0);
    load_cols(ca, S0);
    gather(ca, S0);
    load_vals(ca, S0);
    load_cols(cb, S1);
    rows_of(cb, S1);

    double acc[K][R];
#pragma unroll
    for (int h = 0; h < K; ++h)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[h][r] = 0.0;
    auto step = [&](Set &P, Set &Q) {
        gather(cb, Q);
        load_vals(cb, Q);
        load_cols(cc, P);
        if (ca.w < 0) {
            long_row_mr<VEC>(q, ca.off, alpha, beta, plain, lane);
        } else {
            if (has_slot(ca)) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int h = 0; h < K; ++h) acc[h][r] = fma(P.v[h], P.x[h][r], acc[h][r]);
            }
            if (last_of(ca)) {
#pragma unroll
                for (int h = 0; h < K; ++h) {
                    if (P.r[h] >= 0) {
                        double *yp = Y + static_cast<int64_t>(P.r[h]) * ldy;
                        double o[R];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double a = acc[h][r];
                            o[r] = plain ? a : (beta == 0.0 ? alpha * a : fma(alpha, a, beta * yp[r]));
                        }
                        if constexpr (VEC) {
                            reinterpret_cast<double2 *>(yp)[0] = make_double2(o[0], o[1]);
                            reinterpret_cast<double2 *>(yp)[1] = make_double2(o[2], o[3]);
                        } else {
#pragma unroll
                            for (int r = 0; r < R; ++r) yp[r] = o[r];
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) acc[h][r] = 0.0;
                }
            }
        }
        rows_of(cc, P);
        ca = cb;
        cb = cc;
        advance(cc, dnext);
    };
    while (ca.s < n) {
        step(S0, S1);
        if (ca.s >= n) break;
        step(S1, S0);
    }
}

// ---------------------------------------------------------------------------
// Block vectors, lanes across the right-hand sides: a group of L lanes takes a row
// (V right-hand sides per lane), G = 32/L groups the G next rows of a slice.  One
// row of X is then one contiguous access per group, whatever the width of the pass,
// where a lane per row needs a cache line of its own for every 16 bytes; the value
// and column of a slot are one broadcast load per group.  Each lane runs V chains;
// blocks of a few slot rows of loads, then their FMAs, and the resident warps (32
// per SM) keep the FP64 pipe, which bounds it, busy: Hamiltonian-like 4.2 M rows, 16
// and 32 right-hand sides 1,530 and 3,105 us (2,107 and 4,063 on the tile kernel; one
// FMA per entry and right-hand side takes 1,448 and 2,896), 5-point 1400^2 280 and 552
// (594 and 1,315; 262 and 524), 27-point 101^3, 5: 253 (371; 228).  Every row lies in a
// slice (no long rows).  VEC: the rows of X and Y allow 16-byte accesses (R
// even); otherwise the right-hand sides are loaded one by one and the last lane of a
// group may hold fewer than V.
// ---------------------------------------------------------------------------
struct SellRhsParams {
    SellMrParams m;  // one pass: X and Y at its first right-hand side
    int R, L, G;
};

template <int CNT, int V, bool VEC>
__device__ __forceinline__ void sell_rhs_block(double (&acc)[V], const double *__restrict__ vb,
                                               const int32_t *__restrict__ cb, const double *__restrict__ X,
                                               int64_t ldx, int nv) {
    int32_t c[CNT];
    double v[CNT], x[CNT][V];
#pragma unroll
    for (int u = 0; u < CNT; ++u) c[u] = __ldg(cb + u * kSellC);
#pragma unroll
    for (int u = 0; u < CNT; ++u) v[u] = __ldg(vb + u * kSellC);
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        const double *xp = X + static_cast<int64_t>(c[u]) * ldx;
        if constexpr (VEC) {
#pragma unroll
            for (int r = 0; r < V; r += 2) {
                const double2 t = c[u] >= 0 ? __ldg(reinterpret_cast<const double2 *>(xp + r)) : make_double2(0.0, 0.0);
                x[u][r] = t.x;
                x[u][r + 1] = t.y;
            }
        } else {
#pragma unroll
            for (int r = 0; r < V; ++r) x[u][r] = (c[u] >= 0 && r < nv) ? __ldg(xp + r) : 0.0;
        }
    }
#pragma unroll
    for (int u = 0; u < CNT; ++u)
#pragma unroll
        for (int r = 0; r < V; ++r) acc[r] = fma(v[u], x[u][r], acc[r]);
}

template <int V, bool VEC>
__global__ void __launch_bounds__(512, 2) k_sell_rhs(const SellRhsParams q) {
    constexpr int C = kSellC;
    const SellParams &p = q.m.b;
    const int lane = threadIdx.x & 31, L = q.L, G = q.G;
    if (static_cast<int>(blockIdx.x) >= p.n_ctas) return;
    const int s0 = __ldg(p.cstart + blockIdx.x), n = __ldg(p.cstart + blockIdx.x + 1);
    const int U = (C + G - 1) / G;  // units of G rows per slice
    const int g = lane / L;
    int c = (lane - g * L) * V;     // first right-hand side of the lane
    const int nv = g < G ? min(V, q.R - c) : 0;
    if (nv <= 0) c = 0;             // an idle lane reads what its group's first lane reads
    const double *__restrict__ vals = static_cast<const double *>(p.vals);
    const double *__restrict__ X = q.m.X + c;
    const int64_t ldx = q.m.ldx, ldy = q.m.ldy;
    const double alpha = p.alpha, beta = p.beta;
    const int emode = epi_mode(alpha, beta);
    for (int u = threadIdx.x >> 5; u < (n - s0) * U; u += 16) {
        const int s = s0 + u / U, b = u % U;
        const int2 d = __ldg(p.slices + s);
        double acc[V];
#pragma unroll
        for (int r = 0; r < V; ++r) acc[r] = 0.0;
        int row = -1;
        const int i = b * G + g;
        const bool ok = g < G && i < C;
        const int64_t base = static_cast<int64_t>(d.x) * C + (ok ? i : 0);
        if (ok) row = __ldg(p.srows + static_cast<int64_t>(s) * C + i);
        const double *__restrict__ vb = vals + base;
        const int32_t *__restrict__ cb = p.cols + base;
        constexpr int B = V <= 4 ? 4 : V <= 5 ? 3 : 2;  // slot rows in flight (registers)
        int w = d.y;
        for (; w >= B; w -= B) {
            sell_rhs_block<B, V, VEC>(acc, vb, cb, X, ldx, nv);
            vb += B * C;
            cb += B * C;
        }
        if (B > 3 && w == 3) sell_rhs_block<3, V, VEC>(acc, vb, cb, X, ldx, nv);
        else if (B > 2 && w == 2) sell_rhs_block<2, V, VEC>(acc, vb, cb, X, ldx, nv);
        else if (w == 1) sell_rhs_block<1, V, VEC>(acc, vb, cb, X, ldx, nv);
        if (row >= 0 && nv > 0) {
            double *yp = q.m.Y + static_cast<int64_t>(row) * ldy + c;
#pragma unroll
            for (int r = 0; r < V; ++r)
                if (VEC || r < nv) acc[r] = epi_apply(acc[r], yp + r, alpha, beta, emode);
            if constexpr (VEC) {
#pragma unroll
                for (int r = 0; r < V; r += 2) reinterpret_cast<double2 *>(yp)[r / 2] = make_double2(acc[r], acc[r + 1]);
            } else {
#pragma unroll
                for (int r = 0; r < V; ++r)
                    if (r < nv) yp[r] = acc[r];
            }
        }
    }
}

// Slot-major copy of the regular slices: row h*32 + l of slice s, holding row
// r, has entry rp[r] + j at slot (off + j)*64 + h*32 + l for j < len(r), value 0
// and column -1 after it.  cols_out may be null (values only, after new values),
// vals_out too (columns only).
template <typename VT>
__global__ void __launch_bounds__(256) k_sell_relayout(const int2 *__restrict__ slices,
                                                       const int32_t *__restrict__ srows, int32_t n_slices,
                                                       const int32_t *__restrict__ rp, const VT *__restrict__ val,
                                                       const int32_t *__restrict__ col, VT *__restrict__ vals_out,
                                                       int32_t *__restrict__ cols_out) {
    const int64_t total = static_cast<int64_t>(n_slices) * kSellC;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int2 d = slices[t / kSellC];
        if (d.y <= 0) continue;
        const int hl = static_cast<int>(t % kSellC);
        const int32_t row = srows[t];
        const int32_t k0 = row >= 0 ? rp[row] : 0;
        const int32_t len = row >= 0 ? rp[row + 1] - k0 : 0;
        for (int j = 0; j < d.y; ++j) {
            const int64_t slot = (static_cast<int64_t>(d.x) + j) * kSellC + hl;
            const bool ok = j < len;
            if (vals_out) vals_out[slot] = ok ? val[k0 + j] : VT(0);
            if (cols_out) cols_out[slot] = ok ? col[k0 + j] : -1;
        }
    }
}

template <typename VT, typename XT, typename YT, typename ACC>
struct SellKernel {
    static int grid_limit() {
        static int cached = -1;
        static int cached_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (cached >= 0 && cached_dev == dev) return cached;
        int per_sm = 0, sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sell<VT, XT, YT, ACC, false>, 256, 0) !=
            cudaSuccess)
            return 0;
        cached = per_sm * sms;
        cached_dev = dev;
        return cached;
    }
    // CTAs of a launch over n_slices slices: up to the resident limit, with at
    // least 8 slices each
    static int ctas_for(int32_t n_slices) {
        const int lim = grid_limit();
        if (lim <= 0) return 0;
        const int64_t want = (static_cast<int64_t>(n_slices) + 7) / 8;
        return static_cast<int>(want < lim ? want : lim);
    }
    // k_sell_diag on up to its resident CTAs, 8 half slices per CTA and turn
    template <bool SHORT, bool DOT, bool IND = false>
    static cudaError_t launch_diag(const SellParams &p, const RedOut &o, cudaStream_t s) {
        static int cached = -1;
        static int cached_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (cached < 0 || cached_dev != dev) {
            int per_sm = 0, sms = 0;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sell_diag<VT, XT, YT, ACC, SHORT, DOT, IND>, 256,
                                                              0) != cudaSuccess ||
                per_sm <= 0)
                return cudaErrorInvalidConfiguration;
            cached = per_sm * sms;
            cached_dev = dev;
        }
        const int64_t want = (2 * static_cast<int64_t>(p.n_slices) + 7) / 8;
        const int grid = static_cast<int>(want < cached ? want : cached);
        if (DOT && grid > cg_partials_cap()) return cudaErrorInvalidConfiguration;
        k_sell_diag<VT, XT, YT, ACC, SHORT, DOT, IND><<<grid, 256, 0, s>>>(p, o);
        return cudaGetLastError();
    }
    static cudaError_t launch(const SellParams &p, cudaStream_t s) {
        if (p.n_slices <= 0 || p.n_ctas <= 0) return cudaSuccess;
        if (p.dorder)
            return p.dshort ? launch_diag<true, false>(p, RedOut{}, s) : launch_diag<false, false>(p, RedOut{}, s);
        k_sell<VT, XT, YT, ACC, false><<<p.n_ctas, 256, 0, s>>>(p, RedOut{});
        return cudaGetLastError();
    }
    // y = A x on diagonal slices whose values are read through positions (p.vpos)
    static cudaError_t launch_ind(const SellParams &p, cudaStream_t s) {
        if (p.n_slices <= 0 || p.n_ctas <= 0) return cudaSuccess;
        if (!p.dorder || !p.vpos) return cudaErrorInvalidValue;
        return p.dshort ? launch_diag<true, false, true>(p, RedOut{}, s)
                        : launch_diag<false, false, true>(p, RedOut{}, s);
    }
    // y = A x with the dot x.y reduced into o (the CG step's p.q); needs at least
    // one slice and at most cg_partials_cap() CTAs
    static cudaError_t launch_dot(const SellParams &p, const RedOut &o, cudaStream_t s) {
        if (p.n_slices <= 0 || p.n_ctas <= 0 || p.n_ctas > cg_partials_cap()) return cudaErrorInvalidValue;
        if (p.dorder) return p.dshort ? launch_diag<true, true>(p, o, s) : launch_diag<false, true>(p, o, s);
        k_sell<VT, XT, YT, ACC, true><<<p.n_ctas, 256, 0, s>>>(p, o);
        return cudaGetLastError();
    }
};

}  // namespace spmv
