// Internal declarations shared by the translation units of the library (not part
// of the public ABI in include/spmv.h): the compiled configurations of each
// kernel family and the launchers of the auxiliary kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "types.h"
#include "cg.h"

namespace spmv {

// One compiled configuration of the tile kernel.
struct TileOps {
    cudaError_t (*launch)(const KParams &, int grid, cudaStream_t);
    int (*grid_limit)();   // CTAs resident on the whole GPU (persistent grid)
    TileCfg (*cfg)();
};

// Look up a compiled configuration.  vk/xk/yk: value and vector kinds, acc:
// accumulator, R: group width (1 for a single vector, right-hand sides per group
// for block vectors), E: entries per segment, indirect: values read through a
// permutation (transposed apply), batched: per-tile matrix table.
bool tile_ops(int vk, int xk, int yk, int acc, int R, int E, bool indirect, bool batched,
              TileOps *ops);
bool tile_ops_f64(int R, int E, bool indirect, bool batched, TileOps *ops);
bool tile_ops_f32(int xk, int yk, int acc, int R, int E, bool indirect, bool batched,
                  TileOps *ops);

struct WarpParams;
// One compiled configuration of the warp-chunk kernel (single right-hand side).
struct WarpOps {
    cudaError_t (*launch)(const WarpParams &, int n_chunks, cudaStream_t);
};
bool warp_ops(int vk, int xk, int yk, int acc, int E, bool indirect, bool batched, WarpOps *ops);
bool warp_ops_f64(int E, bool indirect, bool batched, WarpOps *ops);
bool warp_ops_f32(int yk, int acc, int E, bool indirect, bool batched, WarpOps *ops);

struct SlotParams;
// One compiled configuration of the slot-major chunk kernel (plan family 4).
struct SlotOps {
    cudaError_t (*launch)(const SlotParams &, cudaStream_t);
};
// pre: the variant that loads each chunk's row map and old y before its chains
// (row-mapped products).
bool slot_ops(int vk, int xk, int yk, int acc, int E, bool pre, SlotOps *ops);
// The variant whose values arrive by bulk copies into a shared-memory ring
// (plan family 6): FP64 E = 7, 9; FP32 float-float E = 9, 15.
bool slot_ops_tv(int vk, int xk, int yk, int acc, int E, SlotOps *ops);
// The batched variant (vectors of the value type): FP64, FP32 float-float; E = 7.
bool slot_ops_batched(int vk, int acc, int E, SlotOps *ops);
// Slot-major copies of the values (and, when cols_out is not null, the column
// indices) of the regular chunks in `chunks` (ChunkDesc[n_slots / (32E)]).
cudaError_t launch_slot_relayout(const void *chunks, int E, int64_t n_slots, int vk, const void *val,
                                 const int32_t *col, void *vals_out, int32_t *cols_out, cudaStream_t s);
// The slot-major copy of a map over the entries, -1 in the other slots.
cudaError_t launch_slot_map(const void *chunks, int E, int64_t n_slots, const int32_t *map, int32_t *map_out,
                            cudaStream_t s);

struct SellBatchParams;
// The batched launch over members on diagonal slices: FP64, or FP32 storage with short
// FP32 runs (rows of at most 11 entries).
cudaError_t launch_sell_diag_batch(const SellBatchParams &p, int vk, cudaStream_t s);

struct SellParams;
// One compiled configuration of the sorted row-slice kernel (plan family 5):
// (F64, F64, F64) with FP64 FMAs and (F32, F32, F32) with float-float sums.
struct SellOps {
    cudaError_t (*launch)(const SellParams &, cudaStream_t);
    int (*ctas_for)(int32_t n_slices);  // CTAs a launch over n_slices uses
    // values read through positions (p.vpos; diagonal slices); FP32 storage in
    // float-float, as the staged kernel that reads values through a permutation
    cudaError_t (*launch_ind)(const SellParams &, cudaStream_t);
    // y = A x plus the dot x.y reduced into a CG reduction target (FP32
    // storage only; nullptr elsewhere)
    cudaError_t (*launch_dot)(const SellParams &, const RedOut &, cudaStream_t);
};
// max_row: the longest row of the matrix; FP32 storage with the default
// accumulator takes FP32 runs (AccFR) when no row exceeds 11 entries, else FP32
// runs of one block folded into float-float (AccFRF).
bool sell_ops(int vk, int xk, int yk, int acc, SellOps *ops, int32_t max_row = 0x7fffffff);
// Block vectors on the sorted row slices, 4 right-hand sides:
// Y[i*ldy + r] = alpha*sum_j a_ij X[j*ldx + r] + beta*Y[i*ldy + r], r = 0..3
// (b carries the slices, alpha and beta; its x and y are not used).  vec: X, Y,
// ldx and ldy allow 16-byte accesses.
cudaError_t launch_sell_mr(const SellParams &b, const double *X, double *Y, int64_t ldx, int64_t ldy, bool vec,
                           cudaStream_t s);
// The same for R <= kSellMaxRhs right-hand sides with lanes across them.  scattered:
// x gathers find no neighbours in L1.
constexpr int kSellMaxRhs = 32;
cudaError_t launch_sell_rhs(const SellParams &b, const double *X, double *Y, int64_t ldx, int64_t ldy, int R, bool vec,
                            bool scattered, cudaStream_t s);
// Slot-major copies of the values (and, when cols_out is not null, the column
// indices) of the regular slices in `slices` (int2[n_slices]; srows: 32 rows per
// slice) from the CRS arrays rp, val, col.
cudaError_t launch_sell_relayout(const void *slices, const int32_t *srows, int32_t n_slices, const int32_t *rp,
                                 int vk, const void *val, const int32_t *col, void *vals_out, int32_t *cols_out,
                                 cudaStream_t s);

// Exclusive scan of n counts into out[0..n]; sums: scan_sums_len(n) entries of scratch.
cudaError_t launch_scan(const int32_t *in, int64_t n, int32_t *sums, int32_t *out, cudaStream_t s);
int64_t scan_sums_len(int64_t n);
// The row-slice tables of windows of kSellBuildSigma rows: slot rows counted from the
// leading padding on (off: n_slices + 1 entries, off[n_slices] = the slot rows), rows,
// descriptors, places of the diagonals and CTA ranges.  *too_long is set when a row
// has more than kSellBuildMaxRow entries (the tables are then not usable).
constexpr int32_t kSellBuildSigma = 4096;
constexpr int32_t kSellBuildMaxRow = 128;
cudaError_t launch_sell_build(const int32_t *rp, int32_t n_rows, int32_t n_slices, int32_t n_ctas, int32_t *srows,
                              int32_t *width, int32_t *off, int32_t *sums, uint32_t *too_long, void *d, void *dtmp,
                              int32_t *cstart, cudaStream_t s);
// Finds the diagonal slices (in every slot row all 64 rows are stored and column -
// row is one number): their diagonals into diag (int4 elements, from each slice's
// place dtmp[s].w on), place -1 for the others, and all descriptors into dorder,
// the others first.  The slot rows and the number of the diagonal slices are
// added to count[0] and [1].
cudaError_t launch_sell_mark_diag(void *dtmp, int32_t n_slices, const int32_t *srows, const int32_t *cols,
                                  void *diag, uint32_t *count, void *dorder, cudaStream_t s);

// vpos[slot] of the nT slices of A^T = position of the slot's value among the
// values of A's nA slices, -1 in padding (rowpos: n_rows entries of scratch).
// Every row of A lies in its slices (no long rows) and positions fit in int32.
cudaError_t launch_sell_vpos(const void *slicesA, const int32_t *srowsA, int32_t nA, const void *slicesT,
                             const int32_t *srowsT, int32_t nT, const int32_t *rp, const int32_t *rowT,
                             const int32_t *colT, const int32_t *perm, int32_t *rowpos, int32_t *vpos, cudaStream_t s);

// The longest row of the two launches below (every row lies in the slices).
int sell_tile_max_row();
// New values in CRS order (kind sk) into the handle's CRS copy dval (16-byte
// aligned) and the slices p.vals (kind vk).  max_w: the widest slice.
cudaError_t launch_sell_set_values(const SellParams &p, const void *val, int sk, void *dval, int vk, int max_w,
                                   cudaStream_t s);
// gv[k] = (p.alpha*g[row])*x[col], x = p.m.x, over the slices of p (gv in CRS
// order, 16-byte aligned).
cudaError_t launch_sell_grad_val(const SellParams &p, int vk, const void *g, void *gv, int max_w, cudaStream_t s);

// CG on A x = b (x0 = 0) as one cooperative kernel over the row slices of p (order:
// their descriptors with places in p.diag, in slice order; no long rows; max_w: the
// widest slice), tested for ||r|| <= tol*||b|| every kCgCheckEvery iterations.
// vk: kind of the values and vectors; dir, dir2, r: n entries of scratch each (r may
// be b, which is then overwritten); work: 4 * SMs
// doubles, 16-byte aligned; out (4 doubles): r.r, iterations, b.b, 1 after a barrier timed
// out (the GPU taken away for a second between two barriers): x, dir and r are then void.
constexpr int32_t kCgCheckEvery = 8;
bool cg_kernel_fits(int vk, int32_t n_slices, int max_w);
cudaError_t launch_cg(const SellParams &p, const int4 *order, int vk, int max_w, const void *b, void *x, void *dir,
                      void *dir2, void *r, double tol, int32_t max_iter, double *work, double *out, cudaStream_t s);

cudaError_t launch_rowvec(const KParams &p, const int32_t n_rows, int vk, int xk, int yk, int acc,
                          int T, cudaStream_t s);

// out[k] = val[perm[k]] for k < nnz (values of kind vk: FP64 or FP32).
cudaError_t launch_permute(const void *val, const int32_t *perm, void *out, int64_t nnz, int vk, cudaStream_t s);
// out[t] = val[map[t]] for t < n, 0 where map[t] < 0 (map and out 16-byte aligned).
cudaError_t launch_fill_slots(const void *val, const int32_t *map, void *out, int64_t n, int vk, cudaStream_t s);
// The full CRS of a symmetric matrix from its upper triangle (rp, col) and the
// transposed strictly upper part (rowS, colS, permS); mapF: position of each entry's
// value among U's.
cudaError_t launch_expand_sym(int32_t n, const int32_t *rp, const int32_t *col, const int32_t *rowS,
                              const int32_t *colS, const int32_t *permS, int32_t *rpF, int32_t *colF, int32_t *mapF,
                              cudaStream_t s);
// Device-side CRS check; sets *bad to 1 on any violation.
cudaError_t launch_validate(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t *rp, const int32_t *col,
                            int32_t *bad, cudaStream_t s);
// One warp waits on an mbarrier nothing completes, for limit_ns, then records
// kDevErrTimeout in *err.
cudaError_t launch_wait_timeout(uint64_t limit_ns, int32_t *err, cudaStream_t s);
// Halo gather: halo[h] = x[map[h]].
cudaError_t launch_gather(const double *x, const int32_t *map, double *halo, int64_t n,
                          cudaStream_t s);

// grad_val over the warp chunks of A (ChunkDesc table + row-start bitmasks with
// mwp words per chunk): chunks of kGradValE entries per lane, mwp = kGradValWords
// (other tables are rejected with cudaErrorInvalidValue).
constexpr int kGradValE = 7;
constexpr int kGradValWords = 8;
cudaError_t launch_grad_val_chunks(const int32_t *rp, const int32_t *col, const void *chunks,
                                   const uint32_t *masks, int mwp, int32_t n_chunks, int vk,
                                   const void *g, const void *x, double alpha, void *grad_val,
                                   cudaStream_t s);

// Transposed structure: counts, exclusive scan, fill, per-row ordering.
cudaError_t launch_transpose(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t *rp,
                             const int32_t *col, int32_t *rowT, int32_t *colT, int32_t *perm,
                             int32_t *work, cudaStream_t s);

// Transposed structure into caller buffers with the fixed device work array
// (no allocation); n_cols <= transpose_noalloc_max_cols().
cudaError_t launch_transpose_noalloc(int32_t n_rows, int32_t n_cols, int64_t nnz, const int32_t *rp,
                                     const int32_t *col, int32_t *rowT, int32_t *colT, int32_t *perm,
                                     cudaStream_t s);
int64_t transpose_noalloc_max_cols();

// Value conversion (FP64 <-> FP32), n entries.
cudaError_t launch_convert(const void *src, int sk, void *dst, int dk, int64_t n, cudaStream_t s);

// Vector kernels of the CG solvers (see cg.cu).
cudaError_t launch_fill(void *p, int k, double v, int64_t n, cudaStream_t s);

}  // namespace spmv
