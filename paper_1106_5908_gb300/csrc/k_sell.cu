// Compiled configurations of the sorted row-slice kernel (plan family 5) and its
// relayout kernel: FP64 values and vectors, and FP32 storage with FP32 runs
// (every row at most 11 entries, so a lane's chain over a row is a run) or FP32
// runs of one block (4 slot rows) each folded into float-float.
#include "internal.h"
#include "sell_kernel.cuh"

namespace spmv {

bool sell_ops(int vk, int xk, int yk, int acc, SellOps *ops, int32_t max_row) {
    if (vk == kF64 && xk == kF64 && yk == kF64 && acc == kAccF64) {
        ops->launch = &SellKernel<double, double, double, AccF64>::launch;
        ops->ctas_for = &SellKernel<double, double, double, AccF64>::ctas_for;
        ops->launch_dot = nullptr;
        return true;
    }
    if (vk == kF32 && xk == kF32 && yk == kF32 && acc == kAccFF && max_row <= kFRMaxRun) {
        ops->launch = &SellKernel<float, float, float, AccFR>::launch;
        ops->ctas_for = &SellKernel<float, float, float, AccFR>::ctas_for;
        ops->launch_dot = &SellKernel<float, float, float, AccFR>::launch_dot;
        return true;
    }
    if (vk == kF32 && xk == kF32 && yk == kF32 && acc == kAccFF) {
        ops->launch = &SellKernel<float, float, float, AccFRF>::launch;
        ops->ctas_for = &SellKernel<float, float, float, AccFRF>::ctas_for;
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

cudaError_t launch_sell_relayout(const void *slices, const int32_t *srows, int32_t n_slices, const int32_t *rp,
                                 int vk, const void *val, const int32_t *col, void *vals_out, int32_t *cols_out,
                                 cudaStream_t s) {
    if (n_slices <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (static_cast<int64_t>(n_slices) * kSellC + 255) / 256;
    const int grid = static_cast<int>(want < 16LL * sms ? want : 16LL * sms);
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
