// Compiled configurations of the slot-major chunk kernel (plan family 4) and its
// relayout kernel: FP64 values and vectors, and FP32 storage with FP32 runs and
// float-float carries (E = 7, 9, 11: at most 11 entries of a row per lane) or
// float-float accumulation (E = 15).
#include "internal.h"
#include "slot_kernel.cuh"

namespace spmv {

bool slot_ops_batched(int vk, int acc, int E, SlotOps *ops) {
    if (vk == kF64 && acc == kAccF64 && E == 7) {
        ops->launch = &SlotKernel<7, double, double, double, AccF64, kUpdPlain, true>::launch;
        return true;
    }
    if (vk == kF64 && acc == kAccF64 && E == 9) {
        ops->launch = &SlotKernel<9, double, double, double, AccF64, kUpdPlain, true>::launch;
        return true;
    }
    if (vk == kF32 && acc == kAccFF && E == 7) {
        ops->launch = &SlotKernel<7, float, float, float, AccFR, kUpdPlain, true>::launch;
        return true;
    }
    if (vk == kF32 && acc == kAccFF && E == 9) {
        ops->launch = &SlotKernel<9, float, float, float, AccFR, kUpdPlain, true>::launch;
        return true;
    }
    return false;
}

bool slot_ops(int vk, int xk, int yk, int acc, int E, bool pre, SlotOps *ops) {
    if (pre) {
        // row-mapped products (the split's nonlocal part): FP64, E = 7 (E = 9
        // measured no faster there: split 230.9 against 229.4 us)
        if (vk == kF64 && xk == kF64 && yk == kF64 && acc == kAccF64 && E == 7) {
            ops->launch = &SlotKernel<7, double, double, double, AccF64, kUpdMap>::launch;
            return true;
        }
        return false;
    }
#define SPMV_S(VK_, XK_, YK_, ACCK_, E_, VT_, XT_, YT_, ACC_)                                 \
    if (vk == VK_ && xk == XK_ && yk == YK_ && acc == ACCK_ && E == E_) {                     \
        ops->launch = &SlotKernel<E_, VT_, XT_, YT_, ACC_>::launch_any;                          \
        return true;                                                                          \
    }
    SPMV_S(kF64, kF64, kF64, kAccF64, 7, double, double, double, AccF64)
    SPMV_S(kF64, kF64, kF64, kAccF64, 9, double, double, double, AccF64)
    SPMV_S(kF64, kF64, kF64, kAccF64, 11, double, double, double, AccF64)
    SPMV_S(kF64, kF64, kF64, kAccF64, 15, double, double, double, AccF64)
    SPMV_S(kF32, kF32, kF32, kAccFF, 7, float, float, float, AccFR)
    SPMV_S(kF32, kF32, kF32, kAccFF, 9, float, float, float, AccFR)
    SPMV_S(kF32, kF32, kF32, kAccFF, 11, float, float, float, AccFR)
    SPMV_S(kF32, kF32, kF32, kAccFF, 15, float, float, float, AccFF)
#undef SPMV_S
    return false;
}

bool slot_ops_tv(int vk, int xk, int yk, int acc, int E, SlotOps *ops) {
    if (vk == kF64 && xk == kF64 && yk == kF64 && acc == kAccF64) {
        if (E == 7) { ops->launch = &SlotKernelTV<7, double, double, double, AccF64>::launch; return true; }
        if (E == 9) { ops->launch = &SlotKernelTV<9, double, double, double, AccF64>::launch; return true; }
    }
    if (vk == kF32 && xk == kF32 && yk == kF32 && acc == kAccFF) {
        if (E == 9) { ops->launch = &SlotKernelTV<9, float, float, float, AccFF>::launch; return true; }
        if (E == 15) { ops->launch = &SlotKernelTV<15, float, float, float, AccFF>::launch; return true; }
    }
    return false;
}

template <typename VT>
static cudaError_t relayout_as(const void *chunks, int E, int64_t n_slots, const void *val, const int32_t *col,
                               void *vals_out, int32_t *cols_out, VT pad, cudaStream_t s) {
    if (n_slots <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (n_slots + 255) / 256;
    const int grid = static_cast<int>(want < 16LL * sms ? want : 16LL * sms);
    k_slot_relayout<VT><<<grid, 256, 0, s>>>(static_cast<const ChunkDesc *>(chunks), E, n_slots,
                                             static_cast<const VT *>(val), col, static_cast<VT *>(vals_out), cols_out,
                                             pad);
    return cudaGetLastError();
}

cudaError_t launch_slot_relayout(const void *chunks, int E, int64_t n_slots, int vk, const void *val,
                                 const int32_t *col, void *vals_out, int32_t *cols_out, cudaStream_t s) {
    return vk == kF64 ? relayout_as<double>(chunks, E, n_slots, val, col, vals_out, cols_out, 0.0, s)
                      : relayout_as<float>(chunks, E, n_slots, val, col, vals_out, cols_out, 0.0f, s);
}

cudaError_t launch_slot_map(const void *chunks, int E, int64_t n_slots, const int32_t *map, int32_t *map_out,
                            cudaStream_t s) {
    return relayout_as<int32_t>(chunks, E, n_slots, map, nullptr, map_out, nullptr, -1, s);
}

}  // namespace spmv
