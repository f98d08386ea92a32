// Conjugate gradients as one cooperative kernel, for matrices on diagonal row
// slices whose vectors fit in the SMs' shared memory.
//
// A CG iteration on a small grid is all latency: product, dot, update and
// direction as four kernels of a graph take 18.5 us on the 256^2 5-point matrix
// (984 iterations, 8.7 us here), whose bytes would pass in one.  Here one CTA per SM owns a contiguous range of
// half slices for the whole solve.  x, r and q of its rows stay in shared memory
// (with the matrix values, when they fit too), so only p goes through L2; the two
// dots and the new p are three grid barriers per iteration.  Where few half slices
// fall to a CTA, the product forms the new p as it gathers (r + beta p, in every
// place it is needed: one more FMA per entry) and two barriers are enough.  A dot's partial sums
// (one per CTA) are summed by every CTA in the same order, so all CTAs take the
// same steps and the result is deterministic.  The convergence test runs on the
// device every kCgCheckEvery iterations, as the host's does for the other path.
#include <algorithm>

#include "internal.h"
#include "sell_kernel.cuh"

namespace spmv {

namespace {

constexpr int kCgThreads = 1024;

// At a barrier every CTA publishes its partial sum in a slot of its own and polls
// the slots of all, so the sum needs no round trip beside the barrier's.  A slot
// is empty until then (a bit pattern that no sum has).  Slots are written by
// atomic exchanges, which take effect in L2 at once: 152 CTAs meet in 1,700 cycles
// (0.8 us; one counter with release and acquire 2,400; plain stores become visible
// to polling CTAs only after some 10,000).
constexpr unsigned long long kCgEmpty = ~0ull;
constexpr unsigned long long kCgNaN = 0x7ff8000000000000ull;
constexpr unsigned long long kCgNever = 0x7ff4000000000001ull;  // no slot ever holds this signalling NaN
__device__ __forceinline__ unsigned long long slot_exchange(unsigned long long *p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.exch.relaxed.gpu.global.b64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}
__device__ __forceinline__ unsigned long long slot_peek(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// The barriers of one launch: four sets of slots in turn.  Set k (mod 4) is used at
// barrier k; a CTA empties its slot of set k + 2 at barrier k, when all CTAs have
// published for k - 1 and so have read the set's last sums (of k - 2), and before
// it publishes for k + 1, which every CTA waits for ahead of polling set k + 2.
constexpr int kCgMarks = 5;  // slots per lane of the polling warp: up to 160 CTAs
struct Grid {
    unsigned long long *slots;  // 4 * gridDim.x, empty at launch
    unsigned int phase;
    unsigned long long last;    // what emptying a slot returned (lane 0 of warp 0)
    double *s_part;  // kCgThreads doubles of shared memory
    double *s_out;   // 3: the sum, the step made of it, whether all CTAs arrived

    // The sum of v over the grid and the scalar step f(sum), in every thread; a sum
    // orders the CTAs' work (its terms are computed from what they read) but does
    // not make their writes visible.  Only warp 0 adds and divides: every warp
    // instruction takes the FP64 pipe 16 cycles.  false: a bounded wait gave up.
    // PUBLISH: it is a sync() as well.
    template <bool PUBLISH, typename F>
    __device__ __forceinline__ bool sum(double v, F f, double *total, double *step) {
        s_part[threadIdx.x] = v;
        __syncthreads();
        ++phase;
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            double t[4] = {0.0, 0.0, 0.0, 0.0};
            for (int i = lane; i < static_cast<int>(blockDim.x); i += 128)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i + 32 * u < static_cast<int>(blockDim.x)) t[u] += s_part[i + 32 * u];
            unsigned long long m[kCgMarks];
            const bool ok = exchange<PUBLISH>(warp_sum((t[0] + t[1]) + (t[2] + t[3])), lane, m);
            static_assert(kCgMarks == 5, "the sum below");
            const double a = warp_sum(((value(m[0]) + value(m[1])) + (value(m[2]) + value(m[3]))) + value(m[4]));
            const double st = f(a);
            if (lane == 0) {
                s_out[0] = a;
                s_out[1] = st;
                s_out[2] = ok ? 1.0 : 0.0;
            }
        }
        __syncthreads();
        *total = s_out[0];
        *step = s_out[1];
        return s_out[2] != 0.0;
    }
    // All CTAs' earlier writes are visible to all after it.
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        ++phase;
        if (threadIdx.x < 32) {
            unsigned long long m[kCgMarks];
            const bool ok = exchange<true>(0.0, threadIdx.x, m);
            if (threadIdx.x == 0) s_out[2] = ok ? 1.0 : 0.0;
        }
        __syncthreads();
        return s_out[2] != 0.0;
    }

  private:
    static __device__ __forceinline__ double warp_sum(double t) {
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    }
    static __device__ __forceinline__ double value(unsigned long long m) {
        return __longlong_as_double(static_cast<long long>(m));
    }
    // Warp 0: publish t and wait (bounded) for every CTA's slot, this lane's into m.
    // A lane's slots are polled together (one after the other costs a round trip
    // each).  PUBLISH: the CTA's earlier writes are released, the others' acquired.
    template <bool PUBLISH>
    __device__ __forceinline__ bool exchange(double t, int lane, unsigned long long (&m)[kCgMarks]) {
        const int G = gridDim.x;
        unsigned long long *set = slots + (phase & 3u) * G;
        bool ok = true;
        if (lane == 0) {
            if constexpr (PUBLISH) asm volatile("fence.acq_rel.gpu;" ::: "memory");
            unsigned long long v = static_cast<unsigned long long>(__double_as_longlong(t));
            if (v == kCgEmpty || v == kCgNever) v = kCgNaN;
            // the slot emptied at the last barrier is empty now: its exchange has returned
            ok = last != kCgNever;
            if (ok) (void)slot_exchange(set + blockIdx.x, v);
            last = slot_exchange(slots + ((phase + 2) & 3u) * G + blockIdx.x, kCgEmpty);
        }
        uint64_t t0 = 0;
        for (uint32_t it = 0;; ++it) {
            bool all = true;
#pragma unroll
            for (int u = 0; u < kCgMarks; ++u) m[u] = lane + 32 * u < G ? slot_peek(set + lane + 32 * u) : 0ull;
#pragma unroll
            for (int u = 0; u < kCgMarks; ++u) all = all && m[u] != kCgEmpty;
            if (__all_sync(0xffffffffu, all)) break;
            __nanosleep(32);
            if ((it & 63u) == 63u) {
                const uint64_t now = global_timer_ns();
                if (t0 == 0) t0 = now;
                ok = ok && now - t0 <= kWaitLimitNs && it <= kWaitLimitIters * 64u;
            }
            if (__any_sync(0xffffffffu, !ok)) {
                ok = false;
                break;
            }
        }
        if constexpr (PUBLISH) asm volatile("fence.acq_rel.gpu;" ::: "memory");
        return ok;
    }
};

// The operand of the product: p, or (FUSE) r + beta p from the last p.  Both change
// during the kernel: their loads are ordinary ones (never the read-only path).
template <bool FUSE, typename T>
struct CgVec {
    const T *p, *r;
    T beta;
    __device__ __forceinline__ T at(int i) const {
        if constexpr (FUSE) return fma(beta, p[i], r[i]);
        else return p[i];
    }
};

// CNT slot rows of a half slice times p.
template <int CNT, bool DIAG, int VS, typename ACC, typename T, typename V>
__device__ __forceinline__ void cg_block(ACC &acc, const T *v, const int32_t *__restrict__ cb,
                                         const int4 *dp, int row, const V &p) {
    int32_t c[CNT];
    if constexpr (DIAG) {
        const int4 a = dp[0];
        int4 b = make_int4(0, 0, 0, 0);
        if constexpr (CNT > 4) b = dp[1];
        const int32_t g[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = row + g[u];
    } else {
#pragma unroll
        for (int u = 0; u < CNT; ++u) c[u] = __ldg(cb + u * kSellC);
    }
    T vv[CNT], xv[CNT];
#pragma unroll
    for (int u = 0; u < CNT; ++u) vv[u] = v[u * VS];
#pragma unroll
    for (int u = 0; u < CNT; ++u) xv[u] = (DIAG || c[u] >= 0) ? p.at(c[u]) : T(0);
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
        acc.fma(vv[u], xv[u]);
        if (u % kSellU == kSellU - 1 || u == CNT - 1) end_run(acc);
    }
}

template <bool DIAG, int VS, typename ACC, typename T, typename V>
__device__ __forceinline__ void cg_row(ACC &acc, int w, const T *v, const int32_t *__restrict__ cb,
                                       const int4 *dp, int row, const V &p) {
    for (; w >= 8; w -= 8) {
        cg_block<8, DIAG, VS>(acc, v, cb, dp, row, p);
        v += 8 * VS;
        if constexpr (DIAG) dp += 2;
        else cb += 8 * kSellC;
    }
    switch (w) {
        case 7: cg_block<7, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 6: cg_block<6, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 5: cg_block<5, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 4: cg_block<4, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 3: cg_block<3, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 2: cg_block<2, DIAG, VS>(acc, v, cb, dp, row, p); break;
        case 1: cg_block<1, DIAG, VS>(acc, v, cb, dp, row, p); break;
        default: break;
    }
}

// The stored value of a row's sum; a poisoned FP32 sum is formed again from the
// CRS arrays with exact products, as elsewhere, but with ordinary loads of p.
template <typename T, typename ACC, typename V>
__device__ __forceinline__ T cg_result(const ACC &a, const MatRef &m, int row, const V &p) {
    if constexpr (std::is_same<ACC, AccF64>::value) {
        return a.get();
    } else {
        if (!a.poisoned()) return a.h + a.l;
        double s = 0.0;
        for (int k = __ldg(m.rp + row); k < __ldg(m.rp + row + 1); ++k)
            s = fma(widen(__ldg(static_cast<const T *>(m.vs) + k)), widen(p.at(__ldg(m.col + k))), s);
        return narrow<T>(s);
    }
}

// Thread sums of r.r: FP64 FMAs, or float-float for FP32 vectors, as the vector kernels
// of the other path (off the FP64 pipe; out of FP32's range the caller sums the thread's
// terms again).
template <typename T> struct DotAcc { using type = AccF64; };
template <> struct DotAcc<float> { using type = AccFF; };
__device__ __forceinline__ bool dot_poisoned(const AccF64 &) { return false; }
__device__ __forceinline__ bool dot_poisoned(const AccFF &a) { return a.poisoned(); }

__device__ __forceinline__ double step_scale(double a, double *) { return a; }
__device__ __forceinline__ float step_scale(double a, float *) { return __double2float_rn(a); }

}  // namespace

struct CgParams {
    const int4 *order;      // slices: first slot row, width, slice, place in diag (-1: column indices)
    const int32_t *srows;
    const int4 *diag;
    const void *vals;
    const int32_t *cols;
    MatRef m;               // the CRS arrays (FP32 sums out of range)
    int32_t n_half;         // half slices
    int32_t per_cta;        // half slices per CTA
    int32_t max_w;          // the widest slice
    const void *b;          // right-hand side
    void *x, *p;            // the solution (written at the end) and the direction
    void *p2, *r;           // FUSE: the other direction vector and the residual
    unsigned long long *slots;  // 4 per CTA, empty
    double *out;            // rho, iterations, b.b, 1 after a timeout
    double tol;
    int32_t max_iter;
};

// VSM: the matrix values are kept in shared memory too.  FUSE: two barriers (above).
// XG: x stays in global memory (only its own CTA touches it).
template <typename T, typename ACC, bool VSM, bool FUSE, bool XG>
__global__ void __launch_bounds__(kCgThreads, 1) k_cg(const CgParams q) {
    using Dot = typename DotAcc<T>::type;
    constexpr int VS = VSM ? 32 : kSellC;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_part[kCgThreads];
    __shared__ double s_out[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int h0 = blockIdx.x * q.per_cta;
    const int cnt = max(0, min(q.per_cta, q.n_half - h0));
    // per half slice: descriptor, rows, and the rows' x, r and q (and values); per
    // slice: its diagonals
    const int ndg = (q.max_w + 3) / 4;  // int4 per slice
    int4 *s_d = reinterpret_cast<int4 *>(smem), *s_dg = s_d + q.per_cta;
    T *s_r = reinterpret_cast<T *>(s_dg + (q.per_cta / 2 + 1) * ndg), *s_q = s_r + q.per_cta * 32;
    T *s_p = s_q + q.per_cta * 32;  // FUSE
    T *s_x = s_p + (FUSE ? q.per_cta * 32 : 0);  // not XG
    T *s_v = s_x + (XG ? 0 : q.per_cta * 32);
    int32_t *s_row = reinterpret_cast<int32_t *>(s_v + (VSM ? q.per_cta * 32 * q.max_w : 0));
    Grid grid{q.slots, 0u, 0ull, s_part, s_out};
    T *p = static_cast<T *>(q.p), *p2 = static_cast<T *>(q.p2), *r = static_cast<T *>(q.r);
    const T *vals = static_cast<const T *>(q.vals);
    T *x = static_cast<T *>(q.x);

    // x = 0, r = p = b, rho = b.b
    double dot = 0.0;
    for (int l = warp; l < cnt; l += nw) {
        const int h = h0 + l;
        const int4 d = __ldg(q.order + (h >> 1));
        const int row = __ldg(q.srows + static_cast<int64_t>(d.z) * kSellC + (h & 1) * 32 + lane);
        if (lane == 0) s_d[l] = d;
        const int own = (h >> 1) - (h0 >> 1);  // the slice's place in s_dg
        if (d.w >= 0 && lane < (d.y + 3) / 4) s_dg[own * ndg + lane] = __ldg(q.diag + d.w + lane);
        const int i = l * 32 + lane;
        s_row[i] = row;
        // an ordinary load: b may be r, which this kernel writes
        const T b = row >= 0 ? static_cast<const T *>(q.b)[row] : T(0);
        if constexpr (XG) {
            if (row >= 0) x[row] = T(0);
        } else {
            s_x[i] = T(0);
        }
        s_r[i] = b;
        s_q[i] = T(0);
        if (row >= 0) {
            p[row] = FUSE ? T(0) : b;
            if constexpr (FUSE) r[row] = b;
        }
        dot = fma(widen(b), widen(b), dot);
        if constexpr (VSM) {
            const T *src = vals + static_cast<int64_t>(d.x) * kSellC + (h & 1) * 32 + lane;
            for (int j = 0; j < d.y; ++j) s_v[(l * q.max_w + j) * 32 + lane] = __ldg(src + j * kSellC);
        }
    }
    double rho = 0.0, step = 0.0;
    bool ok = grid.sum<true>(dot, [](double t) { return t; }, &rho, &step);
    T be = T(0);  // beta
    const double bb = rho;
    int it = 0;
    while (ok && it < q.max_iter && sqrt(rho) > q.tol * sqrt(bb)) {
        const int stop = min(q.max_iter, it + kCgCheckEvery);
        for (; ok && it < stop; ++it) {
            // q = A p, p.q (in FP64, of exact products for FP32 vectors too)
            AccF64 pq;
            pq.zero();
            const CgVec<FUSE, T> pv{p, r, be};
            for (int l = warp; l < cnt; l += nw) {
                const int4 d = s_d[l];
                const int i = l * 32 + lane, row = s_row[i], half = ((h0 + l) & 1) * 32 + lane;
                const int64_t base = static_cast<int64_t>(d.x) * kSellC + half;
                const T *v = VSM ? s_v + l * q.max_w * 32 + lane : vals + base;
                ACC acc;
                acc.zero();
                if (d.w >= 0)
                    cg_row<true, VS>(acc, d.y, v, static_cast<const int32_t *>(nullptr),
                                     s_dg + (((h0 + l) >> 1) - (h0 >> 1)) * ndg, row, pv);
                else
                    cg_row<false, VS>(acc, d.y, v, q.cols + base, static_cast<const int4 *>(nullptr), row, pv);
                if (row >= 0) {
                    const T y = cg_result<T>(acc, q.m, row, pv), pr = pv.at(row);
                    s_q[i] = y;
                    if constexpr (FUSE) {
                        s_p[i] = pr;
                        p2[row] = pr;
                    }
                    pq.fma(pr, y);
                }
            }
            double tot;
            ok = grid.sum<false>(pq.get(), [rho](double pq) { return pq != 0.0 ? rho / pq : 0.0; }, &tot, &step);
            if (!ok) break;
            // x += alpha p, r -= alpha q, r.r (a zero direction takes no step)
            const T a = step_scale(step, static_cast<T *>(nullptr));
            Dot rr;
            rr.zero();
            for (int l = warp; l < cnt; l += nw) {
                const int i = l * 32 + lane, row = s_row[i];
                if (row >= 0) {
                    const T pr = FUSE ? s_p[i] : p[row];
                    if constexpr (XG) x[row] = fma(a, pr, x[row]);
                    else s_x[i] = fma(a, pr, s_x[i]);
                    const T ri = fma(-a, s_q[i], s_r[i]);
                    s_r[i] = ri;
                    if constexpr (FUSE) r[row] = ri;
                    rr.fma(ri, ri);
                }
            }
            double t = rr.get();
            if (dot_poisoned(rr)) {
                t = 0.0;
                for (int l = warp; l < cnt; l += nw) {
                    const double ri = widen(s_r[l * 32 + lane]);
                    t = fma(ri, ri, t);
                }
            }
            ok = grid.sum<FUSE>(t, [rho](double rr) { return rho != 0.0 ? rr / rho : 0.0; }, &tot, &step);
            if (!ok) break;
            // p = r + beta p
            be = static_cast<T>(step);
            rho = tot;
            if constexpr (FUSE) {
                T *last = p;
                p = p2;
                p2 = last;
            } else {
                for (int l = warp; l < cnt; l += nw) {
                    const int i = l * 32 + lane, row = s_row[i];
                    if (row >= 0) p[row] = fma(be, p[row], s_r[i]);
                }
                ok = grid.sync();
            }
        }
    }
    if constexpr (!XG) {
        for (int l = warp; l < cnt; l += nw) {
            const int row = s_row[l * 32 + lane];
            if (row >= 0) x[row] = s_x[l * 32 + lane];
        }
    }
    if (threadIdx.x == 0) {
        if (!ok) {
            q.out[3] = 1.0;
        } else if (blockIdx.x == 0) {
            q.out[0] = rho;
            q.out[1] = it;
            q.out[2] = bb;
        }
    }
}

namespace {

// Slot rows of half slices per CTA up to which the product forms the new p itself:
// the FMA per entry costs FP64 more than a barrier from about there on (us per
// iteration with and without: 5-point 256^2 8.7 / 9.1, 400^2 13.4 / 12.9, 600^2 17.9 /
// 15.9), FP32 nothing up to the largest that fits (7-point 96^3 16.9 / 17.7).
constexpr int kCgFuse64 = 128;
constexpr int kCgFuse32 = 1536;

struct CgPlan {
    int grid = 0, per_cta = 0, threads = 0;
    bool vsm = false, fuse = false, xg = false;
    size_t smem = 0;
};

// One CTA per SM over the half slices, if a CTA's vectors fit in shared memory;
// the matrix values too when there is room.
bool cg_plan(int vk, int32_t n_half, int max_w, CgPlan *pl) {
    int dev = 0, sms = 0, most = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || n_half <= 0 || sms <= 0 || sms > 32 * kCgMarks) return false;
    const size_t room = static_cast<size_t>(most) - 8 * kCgThreads - 256;  // less the static shared memory
    const size_t vb = vk == kF64 ? 8 : 4;
    pl->per_cta = (n_half + sms - 1) / sms;
    pl->grid = (n_half + pl->per_cta - 1) / pl->per_cta;
    pl->threads = 32 * std::min(kCgThreads / 32, std::max(4, pl->per_cta));
    const size_t rows = static_cast<size_t>(pl->per_cta) * 32;
    const size_t tables = static_cast<size_t>(pl->per_cta) * 16 +
                          static_cast<size_t>(pl->per_cta / 2 + 1) * ((max_w + 3) / 4) * 16 + rows * 4;
    pl->fuse = pl->per_cta * max_w <= (vk == kF64 ? kCgFuse64 : kCgFuse32) && tables + rows * vb * 4 <= room;
    const size_t base = tables + rows * vb * (pl->fuse ? 4 : 3);
    const size_t with = base + rows * max_w * vb, least = tables + rows * vb * 2;
    pl->vsm = with <= room;
    pl->xg = !pl->fuse && base > room;
    pl->smem = pl->vsm ? with : (pl->xg ? least : base);
    return pl->smem <= room;
}

template <typename T, typename ACC, bool VSM, bool FUSE, bool XG = false>
cudaError_t cg_launch_as(const CgParams &q, const CgPlan &pl, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_cg<T, ACC, VSM, FUSE, XG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(pl.smem));
    if (e != cudaSuccess) return e;
    CgParams arg = q;
    void *args[] = {&arg};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(&k_cg<T, ACC, VSM, FUSE, XG>), dim3(pl.grid),
                                       dim3(pl.threads), args, pl.smem, s);
}

template <typename T, typename ACC>
cudaError_t cg_launch(const CgParams &q, const CgPlan &pl, cudaStream_t s) {
    if (pl.fuse)
        return pl.vsm ? cg_launch_as<T, ACC, true, true>(q, pl, s) : cg_launch_as<T, ACC, false, true>(q, pl, s);
    if (pl.xg) return cg_launch_as<T, ACC, false, false, true>(q, pl, s);
    return pl.vsm ? cg_launch_as<T, ACC, true, false>(q, pl, s) : cg_launch_as<T, ACC, false, false>(q, pl, s);
}

}  // namespace

bool cg_kernel_fits(int vk, int32_t n_slices, int max_w) {
    CgPlan pl;
    return cg_plan(vk, 2 * n_slices, max_w, &pl);
}

cudaError_t launch_cg(const SellParams &p, const int4 *order, int vk, int max_w, const void *b, void *x, void *dir,
                      void *dir2, void *r, double tol, int32_t max_iter, double *work, double *out, cudaStream_t s) {
    CgPlan pl;
    if (!cg_plan(vk, 2 * p.n_slices, max_w, &pl)) return cudaErrorInvalidConfiguration;
    CgParams q{};
    q.order = order;
    q.srows = p.srows;
    q.diag = p.diag;
    q.vals = p.vals;
    q.cols = p.cols;
    q.m = p.m;
    q.n_half = 2 * p.n_slices;
    q.per_cta = pl.per_cta;
    q.max_w = max_w;
    q.b = b;
    q.x = x;
    q.p = dir;
    q.p2 = dir2;
    q.r = r;
    q.slots = reinterpret_cast<unsigned long long *>(work);
    q.out = out;
    q.tol = tol;
    q.max_iter = max_iter;
    cudaError_t e = cudaMemsetAsync(work, 0xff, 4 * sizeof(*q.slots) * pl.grid, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(out, 0, 4 * sizeof(double), s);
    if (e != cudaSuccess) return e;
    if (vk == kF64) return cg_launch<double, AccF64>(q, pl, s);
    // FP32 sums as the row-slice kernel forms them: runs over whole rows of at most
    // kFRMaxRun entries, else runs of kSellU entries folded into float-float
    return max_w <= kFRMaxRun ? cg_launch<float, AccFR>(q, pl, s) : cg_launch<float, AccFRF>(q, pl, s);
}

}  // namespace spmv
