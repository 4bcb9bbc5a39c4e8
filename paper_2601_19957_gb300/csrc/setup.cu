// setup.cu -- per-problem constants of the likelihood and the prior box.
//   a_k  = log w_k - (d/2) log 2pi + sum_i log L_k,ii   (normalised Gaussian, Sec. 3.2)
//   c    = (lo + hi) / 2, half = (hi - lo) / 2          (prior centre, Sec. 3.4.1)
//   logV = sum_i log(hi_i - lo_i)                        (prior volume, Sec. 3.2)
// It also validates what only the device can see: lo < hi, L_k,ii > 0, finite values.
#include "sb_internal.cuh"

namespace sb {

template <typename T, typename Op>
__device__ T block_reduce(T v, Op op, T *sh, T identity) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < nw ? sh[lane] : identity;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) sh[0] = v;
    }
    __syncthreads();
    T r = sh[0];
    __syncthreads();
    return r;
}

struct AddOp {
    __device__ double operator()(double a, double b) const { return a + b; }
};
struct MaxOp {
    __device__ long long operator()(long long a, long long b) const { return a > b ? a : b; }
};
struct OrOp {
    __device__ int operator()(int a, int b) const { return a | b; }
};

// The FP64 pipe of an SM takes a warp instruction every 64 cycles per scheduler whatever
// its active lanes, so a short kernel's time is its count of dependent FP64 instructions:
// signs and finiteness are tested on the bit patterns, maxima of positive values on
// integers, and sum_i log v_i is log(prod of mantissas) + (sum of exponents) ln 2 with one
// log per CTA. At d = 1024, K = 8 (device time, cold caches) this launch takes 13 us, the
// constants with a log per coordinate and the check as a launch of its own took 17 + 29.
__device__ __forceinline__ bool pos_finite(double v) {
    const int h = __double2hiint(v);
    return h < 0x7ff00000 && (h > 0 || (h == 0 && __double2loint(v) != 0));
}

// One factor of a log sum: positive finite values go into the product, anything else
// (recorded in the status word) makes the sum its log (NaN or +-inf).
__device__ __forceinline__ void log_factor(double v, double &m, int &e, double &odd, int &has_odd) {
    if (pos_finite(v)) {
        int x;
        m *= frexp(v, &x);
        e += x;
    } else {
        odd += log(v);
        has_odd = 1;
    }
}

// The CTA's log sum, valid in thread 0 (256 threads, at most 4 factors in [1/2, 1) each:
// a warp's product stays above 2^-128, then it is normalised again).
__device__ __forceinline__ double block_log_sum(double m, int e, double odd, int has_odd, double *sh, int *shi) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m *= __shfl_xor_sync(0xffffffffu, m, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (lane == 0) {
        int x;
        sh[wid] = frexp(m, &x);
        shi[wid] = e + x;
    }
    const int any_odd = __syncthreads_or(has_odd);
    double t = 0.0;
    if (wid == 0) {
        m = lane < 8 ? sh[lane] : 1.0;
        e = lane < 8 ? shi[lane] : 0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            m *= __shfl_xor_sync(0xffffffffu, m, o);
            e += __shfl_xor_sync(0xffffffffu, e, o);
        }
        constexpr double kLn2 = 0.693147180559945286, kLn2Lo = 2.3190468138462996e-17;  // ln 2 = sum of both
        t = fma((double)e, kLn2, fma((double)e, kLn2Lo, log(m)));
    }
    __syncthreads();
    if (any_odd) t += block_reduce(odd, AddOp(), sh, 0.0);
    return t;
}

constexpr int kCheckRows = 8;  // rows of L per checking CTA (a warp each)

// Blocks 0 .. K: the box (block 0) and component k = block - 1. Blocks beyond: finiteness
// of the lower triangles of all L_k, a warp per row, eight loads in flight per lane; it
// reads only the triangle (33.6 MB at d = 1024, K = 8: 5 us of HBM) and addresses by row,
// where a flat pass over the squares paid a 64-bit division per element.
__global__ void __launch_bounds__(256) k_setup(ProbView pv) {
    __shared__ double shd[32];
    __shared__ long long shl[32];
    __shared__ int shi[32];
    const int d = pv.d;
    if ((int)blockIdx.x > pv.K) {
        const int lane = threadIdx.x & 31;
        const int64_t row = (int64_t)(blockIdx.x - pv.K - 1) * kCheckRows + (threadIdx.x >> 5);
        if (row >= (int64_t)pv.K * d) return;
        const int i = (int)(row % d);
        const double *p = pv.L + row * d;
        int bad = 0;
        for (int j0 = 0; j0 <= i; j0 += 256) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = j0 + 32 * u + lane;
                v[u] = j <= i ? __ldg(p + j) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) bad |= (__double2hiint(v[u]) & 0x7ff00000) == 0x7ff00000;
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(pv.status, SB_DEV_NONFINITE);
    } else if (blockIdx.x == 0) {
        double m = 1.0, odd = 0.0, wm = 0.0;
        long long wmax = 0;  // bits of the largest positive width
        int bad = 0, e = 0, has_odd = 0;
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            const double lo = pv.lo[i], hi = pv.hi[i];
            const double w = hi - lo;
            if (!isfinite(lo) || !isfinite(hi)) bad |= SB_DEV_NONFINITE;
            if (__double_as_longlong(w) <= 0 || w != w) bad |= SB_DEV_INVALID;
            pv.c[i] = 0.5 * (lo + hi);
            pv.half[i] = 0.5 * (hi - lo);
            log_factor(w, m, e, odd, has_odd);
            const long long wb = __double_as_longlong(w);
            if (w == w && wb > wmax) wmax = wb;  // positive doubles order as their bits
        }
        const double lsum = block_log_sum(m, e, odd, has_odd, shd, shi);
        wm = __longlong_as_double(block_reduce(wmax, MaxOp(), shl, 0ll));
        bad = block_reduce(bad, OrOp(), shi, 0);
        if (threadIdx.x == 0) {
            pv.logV[0] = lsum;
            pv.wmax[0] = wm;
            if (bad) atomicOr(pv.status, bad);
        }
    } else {
        const int k = blockIdx.x - 1;
        const double *Lk = pv.L + (size_t)k * d * d;
        double m = 1.0, odd = 0.0;
        int bad = 0, e = 0, has_odd = 0;
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            const double l = Lk[(size_t)i * d + i];
            if (__double_as_longlong(l) <= 0 || l != l) bad |= SB_DEV_INVALID;
            log_factor(l, m, e, odd, has_odd);
            if (!isfinite(pv.mu[(size_t)k * d + i])) bad |= SB_DEV_NONFINITE;
        }
        const double s = block_log_sum(m, e, odd, has_odd, shd, shi);
        bad = block_reduce(bad, OrOp(), shi, 0);
        if (threadIdx.x == 0) {
            const double lw = pv.log_w[k];
            if (!isfinite(lw)) bad |= SB_DEV_NONFINITE;
            pv.a[k] = (lw - 0.5 * (double)d * SB_LOG_2PI) + s;
            if (bad) atomicOr(pv.status, bad);
        }
    }
}

void launch_setup(const ProbView &pv, cudaStream_t s) {
    note_launch();
    const int64_t rows = (int64_t)pv.K * pv.d;
    k_setup<<<(unsigned)(pv.K + 1 + (rows + kCheckRows - 1) / kCheckRows), 256, 0, s>>>(pv);
}

}  // namespace sb
