// setup.cu -- per-problem constants of the likelihood and the prior box.
//   a_k  = log w_k - (d/2) log 2pi + sum_i log L_k,ii   (normalised Gaussian, Sec. 3.2)
//   c    = (lo + hi) / 2, half = (hi - lo) / 2          (prior centre, Sec. 3.4.1)
//   logV = sum_i log(hi_i - lo_i)                        (prior volume, Sec. 3.2)
// It also validates what only the device can see: lo < hi, L_k,ii > 0, finite values.
#include "sb_internal.cuh"

namespace sb {

// The FP64 pipe of an SM takes a warp instruction every 64 cycles per scheduler whatever
// its active lanes, so a short kernel's time is its count of FP64 instructions: signs and
// finiteness are tested on the bit patterns, maxima of positive values on integers, and
// the reductions add no zeros. The constants and the check (below) are one launch: 46 us of
// device time at d = 1024, K = 8 as two, with caches cold, 13 us now.
__device__ __forceinline__ double block_sum(double v, double *sh) {  // 256 threads; valid in thread 0
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_sum(v);
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < 8 ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    return v;
}

__device__ __forceinline__ bool not_positive(double v) { return __double_as_longlong(v) <= 0 || v != v; }
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

constexpr int kCheckRows = 8;  // rows of L per checking CTA (a warp each)

// Blocks 0 .. K: the box (block 0; its constants are left out where pv.c, pv.half, pv.logV and
// pv.wmax are null, its checks are not) and component k = block - 1. Blocks beyond: finiteness
// of the lower triangles of all L_k, a warp per row, eight loads in flight per lane; it
// reads only the triangle (33.6 MB at d = 1024, K = 8: 5 us of HBM) and addresses by row,
// where a flat pass over the squares paid a 64-bit division per element.
__global__ void __launch_bounds__(256) k_setup(ProbView pv) {
    __shared__ double shd[8];
    __shared__ long long shl[8];
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
            for (int u = 0; u < 8; ++u) bad |= not_finite(v[u]) ? 1 : 0;
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(pv.status, SB_DEV_NONFINITE);
    } else if (blockIdx.x == 0) {
        double lsum = 0.0;
        long long wmax = 0;  // bits of the largest positive width (positive doubles order as their bits)
        int bad = 0;
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            const double lo = pv.lo[i], hi = pv.hi[i];
            const double w = hi - lo;
            if (not_finite(lo) || not_finite(hi)) bad |= SB_DEV_NONFINITE;
            if (not_positive(w)) bad |= SB_DEV_INVALID;
            if (pv.c) {
                pv.c[i] = 0.5 * (lo + hi);
                pv.half[i] = 0.5 * (hi - lo);
            }
            lsum += log(w);
            const long long wb = __double_as_longlong(w);
            if (w == w && wb > wmax) wmax = wb;
        }
        lsum = block_sum(lsum, shd);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long x = __shfl_xor_sync(0xffffffffu, wmax, o);
            wmax = x > wmax ? x : wmax;
        }
        if ((threadIdx.x & 31) == 0) shl[threadIdx.x >> 5] = wmax;
        const int inv = __syncthreads_or(bad & SB_DEV_INVALID), nf = __syncthreads_or(bad & SB_DEV_NONFINITE);
        if (threadIdx.x == 0) {
            for (int w = 0; w < 8; ++w) wmax = shl[w] > wmax ? shl[w] : wmax;
            if (pv.logV) {
                pv.logV[0] = lsum;
                pv.wmax[0] = __longlong_as_double(wmax);
            }
            if (inv || nf) atomicOr(pv.status, (inv ? SB_DEV_INVALID : 0) | (nf ? SB_DEV_NONFINITE : 0));
        }
    } else {
        const int k = blockIdx.x - 1;
        const double *Lk = pv.L + (size_t)k * d * d;
        double s = 0.0;
        int bad = 0;
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            const double l = Lk[(size_t)i * d + i];
            if (not_positive(l)) bad |= SB_DEV_INVALID;
            s += log(l);
            if (not_finite(pv.mu[(size_t)k * d + i])) bad |= SB_DEV_NONFINITE;
        }
        s = block_sum(s, shd);
        const int inv = __syncthreads_or(bad & SB_DEV_INVALID), nf = __syncthreads_or(bad & SB_DEV_NONFINITE);
        if (threadIdx.x == 0) {
            const double lw = pv.log_w[k];
            pv.a[k] = (lw - 0.5 * (double)d * SB_LOG_2PI) + s;
            if (inv || nf || not_finite(lw))
                atomicOr(pv.status, (inv ? SB_DEV_INVALID : 0) | (nf || not_finite(lw) ? SB_DEV_NONFINITE : 0));
        }
    }
}

void launch_setup(const ProbView &pv, cudaStream_t s) {
    note_launch();
    const int64_t rows = (int64_t)pv.K * pv.d;
    k_setup<<<(unsigned)(pv.K + 1 + (rows + kCheckRows - 1) / kCheckRows), 256, 0, s>>>(pv);
}

}  // namespace sb
