// laplace.cu -- FP64 Laplace stage: dedup, Newton polish, filters, log Z.
//
//  * coarse / final deduplication: greedy L-infinity merging in order of
//    decreasing l, ties to the lower index (Sec. 3.5.4, App. A.7); one CTA,
//    each round an argmax over the unassigned points and an early-exit
//    L-infinity test of every unassigned point against the new representative;
//  * Hessian H = -hess l = sum_k r_k P_k - sum_k r_k g_k g_k^T + gbar gbar^T,
//    with P_k = L_k L_k^T precomputed once and g_k = -L_k z_k (the analytic
//    form of the finite-difference Hessian of Sec. 3.7.2 / App. A.4.3);
//    components with r_k == 0 contribute exactly nothing and are skipped;
//  * batched blocked Cholesky H = C C^T (right-looking, 32x32 blocks:
//    diagonal factor, panel triangular solve, trailing update), which also
//    serves as the positive-definiteness (saddle) filter of Sec. 3.6.4;
//  * Newton polish x <- x + t H^{-1} grad l: t = 1 at once when the model
//    increase g^T delta / 2 <= 1e-10 (1 + |l|) (there the descent test is
//    rounding noise), otherwise t halved until l does not drop;
//  * log Z_k = l(x*) + (d/2) log 2pi - sum_i log C_ii (Sec. 3.7.1 with the
//    whitening identity of App. A.8) and log Z = LSE_k log Z_k - log V
//    (Sec. 3.7.3, App. A.10, Sec. 3.2).

#include "sb_laplace.cuh"

namespace sb {

namespace {

constexpr int NB = 32;  // Cholesky block

// ------------------------------------------------------------------ dedup
// Greedy rounds over a grid of co-resident CTAs (cooperative launch). CTA b
// owns points [b*per, (b+1)*per) and their `assigned` flags. Each round:
//   1. every CTA reduces its unassigned points to (max l, lowest index) and
//      publishes it in the round's partial slot (two slots, alternating);
//   2. one grid barrier;
//   3. every CTA reduces the partials itself (same order, same result), so
//      all know the representative without a second barrier; the owner marks
//      it, CTA 0 records it;
//   4. every CTA tests its unassigned points against the representative,
//      one warp per point: coalesced 32-coordinate slices, leaving at the
//      first four that hold a coordinate farther than tau (a warp vote).
// A slot is rewritten two rounds later, after every CTA has passed the
// barrier of the round in between, so it is never overwritten while read.
// The barrier wait is bounded: on timeout the CTA flags SB_DEV_TIMEOUT and
// leaves; every other CTA then times out at its next barrier.
constexpr int DD_THREADS = 256;
constexpr long long kBarrierSpins = 1ll << 22;

__device__ bool grid_barrier(uint32_t *bar, uint32_t n_blocks, int32_t *err) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile uint32_t *gen = bar + 1;
        const uint32_t g = *gen;
        __threadfence();
        int ok = 1;
        if (atomicAdd(bar, 1u) == n_blocks - 1) {
            bar[0] = 0;
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            long long it = 0;
            while (*gen == g) {
                if (++it > kBarrierSpins) {
                    ok = 0;
                    atomicOr(err, SB_DEV_TIMEOUT);
                    break;
                }
                if (it > 4096) __nanosleep(128);  // spin first: most waits are a few microseconds
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// (l, index) order of the greedy: larger l first, ties to the lower index; index < 0 is
// "none". l is compared as order-preserving integers (the FP64 pipe takes 64 cycles per
// warp instruction and scheduler, and a round compares along several reductions).
__device__ __forceinline__ bool dd_better(uint64_t l, int i, uint64_t bl, int bi) {
    return i >= 0 && (bi < 0 || l > bl || (l == bl && i < bi));
}
__device__ __forceinline__ uint64_t dd_key(double l) {  // -0 and +0 alike
    return ordered_bits((__double_as_longlong(l) << 1) == 0 ? 0.0 : l);
}

// |x - b| > tau, decided in FP32 on the rounded operands unless the difference lies within
// their rounding of tau, where FP64 decides (a call: inlined it would be predicated). FP64
// also decides where tau is so small that operands near it may be subnormal in FP32, whose
// rounding is not relative: from 2^-100 on it is below the margin of 2^-20 tau.
static __device__ __noinline__ bool dd_far_exact(double x, double b, double tau) { return fabs(x - b) > tau; }
__device__ __forceinline__ bool dd_far(double x, double b, float bf, double tau, float tf) {
    if (tf < 0x1p-100f) return dd_far_exact(x, b, tau);
    const float xf = f64_to_f32(x), df = fabsf(xf - bf), err = (fabsf(xf) + fabsf(bf)) * 0x1p-23f;
    if (df - err > tf * (1.0f + 0x1p-20f)) return true;
    if (df + err < tf * (1.0f - 0x1p-20f)) return false;
    return dd_far_exact(x, b, tau);
}

__global__ void __launch_bounds__(DD_THREADS) k_dedup(int n, int d, const double *X, const double *ell,
                                                      const int8_t *status, const uint8_t *keep_in, double tau_scale,
                                                      const double *wmax, int cap, int32_t *reps, int32_t *n_reps,
                                                      uint8_t *assigned, double *part_l, int32_t *part_i,
                                                      uint32_t *bar, int32_t *err) {
    extern __shared__ double s_xb[];  // [d] the round's representative, then the same in FP32
    float *s_xf = reinterpret_cast<float *>(s_xb + d);
    __shared__ uint64_t s_l[DD_THREADS / 32];
    __shared__ int s_i[DD_THREADS / 32];
    __shared__ int s_best;
    const int G = gridDim.x;
    const int per = (n + G - 1) / G;
    const int w0 = blockIdx.x * per, w1 = min(n, w0 + per);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double tau = tau_scale * wmax[0];
    const float tf = f64_to_f32(tau);
    uint64_t *part_k = reinterpret_cast<uint64_t *>(part_l);
    for (int w = w0 + threadIdx.x; w < w1; w += DD_THREADS) {
        bool el = finite_bits(ell[w]);
        if (status && status[w] == SB_WALKER_NONFINITE) el = false;
        if (keep_in && !keep_in[w]) el = false;
        assigned[w] = el ? 0 : 1;
    }
    __syncthreads();
    // the best of a warp's lanes, then of the CTA's warps (in every thread)
    auto cta_best = [&](uint64_t &bl, int &bi) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t ol = __shfl_xor_sync(0xffffffffu, bl, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (dd_better(ol, oi, bl, bi)) {
                bl = ol;
                bi = oi;
            }
        }
        if (lane == 0) {
            s_l[wid] = bl;
            s_i[wid] = bi;
        }
        __syncthreads();
        bl = 0;
        bi = -1;
        for (int q = 0; q < DD_THREADS / 32; ++q)
            if (dd_better(s_l[q], s_i[q], bl, bi)) {
                bl = s_l[q];
                bi = s_i[q];
            }
        __syncthreads();
    };
    int count = 0;
    for (int round = 0;; ++round) {
        // 1. this CTA's best unassigned point
        uint64_t bl = 0;
        int bi = -1;
        for (int w = w0 + threadIdx.x; w < w1; w += DD_THREADS) {
            if (assigned[w]) continue;
            const uint64_t l = dd_key(ell[w]);
            if (bi < 0 || l > bl) {  // strided ascending: the first seen has the lower index
                bl = l;
                bi = w;
            }
        }
        cta_best(bl, bi);
        const int slot = (round & 1) * G;
        if (threadIdx.x == 0) {
            part_k[slot + blockIdx.x] = bl;
            part_i[slot + blockIdx.x] = bi;
        }
        // 2.
        if (!grid_barrier(bar, (uint32_t)G, err)) break;
        // 3. the global best from the partials (read past L1: written by other CTAs)
        bl = 0;
        bi = -1;
        for (int q = threadIdx.x; q < G; q += DD_THREADS) {
            const uint64_t l = __ldcg(reinterpret_cast<const unsigned long long *>(part_k + slot + q));
            const int i = __ldcg(part_i + slot + q);
            if (dd_better(l, i, bl, bi)) {
                bl = l;
                bi = i;
            }
        }
        cta_best(bl, bi);
        if (threadIdx.x == 0) {
            s_best = bi;
            if (bi >= 0) {
                if (bi >= w0 && bi < w1) assigned[bi] = 1;
                if (blockIdx.x == 0 && count < cap) reps[count] = bi;
            }
        }
        __syncthreads();
        const int best = s_best;
        if (best < 0) break;
        ++count;
        if (count >= cap) break;
        // 4. L-infinity test of this CTA's unassigned points against the representative
        const double *xb = X + (size_t)best * d;
        for (int i = threadIdx.x; i < d; i += DD_THREADS) {
            s_xb[i] = xb[i];
            s_xf[i] = f64_to_f32(xb[i]);
        }
        __syncthreads();
        for (int w = w0 + wid; w < w1; w += DD_THREADS / 32) {
            if (assigned[w]) continue;
            const double *xw = X + (size_t)w * d;
            bool within = true;
            for (int i0 = 0; i0 < d; i0 += 128) {
                // four slices in flight; the walk leaves at the first that holds a far coordinate
                double v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = i0 + 32 * q + lane;
                    v[q] = i < d ? xw[i] : 0.0;
                }
                bool far = false;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = i0 + 32 * q + lane;
                    far = far || (i < d && dd_far(v[q], s_xb[i], s_xf[i], tau, tf));
                }
                if (__any_sync(0xffffffffu, far)) {
                    within = false;
                    break;
                }
            }
            if (within && lane == 0) assigned[w] = 1;
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_reps = count < cap ? count : cap;
}

__global__ void __launch_bounds__(256) k_gather_rows(int d, const double *X, const int32_t *idx, const int32_t *n_idx,
                                                     double *out, const double *ell, double *ell_out) {
    const int c = blockIdx.x;
    if (c >= *n_idx) return;
    const int w = idx[c];
    for (int i = threadIdx.x; i < d; i += blockDim.x) out[(size_t)c * d + i] = X[(size_t)w * d + i];
    if (threadIdx.x == 0 && ell_out) ell_out[c] = ell[w];
}

// ------------------------------------------------------------------ P_k = L_k L_k^T
// 32 x 32 output tiles (lower ones, mirrored on store), 256 threads with 2 x 2
// outputs each: small tiles keep the deep tiles near the diagonal short, which
// bounds the FP64 critical path when only a few components are formed.
constexpr int PT = 32;
__global__ void __launch_bounds__(256) k_precision(int d, const double *L, double *P, const int32_t *need) {
    // the longest tiles (large j0) first
    const int k = blockIdx.z, i0 = (gridDim.x - 1 - blockIdx.x) * PT, j0 = (gridDim.y - 1 - blockIdx.y) * PT;
    if (j0 > i0) return;
    if (need && !need[k]) return;
    const double *Lk = L + (size_t)k * d * d;
    __shared__ double As[16][PT + 1], Bs[16][PT + 1];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[2][2] = {};
    const int jmax = min(d, j0 + PT);  // P_ij = sum_{l <= min(i,j)} L_il L_jl
    for (int l0 = 0; l0 < jmax; l0 += 16) {
        for (int e = tid; e < 16 * PT; e += 256) {
            const int r = e >> 4, kk = e & 15, l = l0 + kk;
            const int i = i0 + r, j = j0 + r;
            As[kk][r] = (i < d && l < d && l <= i) ? Lk[(size_t)i * d + l] : 0.0;
            Bs[kk][r] = (j < d && l < d && l <= j) ? Lk[(size_t)j * d + l] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const double a0 = As[kk][ty], a1 = As[kk][ty + 16];
            const double b0 = Bs[kk][tx], b1 = Bs[kk][tx + 16];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
    double *Pk = P + (size_t)k * d * d;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int i = i0 + ty + 16 * r, j = j0 + tx + 16 * c;
            if (i < d && j < d) {
                Pk[(size_t)i * d + j] = acc[r][c];
                Pk[(size_t)j * d + i] = acc[r][c];
            }
        }
}

// Components whose P_k the Hessians are about to read: r_ck != 0 at some live
// candidate whose responsibilities are not one-hot, and P_k not formed yet (the
// Hessian skips r == 0 terms and copies L_k at one-hot candidates, so the other
// P_k are never read). Marks them formed.
__global__ void k_precision_need(int K, const double *R, const int32_t *n_c, const int32_t *onehot, int32_t *done,
                                 int32_t *need) {
    const int k = threadIdx.x;
    if (k >= K) return;
    bool any = false;
    for (int c = 0; c < *n_c; ++c) any = any || (R[(size_t)c * K + k] != 0.0 && !(onehot && onehot[c] >= 0));
    const bool nk = any && !done[k];
    need[k] = nk ? 1 : 0;
    if (nk) done[k] = 1;
}

// ------------------------------------------------------------------ per-component gradients
// GK[c][k][i] = -sum_{j<=i} L_k[i][j] z_ck[j]  (zero when r_ck == 0). Grid (candidate,
// component, row slice): the rows of one product are spread over kGradSlices CTAs.
constexpr int kGradSlices = 16;
__global__ void __launch_bounds__(256) k_comp_grads(int d, int K, const double *L, const double *Z, const double *R,
                                                    const int32_t *n_c, double *GK) {
    const int c = blockIdx.x, k = blockIdx.y;
    if (c >= *n_c) return;
    const int per = (d + kGradSlices - 1) / kGradSlices;
    const int i_lo = blockIdx.z * per, i_hi = min(d, i_lo + per);
    const double r = R[(size_t)c * K + k];
    double *g = GK + ((size_t)c * K + k) * d;
    if (r == 0.0) {
        for (int i = i_lo + threadIdx.x; i < i_hi; i += blockDim.x) g[i] = 0.0;
        return;
    }
    extern __shared__ double zs[];
    const double *z = Z + ((size_t)c * K + k) * d;
    for (int i = threadIdx.x; i < i_hi; i += blockDim.x) zs[i] = z[i];
    __syncthreads();
    const double *Lk = L + (size_t)k * d * d;
    // one warp per output row: coalesced reads of L_k rows
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = i_lo + wid; i < i_hi; i += nw) {
        double s = 0.0;
        for (int j = lane; j <= i; j += 32) s += Lk[(size_t)i * d + j] * zs[j];
        s = warp_sum(s);
        if (lane == 0) g[i] = -s;
    }
}

// onehot[c] = k when candidate c's FP64 responsibilities are exactly r_ck = 1 and 0 for
// every other component, else -1. There H = sum_k r_k (P_k - g_k g_k^T) + gbar gbar^T
// with gbar = g_k is exactly P_k = L_k L_k^T, whose Cholesky factor is L_k itself.
__global__ void k_onehot(int K, const double *R, const int32_t *n_c, int cap, int32_t *onehot) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cap) return;
    int k1 = -1;
    bool ok = c < *n_c;
    for (int k = 0; ok && k < K; ++k) {
        const double r = R[(size_t)c * K + k];
        if (r == 1.0 && k1 < 0)
            k1 = k;
        else if (r != 0.0)
            ok = false;
    }
    onehot[c] = ok ? k1 : -1;
}

// H[c][i][i2] = gbar_i gbar_i2 + sum_k r_k (P_k[i][i2] - g_ki g_ki2); at a one-hot
// candidate the lower triangle of its factor L_k instead (the blocked Cholesky skips it)
__global__ void __launch_bounds__(256) k_hessian(int d, int K, const double *P, const double *GK, const double *R,
                                                 const double *gbar, const int32_t *n_c, const int32_t *onehot,
                                                 const double *L, double *H, int32_t *info) {
    const int c = blockIdx.y;
    if (c >= *n_c) return;
    // a fresh factorisation of this candidate follows (candidates past the count keep
    // their factor and its success flag)
    if (blockIdx.x == 0 && threadIdx.x == 0) info[c] = 0;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)d * d) return;
    const int i = (int)(e / d), i2 = (int)(e % d);
    if (onehot && onehot[c] >= 0) {
        H[(size_t)c * d * d + e] = i2 <= i ? L[(size_t)onehot[c] * d * d + e] : 0.0;
        return;
    }
    const double *gb = gbar + (size_t)c * d;
    double h = gb[i] * gb[i2];
    for (int k = 0; k < K; ++k) {
        const double r = R[(size_t)c * K + k];
        if (r == 0.0) continue;
        const double *gk = GK + ((size_t)c * K + k) * d;
        h += r * (P[(size_t)k * d * d + e] - gk[i] * gk[i2]);
    }
    H[(size_t)c * d * d + e] = h;
}

// ------------------------------------------------------------------ blocked Cholesky
// Right-looking, NB x NB blocks, every live candidate of a batch at once, in one
// cooperative launch: for each block step kb, (A) the diagonal block of every
// candidate, (B) its panel blocks below, (C) the trailing blocks, with a bounded grid
// barrier after each phase (a launch per phase and step waited on the previous one's
// launch latency: 96 dependent launches per factorisation at d = 1024). Blocks written
// by one CTA are read by others after a barrier, so every read of H bypasses L1.
//
// The factorisation is a chain through the diagonal blocks, and on it every FP64
// instruction of a warp costs 64 cycles (the pipe's rate per scheduler), so the diagonal
// step is built from as few as possible.
constexpr int CF_THREADS = 256;

// 1 / p: an FP32 reciprocal of the mantissa (within 2^-22) with the negated exponent, then one
// third-order step r + r (e + e^2), e = 1 - p r (error e^3 < 2^-66 before rounding): three
// dependent FP64 instructions instead of a division's.
__device__ __forceinline__ double recip(double p) {
    const uint32_t hi = (uint32_t)__double2hiint(p), e = (hi >> 20) & 0x7ffu;
    if (e - 64u > 1918u) return 1.0 / p;  // near the ends of the range
    const float m = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | ((uint32_t)__double2loint(p) >> 29));
    const uint32_t u = __float_as_uint(__frcp_rn(m));  // in (1/2, 1]: exponent 126 or 127
    const double r = __hiloint2double((int)((hi & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + ((1919u - e) << 20))),
                                      (int)(u << 29));
    const double d = fma(-p, r, 1.0);
    return fma(r, fma(d, d, d), r);
}

// EXACT: with the last bit corrected
template <bool EXACT>
__device__ __forceinline__ double recip_as(double p) {
    const double r = recip(p);
    return EXACT ? fma(r, fma(-p, r, 1.0), r) : r;
}

// EXACT in the functions below (the adjoint, whose dL_k can be 1e-8 of the terms it is the
// difference of): reciprocals as a division rounds them, and updates a_ik -= (a_ij a_kj) /
// a_jj with the product rounded first, one instruction more per column.
//
// Diagonal block kb: A[kb][kb] -= A[kb][kb-1] A[kb][kb-1]^T (upd, the trailing update of the
// step before), then its factor. Threads 0..127 hold the block in registers: lane = row i,
// warp q the columns q, q + 4, ... Step j: the owner warp of column j publishes it unscaled
// and as the multipliers a_ij / a_jj, one barrier of the four warps, and every warp updates
// its later columns, a_ik -= (a_ij / a_jj) a_kj. Columns are scaled by 1 / sqrt(a_jj) at the
// end, all square roots at once. A pivot <= 0 (not positive definite) sets the candidate's
// info to 1 + kb (see chol_live).
template <bool EXACT>
__device__ void diag_block(int d, int kb, bool upd, double *A, int32_t *info_c) {
    __shared__ double a[NB][NB + 1];
    __shared__ double pa[NB][NB + 1];
    __shared__ double col[2][NB], mul[2][NB], piv[NB];
    __shared__ int s_bad;
    const int o = kb * NB, tid = threadIdx.x;
    for (int e = tid; e < NB * NB; e += CF_THREADS) {
        const int i = e / NB, j = e % NB;
        a[i][j] = (o + i < d && o + j < d) ? __ldcg(&A[(size_t)(o + i) * d + o + j])
                                           : (i == j ? 1.0 : 0.0);  // identity padding
        if (upd) pa[i][j] = o + i < d ? __ldcg(&A[(size_t)(o + i) * d + o - NB + j]) : 0.0;
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    if (upd) {
        // the 528 entries of the lower triangle over the threads
        for (int e = tid; e < NB * (NB + 1) / 2; e += CF_THREADS) {
            int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
            while (i * (i + 1) / 2 > e) --i;
            while ((i + 1) * (i + 2) / 2 <= e) ++i;
            const int j = e - i * (i + 1) / 2;
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < NB; ++q) s = fma(pa[i][q], pa[j][q], s);
            a[i][j] -= s;
        }
        __syncthreads();
    }
    if (tid < 128) {
        const int i = tid & 31, q = tid >> 5;
        double x[NB / 4];
#pragma unroll
        for (int t = 0; t < NB / 4; ++t) x[t] = i >= 4 * t + q ? a[i][4 * t + q] : 0.0;
#pragma unroll
        for (int t0 = 0; t0 < NB / 4; ++t0) {
            for (int qo = 0; qo < 4; ++qo) {
                const int j = 4 * t0 + qo, sl = j & 1;
                if (q == qo) {
                    const double p = __shfl_sync(0xffffffffu, x[t0], j);
                    if (i == 0) {
                        piv[j] = p;
                        if (__double_as_longlong(p) <= 0 || p != p) s_bad = 1;
                    }
                    col[sl][i] = x[t0];
                    mul[sl][i] = EXACT ? recip_as<true>(p) : x[t0] * recip(p);
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const double m = mul[sl][i], ci = EXACT ? col[sl][i] : 0.0;
                // the column the next step needs comes first
#pragma unroll
                for (int t = 0; t < NB / 4; ++t)
                    if (t > t0 || (t == t0 && q > qo))
                        x[t] = EXACT ? fma(-(ci * col[sl][4 * t + q]), m, x[t]) : fma(-m, col[sl][4 * t + q], x[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < NB / 4; ++t)
            if (i >= 4 * t + q) a[i][4 * t + q] = x[t];
    }
    __syncthreads();
    if (s_bad) {
        if (tid == 0) *info_c = 1 + kb;
        __syncthreads();
        return;
    }
    if (tid < NB) col[0][tid] = rsqrt(piv[tid]);
    __syncthreads();
    for (int e = tid; e < NB * NB; e += CF_THREADS) {
        const int i = e / NB, j = e % NB;
        if (o + i < d && o + j < d && j <= i) A[(size_t)(o + i) * d + o + j] = a[i][j] * col[0][j];
    }
    __syncthreads();  // the shared blocks are free for the next item
}

// Panel: rows r0 .. r0 + 15 of column block kb, A <- A L_kk^{-T}. Threads 0..127: thread
// (row, part) holds the row's columns part, part + 8, ...; per column j the owner scales by
// 1 / L_jj (reciprocals taken once, in parallel) and publishes it, then every thread
// updates its later columns, two on average (16 rows, not 32, because a warp instruction
// takes its 64 cycles whatever the lanes: eight parts a row halve the chain).
constexpr int TRSM_THREADS = 128, TRSM_ROWS = 16;
template <bool EXACT>
__device__ void trsm_block(int d, int kb, int r0, double *A) {
    __shared__ double l[NB][NB + 1];
    __shared__ double xs[TRSM_ROWS][NB + 1];
    __shared__ double inv[NB];
    const int o = kb * NB;
    for (int e = threadIdx.x; e < NB * NB; e += CF_THREADS) {
        const int i = e / NB, j = e % NB;
        l[i][j] = (o + i < d && o + j < d) ? __ldcg(&A[(size_t)(o + i) * d + o + j]) : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    if (threadIdx.x < NB) inv[threadIdx.x] = recip_as<EXACT>(l[threadIdx.x][threadIdx.x]);
    const int r = threadIdx.x & (TRSM_ROWS - 1), part = threadIdx.x / TRSM_ROWS;  // parts 0..7
    const int row = r0 + r;
    double x[NB / 8];
    if (threadIdx.x < TRSM_THREADS)
#pragma unroll
        for (int q = 0; q < NB / 8; ++q) {
            const int j = part + 8 * q;
            x[q] = (row < d && o + j < d) ? __ldcg(&A[(size_t)row * d + o + j]) : 0.0;
        }
    __syncthreads();
    if (threadIdx.x < TRSM_THREADS) {
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            if (part == (j & 7)) {
                x[j >> 3] *= inv[j];
                xs[r][j] = x[j >> 3];
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            const double xj = xs[r][j];
#pragma unroll
            for (int q = 0; q < NB / 8; ++q)
                if (part + 8 * q > j) x[q] = fma(-xj, l[part + 8 * q][j], x[q]);
        }
#pragma unroll
        for (int q = 0; q < NB / 8; ++q) {
            const int j = part + 8 * q;
            if (row < d && o + j < d) A[(size_t)row * d + o + j] = x[q];
        }
    }
    __syncthreads();  // the shared blocks are free for the next item
}

// Trailing update A[ib][jb] -= A[ib][kb] A[jb][kb]^T for kb < jb <= ib.
__device__ void syrk_block(int d, int kb, int ib, int jb, double *A) {
    __shared__ double pa[NB][NB + 1], pb[NB][NB + 1];
    const int o = kb * NB;
    for (int e = threadIdx.x; e < NB * NB; e += CF_THREADS) {
        const int r = e / NB, q = e % NB;
        const int ia = ib * NB + r, ja = jb * NB + r, col = o + q;
        pa[r][q] = (ia < d && col < d) ? __ldcg(&A[(size_t)ia * d + col]) : 0.0;
        pb[r][q] = (ja < d && col < d) ? __ldcg(&A[(size_t)ja * d + col]) : 0.0;
    }
    __syncthreads();
    const int tx = threadIdx.x % NB, ty = threadIdx.x / NB;  // ty 0..7
#pragma unroll
    for (int rr = 0; rr < NB / 8; ++rr) {
        const int r = ty + 8 * rr;
        const int i = ib * NB + r, j = jb * NB + tx;
        if (i >= d || j >= d || j > i) continue;
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < NB; ++q) s += pa[r][q] * pb[tx][q];
        A[(size_t)i * d + j] = __ldcg(&A[(size_t)i * d + j]) - s;
    }
    __syncthreads();  // the shared blocks are free for the next item
}

// Whether candidate c still takes part in block step kb: not one-hot (a one-hot candidate's
// factor is L_k, copied in place by k_hessian), and no diagonal block up to kb failed. info[c]
// is 0, or 1 + the block that failed. Block kb + 1 is factored beside this step's trailing
// updates, so a reader may see info[c] = 0 or kb + 2 there, in one warp the one and in the
// next the other: both mean "takes part" (its update of the failed candidate is not used),
// so that every thread of a CTA takes the same branch around the block barriers.
__device__ __forceinline__ bool chol_live(int c, int kb, const int32_t *onehot, const int32_t *info) {
    const int32_t failed = *reinterpret_cast<const volatile int32_t *>(&info[c]);
    return !(onehot && onehot[c] >= 0) && (failed == 0 || failed > kb + 1);
}

template <bool EXACT>
__global__ void __launch_bounds__(CF_THREADS) k_chol_coop(int d, double *H, const int32_t *n_c,
                                                         const int32_t *onehot, int32_t *info, uint32_t *bar,
                                                         int32_t *err) {
    // the candidate count is the same value in every CTA, so all CTAs reach every
    // barrier; none is needed when every candidate is one-hot
    const int nc = *n_c;
    if (onehot) {
        bool any = false;
        for (int c = 0; c < nc && !any; ++c) any = onehot[c] < 0;
        if (!any) return;
    }
    const int nblk = (d + NB - 1) / NB;
    for (int c = blockIdx.x; c < nc; c += gridDim.x)
        if (chol_live(c, 0, onehot, info)) diag_block<EXACT>(d, 0, false, H + (size_t)c * d * d, info + c);
    if (!grid_barrier(bar, gridDim.x, err)) return;
    for (int kb = 0; kb + 1 < nblk; ++kb) {
        const int rest = nblk - kb - 1;
        for (int it = blockIdx.x; it < nc * 2 * rest; it += gridDim.x) {
            const int c = it / (2 * rest);
            if (chol_live(c, kb, onehot, info))
                trsm_block<EXACT>(d, kb, (kb + 1) * NB + (it % (2 * rest)) * TRSM_ROWS, H + (size_t)c * d * d);
        }
        if (!grid_barrier(bar, gridDim.x, err)) return;
        // the next diagonal block of every candidate is updated and factored at once, by
        // the first CTAs; the other trailing blocks (ii >= jj, ii > 0) go to the rest
        for (int c = blockIdx.x; c < nc; c += gridDim.x)
            if (chol_live(c, kb, onehot, info)) diag_block<EXACT>(d, kb + 1, true, H + (size_t)c * d * d, info + c);
        const int tri = rest * (rest + 1) / 2 - 1;
        const int skip = (int)gridDim.x > 2 * nc ? nc : 0;  // CTAs that only factor in this phase
        const int b = (int)blockIdx.x - skip, nb = (int)gridDim.x - skip;
        for (int it = b; b >= 0 && it < nc * tri; it += nb) {
            const int c = it / tri, e = it - c * tri + 1;
            if (!chol_live(c, kb, onehot, info)) continue;
            int ii = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
            while (ii * (ii + 1) / 2 > e) --ii;
            while ((ii + 1) * (ii + 2) / 2 <= e) ++ii;
            const int jj = e - ii * (ii + 1) / 2;
            syrk_block(d, kb, kb + 1 + ii, kb + 1 + jj, H + (size_t)c * d * d);
        }
        if (!grid_barrier(bar, gridDim.x, err)) return;
    }
}

// The inverses of the factors' 32 x 32 diagonal blocks, for the solves: the strictly lower
// part of a block's inverse, transposed, goes into the strictly upper part of the block,
// which nothing else uses. A CTA per (block, candidate), a warp per four columns, lanes over
// rows.
__global__ void __launch_bounds__(256) k_chol_dinv(int d, double *H, const int32_t *n_c, const int32_t *info) {
    __shared__ double Cs[NB][NB + 1];
    __shared__ double inv[NB];
    const int c = blockIdx.y, r0 = blockIdx.x * NB;
    if (c >= *n_c || info[c]) return;
    double *C = H + (size_t)c * d * d;
    for (int e = threadIdx.x; e < NB * NB; e += 256) {
        const int i = r0 + e / NB, j = r0 + e % NB;
        Cs[e / NB][e % NB] = i < d && j <= i ? C[(size_t)i * d + j] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    if (threadIdx.x < NB) inv[threadIdx.x] = recip(Cs[threadIdx.x][threadIdx.x]);
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = lane == wid * 4 + q ? 1.0 : 0.0;
    for (int i = wid * 4; i < NB; ++i) {  // rows above the warp's columns stay zero
        const double v = lane > i ? Cs[lane][i] : 0.0, iv = inv[i];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double xi = __shfl_sync(0xffffffffu, b[q], i) * iv;
            b[q] = lane == i ? xi : fma(-v, xi, b[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = r0 + wid * 4 + q, i = r0 + lane;
        if (i < d && i > j) C[(size_t)j * d + i] = b[q];
    }
}

// Solve (C C^T) delta = g for each candidate still polishing and the model
// increase g^T delta / 2 (cooperative launch, one bounded grid barrier per 32-row
// block and direction). The grid is split into slots of Gc CTAs (Gc from the
// candidate count on the device, 1 to 16); slot j serves candidates j, j + slots,
// ... in turn, and CTA q of a slot owns the row blocks J with J % Gc == q of each.
// Forward (C y = g): in step I the owner of block I (already updated by every
// earlier step, by itself) multiplies it by the inverse of the diagonal block (k_chol_dinv) and
// publishes y_I; after the barrier every owner subtracts C_JI y_I from its blocks J > I. The
// owner of block I + 1 has then finished block I + 1's last update before it solves it in step
// I + 1, so one barrier per step suffices. Backward (C^T delta = y) mirrors it
// with (C^T)_JI = (C_IJ)^T for J < I. The right-hand side lives in delta[c]
// (global, read past L1 after barriers). Both products are 32 x 32 by a vector: lane = row,
// warp w the columns 4 w .. 4 w + 3, the eight partial sums added in order; the matrix is
// read into shared memory before the barrier it does not depend on. (A substitution per
// block was 32 dependent steps, 375 us per solve of four candidates at d = 512; 253 now.)
constexpr int CS_THREADS = 256;
__global__ void __launch_bounds__(CS_THREADS) k_chol_solve_coop(int d, const double *H, const double *g,
                                                                const int32_t *n_c, const int32_t *info,
                                                                const uint8_t *active, double *delta, double *pred,
                                                                uint32_t *bar, int32_t *err) {
    __shared__ double M[32][33];
    __shared__ double xs[32];
    __shared__ double part[8];
    __shared__ double red[8][33];
    // the candidate count is the same value in every CTA, so either all CTAs leave
    // here or all reach every grid barrier
    const int ncand = *n_c;
    if (ncand <= 0) return;
    int Gc = (int)gridDim.x / ncand;
    Gc = Gc < 1 ? 1 : (Gc > 16 ? 16 : Gc);
    const int slots = (int)gridDim.x / Gc;
    const int slot = blockIdx.x / Gc, q = blockIdx.x % Gc;
    const int c0 = slot < slots ? slot : ncand;  // CTAs past the last whole slot serve nothing
    const int nb = (d + 31) / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto live = [&](int c) { return !info[c] && active[c]; };
    for (int c = c0; c < ncand; c += slots) {
        if (!live(c)) continue;
        double *y = delta + (size_t)c * d;
        for (int J = q; J < nb; J += Gc)
            for (int i = J * 32 + (int)threadIdx.x; i < min(d, J * 32 + 32); i += CS_THREADS)
                y[i] = g[(size_t)c * d + i];
    }
    __syncthreads();
    // M = the inverse of diagonal block I (upper: its transpose): the strictly lower part from
    // above the diagonal of the block, the diagonal as reciprocals
    auto load_dinv = [&](const double *C, int I, bool upper) {
        const int r0 = I * 32;
        __syncthreads();
        for (int e = threadIdx.x; e < 32 * 32; e += CS_THREADS) {
            const int i = e / 32, j = e % 32;
            const bool in = r0 + i < d && r0 + j < d;
            if (j > i) {
                const double v = in ? C[(size_t)(r0 + i) * d + r0 + j] : 0.0;  // (block^-1)[j][i]
                M[upper ? i : j][upper ? j : i] = v;
                M[upper ? j : i][upper ? i : j] = 0.0;
            } else if (i == j) {
                M[i][i] = in ? recip(C[(size_t)(r0 + i) * d + r0 + i]) : 1.0;
            }
        }
    };
    // M = block C_JI (rows of J), or for the backward pass (C_IJ)^T
    auto load_block = [&](const double *C, int J, int I, bool upper) {
        const int j0 = J * 32, i0 = I * 32;
        __syncthreads();
        for (int e = threadIdx.x; e < 32 * 32; e += CS_THREADS) {
            const int i = e / 32, j = e % 32;
            if (!upper)
                M[i][j] = j0 + i < d && i0 + j < d ? C[(size_t)(j0 + i) * d + i0 + j] : 0.0;
            else
                M[j][i] = i0 + i < d && j0 + j < d ? C[(size_t)(i0 + i) * d + j0 + j] : 0.0;
        }
    };
    // the product M x (x: 32 entries of y from x0, zero past d) in warp 0's lanes
    auto apply = [&](const double *y, int x0) {
        if (threadIdx.x < 32) xs[threadIdx.x] = x0 + (int)threadIdx.x < d ? __ldcg(y + x0 + threadIdx.x) : 0.0;
        __syncthreads();
        double s = M[lane][4 * wid] * xs[4 * wid];
#pragma unroll
        for (int t = 1; t < 4; ++t) s = fma(M[lane][4 * wid + t], xs[4 * wid + t], s);
        red[wid][lane] = s;
        __syncthreads();
        if (wid != 0) return 0.0;
        const double s01 = red[0][lane] + red[1][lane], s23 = red[2][lane] + red[3][lane];
        const double s45 = red[4][lane] + red[5][lane], s67 = red[6][lane] + red[7][lane];
        return (s01 + s23) + (s45 + s67);
    };
    for (int pass = 0; pass < 2; ++pass) {
        const bool upper = pass == 1;
        for (int st = 0; st < nb; ++st) {
            const int I = upper ? nb - 1 - st : st, r0 = I * 32;
            if (I % Gc == q)
                for (int c = c0; c < ncand; c += slots) {
                    if (!live(c)) continue;
                    double *y = delta + (size_t)c * d;
                    load_dinv(H + (size_t)c * d * d, I, upper);
                    __syncthreads();
                    const double v = apply(y, r0);
                    if (wid == 0 && r0 + lane < d) y[r0 + lane] = v;
                    __threadfence();
                }
            // the first block this CTA updates after the barrier
            const int J0 = upper ? q : I + 1 + ((q - (I + 1)) % Gc + Gc) % Gc;
            const bool any = c0 < ncand && (upper ? J0 < I : J0 < nb);
            if (any && live(c0)) load_block(H + (size_t)c0 * d * d, J0, I, upper);
            if (!grid_barrier(bar, gridDim.x, err)) return;
            for (int c = c0; any && c < ncand; c += slots) {
                if (!live(c)) continue;
                const double *C = H + (size_t)c * d * d;
                double *y = delta + (size_t)c * d;
                for (int J = J0; upper ? J < I : J < nb; J += Gc) {
                    if (c != c0 || J != J0) load_block(C, J, I, upper);
                    __syncthreads();
                    const double v = apply(y, r0);
                    if (wid == 0 && J * 32 + lane < d) y[J * 32 + lane] -= v;
                }
            }
            __syncthreads();
        }
    }
    if (!grid_barrier(bar, gridDim.x, err)) return;
    // model increase of l along the Newton step: g^T delta / 2 (first CTA of the slot)
    if (q != 0) return;
    for (int c = c0; c < ncand; c += slots) {
        if (!live(c)) continue;
        const double *y = delta + (size_t)c * d;
        double gd = 0.0;
        for (int i = threadIdx.x; i < d; i += CS_THREADS) gd += g[(size_t)c * d + i] * __ldcg(y + i);
        gd = warp_sum(gd);
        if (lane == 0) part[wid] = gd;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < CS_THREADS / 32; ++w) t += part[w];
            pred[c] = 0.5 * t;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ Newton line search
// mode 0: start (t = 1, trial = x + delta, searching = active & Cholesky ok).
//   A candidate whose Newton step is already below kNewtonXtol (1 + |x|_inf) in
//   max norm has converged: it stays where it is (its H factor is the one at
//   that point) and stops polishing; the others are counted in *n_live.
// mode 1: decide on the evaluated trial (accept if l_t >= l, else halve)
constexpr double kNewtonXtol = 1e-11;
__global__ void __launch_bounds__(256) k_newton_ls(int d, int mode, const int32_t *n_c, const int32_t *info,
                                                   uint8_t *active, uint8_t *searching, int32_t *halvings, double *t,
                                                   double *XC, double *LC, const double *delta, double *XN,
                                                   const double *LN, const double *pred, int32_t *n_live) {
    const int c = blockIdx.x;
    if (c >= *n_c) return;
    __shared__ int s_act;
    __shared__ double s_mx[2][8];
    bool small = false;
    if (mode == 0) {  // max |delta| and max |x| of the candidate
        double md = 0.0, mx = 0.0;
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            md = fmax(md, fabs(delta[(size_t)c * d + i]));
            mx = fmax(mx, fabs(XC[(size_t)c * d + i]));
        }
        md = warp_max(md);
        mx = warp_max(mx);
        if ((threadIdx.x & 31) == 0) {
            s_mx[0][threadIdx.x >> 5] = md;
            s_mx[1][threadIdx.x >> 5] = mx;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < 8; ++q) {
                md = fmax(md, s_mx[0][q]);
                mx = fmax(mx, s_mx[1][q]);
            }
            small = md <= kNewtonXtol * (1.0 + mx);
        }
    }
    if (threadIdx.x == 0) {
        int act = 0;
        if (mode == 0) {
            const int s = active[c] && !info[c] && !small;
            if (!s) active[c] = 0;
            halvings[c] = 0;
            t[c] = 1.0;
            if (s) atomicAdd(n_live, 1);
            if (s && pred[c] <= 1e-10 * (1.0 + fabs(LC[c]))) {
                // quadratic-convergence regime: the descent test is rounding noise, take t = 1
                searching[c] = 0;
                act = 3;
            } else {
                searching[c] = (uint8_t)s;
                act = s ? 2 : 0;  // 2: write the trial
            }
        } else if (searching[c]) {
            if (LN[c] >= LC[c]) {
                searching[c] = 0;
                LC[c] = LN[c];
                act = 1;  // 1: accept
            } else if (halvings[c] + 1 >= 30) {
                searching[c] = 0;
                active[c] = 0;  // no acceptable step: stop polishing this candidate
            } else {
                ++halvings[c];
                t[c] *= 0.5;
                act = 2;
            }
        }
        s_act = act;
    }
    __syncthreads();
    const int act = s_act;
    if (act == 1) {
        for (int i = threadIdx.x; i < d; i += blockDim.x) XC[(size_t)c * d + i] = XN[(size_t)c * d + i];
    } else if (act == 3) {
        for (int i = threadIdx.x; i < d; i += blockDim.x)
            XC[(size_t)c * d + i] = add_rn(XC[(size_t)c * d + i], mul_rn(1.0, delta[(size_t)c * d + i]));
    } else if (act == 2) {
        const double tc = t[c];
        for (int i = threadIdx.x; i < d; i += blockDim.x)
            XN[(size_t)c * d + i] = add_rn(XC[(size_t)c * d + i], mul_rn(tc, delta[(size_t)c * d + i]));
    }
}

// Halvings 1..kHalvings-1 evaluated as one batch: the first acceptable
// halving is the one a sequential search would stop at.
__global__ void __launch_bounds__(256) k_ls_batch_setup(int d, const int32_t *n_c, const uint8_t *searching,
                                                        const double *XC, const double *delta, double *XN2,
                                                        int32_t *rows2, int32_t *n_rows2) {
    const int c = blockIdx.x;
    if (c >= *n_c || !searching[c]) return;
    __shared__ int base;
    if (threadIdx.x == 0) base = atomicAdd(n_rows2, kHalvings - 1);
    __syncthreads();
    double t = 1.0;
    for (int h = 1; h < kHalvings; ++h) {
        t *= 0.5;
        const size_t row = (size_t)c * (kHalvings - 1) + (h - 1);
        for (int i = threadIdx.x; i < d; i += blockDim.x)
            XN2[row * d + i] = add_rn(XC[(size_t)c * d + i], mul_rn(t, delta[(size_t)c * d + i]));
        if (threadIdx.x == 0) rows2[base + h - 1] = (int32_t)row;
    }
}

__global__ void __launch_bounds__(256) k_ls_batch_decide(int d, const int32_t *n_c, uint8_t *searching,
                                                         uint8_t *active, double *XC, double *LC, const double *XN2,
                                                         const double *LN2) {
    const int c = blockIdx.x;
    if (c >= *n_c || !searching[c]) return;
    __shared__ int hsel;
    if (threadIdx.x == 0) {
        int hs = -1;
        for (int h = 1; h < kHalvings; ++h)
            if (LN2[(size_t)c * (kHalvings - 1) + h - 1] >= LC[c]) {
                hs = h;
                break;
            }
        hsel = hs;
    }
    __syncthreads();
    const int h = hsel;
    if (h < 0) {
        if (threadIdx.x == 0) {
            searching[c] = 0;
            active[c] = 0;
        }
        return;
    }
    const size_t row = (size_t)c * (kHalvings - 1) + (h - 1);
    for (int i = threadIdx.x; i < d; i += blockDim.x) XC[(size_t)c * d + i] = XN2[row * d + i];
    __syncthreads();
    if (threadIdx.x == 0) {
        LC[c] = LN2[row];
        searching[c] = 0;
    }
}

// ------------------------------------------------------------------ filters and log Z_k
__global__ void __launch_bounds__(256) k_cand_stats(int d, const double *XC, const double *LC, const double *GC,
                                                    const double *H, const int32_t *info, const double *lo,
                                                    const double *hi, double eps_grad, const int32_t *n_c,
                                                    uint8_t *keep, double *logZk) {
    const int c = blockIdx.x;
    if (c >= *n_c) return;
    __shared__ double s_gm[32], s_ld[32];
    __shared__ int s_in[32];
    double gm = 0.0, ld = 0.0;
    int inside = 1;
    const bool ok = info[c] == 0;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        gm = fmax(gm, fabs(GC[(size_t)c * d + i]));
        const double x = XC[(size_t)c * d + i];
        if (!(x >= lo[i] && x <= hi[i])) inside = 0;
        if (ok) ld += log(H[(size_t)c * d * d + (size_t)i * d + i]);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    gm = warp_max(gm);
    ld = warp_sum(ld);
    inside = __all_sync(0xffffffffu, inside);
    if (lane == 0) {
        s_gm[wid] = gm;
        s_ld[wid] = ld;
        s_in[wid] = inside;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double g = 0.0, l = 0.0;
        int in = 1;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
            g = fmax(g, s_gm[q]);
            l += s_ld[q];
            in &= s_in[q];
        }
        const double ell = LC[c];
        keep[c] = (uint8_t)(ok && isfinite(ell) && g <= eps_grad * (1.0 + fabs(ell)) && in);
        logZk[c] = ok ? (ell + 0.5 * (double)d * SB_LOG_2PI) - l : NAN;
    }
}

// Final dedup of the kept candidates, outputs in order of decreasing l, LSE - log V.
__global__ void __launch_bounds__(1024) k_laplace_final(int d, const double *XC, const double *LC,
                                                        const double *logZk_c, const int32_t *n_c,
                                                        const int32_t *reps, const int32_t *n_reps, const double *logV,
                                                        int cap, double *modes, double *logZk, double *ell_modes,
                                                        int32_t *n_modes, double *logZ, int32_t *dev_status) {
    const int nm = *n_reps;
    for (int t = 0; t < nm && t < cap; ++t) {
        const int c = reps[t];
        for (int i = threadIdx.x; i < d; i += blockDim.x) modes[(size_t)t * d + i] = XC[(size_t)c * d + i];
        if (threadIdx.x == 0) {
            logZk[t] = logZk_c[c];
            if (ell_modes) ell_modes[t] = LC[c];
        }
    }
    if (threadIdx.x == 0) {
        double zmax = -INFINITY;
        for (int t = 0; t < nm; ++t) zmax = fmax(zmax, logZk_c[reps[t]]);
        double lz = -INFINITY;
        if (nm > 0) {
            double s = 0.0;
            for (int t = 0; t < nm; ++t) s += exp(logZk_c[reps[t]] - zmax);
            lz = zmax + log(s) - logV[0];
        } else {
            atomicOr(dev_status, SB_DEV_NO_MODES);
        }
        *logZ = lz;
        *n_modes = nm;
    }
}

}  // namespace

void launch_dedup(int n, int d, const double *X, const double *ell, const int8_t *status, const uint8_t *keep,
                  double tau_scale, const double *wmax, int cap, int32_t *reps, int32_t *n_reps, uint8_t *assigned,
                  const DedupScratch &sc, cudaStream_t s) {
    // one CTA per 32 points up to one per SM (kept small so that concurrent
    // solves on other streams can still be co-resident)
    static const int sms = [] {  // thread-safe one-time query (batched solves use several host threads)
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 1;
    }();
    int G = (n + 31) / 32;
    if (G > sms) G = sms;
    if (G > kDedupMaxGrid) G = kDedupMaxGrid;
    if (G < 1) G = 1;
    cudaMemsetAsync(sc.bar, 0, 2 * sizeof(uint32_t), s);
    void *args[] = {&n, &d, &X, &ell, &status, &keep, &tau_scale, &wmax, &cap, &reps, &n_reps, &assigned,
                    const_cast<double **>(&sc.part_l), const_cast<int32_t **>(&sc.part_i),
                    const_cast<uint32_t **>(&sc.bar), const_cast<int32_t **>(&sc.err)};
    note_launch();
    cudaLaunchCooperativeKernel((const void *)k_dedup, dim3(G), dim3(DD_THREADS), args,
                                (sizeof(double) + sizeof(float)) * d, s);
}

void launch_gather_rows(int d, int cap, const double *X, const int32_t *idx, const int32_t *n_idx, double *out,
                        const double *ell, double *ell_out, cudaStream_t s) {
    note_launch();
    k_gather_rows<<<cap, 256, 0, s>>>(d, X, idx, n_idx, out, ell, ell_out);
}

// Unused shared memory that holds an SM to three CTAs of k_precision, so that its tiles, up to
// d / 32 times different in length, are dealt out as SMs come free (four P_k at d = 512: 371 us
// with every tile resident at once, 274 so).
static int precision_pad() {
    constexpr int kPad = 60 * 1024;
    return allow_smem(k_precision, kPad) == cudaSuccess ? kPad : 0;
}

void launch_onehot(int K, const double *R, const int32_t *n_c, int cap, int32_t *onehot, cudaStream_t s) {
    note_launch();
    k_onehot<<<(cap + 127) / 128, 128, 0, s>>>(K, R, n_c, cap, onehot);
}

void launch_precision_needed(int d, int K, const double *L, const double *R, const int32_t *n_c, int32_t *done,
                             int32_t *need, double *P, cudaStream_t s, const int32_t *onehot) {
    note_launch();
    k_precision_need<<<1, kMaxK, 0, s>>>(K, R, n_c, onehot, done, need);
    dim3 g((d + PT - 1) / PT, (d + PT - 1) / PT, K);
    note_launch();
    k_precision<<<g, 256, precision_pad(), s>>>(d, L, P, need);
}

int laplace_sms();

void launch_hessian_chol(int d, int K, int cap, const double *L, const double *P, const double *Z, const double *R,
                         const double *gbar, const int32_t *n_c, double *GK, double *H, int32_t *info,
                         uint32_t *bar, int32_t *err, cudaStream_t s, const int32_t *onehot, bool exact) {
    note_launch();
    k_comp_grads<<<dim3(cap, K, kGradSlices), 256, sizeof(double) * d, s>>>(d, K, L, Z, R, n_c, GK);
    const int64_t dd = (int64_t)d * d;
    note_launch();
    k_hessian<<<dim3((unsigned)((dd + 255) / 256), cap), 256, 0, s>>>(d, K, P, GK, R, gbar, n_c, onehot, L, H,
                                                                        info);
    auto factor = [&](cudaStream_t fs) {
        ProfScope prof(PROF_CHOLESKY, fs);
        // one CTA per SM (a cooperative grid must be co-resident), no more than the
        // largest phase's items
        const int nblk = (d + NB - 1) / NB;
        const long long items = (long long)cap * (nblk - 1) * nblk / 2;
        int G = laplace_sms();
        if (items < G) G = (int)(items > 0 ? items : 1);
        cudaMemsetAsync(bar, 0, 2 * sizeof(uint32_t), fs);
        void *args[] = {&d, &H, &n_c, &onehot, &info, &bar, &err};
        note_launch();
        cudaLaunchCooperativeKernel((const void *)(exact ? k_chol_coop<true> : k_chol_coop<false>), dim3(G), dim3(CF_THREADS), args, 0, fs);
    };
    // (the kernel leaves at once when every live candidate is one-hot)
    factor(s);
}

int laplace_sms() {
    static const int n = [] {  // thread-safe one-time query
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return n;
}

void launch_chol_solve_coop(int d, int cap, double *H, const double *g, const int32_t *n_c, const int32_t *info,
                            const uint8_t *active, double *delta, double *pred, uint32_t *bar, int32_t *err,
                            cudaStream_t s) {
    // one CTA per SM at most (a cooperative grid must be co-resident), up to 16 per
    // candidate of the cap; the kernel divides them among the live candidates
    int G = laplace_sms();
    if (G > 16 * cap) G = 16 * cap;
    note_launch();
    k_chol_dinv<<<dim3((d + NB - 1) / NB, cap), 256, 0, s>>>(d, H, n_c, info);
    cudaMemsetAsync(bar, 0, 2 * sizeof(uint32_t), s);
    void *args[] = {&d, &H, &g, &n_c, &info, &active, &delta, &pred, &bar, &err};
    note_launch();
    cudaLaunchCooperativeKernel((const void *)k_chol_solve_coop, dim3(G), dim3(CS_THREADS), args, 0, s);
}

__global__ void k_set_eff(int32_t *n_eff, const int32_t *n_reps, const int32_t *n_live) {
    if (threadIdx.x == 0) *n_eff = (!n_live || *n_live > 0) ? *n_reps : 0;
}

void launch_set_eff(int32_t *n_eff, const int32_t *n_reps, const int32_t *n_live, cudaStream_t s) {
    note_launch();
    k_set_eff<<<1, 32, 0, s>>>(n_eff, n_reps, n_live);
}

void launch_newton_ls(int d, int cap, int mode, const int32_t *n_c, const int32_t *info, uint8_t *active,
                      uint8_t *searching, int32_t *halvings, double *t, double *XC, double *LC, const double *delta,
                      double *XN, const double *LN, const double *pred, int32_t *n_live, cudaStream_t s) {
    note_launch();
    k_newton_ls<<<cap, 256, 0, s>>>(d, mode, n_c, info, active, searching, halvings, t, XC, LC, delta, XN, LN,
                                    pred, n_live);
}

void launch_ls_batch_setup(int d, int cap, const int32_t *n_c, const uint8_t *searching, const double *XC,
                           const double *delta, double *XN2, int32_t *rows2, int32_t *n_rows2, cudaStream_t s) {
    cudaMemsetAsync(n_rows2, 0, sizeof(int32_t), s);
    note_launch();
    k_ls_batch_setup<<<cap, 256, 0, s>>>(d, n_c, searching, XC, delta, XN2, rows2, n_rows2);
}

void launch_ls_batch_decide(int d, int cap, const int32_t *n_c, uint8_t *searching, uint8_t *active, double *XC,
                            double *LC, const double *XN2, const double *LN2, cudaStream_t s) {
    note_launch();
    k_ls_batch_decide<<<cap, 256, 0, s>>>(d, n_c, searching, active, XC, LC, XN2, LN2);
}

void launch_cand_stats(int d, int cap, const double *XC, const double *LC, const double *GC, const double *H,
                       const int32_t *info, const double *lo, const double *hi, double eps_grad, const int32_t *n_c,
                       uint8_t *keep, double *logZk, cudaStream_t s) {
    note_launch();
    k_cand_stats<<<cap, 256, 0, s>>>(d, XC, LC, GC, H, info, lo, hi, eps_grad, n_c, keep, logZk);
}

void launch_laplace_final(int d, const double *XC, const double *LC, const double *logZk_c, const int32_t *n_c,
                          const int32_t *reps, const int32_t *n_reps, const double *logV, int cap, double *modes,
                          double *logZk, double *ell_modes, int32_t *n_modes, double *logZ, int32_t *dev_status,
                          cudaStream_t s) {
    note_launch();
    k_laplace_final<<<1, 1024, 0, s>>>(d, XC, LC, logZk_c, n_c, reps, n_reps, logV, cap, modes, logZk, ell_modes,
                                       n_modes, logZ, dev_status);
}

}  // namespace sb
