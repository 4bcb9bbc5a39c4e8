// precheck.cu -- preprocessing: dimensional pathology detection (Sec. 3.4).
//
// The probe needs l at the box centre c and at c +- Delta_i e_i for every i
// (2d + 1 points). Each probe point moves one coordinate, so with
// z_k = L_k^T (x - mu_k):
//     z_k(c + t e_i) = z_k(c) + t L_k[i, :]^T,
//     e_k(c + t e_i) - e_k(c) = -t (z_k(c) . L_k[i, :]) - t^2 |L_k[i, :]|^2 / 2,
// and l(c + t e_i) - l(c) = LSE_k (e_k(c) - l(c) + that change). The whole
// probe is one GEMV per component (z_k(c)) and a dot product and a squared
// norm per row of L_k: O(K d^2) work, two streaming reads of the L_k, and the
// l differences come out without the cancellation of subtracting two l values
// (for one component the difference is the quadratic above exactly).
//
// Then one CTA sorts the finite sensitivities (bitonic, d <= 1024) for the
// median, takes the maximum, classifies (flat: s < eps_flat median; soft:
// s < eps_soft max and not flat) and sums the marginal terms in index order:
// log(2 Delta_i) for a flat coordinate, 1/2 log 2 pi + log(Delta_i / sqrt(s_i))
// for a soft one, and the flagged coordinates' log-volume sum log(2 Delta_i).
#include "sb_precheck.cuh"

namespace sb {

namespace {

// An SM's FP64 pipe takes one warp instruction per 19 cycles (64 per scheduler) whatever
// its active lanes: the two passes over the L_k are bound by their 1.5 K d^2 FMAs (24 us at
// d = 1024, K = 8; the bytes 5 us), the small kernels by their chains of dependent FP64
// instructions, which are spread over lanes (an exponential per lane). Device time of the
// five launches at d = 1024, K = 8 (cold caches): 297 us -> 85 us, the two passes 114 -> 49.
constexpr int PRE_RC = 32;    // rows of L_k per partial of z_k(c)
constexpr int PRE_COLS = 128; // columns per CTA of z_k(c)

// part[k][chunk][j] = sum over rows i of the chunk (i >= j) of L_k[i][j] (c_i - mu_k,i): one
// CTA per 32 x 128 tile of the triangle, so that every SM gets a share of the FMAs (whole
// 64-row chunks: 84 us at d = 1024, K = 8)
__global__ void __launch_bounds__(PRE_COLS) k_pre_z0_part(int d, const double *L, const double *mu, const double *c,
                                                          double *part) {
    __shared__ double dl[PRE_RC];
    const int chunk = blockIdx.y, k = blockIdx.z, nch = gridDim.y;
    const int i0 = chunk * PRE_RC, i1 = min(d, i0 + PRE_RC);
    if ((int)blockIdx.x * PRE_COLS >= i1) return;
    const double *Lk = L + (size_t)k * d * d;
    const double *mk = mu + (size_t)k * d;
    if (threadIdx.x < PRE_RC && i0 + (int)threadIdx.x < d) dl[threadIdx.x] = c[i0 + threadIdx.x] - mk[i0 + threadIdx.x];
    __syncthreads();
    const int j = blockIdx.x * PRE_COLS + threadIdx.x;
    if (j >= i1) return;
    double acc = 0.0;
    if (j <= i0 && i1 - i0 == PRE_RC) {
#pragma unroll 16
        for (int r = 0; r < PRE_RC; ++r) acc = fma(Lk[(size_t)(i0 + r) * d + j], dl[r], acc);
    } else {
        for (int i = max(i0, j); i < i1; ++i) acc = fma(Lk[(size_t)i * d + j], dl[i - i0], acc);
    }
    part[((size_t)k * nch + chunk) * d + j] = acc;
}

// z0[k][j] = sum of the partials of the chunks that reach column j (chunk order), and the
// block's share of |z0_k|^2 (one CTA per component took 31 us at d = 1024, K = 8)
__global__ void __launch_bounds__(PRE_COLS) k_pre_z0_fin(int d, int nch, const double *part, double *z0, double *ssp) {
    __shared__ double sh[PRE_COLS / 32];
    const int k = blockIdx.y, j = blockIdx.x * PRE_COLS + threadIdx.x;
    double z = 0.0;
    if (j < d) {
#pragma unroll 8
        for (int q = j / PRE_RC; q < nch; ++q) z += part[((size_t)k * nch + q) * d + j];
        z0[(size_t)k * d + j] = z;
    }
    const double ss = warp_sum(z * z);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < PRE_COLS / 32; ++w) t += sh[w];
        ssp[(size_t)k * gridDim.x + blockIdx.x] = t;
    }
}

// warp per two rows i, i + 1 of L_k: dot[k][i] = z0_k . L_k[i, :], nrm[k][i] = |L_k[i, :]|^2
// (j <= i). The four sums are reduced together (each exchange halves the values a lane
// holds): 6 FP64 adds for two rows instead of 20.
__global__ void __launch_bounds__(256) k_pre_rows(int d, const double *L, const double *z0, double *dot, double *nrm) {
    const int lane = threadIdx.x & 31;
    const int i = 2 * (blockIdx.x * 8 + (threadIdx.x >> 5)), k = blockIdx.y;
    if (i >= d) return;
    const bool two = i + 1 < d;
    const double *row0 = L + ((size_t)k * d + i) * d;
    const double *row1 = two ? row0 + d : row0;
    const double *zk = z0 + (size_t)k * d;
    double v[4] = {0.0, 0.0, 0.0, 0.0};  // dot and norm of row i, of row i + 1
    for (int j0 = 0; j0 <= i + 1; j0 += 128) {
        double a[4], b[4], z[4], zi[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u + lane;
            a[u] = j <= i ? row0[j] : 0.0;
            b[u] = two && j <= i + 1 ? row1[j] : 0.0;
            z[u] = j <= i + 1 && j < d ? zk[j] : 0.0;
            zi[u] = j <= i ? z[u] : 0.0;  // z0_i+1 is no part of row i (0 times an infinity is NaN)
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j0 + 32 * u > i + 1) break;
            v[0] = fma(a[u], zi[u], v[0]);
            v[1] = fma(a[u], a[u], v[1]);
            v[2] = fma(b[u], z[u], v[2]);
            v[3] = fma(b[u], b[u], v[3]);
        }
    }
    // lanes with bit 16 keep row i + 1, lanes with bit 8 the norm
    const bool h1 = lane & 16, h0 = lane & 8;
    double p0 = (h1 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h1 ? v[0] : v[2], 16);
    double p1 = (h1 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h1 ? v[1] : v[3], 16);
    double q = (h0 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, h0 ? p0 : p1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if ((lane & 7) == 0 && (!h1 || two)) (h0 ? nrm : dot)[(size_t)k * d + i + (h1 ? 1 : 0)] = q;
}

__device__ __forceinline__ double group8_sum(double v) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// up / down changes l(c +- Delta_i e_i) - l(c), s_i = |up| + |down|: eight lanes per
// (coordinate, sign), lane q over the components q, q + 8, ... (an exponential is about 40
// FP64 instructions; K of them in turn in each of d threads on d / 256 CTAs took 55 us)
__global__ void __launch_bounds__(128) k_pre_sens(int d, int K, int nblk, const double *a, const double *ssp,
                                                  const double *dot, const double *nrm, const double *half,
                                                  double *s) {
    __shared__ double s_e[kMaxK];
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        double t = 0.0;
        for (int q = 0; q < nblk; ++q) t += ssp[(size_t)k * nblk + q];
        s_e[k] = a[k] - 0.5 * t;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, q = lane & 7;
    double m0 = -INFINITY;
    for (int k = 0; k < K; ++k) m0 = s_e[k] > m0 ? s_e[k] : m0;
    double s0 = 0.0;
    for (int k = q; k < K; k += 8) s0 += exp(s_e[k] - m0);
    const double l0 = m0 + log(group8_sum(s0));
    const int pair = blockIdx.x * 16 + (threadIdx.x >> 3);  // 2 i + sign
    const int i = pair >> 1;
    const bool live = i < d;
    const double t = live ? ((pair & 1) ? -half[i] : half[i]) : 0.0;
    auto term = [&](int k) {
        return (s_e[k] - l0) - t * dot[(size_t)k * d + i] - 0.5 * t * t * nrm[(size_t)k * d + i];
    };
    double m = -INFINITY;
    if (live)
        for (int k = q; k < K; k += 8) m = fmax(m, term(k));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    double acc = 0.0;
    if (live)
        for (int k = q; k < K; k += 8) acc += exp(term(k) - m);
    acc = group8_sum(acc);
    const double out = live ? fabs(m + log(acc)) : 0.0;
    const double other = __shfl_xor_sync(0xffffffffu, out, 8);  // the other sign of the coordinate
    if (live && (lane & 15) == 0) s[i] = out + other;
}

constexpr int PRE_SORT = 1024;  // >= kMaxD

// One CTA: the sort runs on order-preserving integer keys (FP64 compares share the SM's
// two FP64 lanes) and the marginal terms are summed by a fixed tree; thread 0 walking the
// d terms took most of this kernel's former 98 us at d = 1024.
__global__ void __launch_bounds__(PRE_SORT) k_pre_classify(int d, const double *s, const double *half,
                                                          double eps_flat, double eps_soft, int8_t *cls,
                                                          double *log_int, double *log_vol, int32_t *n_active) {
    __shared__ uint64_t v[PRE_SORT];
    __shared__ double sh_i[PRE_SORT / 32], sh_v[PRE_SORT / 32];
    __shared__ int sh_n[PRE_SORT / 32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const double st = t < d ? s[t] : INFINITY;
    v[t] = ordered_bits(isfinite(st) ? st : INFINITY);
    const int nf = __syncthreads_count(t < d && isfinite(st));
    int n2 = 2;  // the sort covers the power of two that holds d
    while (n2 < d) n2 <<= 1;
    // bitonic sort, ascending (non-finite and padding as +inf at the end)
    for (int size = 2; size <= n2; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const int p = t ^ stride;
            if (t < n2 && p > t) {
                const bool up = (t & size) == 0;
                const uint64_t a = v[t], b = v[p];
                if ((a > b) == up) {
                    v[t] = b;
                    v[p] = a;
                }
            }
            __syncthreads();
        }
    }
    // the inverse of ordered_bits (the sensitivities are >= 0: the sign bit is set)
    auto value = [&](int i) {
        const uint64_t b = v[i];
        return __longlong_as_double((long long)((b >> 63) ? b & 0x7fffffffffffffffull : ~b));
    };
    double med = 0.0, smax = 0.0;
    if (nf > 0) {
        med = (nf & 1) ? value(nf / 2) : 0.5 * (value(nf / 2 - 1) + value(nf / 2));
        smax = value(nf - 1);
    }
    double ti = 0.0, tv = 0.0;
    int act = 0;
    if (t < d) {
        int8_t cl = 0;
        if (isfinite(st)) {
            if (st < eps_flat * med)
                cl = 1;
            else if (st < eps_soft * smax)
                cl = 2;
        }
        cls[t] = cl;
        act = cl == 0;
        if (cl != 0) {
            const double w = log(2.0 * half[t]);
            tv = w;
            ti = cl == 1 ? w : 0.5 * SB_LOG_2PI + log(half[t] / sqrt(st));
        }
    }
    const int na = __popc(__ballot_sync(0xffffffffu, act));
    if (__any_sync(0xffffffffu, t < d && !act)) {  // some coordinate of the warp is flagged
        ti = warp_sum(ti);
        tv = warp_sum(tv);
    }
    if (lane == 0) {
        sh_i[wid] = ti;
        sh_v[wid] = tv;
        sh_n[wid] = na;
    }
    __syncthreads();
    if (t < 32) {
        ti = warp_sum(sh_i[lane]);
        tv = warp_sum(sh_v[lane]);
        int n = sh_n[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        if (lane == 0) {
            *log_int = ti;
            *log_vol = tv;
            *n_active = n;
        }
    }
}

}  // namespace

size_t precheck_scratch_elems(int d, int K) {
    const int nch = (d + PRE_RC - 1) / PRE_RC, nblk = (d + PRE_COLS - 1) / PRE_COLS;
    return (size_t)K * nch * d + 3 * (size_t)K * d + (size_t)K * nblk;
}

void launch_precheck(const ProbView &pv, double eps_flat, double eps_soft, double *scratch, double *s, int8_t *cls,
                     double *log_int, double *log_vol, int32_t *n_active, cudaStream_t st) {
    const int d = pv.d, K = pv.K;
    const int nch = (d + PRE_RC - 1) / PRE_RC, nblk = (d + PRE_COLS - 1) / PRE_COLS;
    double *part = scratch;
    double *z0 = part + (size_t)K * nch * d;
    double *dot = z0 + (size_t)K * d;
    double *nrm = dot + (size_t)K * d;
    double *ssp = nrm + (size_t)K * d;
    note_launch();
    k_pre_z0_part<<<dim3(nblk, nch, K), PRE_COLS, 0, st>>>(d, pv.L, pv.mu, pv.c, part);
    note_launch();
    k_pre_z0_fin<<<dim3(nblk, K), PRE_COLS, 0, st>>>(d, nch, part, z0, ssp);
    note_launch();
    k_pre_rows<<<dim3((d + 15) / 16, K), 256, 0, st>>>(d, pv.L, z0, dot, nrm);
    note_launch();
    k_pre_sens<<<(2 * d + 15) / 16, 128, 0, st>>>(d, K, nblk, pv.a, ssp, dot, nrm, pv.half, s);
    note_launch();
    k_pre_classify<<<1, PRE_SORT, 0, st>>>(d, s, pv.half, eps_flat, eps_soft, cls, log_int, log_vol, n_active);
}

}  // namespace sb
