// small_f64.cu -- FP64 likelihood, gradient and L-BFGS of small problems: a walker stays
// with a few lanes of one warp from its start to its terminal state, in one launch.
//
// What bounds it: the FP64 pipe. A GB300 SM takes one FP64 warp instruction per 19 cycles
// (64 per scheduler), whatever the active lanes and whether or not instructions depend on
// one another (measured), so a GEMM tile gains nothing over a matrix-vector product out of
// shared memory (16 bytes of L_k a cycle keep the pipe full), one warp per scheduler
// nearly fills it, and what counts is the number of warp instructions. Hence:
//  * LPW lanes per walker (8, 16 or 32), 32 / LPW walkers per warp in lockstep: the
//    triangle's diagonal blocks waste LPW / 2 columns per row, a reduction costs
//    log2(LPW) adds for all the warp's walkers together, and so do the scalars;
//  * the packed triangles of every L_k in shared memory (rows at i (i + 1) / 2: 16
//    consecutive rows start in 16 different 8-byte banks, so that both the column and the
//    row pass read without conflicts);
//  * a component whose term is exactly zero is left once that is certain: z_k is formed
//    from its last column slot up (the shortest columns), and when a_k - |z_k part|^2 / 2 lies more than
//    kSkipNats64 = 800 below the term of the walker's leading component, exp() of the
//    difference is 0 in FP64, so neither l, r nor grad l depends on the rest of z_k;
//  * no round ever waits for the slowest walker, and a round is no longer five launches.
// Every sum is formed in the order of the general path (lik_f64.cu, lbfgs.cu), whatever
// LPW: the results are the same bits.
// Measured against that path (GEMM tiles, five launches a round): a whole ChiSao solve at
// d = 64, K = 4, 4096 walkers 231 -> 42 ms, the sunburst solve of one Gaussian at d = 8, 64
// walkers 3.7 -> 0.88 ms, l and grad l at one point (d = 64, K = 4) 363 -> 24 us.
#include "sb_small_f64.cuh"

#include <type_traits>

namespace sb {

namespace {

constexpr double kSkipNats64 = 800.0;  // exp(x) is 0 in FP64 below -745.2
constexpr int kSmemMax = 220 * 1024;
constexpr int kMaxWarps = 8;

// Doubles of a walker group's shared buffer: a vector, l terms and exponentials per
// component, alpha and rho per pair; odd, so that the groups of a warp read their buffers
// from different banks.
__host__ __device__ inline int group_doubles(int d, int K, int m) { return (d + 2 * K + 2 * m) | 1; }
__host__ __device__ inline size_t tri(int d) { return (size_t)d * (d + 1) / 2; }
__host__ __device__ inline size_t problem_doubles(int d, int K) { return (size_t)K * (tri(d) + d + 1); }

// Lanes of the walker group of this lane.
template <int LPW>
__device__ __forceinline__ unsigned group_mask() {
    return (LPW == 32 ? 0xffffffffu : ((1u << (LPW & 31)) - 1u)) << (threadIdx.x & 31 & ~(LPW - 1));
}

struct SmallProb {
    int d, K;
    const double *Ls, *mus, *as;  // shared: packed L_k, mu_k, a_k
};

// Reads L_k, mu_k and a_k into shared memory (packed lower triangles).
__device__ __forceinline__ SmallProb load_problem(int d, int K, const double *L, const double *mu, const double *a,
                                                  double *sh) {
    const size_t T = tri(d);
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5, rows = K * d;
    // a warp takes four rows at a time, so that eight loads or more are in flight per lane
    for (int r0 = (threadIdx.x >> 5) * 4; r0 < rows; r0 += nw * 4) {
        for (int j0 = 0; j0 < d; j0 += 64) {
            double v[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q, i = r % d;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = j0 + 32 * h + lane;
                    v[2 * q + h] = r < rows && j <= i ? __ldg(L + (size_t)r * d + j) : 0.0;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q, k = r / d, i = r - k * d;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = j0 + 32 * h + lane;
                    if (r < rows && j <= i) sh[(size_t)k * T + (size_t)i * (i + 1) / 2 + j] = v[2 * q + h];
                }
            }
        }
    }
    double *mus = sh + K * T;
    for (int e = threadIdx.x; e < K * d; e += blockDim.x) mus[e] = mu[e];
    double *as = mus + K * d;
    for (int e = threadIdx.x; e < K; e += blockDim.x) as[e] = a[e];
    __syncthreads();
    return {d, K, sh, mus, as};
}

// Sum of a walker's per-coordinate products term(v), coordinate l + LPW v in lane l: the
// order of the general path (coordinate i in lane i % 32, slot i / 32; slots in order by
// fused multiply-adds, then a butterfly over the 32 lanes).
template <int LPW, int VPL, typename F>
__device__ __forceinline__ double vec_dot(F mul_add) {
    constexpr int C = 32 / LPW;  // lanes of the general path in one lane here
    double A[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        A[c] = 0.0;
#pragma unroll
        for (int v = c; v < VPL; v += C) A[c] = mul_add(v, A[c]);
    }
    double t = A[0];
    if (C == 4) {
        const double b0 = VPL > 2 ? A[0] + A[C > 2 ? 2 : 0] : A[0];
        const double b1 = VPL > 3 ? A[C > 1 ? 1 : 0] + A[C > 3 ? 3 : 0] : A[C > 1 ? 1 : 0];
        t = VPL > 1 ? b0 + b1 : b0;
    } else if (C == 2) {
        t = VPL > 1 ? A[0] + A[C > 1 ? 1 : 0] : A[0];
    }
#pragma unroll
    for (int o = LPW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// |z|^2 of the slots v >= v0 (zero below) in the order of k_zgemm_f64: per 64-column tile the four columns
// tx + 16 c in order of c, a butterfly over tx, then the tiles in order.
template <int LPW, int VPL>
__device__ __forceinline__ double norm2(const double *z) {
    double q = 0.0;
    constexpr int TV = 64 / LPW;  // slots per tile
#pragma unroll
    for (int t0 = 0; t0 < VPL; t0 += TV) {
        double s;
        if (LPW == 8) {
            double c0 = 0.0, c1 = 0.0;
#pragma unroll
            for (int v = t0; v < t0 + TV && v < VPL; v += 2) {
                c0 = fma(z[v], z[v], c0);
                if (v + 1 < VPL) c1 = fma(z[v + 1], z[v + 1], c1);
            }
            s = VPL > 1 ? c0 + c1 : c0;
        } else if (LPW == 16) {
            s = 0.0;
#pragma unroll
            for (int v = t0; v < t0 + TV && v < VPL; ++v) s = fma(z[v], z[v], s);
#pragma unroll
            for (int o = 8; o > 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        } else {
            const bool up = threadIdx.x & 16;
            s = 0.0;
#pragma unroll
            for (int v = t0; v < t0 + TV && v < VPL; ++v) {
                const double o = __shfl_xor_sync(0xffffffffu, z[v], 16);
                const double a = up ? o : z[v], b = up ? z[v] : o;
                s = fma(a, a, s);
                s = fma(b, b, s);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 8);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        q = VPL > TV ? q + s : s;
    }
    return q;
}

// Column l + LPW v of z = L^T delta: sum over rows i >= column of delta_i L[i][column], i
// ascending.
template <int LPW>
__device__ __forceinline__ double z_column(const double *Lk, const double *dl, int d, int v, int l) {
    const int i0 = v * LPW, i1 = min(i0 + LPW, d);
    const double *p = Lk + (size_t)i0 * (i0 + 1) / 2 + i0 + l;
    double acc = 0.0;
    for (int i = i0; i < i1; ++i) {
        const double e = l <= i - i0 ? *p : 0.0;
        acc = fma(dl[i], e, acc);
        p += i + 1;
    }
#pragma unroll 4
    for (int i = i1; i < d; ++i) {
        acc = fma(dl[i], *p, acc);
        p += i + 1;
    }
    return acc;
}

// acc + row i = l + LPW v of L z: sum over columns j <= i of z_j L[i][j], j ascending.
template <int LPW>
__device__ __forceinline__ double g_row(const double *Lk, const double *z, int d, int v, int l, double acc) {
    const int i0 = v * LPW, i1 = min(i0 + LPW, d);
    const int i = min(i0 + l, d - 1);
    const double *p = Lk + (size_t)i * (i + 1) / 2;
#pragma unroll 4
    for (int j = 0; j < i0; ++j) acc = fma(z[j], p[j], acc);
    for (int j = i0; j < i1; ++j) {
        const double e = j <= i ? p[j] : 0.0;
        acc = fma(z[j], e, acc);
    }
    return acc;
}

// l and (want) sum_k r_k L_k z_k at x for the walker group of this lane, all groups of the
// warp in lockstep (on: the group has a point). lead: the group's leading component of its
// last evaluation, or -1. buf: the group's shared buffer; Zw: [K][d] global scratch.
template <int LPW, int VPL>
__device__ __forceinline__ void evaluate(const SmallProb &P, const double *x, bool on, int &lead, double *buf,
                                         double *Zw, bool want, double &ell, double *g) {
    const int lane = threadIdx.x & 31, l = lane & (LPW - 1);
    const int d = P.d, K = P.K;
    const size_t T = tri(d);
    const int nv = (d + LPW - 1) / LPW;  // slots in use
    double *es = buf + d, *ex = es + K;
    if (K > 1 && nv >= 4 && __any_sync(0xffffffffu, on && lead < 0)) {
        // no leading component yet: the one whose last two column slots leave the largest
        // term (any choice gives the same result; a good one lets the others be left
        // early). With fewer than four slots those two are most of the triangle.
        double top = -INFINITY;
        int guess = 0;
        const int v1 = nv - 1, v0 = nv > 1 ? nv - 2 : 0, i0 = v0 * LPW;
        double xa = 0.0, xb = 0.0;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            if (v == v0) xa = x[v];
            if (v == v1) xb = x[v];
        }
        for (int k = 0; k < K; ++k) {
            const double *mk = P.mus + (size_t)k * d;
            __syncwarp();
            if (i0 + l < d) buf[i0 + l] = xa - mk[i0 + l];
            if (v1 > v0 && i0 + LPW + l < d) buf[i0 + LPW + l] = xb - mk[i0 + LPW + l];
            __syncwarp();
            const double za = z_column<LPW>(P.Ls + k * T, buf, d, v1, l);
            const double zb = v1 > v0 ? z_column<LPW>(P.Ls + k * T, buf, d, v0, l) : 0.0;
            double q = fma(za, za, zb * zb);
#pragma unroll
            for (int o = LPW / 2; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            const double e = fma(-0.5, q, P.as[k]);
            if (e > top) {
                top = e;
                guess = k;
            }
        }
        if (lead < 0) lead = guess;
    }
    uint64_t live = 0;  // components whose term may be above zero (group-uniform)
    double best = -INFINITY;
    const int k_first = on && lead >= 0 ? lead : 0;
    for (int kk = 0; kk < K; ++kk) {
        // the leading component first, then the others in order
        const int k = kk == 0 ? k_first : (kk <= k_first ? kk - 1 : kk);
        const double *Lk = P.Ls + k * T;
        const double *mk = P.mus + (size_t)k * d;
        __syncwarp();
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int i = l + LPW * v;
            if (i < d) buf[i] = sub_rn(x[v], mk[i]);
        }
        __syncwarp();
        double z[VPL];
        bool drop = !on;  // certain to add exactly zero
#pragma unroll
        for (int v = VPL - 1; v >= 0; --v) {
            z[v] = 0.0;
            if (v < nv && !__all_sync(0xffffffffu, drop)) {
                z[v] = z_column<LPW>(Lk, buf, d, v, l);
                // after the first two slots: the part of |z|^2 they hold (any order: a bound)
                if (kk > 0 && v > 0 && v >= nv - 2) {
                    double q = 0.0;
#pragma unroll
                    for (int u = v; u < VPL; ++u) q = fma(z[u], z[u], q);
#pragma unroll
                    for (int o = LPW / 2; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
                    // an infinite |z|^2 stays: its z may hold infinities, which reach grad l
                    const double eb = fma(-0.5 * (1.0 - 1e-10), q, P.as[k]);
                    drop = drop || (finite_bits(q) && eb < best - kSkipNats64);
                }
            }
        }
        if (!__all_sync(0xffffffffu, drop)) {
            const double q = norm2<LPW, VPL>(z);
            const double e = P.as[k] - 0.5 * q;
            if (!drop) {
                if (l == 0) es[k] = e;
                live |= 1ull << k;
                if (e > best) {
                    best = e;
                    lead = k;
                }
                if (want)
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        const int j = l + LPW * v;
                        if (j < d) Zw[(size_t)k * d + j] = z[v];
                    }
            }
        }
    }
    // l = LSE, r: with one live component the sum is exp(0) = 1, l its term and r = 1 (a
    // term that is not finite takes the general formula, which gives NaN)
    __syncwarp();
    const double e1 = live ? es[__ffsll((long long)live) - 1] : 0.0;
    const bool single = __popcll(live) <= 1 && finite_bits(e1);
    if (__all_sync(0xffffffffu, single)) {
        ell = e1;
    } else {
        double emax = -INFINITY;
        for (int k = 0; k < K; ++k)
            if ((live >> k) & 1ull) emax = fmax(emax, es[k]);
        for (int k = l; k < K; k += LPW) ex[k] = ((live >> k) & 1ull) ? exp(es[k] - emax) : 0.0;
        __syncwarp();
        double s = 0.0;
        for (int k = 0; k < K; ++k) s += ex[k];
        ell = emax + log(s);
        __syncwarp();
        for (int k = l; k < K; k += LPW) ex[k] = ex[k] / s;
        __syncwarp();
    }
    if (!want) return;
#pragma unroll
    for (int v = 0; v < VPL; ++v) g[v] = 0.0;
    // the components with r != 0, each group its own next one (ascending)
    uint64_t todo = live;
    while (true) {
        int k = -1;
        double r = 1.0;
        while (todo) {
            const int c = __ffsll((long long)todo) - 1;
            todo &= todo - 1;
            r = single ? 1.0 : ex[c];
            if (r != 0.0) {  // (NaN stays)
                k = c;
                break;
            }
            // r = 0 adds r z = 0 unless z holds an infinity or a NaN
            bool odd = false;
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int j = l + LPW * v;
                if (j < d) odd = odd || !finite_bits(Zw[(size_t)c * d + j]);
            }
            if (__any_sync(group_mask<LPW>(), odd)) {
                k = c;
                break;
            }
        }
        if (__all_sync(0xffffffffu, k < 0)) break;
        __syncwarp();
        if (k >= 0) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int j = l + LPW * v;
                if (j < d) buf[j] = single ? Zw[(size_t)k * d + j] : mul_rn(r, Zw[(size_t)k * d + j]);
            }
        }
        __syncwarp();
        const double *Lk = P.Ls + (k < 0 ? 0 : k) * T;
#pragma unroll
        for (int v = 0; v < VPL; ++v)
            if (v < nv) {
                const double t = g_row<LPW>(Lk, buf, d, v, l, g[v]);
                if (k >= 0 && l + LPW * v < d) g[v] = t;
            }
    }
}

// ------------------------------------------------------------------ points
// RAYS: row n is the ray sample flat0 + n (as in k_zgemm_f64), else a gathered row of X.
template <int LPW, int VPL, bool RAYS>
__global__ void __launch_bounds__(32 * kMaxWarps) k_small_points(LikF64Args a, int warps) {
    extern __shared__ double sh[];
    const int n_rows = a.n_rows_dev ? *a.n_rows_dev : a.n_rows;
    const int lane = threadIdx.x & 31, l = lane & (LPW - 1), warp = threadIdx.x >> 5;
    constexpr int GPW = 32 / LPW;
    const int per = warps * GPW;  // points of a CTA per pass
    if ((int)blockIdx.x >= n_rows) return;
    const SmallProb P = load_problem(a.d, a.K, a.L, a.mu, a.a, sh);
    if (warp >= warps) return;  // it only helped to load
    double *buf = sh + problem_doubles(a.d, a.K) + (size_t)(warp * GPW + lane / LPW) * group_doubles(a.d, a.K, 0);
    // a group takes consecutive rows: ray samples mostly keep their leading component
    const int span = (n_rows + (int)gridDim.x * per - 1) / ((int)gridDim.x * per);
    const int first = (blockIdx.x * per + warp * GPW + lane / LPW) * span;
    int lead = -1;
    for (int q = 0; q < span; ++q) {
        const int n = first + q;
        const bool on = n < n_rows;
        if (!RAYS) lead = -1;
        const int w = on ? (a.rows ? a.rows[n] : n) : 0;
        const int out = a.out_by_walker ? w : n;
        double x[VPL], g[VPL], ell, t = 0.0;
        int r = 0;
        if (RAYS && on) {  // x = c + t_j t_exit u_r, t_j = (j + 1) / n_steps (c_ld: the ray's own c)
            const int64_t flat = a.flat0 + n;
            r = (int)(flat / a.n_steps);
            t = mul_rn(div_rn((double)(flat - (int64_t)r * a.n_steps + 1), (double)a.n_steps), a.texit[r]);
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int i = l + LPW * v;
            x[v] = 0.0;
            if (on && i < a.d) x[v] = RAYS ? add_rn(a.c[(size_t)r * a.c_ld + i], mul_rn(t, a.u[(size_t)r * a.d + i])) : a.X[(size_t)w * a.d + i];
        }
        evaluate<LPW, VPL>(P, x, on, lead, buf, a.Z ? a.Z + (size_t)(on ? out : 0) * a.K * a.d : nullptr,
                           a.G != nullptr, ell, g);
        if (!on) continue;
        if (l == 0) a.ell[out] = a.ell_sign * ell;
        if (a.G)
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int i = l + LPW * v;
                if (i < a.d) a.G[(size_t)out * a.d + i] = a.grad_sign * g[v];
            }
    }
}

// A point per CTA, for fewer points than SMs: a warp per component forms z_k (32 lanes), one warp
// the LSE, and the gradient's 32-row slots go to a warp each, so the four schedulers share
// one point's FP64 instructions. Sums in the same order as in evaluate(). l and grad l at
// one point, d = 64, K = 4: 41 us a call with a warp per point,
// 24 so (the kernel itself 19).
inline size_t point_doubles(int d, int K) { return problem_doubles(d, K) + (size_t)(K + kMaxWarps) * d + 2 * (size_t)K; }
template <int VPL>
__global__ void __launch_bounds__(32 * kMaxWarps) k_small_point(LikF64Args a) {
    extern __shared__ double sh[];
    __shared__ unsigned long long s_odd;  // components whose z is not finite throughout
    __shared__ double s_ell;
    __shared__ unsigned long long s_act;  // components that add to grad l
    __shared__ int s_one;
    const int n_rows = a.n_rows_dev ? *a.n_rows_dev : a.n_rows, n = blockIdx.x;
    if (n >= n_rows) return;
    const int d = a.d, K = a.K, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nv = (d + 31) / 32;
    const size_t T = tri(d);
    const int w = a.rows ? a.rows[n] : n, out = a.out_by_walker ? w : n;
    if (threadIdx.x == 0) s_odd = 0ull;
    const SmallProb P = load_problem(d, K, a.L, a.mu, a.a, sh);
    double *zs = sh + problem_doubles(d, K), *buf = zs + (size_t)K * d + (size_t)warp * d;
    double *es = zs + (size_t)(K + kMaxWarps) * d, *ex = es + K;
    const double *X = a.X + (size_t)w * d;
    for (int k = warp; k < K; k += kMaxWarps) {
        const double *mk = P.mus + (size_t)k * d;
        __syncwarp();
        for (int i = lane; i < d; i += 32) buf[i] = sub_rn(X[i], mk[i]);
        __syncwarp();
        double z[VPL];
        bool odd = false;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            z[v] = v < nv ? z_column<32>(P.Ls + k * T, buf, d, v, lane) : 0.0;
            if (lane + 32 * v < d) zs[(size_t)k * d + lane + 32 * v] = z[v];
            odd = odd || !finite_bits(z[v]);
        }
        const double q = norm2<32, VPL>(z);
        if (lane == 0) es[k] = P.as[k] - 0.5 * q;
        if (__any_sync(0xffffffffu, odd) && lane == 0) atomicOr(&s_odd, 1ull << k);
    }
    __syncthreads();
    if (warp == 0) {
        double emax = -INFINITY;
        for (int k = 0; k < K; ++k) emax = fmax(emax, es[k]);
        // the components whose exponential is not certain to be 0
        uint64_t keep = 0;
        for (int k0 = 0; k0 < K; k0 += 32) {
            const bool far = k0 + lane >= K || es[k0 + lane] < emax - kSkipNats64;
            keep |= (uint64_t)(~__ballot_sync(0xffffffffu, far)) << k0;
        }
        if (__popcll(keep) == 1 && finite_bits(emax)) {
            if (lane == 0) {
                s_ell = emax;
                s_act = keep | s_odd;
                s_one = s_odd == 0ull;
            }
            for (int k = lane; k < K; k += 32) ex[k] = (keep >> k) & 1ull ? 1.0 : 0.0;
        } else {
            for (int k = lane; k < K; k += 32) ex[k] = exp(es[k] - emax);
            __syncwarp();
            double t = 0.0;
            for (int k = 0; k < K; ++k) t += ex[k];
            const double l = emax + log(t);
            __syncwarp();
            uint64_t act = 0;
            for (int k0 = 0; k0 < K; k0 += 32) {
                const int k = k0 + lane;
                const double r = k < K ? ex[k] / t : 0.0;
                if (k < K) ex[k] = r;
                act |= (uint64_t)__ballot_sync(0xffffffffu, k < K && r != 0.0) << k0;
            }
            if (lane == 0) {
                s_ell = l;
                s_act = act | s_odd;
                s_one = 0;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) a.ell[out] = a.ell_sign * s_ell;
    if (!a.G) return;
    const uint64_t act = s_act;
    if (!s_one) {  // r z in place
        for (uint64_t m = act; m; m &= m - 1) {
            const int k = __ffsll((long long)m) - 1;
            for (int j = threadIdx.x; j < d; j += blockDim.x) zs[(size_t)k * d + j] = mul_rn(ex[k], zs[(size_t)k * d + j]);
        }
        __syncthreads();
    }
    for (int v = warp; v < nv; v += kMaxWarps) {
        double g = 0.0;
        for (uint64_t m = act; m; m &= m - 1) {
            const int k = __ffsll((long long)m) - 1;
            g = g_row<32>(P.Ls + k * T, zs + (size_t)k * d, d, v, lane, g);
        }
        const int i = lane + 32 * v;
        if (i < d) a.G[(size_t)out * d + i] = a.grad_sign * g;
    }
}

// ------------------------------------------------------------------ L-BFGS (see lbfgs.cu)
template <int LPW, int VPL>
__global__ void __launch_bounds__(32 * kMaxWarps) k_small_refine(ProbView pv, LbfgsArgs<double> a,
                                                                 const double *starts, int n, double *Z,
                                                                 double *x_out, double *ell_out, int8_t *status_out,
                                                                 int32_t *iters_out, unsigned long long *n_evals,
                                                                 int warps) {
    extern __shared__ double sh[];
    const int lane = threadIdx.x & 31, l = lane & (LPW - 1), warp = threadIdx.x >> 5;
    constexpr int GPW = 32 / LPW;
    const int d = pv.d, K = pv.K, m = a.m;
    const SmallProb P = load_problem(d, K, pv.L, pv.mu, pv.a, sh);
    if (warp >= warps) return;  // it only helped to load
    double *buf = sh + problem_doubles(d, K) + (size_t)(warp * GPW + lane / LPW) * group_doubles(d, K, m);
    double *al = buf + d + 2 * K, *rho = al + m;

    int w = -1;          // the group's walker
    bool more = true;    // walkers may be left
    int lead = -1, it = 0, count = 0, head = 0, bt = 0, attempt = 0, flat = 0, phase = 0;
    double f = 0.0, alpha = 0.0, dphi = 0.0, new_sy = 1.0, new_yy = 1.0;
    unsigned long long evals = 0;
    double x[VPL], g[VPL], p[VPL], xt[VPL], gt[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) x[v] = g[v] = p[v] = xt[v] = gt[v] = 0.0;

    while (true) {
        // groups without a walker take the next one
        if (w < 0 && more) {
            int t = 0;
            if (l == 0) t = atomicAdd(a.n_act, 1);
            t = __shfl_sync(group_mask<LPW>(), t, lane & ~(LPW - 1));
            if (t < n) {
                w = t;
                lead = -1;
                it = count = head = bt = attempt = flat = phase = 0;
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    const int i = l + LPW * v;
                    xt[v] = i < d ? starts[(size_t)w * d + i] : 0.0;
                }
            } else {
                more = false;
            }
        }
        __syncwarp();
        const bool on = w >= 0;
        if (!__any_sync(0xffffffffu, on)) break;
        double ell;
        evaluate<LPW, VPL>(P, xt, on, lead, buf, Z + (size_t)(on ? w : 0) * K * d, true, ell, gt);
        const double ft = -1.0 * ell;
        if (on) ++evals;
        double *S = a.S + (size_t)(on ? w : 0) * m * d, *Y = a.Y + (size_t)(on ? w : 0) * m * d;

        int fin = finite_bits(ft);
#pragma unroll
        for (int v = 0; v < VPL; ++v) fin &= finite_bits(gt[v]) ? 1 : 0;
        {
            const unsigned gm = group_mask<LPW>();
            fin = (__ballot_sync(0xffffffffu, fin) & gm) == gm;
        }
        int status = SB_WALKER_RUNNING;
        bool newiter = false, newdir = false;
        bool accept = false;
        if (on && phase == 0) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                x[v] = xt[v];
                g[v] = gt[v];
            }
            f = ft;
            phase = 1;
            if (!fin)
                status = SB_WALKER_NONFINITE;
            else
                newiter = true;
        } else if (on) {
            const double bound = add_rn(f, mul_rn(mul_rn(a.c1, alpha), dphi));
            accept = fin && ft <= bound;
            if (!accept) {
                ++bt;
                if (bt <= a.max_backtracks) {
                    alpha = mul_rn(alpha, a.backtrack);
#pragma unroll
                    for (int v = 0; v < VPL; ++v) xt[v] = add_rn(x[v], mul_rn(alpha, p[v]));
                } else if (count > 0 && attempt == 0) {
                    count = 0;
                    head = 0;
                    attempt = 1;
                    newdir = true;
                } else {
                    status = SB_WALKER_STALLED;
                }
            }
        }
        __syncwarp();
        if (__any_sync(0xffffffffu, accept)) {
            double sv[VPL], yv[VPL];
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                sv[v] = sub_rn(xt[v], x[v]);
                yv[v] = sub_rn(gt[v], g[v]);
            }
            const double ss = vec_dot<LPW, VPL>([&](int v, double t) { return fma(sv[v], sv[v], t); });
            const double yy = vec_dot<LPW, VPL>([&](int v, double t) { return fma(yv[v], yv[v], t); });
            const double sy = vec_dot<LPW, VPL>([&](int v, double t) { return fma(sv[v], yv[v], t); });
            if (accept) {
                // sy > 1e-10 sqrt(ss) sqrt(yy), the square roots only near the boundary
                const bool clear = sy > 0.0 && sy * sy > 1.01e-20 * (ss * yy);
                if (clear || sy > 1e-10 * sqrt(ss) * sqrt(yy)) {
                    new_sy = sy;  // of the newest pair: gamma = sy / yy
                    new_yy = yy;
                    int slot;
                    if (count < m) {
                        slot = (head + count) % m;
                        ++count;
                    } else {
                        slot = head;
                        head = (head + 1) % m;
                    }
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        const int i = l + LPW * v;
                        if (i < d) {
                            S[(size_t)slot * d + i] = sv[v];
                            Y[(size_t)slot * d + i] = yv[v];
                        }
                    }
                    if (l == 0) rho[slot] = div_rn(1.0, sy);
                }
                flat = (ft >= f) ? flat + 1 : 0;
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    x[v] = xt[v];
                    g[v] = gt[v];
                }
                f = ft;
                ++it;
                newiter = true;
            }
            __syncwarp();
        }
        if (__any_sync(0xffffffffu, newiter)) {
            long long gm = 0;  // |g| of finite values orders as its bits
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const long long b = __double_as_longlong(fabs(g[v]));
                gm = b > gm ? b : gm;
            }
#pragma unroll
            for (int o = LPW / 2; o > 0; o >>= 1) {
                const long long b = __shfl_xor_sync(0xffffffffu, gm, o);
                gm = b > gm ? b : gm;
            }
            if (newiter) {
                if (__longlong_as_double(gm) <= a.gtol * (1.0 + fabs(f)))
                    status = SB_WALKER_CONVERGED;
                else if (flat >= 2)
                    status = SB_WALKER_STALLED;
                else if (it >= a.max_iter)
                    status = SB_WALKER_MAXITER;
                else {
                    attempt = 0;
                    newdir = true;
                }
            }
        }
        __syncwarp();
        if (__any_sync(0xffffffffu, newdir)) {
            // p = -H g by the two-loop recursion over the stored pairs
            const int nc = newdir ? count : 0;
            int cmax = nc;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
            if (cmax > 0) {
                double q[VPL];
#pragma unroll
                for (int v = 0; v < VPL; ++v) q[v] = g[v];
                for (int t = cmax - 1; t >= 0; --t) {
                    const bool has = t < nc;
                    const int slot = has ? (head + t) % m : 0;
                    const double *s = S + (size_t)slot * d, *y = Y + (size_t)slot * d;
                    double sv[VPL], yv[VPL];
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        const int i = l + LPW * v;
                        sv[v] = has && i < d ? s[i] : 0.0;
                        yv[v] = has && i < d ? y[i] : 0.0;
                    }
                    const double sq = vec_dot<LPW, VPL>([&](int v, double u) { return fma(sv[v], q[v], u); });
                    if (has) {
                        const double av = mul_rn(rho[slot], sq);
                        if (l == 0) al[t] = av;
#pragma unroll
                        for (int v = 0; v < VPL; ++v) q[v] = sub_rn(q[v], mul_rn(av, yv[v]));
                    }
                }
                {
                    const double gamma = div_rn(new_sy, new_yy);
#pragma unroll
                    for (int v = 0; v < VPL; ++v) q[v] = mul_rn(gamma, q[v]);
                }
                __syncwarp();
                for (int t = 0; t < cmax; ++t) {
                    const bool has = t < nc;
                    const int slot = has ? (head + t) % m : 0;
                    const double *s = S + (size_t)slot * d, *y = Y + (size_t)slot * d;
                    double sv[VPL], yv[VPL];
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        const int i = l + LPW * v;
                        sv[v] = has && i < d ? s[i] : 0.0;
                        yv[v] = has && i < d ? y[i] : 0.0;
                    }
                    const double yr = vec_dot<LPW, VPL>([&](int v, double u) { return fma(yv[v], q[v], u); });
                    if (has) {
                        const double coef = sub_rn(al[t], mul_rn(rho[slot], yr));
#pragma unroll
                        for (int v = 0; v < VPL; ++v) q[v] = add_rn(q[v], mul_rn(sv[v], coef));
                    }
                }
                if (newdir && nc > 0)
#pragma unroll
                    for (int v = 0; v < VPL; ++v) p[v] = -q[v];
            }
            // steepest descent without history, and again when the direction does not descend
            bool steep = newdir && count == 0;
            double dp = 0.0;
            for (int pass = 0; pass < 2; ++pass) {
                if (__any_sync(0xffffffffu, steep)) {
                    const double gg = vec_dot<LPW, VPL>([&](int v, double t) { return fma(g[v], g[v], t); });
                    if (steep) {
                        const double gn = sqrt(gg);
#pragma unroll
                        for (int v = 0; v < VPL; ++v) p[v] = -div_rn(g[v], gn);
                    }
                    __syncwarp();
                }
                const double t = vec_dot<LPW, VPL>([&](int v, double u) { return fma(g[v], p[v], u); });
                if (pass == 0 || steep) dp = t;
                if (pass == 0) {
                    steep = newdir && !(dp < 0.0);
                    if (steep) {
                        count = 0;
                        head = 0;
                    }
                    if (!__any_sync(0xffffffffu, steep)) break;
                }
            }
            if (newdir) {
                dphi = dp;
                alpha = 1.0;
                bt = 0;
#pragma unroll
                for (int v = 0; v < VPL; ++v) xt[v] = add_rn(x[v], p[v]);
            }
        }
        __syncwarp();
        if (on && status != SB_WALKER_RUNNING) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int i = l + LPW * v;
                if (i < d) x_out[(size_t)w * d + i] = x[v];
            }
            if (l == 0) {
                ell_out[w] = -f;
                status_out[w] = (int8_t)status;
                if (iters_out) iters_out[w] = it;
                atomicAdd(n_evals, evals);
            }
            evals = 0;
            w = -1;
        }
        __syncwarp();
    }
}

__global__ void k_small_init(int32_t *counter, int64_t *n_evals) {
    *counter = 0;
    *n_evals = 0;
}

int sm_count() {
    static const int n = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return n;
}

// Lanes per walker: 8 has the fewest instructions per walker (up to d = 64; 16 beyond), more lanes
// shorten one walker's chain, which counts while there are fewer warps than schedulers
// (4 per SM). d <= 8 leaves wider groups nothing to do.
int lanes_per_walker(int d, int n) {
    int lpw = d <= 64 ? 8 : 16;
    const int schedulers = 4 * sm_count();
    while (lpw < 32 && lpw < d && (long long)n * lpw / 32 < schedulers) lpw *= 2;
    return lpw;
}

// Calls f(integral_constant LPW, integral_constant VPL) for the variant of (d, lpw).
template <typename F>
void with_variant(int d, int lpw, F f) {
    const int vpl = (d + lpw - 1) / lpw;
#define SB_SMALL_CASE(LP, VP) \
    if (lpw == LP && vpl <= VP) return f(std::integral_constant<int, LP>(), std::integral_constant<int, VP>());
    SB_SMALL_CASE(8, 1)
    SB_SMALL_CASE(8, 2)
    SB_SMALL_CASE(8, 4)
    SB_SMALL_CASE(8, 8)
    SB_SMALL_CASE(16, 1)
    SB_SMALL_CASE(16, 2)
    SB_SMALL_CASE(16, 4)
    SB_SMALL_CASE(16, 8)
    SB_SMALL_CASE(32, 1)
    SB_SMALL_CASE(32, 2)
    SB_SMALL_CASE(32, 4)
#undef SB_SMALL_CASE
}

struct Shape {
    int lpw, warps, grid;  // warps: those of a CTA that take walkers
    size_t smem;
};
// One CTA per SM at most (the triangles are loaded once), up to kMaxWarps warps: as few
// warps per CTA as spread the walkers over every SM, bounded by the shared memory.
Shape shape_for(int d, int K, int m, int n) {
    Shape s;
    s.lpw = lanes_per_walker(d, n);
    const int gpw = 32 / s.lpw;
    const long long warps = ((long long)n + gpw - 1) / gpw;
    long long w = (warps + sm_count() - 1) / sm_count();
    const size_t per_warp = sizeof(double) * (size_t)gpw * group_doubles(d, K, m);
    const size_t base = sizeof(double) * problem_doubles(d, K);
    const long long fit = (long long)((kSmemMax - base) / per_warp);
    if (w > kMaxWarps) w = kMaxWarps;
    if (w > fit) w = fit;
    if (w < 1) w = 1;
    s.warps = (int)w;
    const long long g = (warps + w - 1) / w;
    s.grid = (int)(g < sm_count() ? g : sm_count());
    s.smem = base + per_warp * (size_t)w;
    return s;
}

}  // namespace

bool small_f64_fits(int d, int K, int m) {
    // four warps of the widest grouping (8 lanes a walker: four groups a warp)
    return d <= 128 && sizeof(double) * (problem_doubles(d, K) + 16 * (size_t)group_doubles(d, K, m)) <= (size_t)kSmemMax;
}

void launch_small_refine_f64(const ProbView &pv, const LbfgsArgs<double> &a, const double *starts, int n, double *Z,
                             double *x_out, double *ell_out, int8_t *status_out, int32_t *iters_out,
                             int64_t *n_evals, cudaStream_t s) {
    const Shape sp = shape_for(pv.d, pv.K, a.m, n);
    note_launch();
    k_small_init<<<1, 1, 0, s>>>(a.n_act, n_evals);
    ProfScope prof(PROF_LBFGS_STEP, s);
    with_variant(pv.d, sp.lpw, [&](auto LP, auto VP) {
        auto *k = k_small_refine<decltype(LP)::value, decltype(VP)::value>;
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        note_launch();
        k<<<sp.grid, 32 * kMaxWarps, sp.smem, s>>>(pv, a, starts, n, Z, x_out, ell_out, status_out, iters_out,
                                                   reinterpret_cast<unsigned long long *>(n_evals), sp.warps);
    });
}

void launch_small_points_f64(const LikF64Args &a, bool rays, cudaStream_t s) {
    if (a.n_rows <= 0) return;
    ProfScope prof(PROF_F64_Z, s);
    const size_t pt = sizeof(double) * point_doubles(a.d, a.K);
    if (!rays && a.n_rows <= sm_count() && pt <= (size_t)kSmemMax) {
        auto launch = [&](auto VP) {
            auto *k = k_small_point<decltype(VP)::value>;
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
            note_launch();
            k<<<a.n_rows, 32 * kMaxWarps, pt, s>>>(a);
        };
        if (a.d <= 32) return launch(std::integral_constant<int, 1>());
        if (a.d <= 64) return launch(std::integral_constant<int, 2>());
        return launch(std::integral_constant<int, 4>());
    }
    const Shape sp = shape_for(a.d, a.K, 0, a.n_rows);
    with_variant(a.d, sp.lpw, [&](auto LP, auto VP) {
        auto *k = rays ? k_small_points<decltype(LP)::value, decltype(VP)::value, true>
                       : k_small_points<decltype(LP)::value, decltype(VP)::value, false>;
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        note_launch();
        k<<<sp.grid, 32 * kMaxWarps, sp.smem, s>>>(a, sp.warps);
    });
}

}  // namespace sb
