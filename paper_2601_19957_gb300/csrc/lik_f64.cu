// lik_f64.cu -- FP64 batched log-likelihood and gradient on CUDA cores.
//
// For a batch of points x_n (gathered walker rows, or ray samples generated on
// the fly) and components k:
//   z_nk = L_k^T (x_n - mu_k)                      (a triangular GEMM per k)
//   e_nk = a_k - |z_nk|^2 / 2,  l_n = LSE_k e_nk,  r_nk = softmax_k e_nk
//   grad l_n = -sum_k r_nk L_k z_nk                 (a second triangular GEMM)
// The Gaussian-mixture likelihood is the paper's problem statement (Sec. 3.2);
// the analytic gradient replaces its finite differences (App. A.4.1).
//
// FP64 throughput bounds this path (an SM takes one FP64 warp instruction per 19 cycles); it
// exists as the exact reference path and the plain-FP64 comparator of the tensor-core path.
//
// Tiling: 8 R points x 64 output coordinates per CTA (R = 4; R = 1 for the short row lists
// below, whose few tiles would otherwise be the launch's tail), reduction chunks of 16, 128
// threads with an R x 4 register tile each (columns tx + 16 c). Only the
// triangle that L_k occupies is visited: the z GEMM for output column block [j0, j0 + 64)
// reads rows i >= j0 of L_k, the gradient GEMM for output block [i0, i0 + 64) columns j < i0 +
// 64, and inside a diagonal block the 16-column groups that lie wholly outside the
// triangle are left out (6 of 16).
//
// Grouped evaluation (K >= 2, more than one column block, and enough rows): the last column
// block of every z_k, the cheapest, gives part of |z_k|^2; the row's component with the largest
// a_k - |part|^2 / 2 leads and is finished first; another component is finished only when it
// could still come within kSkipNats64 nats of the leading term. exp() of the difference is
// exactly 0 in FP64 otherwise, so neither l, r nor grad l depends on the rest of its z_k.
// Rows are listed per component, so the tiles hold rows that need the same L_k, and the
// gradient runs over the components with r != 0 only. Each sum keeps the order of the full
// evaluation, so the results are the same bits. l and grad l at 4096 points, d = 256, K = 4:
// 3227 us -> 819 us (the FP64 pipe's floor for every component in full is 2.0 ms).
#include "sb_internal.cuh"
#include "sb_small_f64.cuh"

#include <type_traits>

namespace sb {

namespace {
constexpr int BM = 32, BN = 64, BK = 16;  // BM: rows of an R = 4 tile
constexpr int NT = 128;                   // threads of a tile
constexpr int kGroupMinRows = 256;     // fewer rows: the grouping's launches cost more than they save
constexpr double kSkipNats64 = 800.0;  // exp(x) is 0 in FP64 below -745.2

enum { SRC_GATHER = 0, SRC_RAYS = 1 };

__device__ __forceinline__ int rows_of(const LikF64Args &a) { return a.n_rows_dev ? *a.n_rows_dev : a.n_rows; }

// Row lists of the grouped evaluation, in the caller's integer scratch a.grp.
struct Lists {
    int32_t *lead;           // [n] leading component
    int32_t *l1, *l2, *lg;   // [K][n] rows led by k; rows that need k besides; rows with r_k = 1 alone
    int32_t *lm;             // [n] rows with several r != 0
    int32_t *c1, *c2, *cg, *cm;  // their lengths [K], [K], [K], [1]
    uint64_t *mask;          // [n] components evaluated in full
};
__host__ __device__ inline Lists lists_of(int32_t *p, int n, int K) {
    Lists L;
    L.mask = reinterpret_cast<uint64_t *>(p);  // 256-byte aligned
    p += 2 * (size_t)n;
    L.c1 = p;
    L.c2 = p + K;
    L.cg = p + 2 * K;
    L.cm = p + 3 * K;
    p += 3 * K + 1;
    L.lead = p;
    L.l1 = p + n;
    L.l2 = L.l1 + (size_t)K * n;
    L.lg = L.l2 + (size_t)K * n;
    L.lm = L.lg + (size_t)K * n;
    return L;
}

// The (component, first list entry) of row tile t over lists of lengths cnt[0 .. K), or
// k = -1 past the last tile.
template <int ROWS>
__device__ __forceinline__ int list_tile(const int32_t *cnt, int K, int t, int &r0) {
    for (int k = 0; k < K; ++k) {
        const int nt = (cnt[k] + ROWS - 1) / ROWS;
        if (t < nt) {
            r0 = t * ROWS;
            return k;
        }
        t -= nt;
    }
    return -1;
}

// z of one tile: 8 R rows x columns [64 jt, 64 jt + 64) of component k. LISTED: the rows are
// entries of the list of k (row tile from cnt), else rows 8 R blockIdx.x .. of all rows.
// jt = jt0 + blockIdx.y (ascending: the longest column block first).
// Returns false past the last tile.
template <int SRC, bool STORE_Z, bool LISTED, int R>
__device__ __forceinline__ bool z_tile(const LikF64Args &a, int tile, int jt0, const int32_t *list,
                                       const int32_t *cnt) {
    constexpr int BM = 8 * R;
    const int n_rows = rows_of(a);
    const int d = a.d, K = a.K, nJT = (d + BN - 1) / BN;
    int k = blockIdx.z, n0 = tile * BM, n_end = n_rows;
    if (LISTED) {
        k = list_tile<BM>(cnt, K, tile, n0);
        if (k < 0) return false;
        n_end = cnt[k];
        list += (size_t)k * a.n_rows;
    }
    if (n0 >= n_end) return false;
    const int jt = jt0 + blockIdx.y, j0 = jt * BN;
    const double *Lk = a.L + (size_t)k * d * d;
    const double *mk = a.mu + (size_t)k * d;

    __shared__ double As[BK][BM + 1];
    __shared__ double Bs[BK][BN];
    __shared__ const double *s_src[BM];
    __shared__ double s_scale[BM];
    __shared__ int s_out[BM];

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < BM) {
        const bool valid = n0 + tid < n_end;
        const int n = valid ? (LISTED ? list[n0 + tid] : n0 + tid) : 0;
        if (SRC == SRC_GATHER) {
            const int w = valid ? (a.rows ? a.rows[n] : n) : 0;
            s_src[tid] = a.X + (size_t)w * d;
            s_out[tid] = valid ? (a.out_by_walker ? w : n) : -1;
            s_scale[tid] = 0.0;
        } else {
            const int64_t flat = a.flat0 + n;
            const int r = valid ? (int)(flat / a.n_steps) : 0;
            const int j = valid ? (int)(flat % a.n_steps) : 0;
            s_src[tid] = a.u + (size_t)r * d;
            // t_j * t_exit with t_j = (j+1)/n_steps (ray grid reading, Sec. 3.5.2)
            s_scale[tid] = valid ? mul_rn(div_rn((double)(j + 1), (double)a.n_steps), a.texit[r]) : 0.0;
            s_out[tid] = valid ? n : -1;
        }
    }
    __syncthreads();

    double acc[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

    auto chunk = [&](int i0, auto NC) {  // the first NC column groups
        constexpr int nc = decltype(NC)::value;
#pragma unroll
        for (int q = 0; q < BM * BK / NT; ++q) {
            const int e = tid + NT * q;
            const int row = e >> 4, kk = e & 15, i = i0 + kk;
            double v = 0.0;
            if (s_out[row] >= 0 && i < d) {
                double x;
                if (SRC == SRC_GATHER) {
                    x = s_src[row][i];
                } else {
                    x = add_rn(a.c[i], mul_rn(s_scale[row], s_src[row][i]));
                }
                v = sub_rn(x, mk[i]);
            }
            As[kk][row] = v;
        }
#pragma unroll
        for (int q = 0; q < BN * BK / NT; ++q) {
            const int e = tid + NT * q;
            const int kk = e >> 6, col = e & 63, i = i0 + kk, j = j0 + col;
            Bs[kk][col] = (i < d && j < d && j <= i) ? Lk[(size_t)i * d + j] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double av[R], bv[nc];
#pragma unroll
            for (int r = 0; r < R; ++r) av[r] = As[kk][ty + 8 * r];
#pragma unroll
            for (int c = 0; c < nc; ++c) bv[c] = Bs[kk][tx + 16 * c];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < nc; ++c) acc[r][c] = fma(av[r], bv[c], acc[r][c]);
        }
        __syncthreads();
    };
    // the diagonal block: rows i of chunk q meet the column groups c <= q only
    chunk(j0, std::integral_constant<int, 1>());
    if (j0 + BK < d) chunk(j0 + BK, std::integral_constant<int, 2>());
    if (j0 + 2 * BK < d) chunk(j0 + 2 * BK, std::integral_constant<int, 3>());
    for (int i0 = j0 + 3 * BK; i0 < d; i0 += BK) chunk(i0, std::integral_constant<int, 4>());

#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int row = ty + 8 * r;
        const int out = s_out[row];
        double q = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j = j0 + tx + 16 * c;
            if (j < d) q += acc[r][c] * acc[r][c];
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (out >= 0) {
            if (tx == 0) a.qpart[((size_t)out * K + k) * nJT + jt] = q;
            if (STORE_Z) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int j = j0 + tx + 16 * c;
                    if (j < d) a.Z[((size_t)out * K + k) * d + j] = acc[r][c];
                }
            }
        }
    }
    return true;
}

template <int SRC, bool STORE_Z>
__global__ void __launch_bounds__(NT) k_zgemm_f64(LikF64Args a, int jt0) {
    z_tile<SRC, STORE_Z, false, 4>(a, blockIdx.x, jt0, nullptr, nullptr);
}
// The lists' lengths are known on the device only: CTAs go from tile to tile.
template <bool STORE_Z, int R>
__global__ void __launch_bounds__(NT) k_zgemm_f64_listed(LikF64Args a, const int32_t *list, const int32_t *cnt) {
    for (int t = blockIdx.x; z_tile<SRC_GATHER, STORE_Z, true, R>(a, t, 0, list, cnt); t += gridDim.x)
        __syncthreads();  // the shared tiles are free for the next one
}

// The row's places in the lists of the components of `mask`: one atomic per warp and component
// (the order inside a list does not reach the results, which are stored by row).
__device__ __forceinline__ void append(uint64_t mask, int n, int K, int cap, int32_t *list, int32_t *cnt) {
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < K; ++c) {
        const unsigned m = __ballot_sync(0xffffffffu, (mask >> c) & 1ull);
        if (!m) continue;
        int base = 0;
        if (lane == __ffs(m) - 1) base = atomicAdd(&cnt[c], __popc(m));
        base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
        if ((m >> lane) & 1u) list[(size_t)c * cap + base + __popc(m & ((1u << lane) - 1u))] = n;
    }
}

__device__ __forceinline__ int out_row(const LikF64Args &a, int n) {
    return a.out_by_walker ? (a.rows ? a.rows[n] : n) : n;
}

// The leading component of each row from the last column block's part of |z_k|^2.
__global__ void __launch_bounds__(128) k_grp_lead(LikF64Args a, Lists L) {
    const int n_rows = rows_of(a);
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int K = a.K, nJT = (a.d + BN - 1) / BN;
    int lead = 0;
    if (n < n_rows) {
        const double *qp = a.qpart + (size_t)out_row(a, n) * K * nJT + nJT - 1;
        double top = -INFINITY;
        for (int k = 0; k < K; ++k) {
            const double e = fma(-0.5, qp[(size_t)k * nJT], a.a[k]);
            if (e > top) {
                top = e;
                lead = k;
            }
        }
        L.lead[n] = lead;
    }
    append(n < n_rows ? 1ull << lead : 0ull, n, K, a.n_rows, L.l1, L.c1);
}

// The components a row needs besides its leading one (see the header).
__global__ void __launch_bounds__(128) k_grp_need(LikF64Args a, Lists L) {
    const int n_rows = rows_of(a);
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int K = a.K, nJT = (a.d + BN - 1) / BN;
    uint64_t mask = 0;
    if (n < n_rows) {
        const double *qp = a.qpart + (size_t)out_row(a, n) * K * nJT;
        const int j = L.lead[n];
        double q = 0.0;
        for (int t = 0; t < nJT; ++t) q += qp[(size_t)j * nJT + t];
        const double low = (a.a[j] - 0.5 * q) - kSkipNats64;
        for (int k = 0; k < K; ++k) {
            const double ql = qp[(size_t)k * nJT + nJT - 1];
            const bool skip = k != j && finite_bits(ql) && fma(-0.5 * (1.0 - 1e-10), ql, a.a[k]) < low;
            if (!skip) mask |= 1ull << k;
        }
        L.mask[n] = mask;
        mask &= ~(1ull << j);
    }
    append(mask, n, K, a.n_rows, L.l2, L.c2);
}

// Per point: l = LSE_k (a_k - q_k/2) and the responsibilities r_k. GROUPED: over the
// components evaluated in full (the others add exact zeros), and with a.G also the
// gradient's row lists.
template <bool GROUPED>
__global__ void __launch_bounds__(128) k_lse_f64(LikF64Args a, Lists L) {
    const int n_rows = rows_of(a);
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int K = a.K, nJT = (a.d + BN - 1) / BN;
    int one = -1;
    bool multi = false;
    if (n < n_rows) {
        const int out = out_row(a, n);
        const uint64_t mask = GROUPED ? L.mask[n] : ~0ull;
        const double *qr = a.qpart + (size_t)out * K * nJT;
        auto term = [&](int k) {
            const double *qp = qr + (size_t)k * nJT;
            double q = 0.0;
            for (int t = 0; t < nJT; ++t) q += qp[t];
            return a.a[k] - 0.5 * q;
        };
        const int k1 = GROUPED ? __ffsll((long long)mask) - 1 : 0;
        if (GROUPED && (mask & (mask - 1)) == 0 && finite_bits(term(k1))) {
            // one component left: its exponential, and the sum, are 1
            a.ell[out] = a.ell_sign * term(k1);
            if (a.R)
                for (int k = 0; k < K; ++k) a.R[(size_t)out * K + k] = k == k1 ? 1.0 : 0.0;
            one = k1;
        } else {
            double e[kMaxK];
            double emax = -INFINITY;
            for (int k = 0; k < K; ++k) {
                if (GROUPED && !((mask >> k) & 1ull)) continue;
                e[k] = term(k);
                emax = fmax(emax, e[k]);
            }
            double ssum = 0.0;
            for (int k = 0; k < K; ++k) {
                if (GROUPED && !((mask >> k) & 1ull)) continue;
                e[k] = exp(e[k] - emax);
                ssum += e[k];
            }
            a.ell[out] = a.ell_sign * (emax + log(ssum));
            int cnt = 0;
            if (a.R)
                for (int k = 0; k < K; ++k) {
                    const double r = GROUPED && !((mask >> k) & 1ull) ? 0.0 : e[k] / ssum;
                    a.R[(size_t)out * K + k] = r;
                    if (r != 0.0) {
                        ++cnt;
                        one = r == 1.0 ? k : -2;
                    }
                }
            multi = cnt != 1 || one < 0;
        }
    }
    if (GROUPED && a.G) {
        append(n < n_rows && !multi ? 1ull << one : 0ull, n, K, a.n_rows, L.lg, L.cg);
        append(multi ? 1ull : 0ull, n, 1, a.n_rows, L.lm, L.cm);
    }
}

// grad: out[n][i] = sign * sum_k sum_{j<=i} r_nk z_nk[j] L_k[i][j]  (= -sign * grad l).
// ROWS_ALL: every row and component; ROWS_ONE: the rows of the list of each component,
// whose r is 1 there and 0 elsewhere; ROWS_MULTI: the listed rows, components with r = 0 left out.
enum { ROWS_ALL = 0, ROWS_ONE = 1, ROWS_MULTI = 2 };
template <int MODE, int R>
struct GradTile {
    static constexpr int BM = 8 * R;
    double As[BK][BM + 1];
    double Bs[BK][BN + 1];
    int s_out[BM];
};
template <int MODE, int R>
__device__ __forceinline__ bool grad_tile(const LikF64Args &a, int tile, const int32_t *list, const int32_t *cnt,
                                          GradTile<MODE, R> &sm) {
    constexpr int BM = 8 * R;
    auto &As = sm.As;
    auto &Bs = sm.Bs;
    auto &s_out = sm.s_out;
    const int d = a.d, K = a.K;
    int n0 = tile * BM, n_end = rows_of(a), k_lo = 0, k_hi = K;
    if (MODE == ROWS_ONE) {
        k_lo = list_tile<BM>(cnt, K, tile, n0);
        if (k_lo < 0) return false;
        k_hi = k_lo + 1;
        n_end = cnt[k_lo];
        list += (size_t)k_lo * a.n_rows;
    } else if (MODE == ROWS_MULTI) {
        n_end = *cnt;
    }
    if (n0 >= n_end) return false;
    const int i0 = (gridDim.y - 1 - blockIdx.y) * BN;  // the longest column range first

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < BM) {
        const bool valid = n0 + tid < n_end;
        s_out[tid] = valid ? out_row(a, MODE == ROWS_ALL ? n0 + tid : list[n0 + tid]) : -1;
    }
    __syncthreads();

    double acc[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

    for (int k = k_lo; k < k_hi; ++k) {
        if (MODE == ROWS_MULTI) {
            const bool on = tid < BM && s_out[tid] >= 0 && a.R[(size_t)s_out[tid] * K + k] != 0.0;
            if (!__syncthreads_or(on)) continue;
        }
        const double *Lk = a.L + (size_t)k * d * d;
        auto chunk = [&](int j0, auto C0) {  // the column groups from C0 on
            constexpr int c0 = decltype(C0)::value;
#pragma unroll
            for (int q = 0; q < BM * BK / NT; ++q) {
                const int e = tid + NT * q;
                const int row = e >> 4, kk = e & 15, j = j0 + kk;
                const int out = s_out[row];
                double v = 0.0;
                if (out >= 0 && j < d) {
                    if (MODE == ROWS_ONE) {
                        v = a.Z[((size_t)out * K + k) * d + j];
                    } else {
                        const double r = a.R[(size_t)out * K + k];
                        if (MODE == ROWS_ALL || r != 0.0) v = r * a.Z[((size_t)out * K + k) * d + j];
                    }
                }
                As[kk][row] = v;
            }
            {
                // 64 columns (rows i of L_k) x 16 j: each thread loads 8 consecutive j of one row
                const int col = tid >> 1, kq = (tid & 1) * 8;
                const int i = i0 + col;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int j = j0 + kq + t;
                    Bs[kq + t][col] = (i < d && j < d && j <= i) ? Lk[(size_t)i * d + j] : 0.0;
                }
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                double av[R], bv[4];
#pragma unroll
                for (int r = 0; r < R; ++r) av[r] = As[kk][ty + 8 * r];
#pragma unroll
                for (int c = c0; c < 4; ++c) bv[c] = Bs[kk][tx + 16 * c];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = c0; c < 4; ++c) acc[r][c] = fma(av[r], bv[c], acc[r][c]);
            }
            __syncthreads();
        };
        for (int j0 = 0; j0 <= i0 && j0 < d; j0 += BK) chunk(j0, std::integral_constant<int, 0>());
        // the rest of the diagonal block: columns j of chunk q reach the rows of groups c >= q only
        if (i0 + BK < d) chunk(i0 + BK, std::integral_constant<int, 1>());
        if (i0 + 2 * BK < d) chunk(i0 + 2 * BK, std::integral_constant<int, 2>());
        if (i0 + 3 * BK < d) chunk(i0 + 3 * BK, std::integral_constant<int, 3>());
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int out = s_out[ty + 8 * r];
        if (out < 0) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int i = i0 + tx + 16 * c;
            if (i < d) a.G[(size_t)out * d + i] = a.grad_sign * acc[r][c];
        }
    }
    return true;
}
__global__ void __launch_bounds__(NT) k_ggemm_f64(LikF64Args a) {
    __shared__ GradTile<ROWS_ALL, 4> sm;
    grad_tile<ROWS_ALL, 4>(a, blockIdx.x, nullptr, nullptr, sm);
}
// The gradient of the grouped evaluation: first the tiles of the rows with several
// components (8 rows each: up to K times as long as the others'), on n_multi CTAs.
__global__ void __launch_bounds__(NT) k_ggemm_f64_grouped(LikF64Args a, Lists L, int n_multi) {
    __shared__ union {
        GradTile<ROWS_MULTI, 1> m;
        GradTile<ROWS_ONE, 4> o;
    } sm;
    if ((int)blockIdx.x < n_multi) {
        for (int t = blockIdx.x; grad_tile<ROWS_MULTI, 1>(a, t, L.lm, L.cm, sm.m); t += n_multi) __syncthreads();
    } else {
        grad_tile<ROWS_ONE, 4>(a, blockIdx.x - n_multi, L.lg, L.cg, sm.o);
    }
}
// ------------------------------------------------------------------ few points (GEMV shape)
// For a handful of points (the Laplace stage's candidates) a 64-row GEMM tile
// does 64 rows of FP64 work for each real row. These kernels spread the work
// over (column block, component, point block) instead, with the same outputs,
// layouts and a fixed summation order.
constexpr int FEW_CB = 8;  // points per CTA

// z_k[j] for the 64 columns j of one tile, one component and CB points: thread
// (column, row group of 4) accumulates rows i = i0 + rg, i0 + rg + 4, ... of
// L_k (coalesced row segments), then the four row groups are summed in a
// fixed order.
struct FewZShared {
    double dl[FEW_CB][64];  // delta = x - mu_k for 64 rows i of the current chunk
    double part[4][FEW_CB][64];
    double red[FEW_CB][2];
    int s_src[FEW_CB], s_out[FEW_CB];
};

template <int CB>
__device__ __forceinline__ void few_z_body(const LikF64Args &a, int jt, int k, int c0, FewZShared &sm) {
    const int d = a.d, K = a.K, nJT = (d + 63) / 64, j0 = jt * 64;
    const int tx = threadIdx.x & 63, rg = threadIdx.x >> 6;
    auto &dl = sm.dl;
    auto &part = sm.part;
    auto &red = sm.red;
    auto &s_src = sm.s_src;
    auto &s_out = sm.s_out;
    if (threadIdx.x < CB) {
        const int n = c0 + threadIdx.x;
        const int w = a.rows ? a.rows[n] : n;
        s_src[threadIdx.x] = w;
        s_out[threadIdx.x] = a.out_by_walker ? w : n;
    }
    __syncthreads();
    const double *Lk = a.L + (size_t)k * d * d;
    const double *mk = a.mu + (size_t)k * d;
    const int j = j0 + tx;
    double acc[CB];
#pragma unroll
    for (int c = 0; c < CB; ++c) acc[c] = 0.0;
    for (int i0 = j0; i0 < d; i0 += 64) {
        for (int e = threadIdx.x; e < CB * 64; e += 256) {
            const int c = e >> 6, ii = e & 63, i = i0 + ii;
            dl[c][ii] = i < d ? sub_rn(a.X[(size_t)s_src[c] * d + i], mk[i]) : 0.0;
        }
        __syncthreads();
        const int imax = min(64, d - i0);
        for (int ii = rg; ii < imax; ii += 4) {
            const int ig = i0 + ii;
            const double l = (j < d && j <= ig) ? Lk[(size_t)ig * d + j] : 0.0;
#pragma unroll
            for (int c = 0; c < CB; ++c) acc[c] = fma(dl[c][ii], l, acc[c]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < CB; ++c) part[rg][c][tx] = acc[c];
    __syncthreads();
    if (rg == 0) {
        // |z|^2 over the 64 columns: warp shuffles, then the two warps through shared memory
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            const double z = ((part[0][c][tx] + part[1][c][tx]) + part[2][c][tx]) + part[3][c][tx];
            acc[c] = z;
            double q = (j < d) ? z * z : 0.0;
            q = warp_sum(q);
            if ((tx & 31) == 0) red[c][tx >> 5] = q;
        }
        asm volatile("bar.sync 1, 64;" ::: "memory");  // the two warps of row group 0
        if (tx < CB) a.qpart[((size_t)s_out[tx] * K + k) * nJT + jt] = red[tx][0] + red[tx][1];
        if (a.Z && j < d)
#pragma unroll
            for (int c = 0; c < CB; ++c) a.Z[((size_t)s_out[c] * K + k) * d + j] = acc[c];
    }
}

__global__ void __launch_bounds__(256) k_few_z(LikF64Args a) {
    __shared__ FewZShared sm;
    const int n_rows = rows_of(a);
    const int c0 = blockIdx.z * FEW_CB;
    if (c0 >= n_rows) return;
    switch (min(FEW_CB, n_rows - c0)) {  // the live point count of this CTA (device-side)
        case 1: few_z_body<1>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 2: few_z_body<2>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 3: few_z_body<3>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 4: few_z_body<4>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 5: few_z_body<5>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 6: few_z_body<6>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        case 7: few_z_body<7>(a, blockIdx.x, blockIdx.y, c0, sm); break;
        default: few_z_body<8>(a, blockIdx.x, blockIdx.y, c0, sm); break;
    }
}

// grad: out[n][i] = sign * sum_k sum_{j<=i} r_nk z_nk[j] L_k[i][j]; warp per row i,
// CB points; components with r == 0 at every point of the CTA are skipped.
template <int CB>
__device__ __forceinline__ void few_g_body(const LikF64Args &a, int c0, int *s_out) {
    const int d = a.d, K = a.K;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = blockIdx.x * 8 + wid;
    if (threadIdx.x < CB) {
        const int n = c0 + threadIdx.x;
        s_out[threadIdx.x] = a.out_by_walker ? (a.rows ? a.rows[n] : n) : n;
    }
    __syncthreads();
    if (i >= d) return;
    double acc[CB];
#pragma unroll
    for (int c = 0; c < CB; ++c) acc[c] = 0.0;
    for (int k = 0; k < K; ++k) {
        double rk[CB];
        const double *zk[CB];
        bool any = false;
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            const int o = s_out[c];
            rk[c] = a.R[(size_t)o * K + k];
            zk[c] = a.Z + ((size_t)o * K + k) * d;
            any = any || rk[c] != 0.0;
        }
        if (!any) continue;
        const double *Lrow = a.L + (size_t)k * d * d + (size_t)i * d;
        for (int j = lane; j <= i; j += 32) {
            const double l = Lrow[j];
#pragma unroll
            for (int c = 0; c < CB; ++c) acc[c] = fma(rk[c] * zk[c][j], l, acc[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < CB; ++c) {
        const double v = warp_sum(acc[c]);
        if (lane == 0) a.G[(size_t)s_out[c] * d + i] = a.grad_sign * v;
    }
}

__global__ void __launch_bounds__(256) k_few_g(LikF64Args a) {
    __shared__ int s_out[FEW_CB];
    const int n_rows = rows_of(a);
    const int c0 = blockIdx.y * FEW_CB;
    if (c0 >= n_rows) return;
    switch (min(FEW_CB, n_rows - c0)) {
        case 1: few_g_body<1>(a, c0, s_out); break;
        case 2: few_g_body<2>(a, c0, s_out); break;
        case 3: few_g_body<3>(a, c0, s_out); break;
        case 4: few_g_body<4>(a, c0, s_out); break;
        case 5: few_g_body<5>(a, c0, s_out); break;
        case 6: few_g_body<6>(a, c0, s_out); break;
        case 7: few_g_body<7>(a, c0, s_out); break;
        default: few_g_body<8>(a, c0, s_out); break;
    }
}

}  // namespace

size_t lik_f64_qpart_elems(int d, int K, int rows) { return (size_t)rows * K * ((d + BN - 1) / BN); }

size_t lik_f64_group_elems(int K, int rows) { return 4 * (size_t)rows + 3 * (size_t)K * rows + 3 * (size_t)K + 4; }

namespace {
template <int SRC, bool STORE_Z>
void z_all(const LikF64Args &a, int jt0, int njt, cudaStream_t s) {
    const dim3 g((a.n_rows + BM - 1) / BM, njt, a.K);
    ProfScope prof(PROF_F64_Z, s);
    note_launch();
    k_zgemm_f64<SRC, STORE_Z><<<g, NT, 0, s>>>(a, jt0);
}

// The listed rows (at most `total` over the K lists, whose last tiles may be short).
template <bool STORE_Z, int R>
void z_listed(const LikF64Args &a, int njt, const int32_t *list, const int32_t *cnt, long long total,
              cudaStream_t s) {
    const long long tiles = total / (8 * R) + a.K;
    ProfScope prof(PROF_F64_Z, s);
    note_launch();
    k_zgemm_f64_listed<STORE_Z, R><<<dim3((unsigned)(tiles < 1216 ? tiles : 1216), njt), NT, 0, s>>>(a, list, cnt);
}

// l (and grad l when a.G is given) in groups of rows per component.
template <bool GRAD>
void points_grouped(const LikF64Args &a, cudaStream_t s) {
    const int n = a.n_rows, K = a.K, nJT = (a.d + BN - 1) / BN;
    const Lists L = lists_of(a.grp, n, K);
    cudaMemsetAsync(L.c1, 0, sizeof(int32_t) * (3 * K + 1), s);
    const unsigned gr = (unsigned)((n + 127) / 128);
    z_all<SRC_GATHER, GRAD>(a, nJT - 1, 1, s);
    note_launch();
    k_grp_lead<<<gr, 128, 0, s>>>(a, L);
    z_listed<GRAD, 4>(a, nJT - 1, L.l1, L.c1, n, s);
    note_launch();
    k_grp_need<<<gr, 128, 0, s>>>(a, L);
    z_listed<GRAD, 1>(a, nJT - 1, L.l2, L.c2, (long long)(K - 1) * n, s);
    note_launch();
    k_lse_f64<true><<<gr, 128, 0, s>>>(a, L);
    if (!GRAD) return;
    ProfScope prof(PROF_F64_GRAD, s);
    note_launch();
    const int n_multi = (n + 7) / 8 < 608 ? (n + 7) / 8 : 608;
    // unused shared memory holds an SM to two CTAs, so that the tiles, up to nJT times
    // different in length, are dealt out as SMs come free (all resident at once: 484 us at
    // 4096 points, d = 256, K = 4, 304 us so; 287 us of FP64 instructions)
    constexpr int kPad = 96 * 1024;
    const int pad = allow_smem(k_ggemm_f64_grouped, kPad) == cudaSuccess ? kPad : 0;
    k_ggemm_f64_grouped<<<dim3(n_multi + n / BM + K, nJT), NT, pad, s>>>(a, L, n_multi);
}
}  // namespace

void launch_lik_f64_z(const LikF64Args &a, cudaStream_t s) {
    if (a.n_rows <= 0) return;
    z_all<SRC_GATHER, true>(a, 0, (a.d + BN - 1) / BN, s);
}

void launch_lik_f64_rays(const LikF64Args &a, cudaStream_t s) {
    if (a.n_rows <= 0) return;
    if (small_f64_fits(a.d, a.K, 0)) return launch_small_points_f64(a, true, s);
    z_all<SRC_RAYS, false>(a, 0, (a.d + BN - 1) / BN, s);
    note_launch();
    k_lse_f64<false><<<(a.n_rows + 127) / 128, 128, 0, s>>>(a, Lists{});
}

// Routes: small problems whole in shared memory (small_f64.cu); several components over
// several column blocks and at least kGroupMinRows rows in groups per component (when the
// caller gives the scratch); else every row and component.
void launch_lik_f64_points(const LikF64Args &a0, bool want_grad, cudaStream_t s) {
    if (a0.n_rows <= 0) return;
    LikF64Args a = a0;
    if (!want_grad) a.G = nullptr;
    if (small_f64_fits(a.d, a.K, 0)) return launch_small_points_f64(a, false, s);
    const int nJT = (a.d + BN - 1) / BN;
    if (a.grp && a.K >= 2 && nJT >= 2 && a.n_rows >= kGroupMinRows)
        return want_grad ? points_grouped<true>(a, s) : points_grouped<false>(a, s);
    if (want_grad)
        z_all<SRC_GATHER, true>(a, 0, nJT, s);
    else
        z_all<SRC_GATHER, false>(a, 0, nJT, s);
    note_launch();
    k_lse_f64<false><<<(a.n_rows + 127) / 128, 128, 0, s>>>(a, Lists{});
    if (!want_grad) return;
    ProfScope prof(PROF_F64_GRAD, s);
    note_launch();
    k_ggemm_f64<<<dim3((a.n_rows + BM - 1) / BM, nJT), NT, 0, s>>>(a);
}

}  // namespace sb

namespace sb {
void launch_lik_f64_few(const LikF64Args &a, bool want_grad, cudaStream_t s) {
    if (a.n_rows <= 0) return;
    const int nJT = (a.d + 63) / 64;
    const int cb = (a.n_rows + 7) / 8;
    {
        ProfScope prof(PROF_F64_Z, s);
        note_launch();
        k_few_z<<<dim3(nJT, a.K, cb), 256, 0, s>>>(a);
    }
    note_launch();
    k_lse_f64<false><<<(a.n_rows + 127) / 128, 128, 0, s>>>(a, Lists{});
    if (want_grad) {
        ProfScope prof(PROF_F64_GRAD, s);
        note_launch();
        k_few_g<<<dim3((a.d + 7) / 8, cb), 256, 0, s>>>(a);
    }
}
}  // namespace sb
