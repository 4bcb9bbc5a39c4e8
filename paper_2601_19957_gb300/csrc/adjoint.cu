// adjoint.cu -- FP64 adjoint of log Z with respect to the component means and
// precision Cholesky factors (mu_k, L_k), for torch.autograd.
//
// log Z = LSE_m log Z_m - log V with log Z_m = l(x*_m) + (d/2) log 2pi - 1/2 log det H_m
// (Sec. 3.7.1, App. A.3, A.8) and x*_m a stationary point of l. With
// pi_m = softmax_m log Z_m and W = H^-1 at x*:
//
//   d log Z_m / d phi = d/dphi [ l - 1/2 log det H - 1/2 v^T grad l ]   (x = x*, v held fixed)
//   v = W t,  t = grad_x log det H = (tr(W dH/dx_i))_i
//
// The last term is the implicit shift of the mode, dx*/dphi = W d(grad l)/dphi,
// which moves log det H (l itself is stationary). Reverse-mode through the
// mixture pieces at x (delta_k = x - mu_k, z_k = L_k^T delta_k, r = softmax(e),
// g_k = -L_k z_k, gbar = sum r_k g_k, H = sum_k r_k (P_k - g_k g_k^T) + gbar gbar^T):
//
//   c       = -W gbar - v/2
//   beta_k  = -1/2 [tr(W P_k) - g_k^T W g_k] + c^T g_k
//   eps_k   = r_k + r_k (beta_k - sum_j r_j beta_j)                       (adjoint of e_k)
//   gam_k   = r_k (W g_k + c)                                             (adjoint of g_k)
//   dmu_k   = -eps_k g_k + P_k gam_k
//   dL_k    = lower[ eps_k (diag(1/L_ii) - delta_k z_k^T) - gam_k z_k^T - delta_k (L_k^T gam_k)^T - r_k W L_k ]
//
// and t from the same reverse pass applied to log det H alone:
//   beta'_k = tr(W P_k) - g_k^T W g_k + 2 gbar^T W g_k,  eps'_k = r_k (beta'_k - sum_j r_j beta'_j)
//   gam'_k  = 2 r_k W (gbar - g_k),  t = sum_k (eps'_k g_k - P_k gam'_k).
// tr(W P_k) = <W L_k, L_k>_F. Components with r_k == 0 contribute exactly zero
// and are skipped. H is recomputed at every mode (not stored by the forward),
// factored H = C C^T, and C^-1 is formed once (its 32 x 32 diagonal blocks by
// substitution, then pairs of blocks merged level by level) for the vectors, W v = C^-T (C^-1
// v); W L_k comes from triangular solves (k_adj_solve says why). At a one-hot mode (r_k = 1, the other r
// exactly 0) H = P_k and C = L_k, so W L_k = L_k^-T: tr(W P_k) = d and lower[W L_k] =
// diag(1 / L_ii), with no solve. Products with P_k are formed as L_k (L_k^T v); P_k itself
// is built only for the Hessian of a mode that is not one-hot. Nothing is read back to
// the host: every skip is decided from R and the one-hot flag on the device. Modes go
// through the kernels in groups (adjoint_group), since one mode's factor, inverse and vector
// steps leave most of the chip idle; their shares are added to dmu and dL in mode order.
//
// The bound is the FP64 pipe (one warp instruction per 19 cycles and SM): per mode K d^3 /
// 3 fused multiply-adds in the two solves, d^3 / 6 each in the factor and its inverse.
#include "sb_adjoint.cuh"

namespace sb {

namespace {

constexpr int TB = 32;  // output tile and K chunk of the GEMMs, block of the inverse's first level

// ------------------------------------------------------------------ C^-1 and the GEMMs
// 32 x 32 output tiles, 256 threads with 2 x 2 outputs each, K chunks of 32: the longest
// tile (a whole row of the triangle) is then d warp instructions per warp and output pair,
// a sixth of the GEMM's time at d = 512; 64 x 64 tiles would put half of it on one SM.
struct TileBuf {
    double A[TB][TB + 1], B[TB][TB + 1];
};

// acc += sum over l in [l0, l1) of a(i, l) b(l, j) for the tile's rows i0 + ty (+16) and columns j0 + tx (+16);
// a and b return zero outside their triangles.
template <typename FA, typename FB>
__device__ __forceinline__ void tile_gemm(TileBuf &sm, int l0, int l1, double (&acc)[2][2], FA a, FB b) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int l = l0; l < l1; l += TB) {
#pragma unroll
        for (int e = tid; e < TB * TB; e += 256) {
            const int r = e >> 5, c = e & 31;
            sm.A[r][c] = a(r, l + c);  // A[row][l]
            sm.B[r][c] = b(l + r, c);  // B[l][column]
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TB; ++q) {
            const double a0 = sm.A[ty][q], a1 = sm.A[ty + 16][q];
            const double b0 = sm.B[q][tx], b1 = sm.B[q][tx + 16];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
        __syncthreads();
    }
}

// The inverses of the 32 x 32 diagonal blocks of C (identity past d): a warp per four
// columns, lanes over rows, multiplication by the diagonal's reciprocals. (The merges fill
// the blocks below; those above the diagonal are not read.)
__global__ void __launch_bounds__(256) k_inv_diag(int d, const double *C, double *Ci) {
    __shared__ double Cs[TB][TB + 1];
    __shared__ double inv[TB];
    const int r0 = blockIdx.x * TB;
    C += (size_t)blockIdx.y * d * d;  // mode
    Ci += (size_t)blockIdx.y * d * d;
    for (int e = threadIdx.x; e < TB * TB; e += 256) {
        const int i = r0 + e / TB, j = r0 + e % TB;
        Cs[e / TB][e % TB] = i < d && j <= i ? C[(size_t)i * d + j] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    if (threadIdx.x < TB) inv[threadIdx.x] = 1.0 / Cs[threadIdx.x][threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = lane == wid * 4 + q ? 1.0 : 0.0;
    for (int i = wid * 4; i < TB; ++i) {  // rows above the warp's columns stay zero
        const double c = lane > i ? Cs[lane][i] : 0.0, iv = inv[i];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double xi = __shfl_sync(0xffffffffu, b[q], i) * iv;
            b[q] = lane == i ? xi : fma(-c, xi, b[q]);
        }
    }
    const int i = r0 + lane;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = r0 + wid * 4 + q;
        if (i < d && j < d) Ci[(size_t)i * d + j] = b[q];
    }
}

// One level of the merge [A 0; B D]^-1 = [A^-1 0; -D^-1 B A^-1, D^-1] for every pair of
// blocks of s rows and mode (blockIdx.z): pass 0 T = B A^-1, pass 1 Ci = -D^-1 T.
template <int PASS>
__global__ void __launch_bounds__(256) k_inv_merge(int d, int s, const double *C, double *Ci, double *T) {
    __shared__ TileBuf sm;
    const int pairs = (d + 2 * s - 1) / (2 * s), mo = blockIdx.z / pairs;
    C += (size_t)mo * d * d;
    Ci += (size_t)mo * d * d;
    T += (size_t)mo * d * d;
    const int p0 = (blockIdx.z % pairs) * 2 * s, q0 = p0 + s;  // first rows of the A and the D block
    const int i0 = q0 + blockIdx.y * TB, j0 = p0 + blockIdx.x * TB;
    if (i0 >= d) return;
    double acc[2][2] = {};
    if (PASS == 0) {
        tile_gemm(
            sm, j0, q0, acc, [&](int r, int l) { return i0 + r < d ? C[(size_t)(i0 + r) * d + l] : 0.0; },
            [&](int l, int c) { return j0 + c <= l ? Ci[(size_t)l * d + j0 + c] : 0.0; });
    } else {
        tile_gemm(
            sm, q0, min(d, i0 + TB), acc,
            [&](int r, int l) { return i0 + r < d && l <= i0 + r ? Ci[(size_t)(i0 + r) * d + l] : 0.0; },
            [&](int l, int c) { return l < d ? T[(size_t)l * d + j0 + c] : 0.0; });
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int i = i0 + ty + 16 * r, j = j0 + tx + 16 * c;
            if (i < d) (PASS == 0 ? T : Ci)[(size_t)i * d + j] = PASS == 0 ? acc[r][c] : -acc[r][c];
        }
}

void launch_tri_inverse(int d, int nm, const double *C, double *Ci, double *T, cudaStream_t st) {
    note_launch();
    k_inv_diag<<<dim3((d + TB - 1) / TB, nm), 256, 0, st>>>(d, C, Ci);
    for (int s = TB; s < d; s *= 2) {
        const int pairs = (d + 2 * s - 1) / (2 * s);
        const dim3 g(s / TB, s / TB, pairs * nm);
        note_launch();
        k_inv_merge<0><<<g, 256, 0, st>>>(d, s, C, Ci, T);
        note_launch();
        k_inv_merge<1><<<g, 256, 0, st>>>(d, s, C, Ci, T);
    }
}

// Whether W L_k is formed for component k: r_k > 0 and the mode is not one-hot.
__device__ __forceinline__ bool needs_product(const double *R, const int32_t *onehot, int k) {
    return R[k] != 0.0 && onehot[0] < 0;
}

// W L_k = C^-T (C^-1 L_k) by triangular solves, rows from each column's own block down (the
// lower triangle is all that is used).
// One CTA takes 16 columns of one component and mode through both solves: per 32-row block
// the products with the blocks solved before are subtracted one after the other (each summed
// from zero), then the diagonal block is solved by substitution. Near a one-hot mode
// eps / L_ii - r (W L_k)_ii and its off-diagonal part cancel to about r_j of another
// component, 1e-5 to 1e-8 of the terms, so the rounding of these solves shows in dL_k: the
// products with an explicit C^-1 take as long at d = 512, but their dL lies up to 1.5e-9 of
// its norm from that of the solves.
// Bound by the FP64 pipe: two outputs per thread; in the substitution a warp takes two columns,
// lane = (column, row of a half block), 80 warp instructions instead of 128 with a row per
// lane. 16 columns, not 32, because the first column tile is the longest chain of all, and
// two CTAs per SM (unused shared memory), so that the chains, which differ in length by nb
// squared, are dealt out as SMs come free, the longest first. d = 512, K = 4, four modes:
// 2.0 ms (2.06 for the two products).
constexpr int SC = 16;  // columns per CTA
__global__ void __launch_bounds__(256) k_adj_solve(int d, int K, const double *C, const double *L, const double *R,
                                                   const int32_t *onehot, double *X) {
    __shared__ double As[TB][TB + 1];
    __shared__ double Xs[TB][SC + 1];
    __shared__ double Bs[TB][SC + 1];
    __shared__ double inv[TB];
    const int k = blockIdx.x % K, mo = blockIdx.x / K;
    if (!needs_product(R + (size_t)mo * K, onehot + mo, k)) return;
    C += (size_t)mo * d * d;
    X += ((size_t)mo * K + k) * d * d;
    const double *Lk = L + (size_t)k * d * d;
    const int c0 = blockIdx.y * SC, I0 = c0 / TB, nb = (d + TB - 1) / TB;
    const int tid = threadIdx.x, tc = tid & (SC - 1), tr = tid / SC;  // rows tr and tr + 16
    const int lane = tid & 31, wid = tid >> 5;
    // the block (I, J) of C, or of C^T for upper, into registers: A[i][q] of the product;
    // and rows of X block J
    auto load = [&](int I, int J, bool upper, double (&a)[4], double (&x)[2]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = (tid >> 5) + 8 * e;
            const int gi = (upper ? J : I) * TB + r, gj = (upper ? I : J) * TB + lane;
            a[e] = gi < d && gj < d ? C[(size_t)gi * d + gj] : 0.0;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int gr = J * TB + tr + 16 * e;
            x[e] = gr < d && c0 + tc < d ? X[(size_t)gr * d + c0 + tc] : 0.0;
        }
    };
    for (int pass = 0; pass < 2; ++pass) {
        const bool upper = pass;
        for (int s = I0; s < nb; ++s) {
            const int I = upper ? nb - 1 - (s - I0) : s, step = upper ? -1 : 1;
            double b[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int gi = I * TB + tr + 16 * e, gc = c0 + tc;
                b[e] = 0.0;
                if (gi < d && gc < d) b[e] = upper ? X[(size_t)gi * d + gc] : gc <= gi ? Lk[(size_t)gi * d + gc] : 0.0;
            }
            double dinv = 1.0;
            if (wid == 0 && I * TB + lane < d) dinv = 1.0 / C[(size_t)(I * TB + lane) * (d + 1)];
            double a[4], x[2];
            int J = upper ? nb - 1 : I0;
            if (J != I) load(I, J, upper, a, x);
            for (; J != I; J += step) {
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = (tid >> 5) + 8 * e;
                    As[upper ? lane : r][upper ? r : lane] = a[e];
                }
                Xs[tr][tc] = x[0];
                Xs[tr + 16][tc] = x[1];
                __syncthreads();
                if (J + step != I) load(I, J + step, upper, a, x);
                double acc[2] = {};
#pragma unroll
                for (int q = 0; q < TB; ++q) {
                    const double xq = Xs[q][tc];
                    acc[0] = fma(As[tr][q], xq, acc[0]);
                    acc[1] = fma(As[tr + 16][q], xq, acc[1]);
                }
                b[0] -= acc[0];
                b[1] -= acc[1];
            }
            // the diagonal block (identity past d)
            __syncthreads();
            for (int e = tid; e < TB * TB; e += 256) {
                const int r = e / TB, c = e % TB, gi = I * TB + r, gj = I * TB + c;
                const double v = gi < d && gj < d ? C[(size_t)gi * d + gj] : r == c ? 1.0 : 0.0;
                As[upper ? c : r][upper ? r : c] = v;
            }
            if (wid == 0) inv[lane] = dinv;
            Bs[tr][tc] = b[0];
            Bs[tr + 16][tc] = b[1];
            __syncthreads();
            {
                const int col = 2 * wid + (lane >> 4), r = lane & 15, base = lane & 16;
                double lo = Bs[r][col], hi = Bs[r + 16][col];  // rows r and r + 16
                if (!upper) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const double xi = __shfl_sync(0xffffffffu, lo, base | i) * inv[i];
                        const double t = fma(-As[r][i], xi, lo);
                        lo = r == i ? xi : r > i ? t : lo;
                        hi = fma(-As[r + 16][i], xi, hi);
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const double xi = __shfl_sync(0xffffffffu, hi, base | i) * inv[i + 16];
                        const double t = fma(-As[r + 16][i + 16], xi, hi);
                        hi = r == i ? xi : r > i ? t : hi;
                    }
                } else {
#pragma unroll
                    for (int i = 15; i >= 0; --i) {
                        const double xi = __shfl_sync(0xffffffffu, hi, base | i) * inv[i + 16];
                        const double t = fma(-As[r + 16][i + 16], xi, hi);
                        hi = r == i ? xi : r < i ? t : hi;
                        lo = fma(-As[r][i + 16], xi, lo);
                    }
#pragma unroll
                    for (int i = 15; i >= 0; --i) {
                        const double xi = __shfl_sync(0xffffffffu, lo, base | i) * inv[i];
                        const double t = fma(-As[r][i], xi, lo);
                        lo = r == i ? xi : r < i ? t : lo;
                    }
                }
                Bs[r][col] = lo;
                Bs[r + 16][col] = hi;
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int gi = I * TB + tr + 16 * e, gc = c0 + tc;
                const double v = Bs[tr + 16 * e][tc];
                if (gi < d && gc < d) X[(size_t)gi * d + gc] = v;
            }
            __syncthreads();  // the rows are written before a later block reads them
        }
    }
}

// tr(W P_k) = <W L_k, L_k>_F over the lower triangle, a CTA per component and mode. About d in
// size, and at the mode's own component eps_k is what remains of it after the cancellation
// above, so it is one sum in a fixed order, 130 us at d = 512.
__global__ void __launch_bounds__(256) k_adj_trace(int d, int K, const double *X, const double *L, const double *R,
                                                   const int32_t *onehot, double *tr) {
    __shared__ double sh[8];
    const int k = blockIdx.x % K, mo = blockIdx.x / K;
    if (!needs_product(R + (size_t)mo * K, onehot + mo, k)) return;
    X += ((size_t)mo * K + k) * d * d;
    L += (size_t)k * d * d;
    constexpr int kBatch = 32;  // loads in flight per thread and matrix
    const int di = 256 / d, dj = 256 % d;
    int i = threadIdx.x / d, j = threadIdx.x % d;
    double s = 0.0;
    while (i < d) {
        double a[kBatch], b[kBatch];
        bool in[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            in[q] = i < d && j <= i;
            a[q] = in[q] ? X[(size_t)i * d + j] : 0.0;
            b[q] = in[q] ? L[(size_t)i * d + j] : 0.0;
            i += di;
            j += dj;
            if (j >= d) {
                j -= d;
                ++i;
            }
        }
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
            if (__any_sync(__activemask(), in[q])) s = in[q] ? fma(a[q], b[q], s) : s;
    }
    __syncwarp();
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        tr[blockIdx.x] = t;
    }
}

// dL_k += pi lower[ eps (diag(1/L) - delta z^T) - gam z^T - delta u^T - r W L_k ] with u =
// L^T gam (at a one-hot mode lower[W L_k] = diag(1 / L_ii)), the modes in order.
__global__ void __launch_bounds__(256) k_adj_dL(int d, int nm, const double *pi, const double *R, const double *eps,
                                                const int32_t *onehot, const double *L, const double *x,
                                                const double *mu, const double *Z, const double *gam,
                                                const double *U, const double *X, double *dL) {
    const int k = blockIdx.z, K = gridDim.z, i = blockIdx.y, j = blockIdx.x * 256 + threadIdx.x;
    if (j > i) return;
    const size_t e = (size_t)i * d + j, ek = (size_t)k * d * d + e;
    double sum = dL[ek];
    for (int mo = 0; mo < nm; ++mo) {
        const size_t mk = (size_t)mo * K + k, kd = mk * d;
        const double rk = R[mk];
        if (rk == 0.0) continue;
        const double ep = eps[mk], di = x[(size_t)mo * d + i] - mu[(size_t)k * d + i], zj = Z[kd + j];
        const double wl = onehot[mo] >= 0 ? (i == j ? 1.0 / L[ek] : 0.0) : X[mk * d * d + e];
        double v = -ep * di * zj - gam[kd + i] * zj - di * U[kd + j] - rk * wl;
        if (i == j) v += ep / L[ek];
        sum += pi[mo] * v;
    }
    dL[ek] = sum;
}

// ------------------------------------------------------------------ per-mode vector algebra
// Vectors are rows of [mode][nv][d]. Rows of V: 0 .. K-1 = g_k (active only, else 0), K = gbar.
__global__ void k_pack_rhs(int d, int K, const double *GK, const double *gbar, const double *R, double *V) {
    const int c = blockIdx.y, mo = blockIdx.z;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d) return;
    double v = gbar[(size_t)mo * d + i];
    if (c < K) v = R[(size_t)mo * K + c] != 0.0 ? GK[((size_t)mo * K + c) * d + i] : 0.0;
    V[((size_t)mo * (K + 1) + c) * d + i] = v;
}

// Where a vector kernel finds its operands: matrix T + mode tm + vector tc, vectors
// V + mode vm + vector d (skipped where R[mode rm + c] == 0, c < K).
struct VecArgs {
    const double *T;
    size_t tm, tc;
    const double *V;
    size_t vm;
    const double *R;
    int K;
    double *Y;
    size_t ym;
};

// y = T v for a lower triangular matrix, a warp per row; vector c = blockIdx.y, mode blockIdx.z.
__global__ void __launch_bounds__(256) k_adj_lower(int d, VecArgs a) {
    const int c = blockIdx.y, mo = blockIdx.z;
    if (a.R && c < a.K && a.R[(size_t)mo * a.K + c] == 0.0) return;
    const int lane = threadIdx.x & 31, i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= d) return;
    const double *row = a.T + mo * a.tm + c * a.tc + (size_t)i * d, *v = a.V + mo * a.vm + (size_t)c * d;
    double s = 0.0;
#pragma unroll 4
    for (int j = lane; j <= i; j += 32) s = fma(row[j], v[j], s);
    s = warp_sum(s);
    if (lane == 0) a.Y[mo * a.ym + (size_t)c * d + i] = s;
}

// dmu_k += pi (-eps_k g_k + y_k) with y_k = L_k u_k, the group's modes in turn: a warp per (i, k).
__global__ void __launch_bounds__(256) k_adj_dmu(int d, int nm, const double *L, const double *U, const double *R,
                                                 const double *pi, const double *eps, const double *GK, double *dmu) {
    const int k = blockIdx.y, K = gridDim.y;
    const int lane = threadIdx.x & 31, i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= d) return;
    const double *row = L + (size_t)k * d * d + (size_t)i * d;
    double sum = dmu[(size_t)k * d + i];
    for (int mo = 0; mo < nm; ++mo) {
        const size_t mk = (size_t)mo * K + k;
        if (R[mk] == 0.0) continue;
        const double *v = U + mk * d;
        double s = 0.0;
#pragma unroll 4
        for (int j = lane; j <= i; j += 32) s = fma(row[j], v[j], s);
        s = warp_sum(s);
        sum += pi[mo] * (-eps[mk] * GK[mk * d + i] + s);
    }
    if (lane == 0) dmu[(size_t)k * d + i] = sum;
}

// y = T^T v (diff: v = gbar row - v, the row K of the same mode): a CTA per 32 columns, a lane per column, the eight
// warps over interleaved rows, partials summed in a fixed order.
__global__ void __launch_bounds__(256) k_adj_upper(int d, VecArgs a, bool diff) {
    __shared__ double part[8][32];
    const int c = blockIdx.y, mo = blockIdx.z;
    if (a.R && c < a.K && a.R[(size_t)mo * a.K + c] == 0.0) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, j0 = blockIdx.x * 32, j = j0 + lane;
    const double *Tc = a.T + mo * a.tm + c * a.tc, *v = a.V + mo * a.vm + (size_t)c * d;
    const double *w = a.V + mo * a.vm + (size_t)a.K * d;
    double s = 0.0;
    if (j < d) {
#pragma unroll 4
        for (int i = j0 + wid; i < d; i += 8) {
            const double t = i >= j ? Tc[(size_t)i * d + j] : 0.0;
            s = fma(t, diff ? w[i] - v[i] : v[i], s);
        }
    }
    part[wid][lane] = s;
    __syncthreads();
    if (wid == 0 && j < d) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) t += part[q][lane];
        a.Y[mo * a.ym + (size_t)c * d + j] = t;
    }
}

// One CTA of 1024 threads per mode: given WV (rows W g_0 .. W g_{K-1}, W gbar) and
// tr(W P_k), form t (stage 0), or with Wt known form eps and gam (stage 1). A warp per
// component for the inner products.
__global__ void __launch_bounds__(1024) k_adj_stage(int stage, int d, int K, const double *R,
                                                    const int32_t *onehot, const double *GK, const double *gbar,
                                                    const double *WV, const double *trp, const double *PY,
                                                    const double *Wt, double *t_out, double *eps, double *gam) {
    __shared__ double s_beta[kMaxK];
    const int mo = blockIdx.x;
    R += (size_t)mo * K;
    GK += (size_t)mo * K * d;
    gbar += (size_t)mo * d;
    WV += (size_t)mo * (K + 1) * d;
    trp += (size_t)mo * K;
    if (stage == 0) {
        PY += (size_t)mo * K * d;
        t_out += (size_t)mo * d;
    } else {
        Wt += (size_t)mo * d;
        eps += (size_t)mo * K;
        gam += (size_t)mo * K * d;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double *Wg = WV + (size_t)K * d;  // W gbar
    const bool oh = onehot[mo] >= 0;
    for (int k = wid; k < K; k += 32) {
        double beta = 0.0;
        if (R[k] != 0.0) {
            const double *gk = GK + (size_t)k * d, *wgk = WV + (size_t)k * d;
            double a1 = 0.0, a2 = 0.0;
            for (int i = lane; i < d; i += 32) {
                a1 = fma(gk[i], wgk[i], a1);  // g_k^T W g_k
                // gbar^T W g_k, or c^T g_k with c = -W gbar - W t / 2
                a2 = stage == 0 ? fma(gbar[i], wgk[i], a2) : fma(fma(-0.5, Wt[i], -Wg[i]), gk[i], a2);
            }
            a1 = warp_sum(a1);
            a2 = warp_sum(a2);
            const double tr = oh ? (double)d : trp[k];
            beta = stage == 0 ? (tr - a1 + 2.0 * a2) : (-0.5 * (tr - a1) + a2);
        }
        if (lane == 0) s_beta[k] = beta;
    }
    __syncthreads();
    double sb = 0.0;
    for (int k = 0; k < K; ++k) sb += R[k] * s_beta[k];
    if (stage == 0) {
        // t = sum_k eps'_k g_k - P_k gam'_k,  gam'_k = 2 r_k W (gbar - g_k)
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            double ti = 0.0;
            for (int k = 0; k < K; ++k) {
                const double r = R[k];
                if (r == 0.0) continue;
                const double e1 = r * (s_beta[k] - sb);
                ti += e1 * GK[(size_t)k * d + i];
                // (P_k gam'_k)_i = 2 r (P_k (W gbar - W g_k))_i, formed apart (PY)
                ti -= 2.0 * r * PY[(size_t)k * d + i];
            }
            t_out[i] = ti;
        }
    } else {
        if ((int)threadIdx.x < K) {
            const int k = threadIdx.x;
            eps[k] = R[k] == 0.0 ? 0.0 : R[k] + R[k] * (s_beta[k] - sb);
        }
        for (int i = threadIdx.x; i < d; i += blockDim.x) {
            const double c = -Wg[i] - 0.5 * Wt[i];
            for (int k = 0; k < K; ++k) gam[(size_t)k * d + i] = R[k] == 0.0 ? 0.0 : R[k] * (WV[(size_t)k * d + i] + c);
        }
    }
}

__global__ void k_softmax_pi(int n, const double *logZk, double g, double *pi) {
    if (threadIdx.x != 0) return;
    double mx = -INFINITY;
    for (int i = 0; i < n; ++i) mx = fmax(mx, logZk[i]);
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += exp(logZk[i] - mx);
    for (int i = 0; i < n; ++i) pi[i] = g * exp(logZk[i] - mx) / s;
}

}  // namespace

int adjoint_group(int K) {
    const int g = 32 / K;
    return g < 1 ? 1 : (g > 4 ? 4 : g);
}

void adjoint_carve(Carver &cv, AdjWs &w, int d, int K, int group) {
    const size_t nJT = (d + 63) / 64, dd = (size_t)d * d, g = group > 0 ? group : 1;
    w.group = (int)g;
    w.P = cv.take<double>(K * dd);
    w.H = cv.take<double>(g * dd);
    w.Ci = group > 0 ? cv.take<double>(g * dd) : w.P;
    w.X = cv.take<double>(g * K * dd);
    w.trp = cv.take<double>(g * K);
    w.Z = cv.take<double>(g * K * d);
    w.R = cv.take<double>(g * K);
    w.qpart = cv.take<double>(g * K * nJT);
    w.gbar = cv.take<double>(g * d);
    w.ell = cv.take<double>(g);
    w.GK = cv.take<double>(g * K * d);
    w.V = cv.take<double>(g * d * (K + 1));
    w.Y = cv.take<double>(g * d * (K + 1));
    w.T = cv.take<double>(g * d);
    w.eps = cv.take<double>(g * K);
    w.gam = cv.take<double>(g * K * d);
    w.pi = cv.take<double>(kMaxAdjModes);
    w.info = cv.take<int32_t>(g);
    w.count = cv.take<int32_t>(1);
    w.onehot = cv.take<int32_t>(g);
    w.p_done = cv.take<int32_t>(kMaxK);
    w.p_need = cv.take<int32_t>(kMaxK);
    w.bar = cv.take<uint32_t>(2);
}

__global__ void k_set_count(int32_t *p, int v) {
    if (threadIdx.x == 0) *p = v;
}

sb_status adjoint_run(const ProbView &pv, const AdjWs &w, const double *modes, const double *logZk, int n_modes,
                      double grad_logZ, double *dmu, double *dL, cudaStream_t s) {
    const int d = pv.d, K = pv.K, group = w.group;
    if (n_modes < 1 || n_modes > kMaxAdjModes) return SB_ERR_INVALID_ARG;
    SB_CUDA_TRY(cudaMemsetAsync(dmu, 0, sizeof(double) * K * d, s));
    SB_CUDA_TRY(cudaMemsetAsync(dL, 0, sizeof(double) * (size_t)K * d * d, s));
    SB_CUDA_TRY(cudaMemsetAsync(w.p_done, 0, sizeof(int32_t) * kMaxK, s));
    note_launch();
    k_softmax_pi<<<1, 32, 0, s>>>(n_modes, logZk, grad_logZ, w.pi);
    const int tiles = (d + SC - 1) / SC;
    const unsigned rows8 = (unsigned)((d + 7) / 8), cols32 = (unsigned)((d + 31) / 32);
    const size_t dd = (size_t)d * d, dK = (size_t)d * K, dV = (size_t)d * (K + 1);
    constexpr int kPad = 80 * 1024;  // two CTAs of k_adj_solve per SM
    SB_CUDA_TRY(cudaFuncSetAttribute(k_adj_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, kPad));
    for (int m0 = 0; m0 < n_modes; m0 += group) {
        const int nm = n_modes - m0 < group ? n_modes - m0 : group;
        const double *x = modes + (size_t)m0 * d;
        const double *pi = w.pi + m0;
        if (w.Ci == w.P) SB_CUDA_TRY(cudaMemsetAsync(w.p_done, 0, sizeof(int32_t) * kMaxK, s));
        note_launch();
        k_set_count<<<1, 32, 0, s>>>(w.count, nm);
        // W v for the nv vectors per mode of V (stride vm; those with R == 0 skipped, zero and unread)
        auto apply_W = [&](int nv, const double *V, size_t vm, double *out, size_t om, const double *R) {
            note_launch(2);
            k_adj_lower<<<dim3(rows8, nv, nm), 256, 0, s>>>(d, VecArgs{w.Ci, dd, 0, V, vm, R, K, w.Y, dV});
            k_adj_upper<<<dim3(cols32, nv, nm), 256, 0, s>>>(d, VecArgs{w.Ci, dd, 0, w.Y, dV, R, K, out, om}, false);
        };
        // l, grad l, z_k, r_k at x (FP64 likelihood kernels), then g_k, H and H = C C^T
        // (at a one-hot mode C = L_k is copied, as in the Laplace stage), C^-1
        LikF64Args la{};
        la.d = d;
        la.K = K;
        la.mu = pv.mu;
        la.L = pv.L;
        la.a = pv.a;
        la.X = x;
        la.n_rows = nm;
        la.qpart = w.qpart;
        la.Z = w.Z;
        la.R = w.R;
        la.ell = w.ell;
        la.ell_sign = 1.0;
        la.G = w.gbar;
        la.grad_sign = -1.0;
        la.out_by_walker = 0;
        launch_lik_f64_few(la, true, s);
        launch_onehot(K, w.R, w.count, nm, w.onehot, s);
        launch_precision_needed(d, K, pv.L, w.R, w.count, w.p_done, w.p_need, w.P, s, w.onehot);
        launch_hessian_chol(d, K, nm, pv.L, w.P, w.Z, w.R, w.gbar, w.count, w.GK, w.H, w.info, w.bar, pv.status, s,
                            w.onehot, true);
        launch_tri_inverse(d, nm, w.H, w.Ci, w.X, s);
        // W [g_0 .. g_{K-1}, gbar] in place; X_k = W L_k and tr(W P_k)
        note_launch();
        k_pack_rhs<<<dim3((d + 255) / 256, K + 1, nm), 256, 0, s>>>(d, K, w.GK, w.gbar, w.R, w.V);
        apply_W(K + 1, w.V, dV, w.V, dV, w.R);
        note_launch();
        k_adj_solve<<<dim3(K * nm, tiles), 256, kPad, s>>>(d, K, w.H, pv.L, w.R, w.onehot, w.X);
        note_launch();
        k_adj_trace<<<K * nm, 256, 0, s>>>(d, K, w.X, pv.L, w.R, w.onehot, w.trp);
        // P_k (W gbar - W g_k) = L_k (L_k^T (W gbar - W g_k))
        note_launch(2);
        k_adj_upper<<<dim3(cols32, K, nm), 256, 0, s>>>(d, VecArgs{pv.L, 0, dd, w.V, dV, w.R, K, w.Y, dK}, true);
        k_adj_lower<<<dim3(rows8, K, nm), 256, 0, s>>>(d, VecArgs{pv.L, 0, dd, w.Y, dK, w.R, K, w.gam, dK});
        // t = grad_x log det H, then v = W t in place, then c, eps_k, gam_k
        note_launch();
        k_adj_stage<<<nm, 1024, 0, s>>>(0, d, K, w.R, w.onehot, w.GK, w.gbar, w.V, w.trp, w.gam, nullptr, w.T,
                                        nullptr, nullptr);
        apply_W(1, w.T, d, w.T, d, nullptr);
        note_launch();
        k_adj_stage<<<nm, 1024, 0, s>>>(1, d, K, w.R, w.onehot, w.GK, w.gbar, w.V, w.trp, nullptr, w.T, nullptr,
                                        w.eps, w.gam);
        // u_k = L_k^T gam_k, dmu_k += pi (-eps_k g_k + L_k u_k), dL_k
        note_launch(3);
        k_adj_upper<<<dim3(cols32, K, nm), 256, 0, s>>>(d, VecArgs{pv.L, 0, dd, w.gam, dK, w.R, K, w.Y, dK}, false);
        k_adj_dmu<<<dim3(rows8, K), 256, 0, s>>>(d, nm, pv.L, w.Y, w.R, pi, w.eps, w.GK, dmu);
        k_adj_dL<<<dim3((d + 255) / 256, d, K), 256, 0, s>>>(d, nm, pi, w.R, w.eps, w.onehot, pv.L, x, pv.mu, w.Z,
                                                             w.gam, w.Y, w.X, dL);
    }
    SB_CUDA_TRY(cudaGetLastError());
    SB_CUDA_TRY(cudaStreamSynchronize(s));  // the call returns with its results written
    return SB_OK;
}

}  // namespace sb
