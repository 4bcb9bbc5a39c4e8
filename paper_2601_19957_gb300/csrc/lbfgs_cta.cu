// lbfgs_cta.cu -- FP32 batched L-BFGS step, one CTA per walker (mixed-precision path).
//
// Same state machine as the warp-per-walker kernel (Armijo backtracking,
// history reset and one retry, curvature skip, CONVERGED / STALLED / MAXITER;
// Sec. 3.6.2, App. A.5), but the direction p = -H_k grad f is formed through
// the compact representation of the L-BFGS inverse Hessian (Byrd, Nocedal &
// Schnabel, Math. Prog. 63, 1994, Thm. 2.2):
//
//   H_k = gamma I + [S  gamma Y] [ R^-T (D + gamma Y^T Y) R^-1   -R^-T ] [ S^T       ]
//                               [ -R^-1                          0     ] [ gamma Y^T ]
//
// with S, Y the stored pairs (oldest first), R_ij = s_i^T y_j (i <= j),
// D = diag(s_i^T y_i), gamma = s^T y / y^T y of the newest pair. It is the
// same matrix the two-loop recursion applies (App. A.5), so the direction is
// identical in exact arithmetic; what changes is the data flow. The two-loop
// walks the pairs with a serial dependency (each alpha_i needs the q left by
// the previous pair). Here one pass computes all inner products S^T g, Y^T g
// and the new pair's column of R and row and column of Y^T Y at once
// (independent loads, several pairs in flight), m x m matrix-vector products
// with R^-1 (kept per walker, one new column per appended pair) give the
// coefficients, and a second pass forms p = -gamma g - S a + gamma Y w. R^-1,
// Y^T Y and D live per walker in HBM and are updated incrementally, so the
// history S, Y is read twice per iteration (the second read mostly from L2)
// and never re-walked. The pairs are stored in bf16, and the first pass runs
// on the tensor cores (mma.sync, the pairs as the B operand; g split into
// three bf16 terms).
//
// A walker's step is a chain of dependent phases (reductions, the m x m
// solve), so the SM is kept busy by several walkers at once: CT threads per
// walker, thread t owning the 8 consecutive coordinates from 8 t (one 16-byte
// chunk of a stored bf16 row).
//
// What bounds it at d = 1024, m = 20: HBM for the pairs (4.9 of 6.8 TB/s) and the
// instructions of a visit, 2890 per warp. They were 4570 with the pairs walked in
// the order of their age (a wrap test per row and per entry of the m x m state), one
// FMA per coordinate and a shuffle tree per reduced value: 8192 walkers 235 us, 195 so.
#include <cuda_bf16.h>

#include <mutex>

#include "sb_lbfgs.cuh"

namespace sb {

namespace {

// CT: threads per walker, eight coordinates each, so CT = 32, 64 and 128 serve d <= 256, 512
// and 1024. A visit is a chain of phases whose length hardly depends on d, so what counts is
// the walkers per SM: threads past d would only repeat the chain (with 128 threads for every
// d a batch of 64 problems with d <= 512 took 234 ms, 186 with the width that fits d).
template <int CT>
struct Cfg {
    static constexpr int NW = CT / 32;            // warps per walker
    static constexpr int VPT = 2;                 // float4 groups per thread
    static constexpr int MAXD = 4 * VPT * CT;     // largest d
    static constexpr int MINB = 512 / CT;         // CTAs per SM (registers)
    // ring of the stored pairs: DB slots of PGB pairs (one 8-column tensor-core tile
    // of s, y vectors), each stored row up to MAXD bf16 coordinates plus 16 bytes:
    // row r of a slot starts 16 r bytes further into the 128-byte bank window than
    // row 0, so the same 16-byte chunk of the 8 rows falls in 8 different bank groups
    static constexpr int PGB = 4;
    static constexpr int DB = 3;
    static constexpr int ROW_B = MAXD * 2 + 16;
    static constexpr int SLOT_B = 2 * PGB * ROW_B;
    static constexpr int RING_B = DB * SLOT_B;
};

// Vector accesses need 16-byte aligned rows: d % 4 == 0 (rows start at multiples of d).
__device__ __forceinline__ float4 ld4(const float *p, int i0, int d) {
    if (((d & 3) == 0) && i0 + 3 < d) return *reinterpret_cast<const float4 *>(p + i0);
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 + 0 < d) r.x = p[i0 + 0];
    if (i0 + 1 < d) r.y = p[i0 + 1];
    if (i0 + 2 < d) r.z = p[i0 + 2];
    if (i0 + 3 < d) r.w = p[i0 + 3];
    return r;
}
__device__ __forceinline__ void st4(float *p, int i0, int d, float4 v) {
    if (((d & 3) == 0) && i0 + 3 < d) {
        *reinterpret_cast<float4 *>(p + i0) = v;
        return;
    }
    if (i0 + 0 < d) p[i0 + 0] = v.x;
    if (i0 + 1 < d) p[i0 + 1] = v.y;
    if (i0 + 2 < d) p[i0 + 2] = v.z;
    if (i0 + 3 < d) p[i0 + 3] = v.w;
}
__device__ __forceinline__ float dot4(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }
__device__ __forceinline__ float4 axpy4(float a, float4 x, float4 y) {
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// Per-thread asynchronous copies global -> shared (16 bytes of a stored row, L2 only;
// 4 bytes of the m x m state). A thread completes its own copy groups
// (cp.async.wait_group); a warp barrier then makes them visible to the warp.
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// The stored pairs are bf16 (half the bytes of the stream that bounds the
// step). Inner products, R and Y^T Y are formed from the stored (rounded)
// vectors, so the direction applies the exact L-BFGS matrix of the pairs as
// stored.
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}
__device__ __forceinline__ float4 unpack4(uint32_t lo, uint32_t hi) {
    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162 *>(&lo);
    const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162 *>(&hi);
    return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}

__device__ __forceinline__ uint64_t dup2(float c) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(c));
    return r;
}
// acc += c x for the two bf16 of one word, exactly widened
__device__ __forceinline__ void fma_bf16x2(uint64_t &acc, uint64_t c, uint32_t x) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(x << 16), "r"(x & 0xffff0000u));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(c), "l"(v));
}

template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Four 8 x 8 bf16 matrices from shared memory; lane l gives the address of row
// l % 8 of matrix l / 8 (16 bytes) and receives row l / 4, columns 2 (l % 4),
// 2 (l % 4) + 1 of each matrix.
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void *row) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(row))
                 : "memory");
}
// D += A B for a 16 x 16 bf16 A whose rows 8..15 are zero (a0: row l / 4,
// k = 2 (l % 4) + {0, 1}; a2: the same row, k + 8), a 16 x 8 bf16 B (b0: k =
// 2 (l % 4) + {0, 1}, column l / 4; b1: k + 8) and FP32 accumulation; d0, d1
// are row l / 4, columns 2 (l % 4) + {0, 1}.
__device__ __forceinline__ void mma_rows8(float (&d)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1));
}
// v = hi + mid + lo with each term a bf16 (the remainders are exact in FP32), so
// products with bf16 vectors accumulate to FP32 accuracy on the tensor cores.
__device__ __forceinline__ void split3_bf16(float v, float &hi, float &mid, float &lo) {
    hi = __bfloat162float(__float2bfloat16_rn(v));
    const float r = v - hi;
    mid = __bfloat162float(__float2bfloat16_rn(r));
    lo = r - mid;
}

// A vector of d coordinates as this thread's VPT float4 groups: thread t holds
// the 4 VPT consecutive coordinates from 4 VPT t, so its share of a bf16 row is
// one 16-byte chunk and a warp's copy instruction covers 512 contiguous bytes.
template <int CT>
struct Vec {
    float4 v[Cfg<CT>::VPT];
    __device__ __forceinline__ static int i0(int q) { return 4 * (Cfg<CT>::VPT * (int)threadIdx.x + q); }
    // EVEN: d % (4 VPT) == 0, so a thread holds all of its coordinates or none
    template <bool EVEN>
    __device__ __forceinline__ void load(const float *p, int d) {
        if (EVEN) {
            const bool own = i0(0) < d;
#pragma unroll
            for (int q = 0; q < Cfg<CT>::VPT; ++q)
                v[q] = own ? *reinterpret_cast<const float4 *>(p + i0(q)) : zero4();
        } else {
#pragma unroll
            for (int q = 0; q < Cfg<CT>::VPT; ++q) v[q] = ld4(p, i0(q), d);
        }
    }
    template <bool EVEN>
    __device__ __forceinline__ void store(float *p, int d) const {
        if (EVEN) {
            if (i0(0) < d)
#pragma unroll
                for (int q = 0; q < Cfg<CT>::VPT; ++q) *reinterpret_cast<float4 *>(p + i0(q)) = v[q];
        } else {
#pragma unroll
            for (int q = 0; q < Cfg<CT>::VPT; ++q) st4(p, i0(q), d, v[q]);
        }
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int q = 0; q < Cfg<CT>::VPT; ++q) v[q] = zero4();
    }
};
template <int CT>
__device__ __forceinline__ float dotv(const Vec<CT> &a, const Vec<CT> &b) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < Cfg<CT>::VPT; ++q) s += dot4(a.v[q], b.v[q]);
    return s;
}
// y += c x
template <int CT>
__device__ __forceinline__ void axpyv(float c, const Vec<CT> &x, Vec<CT> &y) {
#pragma unroll
    for (int q = 0; q < Cfg<CT>::VPT; ++q) y.v[q] = axpy4(c, x.v[q], y.v[q]);
}
// a + c b
template <int CT>
__device__ __forceinline__ Vec<CT> lincomb(const Vec<CT> &a, float c, const Vec<CT> &b) {
    Vec<CT> r;
#pragma unroll
    for (int q = 0; q < Cfg<CT>::VPT; ++q) r.v[q] = axpy4(c, b.v[q], a.v[q]);
    return r;
}
template <int CT>
__device__ __forceinline__ Vec<CT> subv(const Vec<CT> &a, const Vec<CT> &b) {
    Vec<CT> r;
#pragma unroll
    for (int q = 0; q < Cfg<CT>::VPT; ++q)
        r.v[q] = make_float4(a.v[q].x - b.v[q].x, a.v[q].y - b.v[q].y, a.v[q].z - b.v[q].z, a.v[q].w - b.v[q].w);
    return r;
}
// bits of the largest |a_i|: 0x7f800000 and more when some a_i is infinite or NaN
template <int CT>
__device__ __forceinline__ uint32_t absmax_bits(const Vec<CT> &a) {
    uint32_t m = 0;
    auto up = [&](float v) { m = max(m, __float_as_uint(v) & 0x7fffffffu); };
#pragma unroll
    for (int q = 0; q < Cfg<CT>::VPT; ++q) {
        up(a.v[q].x);
        up(a.v[q].y);
        up(a.v[q].z);
        up(a.v[q].w);
    }
    return m;
}
template <int CT>
__device__ __forceinline__ uint4 pack_bf16(const Vec<CT> &v) {
    return make_uint4(pack2(v.v[0].x, v.v[0].y), pack2(v.v[0].z, v.v[0].w), pack2(v.v[1].x, v.v[1].y),
                      pack2(v.v[1].z, v.v[1].w));
}
template <int CT>
__device__ __forceinline__ Vec<CT> unpack_bf16(uint4 p) {
    Vec<CT> r;
    r.v[0] = unpack4(p.x, p.y);
    r.v[1] = unpack4(p.z, p.w);
    return r;
}

// Sums of per-thread values over the CTA; every thread gets the totals. One barrier:
// callers alternate between two scratch buffers, so a buffer is never rewritten before
// every thread has read it (the next call's barrier orders it). Several values share the
// shuffles: each step that halves the lanes of a value halves the values of a lane too.
template <int CT>
__device__ __forceinline__ float2 block_sum2(float a, float b, float4 *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool hi = lane & 16;
    float v = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
    for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) == 0) reinterpret_cast<float *>(sh + wid)[lane >> 4] = v;
    __syncthreads();
    float2 t = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < Cfg<CT>::NW; ++q) {
        const float2 u = *reinterpret_cast<const float2 *>(sh + q);
        t.x += u.x;
        t.y += u.y;
    }
    return t;
}
// three sums and the largest of mx
template <int CT>
__device__ __forceinline__ float3 block_sum3_max(float a, float b, float c, uint32_t &mx, float4 *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool b4 = lane & 16, b3 = lane & 8;
    const float ab = (b4 ? b : a) + __shfl_xor_sync(0xffffffffu, b4 ? a : b, 16);
    c += __shfl_xor_sync(0xffffffffu, c, 16);
    float v = (b3 ? c : ab) + __shfl_xor_sync(0xffffffffu, b3 ? ab : c, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    mx = __reduce_max_sync(0xffffffffu, mx);
    // lane 0 holds a, 16 b, 8 c; lane 24 writes the maximum
    if ((lane & 7) == 0)
        reinterpret_cast<float *>(sh + wid)[lane == 24 ? 3 : b3 ? 2 : b4 ? 1 : 0] = lane == 24 ? __uint_as_float(mx) : v;
    __syncthreads();
    float3 t = make_float3(0.f, 0.f, 0.f);
    mx = 0;
#pragma unroll
    for (int q = 0; q < Cfg<CT>::NW; ++q) {
        const float4 u = sh[q];
        t.x += u.x;
        t.y += u.y;
        t.z += u.z;
        mx = max(mx, __float_as_uint(u.w));
    }
    return t;
}

// The dynamic shared memory of the step kernel: the pair ring (Cfg RING_B bytes), pass 2's
// coefficient pairs, R^-1 and Y^T Y (row stride ld), pass 1's per-warp partial sums and the
// m-vectors S^T g, Y^T g, w, D = diag(S^T Y) and the new pair's column of R. Addresses are
// formed from the array and m (registers), not kept in shared memory, so that no access
// waits on a pointer load.
extern __shared__ __align__(16) float4 lb_dyn[];
__device__ __forceinline__ unsigned char *ring_base() { return reinterpret_cast<unsigned char *>(lb_dyn); }

// Row stride of the m x m matrices: as in HBM (one linear copy) unless m is a multiple of 8,
// whose rows would share banks.
__host__ __device__ __forceinline__ int mm_ld(int m) { return (m & 7) ? m : m + 4; }
// Pass 1's partial sums per ring group and warp: two rows (g, y_new) x the group's 2 PGB
// vectors.
template <int CT>
__host__ __device__ __forceinline__ int p1_floats(int m) {
    return (m + Cfg<CT>::PGB - 1) / Cfg<CT>::PGB * Cfg<CT>::NW * 2 * 2 * Cfg<CT>::PGB;
}
// Floats of the dynamic area after the ring.
template <int CT>
__host__ __device__ __forceinline__ int mm_floats(int m) {
    return 2 * m * mm_ld(m) + p1_floats<CT>(m) + 7 * m;
}
template <int CT>
struct Lay {
    int m, ld;
    __device__ __forceinline__ explicit Lay(int m_) : m(m_), ld(mm_ld(m_)) {}
    __device__ __forceinline__ float2 *cf() const { return reinterpret_cast<float2 *>(ring_base() + Cfg<CT>::RING_B); }
    // 16-byte aligned when m is even
    __device__ __forceinline__ float *RI() const { return reinterpret_cast<float *>(cf() + m); }
    __device__ __forceinline__ float *YY() const { return RI() + m * ld; }
    __device__ __forceinline__ float *p1() const { return YY() + m * ld; }
    __device__ __forceinline__ float *u1() const { return p1() + p1_floats<CT>(m); }
    __device__ __forceinline__ float *u2() const { return u1() + m; }
    __device__ __forceinline__ float *nr() const { return u2() + m; }
    __device__ __forceinline__ float *cw() const { return nr() + m; }
    __device__ __forceinline__ float *dg() const { return cw() + m; }
};

template <int CT>
struct Shared {
    float4 red2[2][Cfg<CT>::NW];  // reduction scratch, used alternately (see block_sum2)
    uint4 zero16;                 // a zero row for the unused rows of the tensor-core operand
};

// The m x m state of a walker, indexed by the slots the pairs sit in (as the ring below and
// both passes are: the pairs enter only sums, so their order does not matter, and slots
// 0 .. count - 1 are one contiguous piece): R^-1, the inverse of R = upper(S^T Y), with
// zeros below its diagonal in the pairs' order of age, Y^T Y, and D_i = s_i . y_i (in
// rho). R^-1 is kept instead of R because the history changes only by appending a pair
// (one new column of R^-1, a triangular matvec) and dropping the oldest (the inverse of
// R's trailing block is the trailing block of R^-1), so the direction needs matvecs, not
// substitutions.
//
// Starts the copies of the walker's R^-1, Y^T Y and D into shared memory (waited for before
// the solve). A new pair's row and column are written by new_mm and the solve.
template <int CT>
__device__ __forceinline__ void fetch_mm(const Lay<CT> &L, const float *mri, const float *myy, const float *dw,
                                         int count, int m) {
    float *RI = L.RI(), *YY = L.YY(), *dg = L.dg();
    const int t = threadIdx.x;
    if (m & 1) {
        for (int e = t; e < count * m; e += CT) {
            cp_async4(RI + e, mri + e);
            cp_async4(YY + e, myy + e);
        }
    } else if (m & 7) {  // m^2 is a multiple of 4: the last chunk stays inside
#pragma unroll 1
        for (int e = 4 * t; e < count * m; e += 4 * CT) {
            cp_async16(RI + e, mri + e);
            cp_async16(YY + e, myy + e);
        }
    } else {
        for (int i = t >> 5; i < count; i += Cfg<CT>::NW)
            for (int j = 4 * (t & 31); j < m; j += 128) {
                cp_async16(RI + i * L.ld + j, mri + i * m + j);
                cp_async16(YY + i * L.ld + j, myy + i * m + j);
            }
    }
    for (int i = t; i < count; i += CT) cp_async4(dg + i, dw + i);
}
// Pass 1's totals (the warps' sums in warp order): u1 = S^T g, u2 = Y^T g and, when a pair
// was appended (slot sc), its column of R (s_i . y_new, into nr; D_new into dg and HBM) and
// its row and column of Y^T Y (shared memory and HBM). R^-1's new column is formed by the
// solver. Returns the algorithmic bytes of m x m state of this visit.
template <int CT>
__device__ __forceinline__ uint64_t new_mm(const Lay<CT> &L, float *myy, float *dw, int count, int m, int sc) {
    constexpr int PG = Cfg<CT>::PGB, NW = Cfg<CT>::NW;
    const float *p1 = L.p1();
    const int n = (sc >= 0 ? 4 : 2) * count;
#pragma unroll 1
    for (int e = threadIdx.x; e < n; e += CT) {
        // role: 0 s.g, 1 y.g, 2 s.y_new, 3 y.y_new
        const int role = (e >= count) + (e >= 2 * count) + (e >= 3 * count), i = e - role * count;
        const float *src = p1 + ((i / PG) * NW * 2 + (role >> 1)) * (2 * PG) + 2 * (i % PG) + (role & 1);
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < NW; ++q) v += src[q * 2 * 2 * PG];
        if (role < 3) {
            L.u1()[role * m + i] = v;  // u1, u2, nr
            if (role == 2 && i == sc) L.dg()[sc] = dw[sc] = v;
        } else {
            L.YY()[i * L.ld + sc] = L.YY()[sc * L.ld + i] = v;
            myy[i * m + sc] = myy[sc * m + i] = v;
        }
    }
    const uint64_t c = count;
    return (c * (c + 1) / 2 + c * c + c) * 4 + (sc >= 0 ? (uint64_t)(3 * c) * 4 : 0);
}

// The m x m part, on the whole CTA, with R^-1 in shared memory: when a pair was appended
// (slot sc) R^-1's new column, v_i = -(sum_k RI_ik R_k,sc) / D_sc, v_sc = 1 / D_sc, and its
// row, zero elsewhere (also written to HBM); w = R^-1 u1 (the new column's term added
// apart), gamma = D / (y^T y) of the newest pair (slot sn), tv = D w + gamma Y^T Y w -
// gamma u2 and a = R^-T tv. Each entry is a dot product over G threads (strided terms,
// then a fixed-order shuffle sum), one barrier between the stages. Every thread calls it.
// Leaves (-a_i, gamma w_i) in cf; returns gamma.
template <int CT>
__device__ __forceinline__ float solve_mm(const Lay<CT> &L, int c, int sc, int sn, float *mri, int m) {
    const int lg = c <= 32 ? 2 : (c <= 64 ? 1 : 0), G = 1 << lg;  // threads per entry (the same for every CT)
    const int p = (int)threadIdx.x & (G - 1), i0 = (int)threadIdx.x >> lg, E = CT >> lg;  // E entries at a time
    const int LD = L.ld;
    float *RI = L.RI();
    const float *YY = L.YY();
    float *tv = L.p1();  // pass 1's partial sums are consumed before the solve
    const float *nr = L.nr(), *u1 = L.u1(), *u2 = L.u2(), *dg = L.dg();
    float *cw = L.cw();
    auto gsum = [&](float v) {  // every lane calls it: full-warp shuffles
        if (G >= 2) v += __shfl_xor_sync(0xffffffffu, v, 1);
        if (G >= 4) v += __shfl_xor_sync(0xffffffffu, v, 2);
        return v;
    };
#pragma unroll 1
    for (int i = i0, b = 0; b < c; b += E, i += E) {
        float t = 0.f, r = 0.f;
        if (i < c && i != sc) {
#pragma unroll 1
            for (int k = p; k < c; k += G) {
                const float ri = RI[i * LD + k];
                if (k != sc) {  // the slot's old column
                    t = fmaf(ri, u1[k], t);
                    if (sc >= 0) r = fmaf(ri, nr[k], r);
                }
            }
        }
        t = gsum(t);
        if (sc >= 0) {
            r = gsum(r);
            if (p == 0 && i < c) {
                const float dn = nr[sc], v = i == sc ? 1.f / dn : -r / dn;
                t = fmaf(v, u1[sc], t);
                RI[i * LD + sc] = v;
                mri[i * m + sc] = v;
                if (i != sc) {
                    RI[sc * LD + i] = 0.f;
                    mri[sc * m + i] = 0.f;
                }
            }
        }
        if (p == 0 && i < c) cw[i] = t;
    }
    __syncthreads();
    const float gam = dg[sn] / YY[sn * LD + sn];
#pragma unroll 1
    for (int i = i0, b = 0; b < c; b += E, i += E) {
        float t = 0.f;
        if (i < c)
#pragma unroll 1
            for (int j = p; j < c; j += G) t = fmaf(YY[i * LD + j], cw[j], t);
        t = gsum(t);
        if (p == 0 && i < c) tv[i] = dg[i] * cw[i] + gam * t - gam * u2[i];
    }
    __syncthreads();
#pragma unroll 1
    for (int i = i0, b = 0; b < c; b += E, i += E) {
        float t = 0.f;
        if (i < c)
#pragma unroll 1
            for (int k = p; k < c; k += G) t = fmaf(RI[k * LD + i], tv[k], t);
        t = gsum(t);
        if (p == 0 && i < c) L.cf()[i] = make_float2(-t, gam * cw[i]);
    }
    __syncthreads();
    return gam;
}

using bf16 = __nv_bfloat16;

// Stores this thread's chunk of a history row (coordinates past d are zero in the vector):
// 8 consecutive coordinates, one 16-byte store, for every chunk inside the row pitch.
__device__ __forceinline__ void store_hist(uint4 v, bf16 *row, int ldh) {
    const int e0 = 8 * (int)threadIdx.x;
    if (e0 < ldh) *reinterpret_cast<uint4 *>(row + e0) = v;
}

// The ring the stored pairs stream through (Cfg: DB slots of PGB pairs; row 2 q + v of
// a slot is vector v (0: s, 1: y) of its pair q). Each thread copies and reads its own
// 16-byte chunk of every row (cp.async); pass 1's tensor-core operands also read the
// chunks of the other lanes of the warp, after a warp barrier. Every issue commits one
// copy group (empty when there is nothing to copy), so a wait for the group issued
// D - 1 issues earlier is cp.async.wait_group D - 1.
template <int CT>
struct Ring {
    static constexpr int PG = Cfg<CT>::PGB, D = Cfg<CT>::DB;
    static_assert(Cfg<CT>::VPT == 2, "one 16-byte bf16 chunk (8 coordinates) per stored vector and thread");
    int ldh, J, cn;  // row pitch, pairs (slots 0 .. J - 1), slot of the new pair (or -1)
    const bf16 *S, *Y;
    uint4 s_new, y_new;
    bool known;  // s_new and y_new are (before the trial is judged only the slot is)

    __device__ __forceinline__ unsigned char *row(int sl, int r) const {
        return ring_base() + sl * Cfg<CT>::SLOT_B + r * Cfg<CT>::ROW_B;
    }
    // this thread's chunk of row r of slot sl
    __device__ __forceinline__ uint4 *chunk(int sl, int r) const {
        return reinterpret_cast<uint4 *>(row(sl, r)) + threadIdx.x;
    }
    // Group k (slots k PG .. k PG + PG - 1 below J; none for k < 0) into ring slot sl. The
    // visit's new pair comes from registers (s_new, y_new), not HBM.
    __device__ __forceinline__ void issue(int k, int sl) const {
        const int e0 = Vec<CT>::i0(0);
        if (k >= 0 && e0 < ldh) {
            const int j0 = k * PG;
            const bf16 *s = S + (size_t)(j0 * ldh + e0), *y = Y + (size_t)(j0 * ldh + e0);
            if (j0 + PG <= J && (unsigned)(cn - j0) >= (unsigned)PG) {
#pragma unroll
                for (int q = 0; q < PG; ++q, s += ldh, y += ldh) {
                    cp_async16(chunk(sl, 2 * q), s);
                    cp_async16(chunk(sl, 2 * q + 1), y);
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < PG && j0 + q < J; ++q, s += ldh, y += ldh) {
                    if (j0 + q == cn) {
                        if (known) {
                            *chunk(sl, 2 * q) = s_new;
                            *chunk(sl, 2 * q + 1) = y_new;
                        }
                    } else {
                        cp_async16(chunk(sl, 2 * q), s);
                        cp_async16(chunk(sl, 2 * q + 1), y);
                    }
                }
            }
        }
        cp_async_commit();
    }
    // The first D - 1 groups after the trial is judged: the new pair's row, or, when its slot sp
    // keeps its old pair, that row.
    __device__ __forceinline__ void settle(int sp) const {
        if (sp >= (D - 1) * PG) return;
        const int sl = sp / PG, q = sp % PG, e0 = Vec<CT>::i0(0);
        if (cn == sp) {
            if (e0 < ldh) {
                *chunk(sl, 2 * q) = s_new;
                *chunk(sl, 2 * q + 1) = y_new;
            }
        } else if (sp < J) {
            if (e0 < ldh) {
                cp_async16(chunk(sl, 2 * q), S + (size_t)(sp * ldh + e0));
                cp_async16(chunk(sl, 2 * q + 1), Y + (size_t)(sp * ldh + e0));
            }
            cp_async_commit();
            cp_async_wait<0>();
        }
    }
    // the group issued D - 1 issues ago has landed, and is visible to the warp
    __device__ __forceinline__ void wait() const {
        cp_async_wait<D - 1>();
        __syncwarp();
    }
    // p += c.x s + c.y y for pair q of ring slot sl, on this thread's coordinates
    __device__ __forceinline__ void add(int sl, int q, float2 c, uint64_t (&p)[4]) const {
        const uint4 a4 = *chunk(sl, 2 * q), b4 = *chunk(sl, 2 * q + 1);
        const uint64_t cs = dup2(c.x), cy = dup2(c.y);
        fma_bf16x2(p[0], cs, a4.x);
        fma_bf16x2(p[1], cs, a4.y);
        fma_bf16x2(p[2], cs, a4.z);
        fma_bf16x2(p[3], cs, a4.w);
        fma_bf16x2(p[0], cy, b4.x);
        fma_bf16x2(p[1], cy, b4.y);
        fma_bf16x2(p[2], cy, b4.z);
        fma_bf16x2(p[3], cy, b4.w);
    }
};

// Direction for walker state st (pairs in slots 0 .. count - 1). When sc = ring.cn >= 0 the
// pair in that slot was stored this visit and its column of R, row and column of
// Y^T Y come from the same pass. sp: the slot the caller left out when it started the first
// D - 1 groups. Writes P and the unit trial X + P; updates st.dphi / alpha / bt and possibly
// resets the history (steepest descent when p is not a descent direction). Returns the
// algorithmic bytes moved.
//
// Pass 1 streams the slots upwards; at its end the ring holds the last min(groups, DB)
// groups, so pass 2 walks the groups downwards: those are read where they are, and each
// ring slot it frees is refilled with the group DB below (the same ring slot, g mod DB), the
// only ones read from HBM (L2) again.
template <int CT, bool EVEN>
__device__ uint64_t direction(const LbfgsArgs<float> &a, int w, WalkerState<float> &st, int sp, const Vec<CT> &g_in,
                              const Vec<CT> &x_in, const Ring<CT> &ring, float *mri_w, float *myy_w, Shared<CT> &sh,
                              const Lay<CT> &L, int &par) {
    using RG = Ring<CT>;
    constexpr int PG = RG::PG, D = RG::D, NW = Cfg<CT>::NW;
    const int d = a.d, m = a.m;
    const int count = st.count;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t bytes = 0;
    Vec<CT> p;
    p.zero();
    // x and g are stored at X, G by the caller; they are read back after pass 1
    // instead of being held through it
    Vec<CT> g = g_in, x = x_in;
    if (count > 0) {
        const int ng = (count + PG - 1) / PG;
        const int sc = ring.cn;
        float *dw = a.rho + (size_t)w * m;
        ring.settle(sp);
        float *p1 = L.p1();
        {
            // Pass 1 on the tensor cores: per warp (its 256 coordinates, 16 k-steps of
            // 16) and group (8 stored vectors s_0 y_0 .. s_3 y_3 as the columns of B),
            // D = A B with the rows of A = (g_hi, g_mid, g_lo, y_new, 0 ..) at the same
            // coordinates. The A fragments are staged once through this warp's
            // own chunks of ring slot D - 1 (free until group D - 1 is issued into it).
            {
                float hi[8], mi[8], lo[8];
                const float gv[8] = {g.v[0].x, g.v[0].y, g.v[0].z, g.v[0].w, g.v[1].x, g.v[1].y, g.v[1].z, g.v[1].w};
#pragma unroll
                for (int e = 0; e < 8; ++e) split3_bf16(gv[e], hi[e], mi[e], lo[e]);
                *ring.chunk(D - 1, 0) =
                    make_uint4(pack2(hi[0], hi[1]), pack2(hi[2], hi[3]), pack2(hi[4], hi[5]), pack2(hi[6], hi[7]));
                *ring.chunk(D - 1, 1) =
                    make_uint4(pack2(mi[0], mi[1]), pack2(mi[2], mi[3]), pack2(mi[4], mi[5]), pack2(mi[6], mi[7]));
                *ring.chunk(D - 1, 2) =
                    make_uint4(pack2(lo[0], lo[1]), pack2(lo[2], lo[3]), pack2(lo[4], lo[5]), pack2(lo[6], lo[7]));
                *ring.chunk(D - 1, 3) = ring.y_new;  // as stored; zero when there is none
            }
            __syncwarp();
            const int mi8 = lane >> 3, ri8 = lane & 7;  // ldmatrix: matrix and row this lane addresses
            const int u0 = 16 * (32 * wid + 2 * (mi8 >> 1) + (mi8 & 1));  // its byte in the row at k-step 0
            uint32_t af[16][2];                         // A fragments (a0, a2) per k-step
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                const void *src = ri8 < 4 ? (const void *)(ring.row(D - 1, ri8) + u0 + 32 * c) : (const void *)&sh.zero16;
                uint32_t r[4];
                ldsm_x4(r, src);
                af[c][0] = r[0];
                af[c][1] = r[1];
                af[c + 1][0] = r[2];
                af[c + 1][1] = r[3];
            }
            int nk = (d - 256 * wid + 15) / 16;  // k-steps of this warp inside d (warp-uniform)
            nk = nk < 0 ? 0 : (nk > 16 ? 16 : nk);
            const int gid = lane >> 2, tig = lane & 3;
            __syncwarp();
            ring.issue(D - 1, D - 1);
            int sl = 0;
#pragma unroll 1
            for (int k = 0; k < ng; ++k) {
                ring.wait();
                // B rows: the group's 8 stored vectors (pair n / 2, s or y); the k-steps
                // accumulate into four independent sets (k-step mod 4), summed after, so
                // that the MMAs are not one dependent chain
                float a4[4][4] = {};
                const unsigned char *br = ring.row(sl, ri8) + u0;
                auto step = [&](int c) {
                    uint32_t b[4];
                    ldsm_x4(b, br + 32 * c);
                    mma_rows8(a4[c & 3], af[c][0], af[c][1], b[0], b[1]);
                    mma_rows8(a4[(c + 1) & 3], af[c + 1][0], af[c + 1][1], b[2], b[3]);
                };
                if (nk == 16) {
#pragma unroll
                    for (int c = 0; c < 16; c += 2) step(c);
                } else {
                    // past d both operands are zero
#pragma unroll
                    for (int c = 0; c < 16; c += 2)
                        if (c < nk) step(c);
                }
                float acc[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) acc[e] = (a4[0][e] + a4[1][e]) + (a4[2][e] + a4[3][e]);
                // g . v = (g_hi + g_mid) . v + g_lo . v from rows 0, 1, 2
                const float h0 = __shfl_down_sync(0xffffffffu, acc[0], 4);
                const float l0 = __shfl_down_sync(0xffffffffu, acc[0], 8);
                const float h1 = __shfl_down_sync(0xffffffffu, acc[1], 4);
                const float l1 = __shfl_down_sync(0xffffffffu, acc[1], 8);
                if (gid == 0 || gid == 3) {
                    const float2 o = gid == 0 ? make_float2((acc[0] + h0) + l0, (acc[1] + h1) + l1)
                                              : make_float2(acc[0], acc[1]);
                    *reinterpret_cast<float2 *>(p1 + ((k * NW + wid) * 2 + (gid != 0)) * (2 * PG) + 2 * tig) = o;
                }
                __syncwarp();  // the warp has read the group before its slot is refilled
                ring.issue(k + D < ng ? k + D : -1, sl);
                sl = sl == D - 1 ? 0 : sl + 1;
            }
        }
        cp_async_wait<0>();  // the m x m state
        __syncthreads();
        bytes += new_mm<CT>(L, myy_w, dw, count, m, sc);
        g.template load<EVEN>(a.G + (size_t)w * d, d);
        x.template load<EVEN>(a.X + (size_t)w * d, d);
        __syncthreads();
        int sn = st.head + count - 1;  // the newest pair's slot
        if (sn >= m) sn -= m;
        const float gam = solve_mm<CT>(L, count, sc, sn, mri_w, m);
        // pass 2: p = -gamma g - S a + gamma Y w, the groups downwards
        uint64_t p2[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float4 t = make_float4(-gam * g.v[q].x, -gam * g.v[q].y, -gam * g.v[q].z, -gam * g.v[q].w);
            asm("mov.b64 %0, {%1, %2};" : "=l"(p2[2 * q]) : "f"(t.x), "f"(t.y));
            asm("mov.b64 %0, {%1, %2};" : "=l"(p2[2 * q + 1]) : "f"(t.z), "f"(t.w));
        }
        const int r0 = ng > D ? ng - D : 0;  // groups below r0 are no longer in the ring
        const float2 *cf = L.cf();
        int sl = (ng - 1) % D;
#pragma unroll 1
        for (int k = ng - 1; k >= 0; --k) {
            if (k < r0) ring.wait();
            const int n = count - k * PG;
            if (n >= PG) {
#pragma unroll
                for (int q = 0; q < PG; ++q) ring.add(sl, q, cf[k * PG + q], p2);
            } else {
#pragma unroll 1
                for (int q = 0; q < n; ++q) ring.add(sl, q, cf[k * PG + q], p2);
            }
            ring.issue(k - D, sl);  // this thread's own chunks, just read
            sl = sl == 0 ? D - 1 : sl - 1;
        }
        cp_async_wait<0>();  // (only empty groups remain) the ring is free for the next walker
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            asm("mov.b64 {%0, %1}, %2;" : "=f"(p.v[q].x), "=f"(p.v[q].y) : "l"(p2[2 * q]));
            asm("mov.b64 {%0, %1}, %2;" : "=f"(p.v[q].z), "=f"(p.v[q].w) : "l"(p2[2 * q + 1]));
        }
        // the two-loop recursion's history traffic: each pair read in both passes
        bytes += (uint64_t)4 * count * d * sizeof(bf16);
    }
    float2 dp = make_float2(0.f, 0.f);  // grad f . p and |p|^2
    if (count > 0) dp = block_sum2<CT>(dotv(g, p), dotv(p, p), sh.red2[par++ & 1]);
    if (count == 0 || !(dp.x < 0.f)) {
        st.count = 0;
        st.head = 0;
        const float gn = sqrtf(block_sum2<CT>(dotv(g, g), 0.f, sh.red2[par++ & 1]).x);
#pragma unroll
        for (int q = 0; q < Cfg<CT>::VPT; ++q)
            p.v[q] = make_float4(-g.v[q].x / gn, -g.v[q].y / gn, -g.v[q].z / gn, -g.v[q].w / gn);
        dp = block_sum2<CT>(dotv(g, p), dotv(p, p), sh.red2[par++ & 1]);
    }
    st.dphi = dp.x;
    st.pn = sqrtf(dp.y);
    st.alpha = 1.f;
    st.bt = 0;
    p.template store<EVEN>(a.P + (size_t)w * d, d);
    lincomb(x, 1.f, p).template store<EVEN>(a.XT + (size_t)w * d, d);
    return bytes + (uint64_t)8 * d;
}

// Algorithmic bytes of the L-BFGS step launches (added only while counting is on).
__device__ unsigned long long g_lbfgs_bytes;

template <int CT, bool EVEN>
__global__ void __launch_bounds__(CT, Cfg<CT>::MINB) k_lbfgs_cta(LbfgsArgs<float> a, float *MRI, float *MYY,
                                                                int count_bytes) {
    __shared__ Shared<CT> sh;
    const int d = a.d, m = a.m, ldh = hist_ld(d);
    const Lay<CT> L(m);
    // the ring starts zeroed: chunks past the row pitch are never copied into and must
    // read as zeros where a k-step of pass 1 straddles the end of the coordinates
    for (int e = threadIdx.x; e < Cfg<CT>::RING_B / 16; e += CT) lb_dyn[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x == 0) {
        sh.zero16 = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    const int n_act = *a.n_act;
    int par = 0;  // alternation of the reduction scratch (identical in every thread)
    uint64_t bytes = 0;
    // the next visit's walker id is loaded one visit ahead, so a visit's first
    // loads (state, vectors) do not wait behind the active-list read
    int w_next = (int)blockIdx.x < n_act ? a.act[blockIdx.x] : 0;
    for (int n = blockIdx.x; n < n_act; n += gridDim.x) {
        const int w = w_next;
        if (n + (int)gridDim.x < n_act) w_next = a.act[n + gridDim.x];
        WalkerState<float> st = a.st[w];  // same address in every thread: one broadcast load
        const float ft = a.FT[w];
        const float alpha0 = st.alpha, pn0 = st.pn;
        float dnext = -1.f;  // bound on |new trial - this visit's trial| (see k_tc_need)
        float *X = a.X + (size_t)w * d;
        float *G = a.G + (size_t)w * d;
        Vec<CT> x, g, xt, gt;
        x.template load<EVEN>(X, d);
        g.template load<EVEN>(G, d);
        xt.template load<EVEN>(a.XT + (size_t)w * d, d);
        gt.template load<EVEN>(a.GT + (size_t)w * d, d);
        bytes += (uint64_t)16 * d + 4 + 2 * sizeof(WalkerState<float>);
        // Most trials are accepted with a new pair, so the first groups of the history and
        // the m x m state are started before the trial is judged, all but the slot the
        // pair would take (sp); they land while the vectors are read and reduced.
        const int sp = st.count < m ? st.count : st.head;
        Ring<CT> ring{ldh, sp < st.count ? st.count : sp + 1, sp, reinterpret_cast<const bf16 *>(a.S) + (size_t)w * m * ldh,
                      reinterpret_cast<const bf16 *>(a.Y) + (size_t)w * m * ldh, make_uint4(0u, 0u, 0u, 0u),
                      make_uint4(0u, 0u, 0u, 0u), false};
        float *mri_w = MRI + (size_t)w * m * m, *myy_w = MYY + (size_t)w * m * m;
#pragma unroll
        for (int k = 0; k < Cfg<CT>::DB - 1; ++k) ring.issue(k, k);
        fetch_mm<CT>(L, mri_w, myy_w, a.rho + (size_t)w * m, st.count, m);  // joins the next copy group
        // finiteness of the trial gradient, the candidate pair (as it will be stored) and its
        // inner products, and max |grad| at the trial, all in one reduction
        const uint4 s_new = pack_bf16<CT>(subv(xt, x)), y_new = pack_bf16<CT>(subv(gt, g));
        uint32_t gm_bits = absmax_bits<CT>(gt);
        float3 r3;
        {
            const Vec<CT> s4 = unpack_bf16<CT>(s_new), y4 = unpack_bf16<CT>(y_new);
            r3 = block_sum3_max<CT>(dotv(s4, s4), dotv(y4, y4), dotv(s4, y4), gm_bits, sh.red2[par++ & 1]);
        }
        if (EVEN && n + (int)gridDim.x < n_act && threadIdx.x < 4) {
            // the next walker's vectors into L2 (rows are whole 32-byte pieces); its pairs are
            // too many for that (the solve 147 -> 157 ms with them, 132.5 -> 131.2 without)
            const float *v = threadIdx.x == 0 ? a.X : threadIdx.x == 1 ? a.G : threadIdx.x == 2 ? a.XT : a.GT;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(v + (size_t)w_next * d),
                         "r"((uint32_t)d * 4u)
                         : "memory");
        }
        const bool finite = isfinite(ft) && gm_bits < 0x7f800000u;
        const float gm = __uint_as_float(gm_bits);
        bool newiter = false;
        ring.known = true;
        ring.cn = -1;
        if (st.phase == 0) {
            x = xt;
            g = gt;
            x.template store<EVEN>(X, d);
            g.template store<EVEN>(G, d);
            bytes += (uint64_t)8 * d;
            st.f = ft;
            st.phase = 1;
            if (!finite)
                st.status = SB_WALKER_NONFINITE;
            else
                newiter = true;
        } else if (finite && ft <= st.f + (a.c1 * st.alpha) * st.dphi) {
            if (r3.z > 1e-10f * sqrtf(r3.x) * sqrtf(r3.y)) {
                int slot;
                if (st.count < m) {
                    slot = st.count;  // the slots fill upwards from 0
                    ++st.count;
                } else {
                    slot = st.head;
                    st.head = slot + 1 == m ? 0 : slot + 1;
                }
                store_hist(s_new, reinterpret_cast<bf16 *>(a.S) + ((size_t)w * m + slot) * ldh, ldh);
                store_hist(y_new, reinterpret_cast<bf16 *>(a.Y) + ((size_t)w * m + slot) * ldh, ldh);
                bytes += (uint64_t)2 * d * sizeof(bf16);
                ring.s_new = s_new;
                ring.y_new = y_new;
                ring.cn = slot;
            }
            ring.J = st.count;
            st.flat = (ft >= st.f) ? st.flat + 1 : 0;
            x = xt;
            g = gt;
            x.template store<EVEN>(X, d);
            g.template store<EVEN>(G, d);
            bytes += (uint64_t)8 * d;
            st.f = ft;
            ++st.it;
            newiter = true;
        } else {
            ++st.bt;
            if (st.bt <= a.max_backtracks) {
                st.alpha *= a.backtrack;
                Vec<CT> p;
                p.template load<EVEN>(a.P + (size_t)w * d, d);
                lincomb(x, st.alpha, p).template store<EVEN>(a.XT + (size_t)w * d, d);
                bytes += (uint64_t)8 * d;
                dnext = (alpha0 - st.alpha) * st.pn;
            } else if (st.count > 0 && st.attempt == 0) {
                st.count = 0;
                st.head = 0;
                st.attempt = 1;
                bytes += direction<CT, EVEN>(a, w, st, sp, g, x, ring, mri_w, myy_w, sh, L, par);
                dnext = st.pn + alpha0 * pn0;  // from the old trial back to x, then out
            } else {
                st.status = SB_WALKER_STALLED;
            }
        }
        if (newiter) {
            if (gm <= a.gtol * (1.f + fabsf(st.f))) {
                st.status = SB_WALKER_CONVERGED;
            } else if (st.flat >= 2) {
                st.status = SB_WALKER_STALLED;
            } else if (st.it >= a.max_iter) {
                st.status = SB_WALKER_MAXITER;
            } else {
                st.attempt = 0;
                bytes += direction<CT, EVEN>(a, w, st, sp, g, x, ring, mri_w, myy_w, sh, L, par);
                dnext = st.pn;  // x is this visit's trial
            }
        }
        if (threadIdx.x == 0) {
            a.st[w] = st;
            if (a.dist && dnext >= 0.f) a.dist[w] = dnext * 1.0001f;  // margin for the rounding of |p|
        }
        cp_async_wait_all();  // what a rejected or last trial did not use
        // No barrier before the next walker: a thread's ring chunks are read by
        // other lanes only in pass 1, behind warp barriers, and every copy group has
        // completed. The reduction scratch alternates, and every other shared array
        // is rewritten only after the next walker's first reduction barrier.
    }
    if (count_bytes && threadIdx.x == 0 && bytes) atomicAdd(&g_lbfgs_bytes, (unsigned long long)bytes);
}

// The active list of the mixed path, compacted and grouped by each walker's dominant
// component (key[w], the component of the largest term at its latest evaluation;
// -1 goes last), keeping the list order inside a group: the evaluation round skips
// (128-row block, component) pairs no row of the block needs, and walkers of
// different basins interleaved in one block would make every block need every
// component. Skipped terms are exactly zero, so the grouping changes no result.
// Two launches over G CTAs, CTA c owning the list entries [c R, (c + 1) R), R = E x
// threads, E consecutive entries per thread (lane, then warp, then CTA order is list
// order). The first gathers every entry's walker, status and key (independent loads,
// spread over the GPU), packs (bucket, walker) into tmp and counts the buckets per
// CTA; the second reads the G x buckets count table, so CTA c knows where each
// bucket starts and how many entries of it the CTAs before c hold, ranks its entries
// per warp and places each in act. tmp decouples the two, as entries move between
// CTAs' ranges.
constexpr int kSortBuckets = kMaxK + 1;
constexpr int kCompactE = 16;        // most entries per thread
constexpr int kCkThreads = 256;      // threads per CTA
constexpr int kCkMinBlocks = 64;     // CTAs for a short list (one entry per thread up to 16384)
constexpr int kPackShift = 25;       // packed entry: bucket << 25 | walker
constexpr uint32_t kPackDrop = 0xffffffffu;  // a dropped entry (bucket field 127)
static_assert(kSortBuckets < 127, "the bucket field holds 7 bits");

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Buckets present in this warp's entries (bit b for bucket b < nb).
__device__ __forceinline__ uint64_t warp_buckets(const uint32_t (&pk)[kCompactE], int E, int nb) {
    uint64_t present = 0;
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) {
        const uint32_t b = pk[e] >> kPackShift;
        if (e < E && b < (uint32_t)nb) present |= 1ull << b;
    }
    return (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)present) |
           ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(present >> 32)) << 32);
}
__device__ __forceinline__ int count_bucket(const uint32_t (&pk)[kCompactE], int E, int b) {
    int cnt = 0;
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) cnt += (e < E && (pk[e] >> kPackShift) == (uint32_t)b);
    return cnt;
}
// entries per thread for prev entries over G CTAs
__device__ __forceinline__ int compact_E(int prev, int G) {
    const int per = G * kCkThreads;
    return (prev + per - 1) / per;
}

// cnt: [G][nb] bucket counts, then cnt[G nb] = the list length before compaction
__global__ void __launch_bounds__(kCkThreads) k_compact_count(const WalkerState<float> *st, const int32_t *act,
                                                              const int32_t *n_act, const int32_t *key, int K,
                                                              uint32_t *tmp, int32_t *cnt) {
    __shared__ int total[kSortBuckets];
    const int prev = *n_act, G = (int)gridDim.x, nb = K + 1;
    const int E = compact_E(prev, G);
    const int lane = threadIdx.x & 31;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) total[b] = 0;
    __syncthreads();
    const int s0 = ((int)blockIdx.x * kCkThreads + (int)threadIdx.x) * E;
    int w[kCompactE];
    uint32_t pk[kCompactE];
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) w[e] = (e < E && s0 + e < prev) ? act[s0 + e] : -1;
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) {
        const bool run = w[e] >= 0 && st[w[e]].status == SB_WALKER_RUNNING;
        const int k = w[e] >= 0 ? key[w[e]] : -1;
        const int b = (k >= 0 && k < K) ? k : K;
        pk[e] = run ? ((uint32_t)b << kPackShift) | (uint32_t)w[e] : kPackDrop;
        if (e < E && s0 + e < prev) tmp[s0 + e] = pk[e];
    }
    for (uint64_t m = warp_buckets(pk, E, nb); m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        const int sum = __reduce_add_sync(0xffffffffu, count_bucket(pk, E, b));
        if (lane == 0) atomicAdd(&total[b], sum);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) cnt[(size_t)blockIdx.x * nb + b] = total[b];
    if (blockIdx.x == 0 && threadIdx.x == 0) cnt[(size_t)G * nb] = prev;
}

__global__ void __launch_bounds__(kCkThreads) k_compact_place(int32_t *act, int32_t *n_act, int64_t *n_evals, int K,
                                                              const uint32_t *tmp, const int32_t *cnt) {
    constexpr int NW = kCkThreads / 32;
    __shared__ int off[kSortBuckets];             // this CTA's first slot of each bucket
    __shared__ int wtot[NW][kSortBuckets], woff[NW][kSortBuckets];
    const int G = (int)gridDim.x, nb = K + 1, c = (int)blockIdx.x;
    const int prev = cnt[(size_t)G * nb];
    const int E = compact_E(prev, G);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid == 0) {
        // per bucket: all CTAs' total and the CTAs before c; then the exclusive sums of
        // the totals, 32 buckets at a time
        int carry = 0;
        for (int b0 = 0; b0 < nb; b0 += 32) {
            const int b = b0 + lane;
            int tot = 0, before = 0;
            if (b < nb)
                for (int q = 0; q < G; ++q) {
                    const int v = cnt[(size_t)q * nb + b];
                    tot += v;
                    before += q < c ? v : 0;
                }
            const int incl = warp_incl_scan(tot);
            if (b < nb) off[b] = carry + incl - tot + before;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (c == 0 && lane == 0) {
            *n_act = carry;
            if (n_evals) *n_evals += prev;
        }
    }
    const int s0 = (c * kCkThreads + (int)threadIdx.x) * E;
    uint32_t pk[kCompactE];
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) pk[e] = (e < E && s0 + e < prev) ? tmp[s0 + e] : kPackDrop;
    const uint64_t wpres = warp_buckets(pk, E, nb);
    for (int b = lane; b < nb; b += 32) wtot[wid][b] = 0;
    __syncwarp();
    for (uint64_t m = wpres; m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        const int incl = warp_incl_scan(count_bucket(pk, E, b));
        if (lane == 31) wtot[wid][b] = incl;
    }
    __syncthreads();
    // per bucket: the warps' offsets (a scan over the NW warps' totals)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        int run = off[b];
        for (int q = 0; q < NW; ++q) {
            woff[q][b] = run;
            run += wtot[q][b];
        }
    }
    __syncthreads();
    for (uint64_t m = wpres; m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        const int n_b = count_bucket(pk, E, b);
        int pos = woff[wid][b] + warp_incl_scan(n_b) - n_b;
#pragma unroll
        for (int e = 0; e < kCompactE; ++e)
            if (e < E && (pk[e] >> kPackShift) == (uint32_t)b) act[pos++] = (int32_t)(pk[e] & ((1u << kPackShift) - 1u));
    }
}

// The same for a list that one CTA holds in registers (kCkThreads kCompactE entries), in one
// launch: a short round is bound by the rate at which its kernels start.
__global__ void __launch_bounds__(kCkThreads) k_compact_one(const WalkerState<float> *st, int32_t *act, int32_t *n_act,
                                                            int64_t *n_evals, const int32_t *key, int K) {
    constexpr int NW = kCkThreads / 32;
    __shared__ int wtot[NW][kSortBuckets], start[kSortBuckets + 1];
    const int prev = *n_act, nb = K + 1;
    const int E = compact_E(prev, 1);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int s0 = (int)threadIdx.x * E;
    int w[kCompactE];
    uint32_t pk[kCompactE];
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) w[e] = (e < E && s0 + e < prev) ? act[s0 + e] : -1;
#pragma unroll
    for (int e = 0; e < kCompactE; ++e) {
        const bool run = w[e] >= 0 && st[w[e]].status == SB_WALKER_RUNNING;
        const int k = w[e] >= 0 ? key[w[e]] : -1;
        const int b = (k >= 0 && k < K) ? k : K;
        pk[e] = run ? ((uint32_t)b << kPackShift) | (uint32_t)w[e] : kPackDrop;
    }
    for (int b = lane; b < nb; b += 32) wtot[wid][b] = 0;
    __syncwarp();
    const uint64_t wpres = warp_buckets(pk, E, nb);
    for (uint64_t m = wpres; m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        const int sum = __reduce_add_sync(0xffffffffu, count_bucket(pk, E, b));
        if (lane == 0) wtot[wid][b] = sum;
    }
    __syncthreads();  // every entry is read before any is written
    if (wid == 0) {
        int carry = 0;
        for (int b0 = 0; b0 < nb; b0 += 32) {
            const int b = b0 + lane;
            int tot = 0;
            if (b < nb)
                for (int q = 0; q < NW; ++q) tot += wtot[q][b];
            const int incl = warp_incl_scan(tot);
            if (b < nb) start[b] = carry + incl - tot;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) {
            *n_act = carry;
            if (n_evals) *n_evals += prev;
        }
    }
    __syncthreads();
    for (uint64_t m = wpres; m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        const int n_b = count_bucket(pk, E, b);
        int pos = start[b] + warp_incl_scan(n_b) - n_b;
        for (int q = 0; q < wid; ++q) pos += wtot[q][b];
#pragma unroll
        for (int e = 0; e < kCompactE; ++e)
            if (e < E && (pk[e] >> kPackShift) == (uint32_t)b) act[pos++] = (int32_t)(pk[e] & ((1u << kPackShift) - 1u));
    }
}

}  // namespace

int lbfgs_compact_blocks(int n) {
    const int per = kCkThreads * kCompactE;
    const int need = (n + per - 1) / per;
    return need > kCkMinBlocks ? need : kCkMinBlocks;
}

size_t lbfgs_compact_cnt_elems(int n) { return (size_t)lbfgs_compact_blocks(n) * kSortBuckets + 1; }

void launch_lbfgs_compact_by_key(const LbfgsArgs<float> &a, int n, int64_t *n_evals, const int32_t *key, int K,
                                 int32_t *tmp, int32_t *cnt, cudaStream_t s) {
    if (n <= kCkThreads * kCompactE) {
        note_launch();
        k_compact_one<<<1, kCkThreads, 0, s>>>(a.st, a.act, a.n_act, n_evals, key, K);
        return;
    }
    const int G = lbfgs_compact_blocks(n);
    note_launch();
    k_compact_count<<<G, kCkThreads, 0, s>>>(a.st, a.act, a.n_act, key, K, reinterpret_cast<uint32_t *>(tmp), cnt);
    note_launch();
    k_compact_place<<<G, kCkThreads, 0, s>>>(a.act, a.n_act, n_evals, K, reinterpret_cast<const uint32_t *>(tmp), cnt);
}

bool lbfgs_compact_by_key_fits(int n) { return n >= 0 && n < (1 << kPackShift); }

namespace {
template <int CT, bool EVEN>
void launch_step(const LbfgsArgs<float> &a, int n, float *MRI, float *MYY, int num_sms, cudaStream_t s) {
    const int count_bytes = prof_class_on(PROF_LBFGS_STEP) ? 1 : 0;
    const size_t dyn = (size_t)Cfg<CT>::RING_B + sizeof(float) * mm_floats<CT>(a.m);
    static std::once_flag once;  // batched solves launch from several host threads
    std::call_once(once, [] {
        const size_t most = (size_t)Cfg<CT>::RING_B + sizeof(float) * mm_floats<CT>(kMaxM);
        cudaFuncSetAttribute(k_lbfgs_cta<CT, EVEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    });
    // as many CTAs as stay resident: each goes from walker to walker
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_lbfgs_cta<CT, EVEN>, CT, dyn) != cudaSuccess || per < 1)
        per = 1;
    int grid = num_sms * per;
    if (grid > n) grid = n > 0 ? n : 1;
    note_launch();
    k_lbfgs_cta<CT, EVEN><<<grid, CT, dyn, s>>>(a, MRI, MYY, count_bytes);
}
template <int CT>
void launch_step_ct(const LbfgsArgs<float> &a, int n, float *MRI, float *MYY, int num_sms, cudaStream_t s) {
    // d a multiple of 8 (one whole 16-byte chunk per thread or none): no per-element bounds
    if (a.d % (4 * Cfg<CT>::VPT) == 0)
        launch_step<CT, true>(a, n, MRI, MYY, num_sms, s);
    else
        launch_step<CT, false>(a, n, MRI, MYY, num_sms, s);
}
}  // namespace

void launch_lbfgs_step_cta(const LbfgsArgs<float> &a, int n, float *MRI, float *MYY, int num_sms, cudaStream_t s) {
    ProfScope prof(PROF_LBFGS_STEP, s);
    if (a.d <= Cfg<32>::MAXD)
        launch_step_ct<32>(a, n, MRI, MYY, num_sms, s);
    else if (a.d <= Cfg<64>::MAXD)
        launch_step_ct<64>(a, n, MRI, MYY, num_sms, s);
    else
        launch_step_ct<128>(a, n, MRI, MYY, num_sms, s);
}

double lbfgs_bytes_take() {
    unsigned long long v = 0, z = 0;
    if (cudaDeviceSynchronize() != cudaSuccess) return -1.0;
    if (cudaMemcpyFromSymbol(&v, g_lbfgs_bytes, sizeof(v)) != cudaSuccess) return -1.0;
    if (cudaMemcpyToSymbol(g_lbfgs_bytes, &z, sizeof(z)) != cudaSuccess) return -1.0;
    return (double)v;
}

}  // namespace sb
