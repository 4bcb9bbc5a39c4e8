// rays.cu -- sunburst ray directions and start selection (Sec. 3.5.1-3.5.2, Sec. 4.1).
//
// Directions: ray r, coordinate pair p draws one Philox4x32-10 block with
// counter (p, r, 'RAYS', 0) and key (seed lo, seed hi); its two 64-bit words
// give two uniforms, Box-Muller gives two standard normals, and the vector is
// scaled to unit length (uniform on S^{d-1}). t_exit,r = min_i half_i / |u_ri|
// is the distance from the box centre to the box surface along u_r.
//
// Start selection takes the n_starts smallest keys (tier, rank, -l, flat):
// tier 0 marks a discrete local maximum of l along its ray (the sign change of
// the ray derivative, Sec. 4.1), rank is the position of l inside its ray.
// The cut is found exactly: a histogram over (tier, rank) buckets picks the
// bucket holding the n_starts-th key, then a 12-pass 8-bit radix select over
// the 96-bit key (order-preserving bits of -l, flat index) inside that bucket.
// Selected samples are emitted in ascending flat index by an ordered scan.
#include "sb_internal.cuh"

namespace sb {

namespace {

__global__ void __launch_bounds__(256) k_ray_dirs(int d, int n_rays, uint32_t k0, uint32_t k1, const double *half,
                                                  double *u, double *texit) {
    const int lane = threadIdx.x & 31;
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= n_rays) return;
    double *ur = u + (size_t)r * d;
    const int npairs = (d + 1) / 2;
    double ss = 0.0;
    for (int p = lane; p < npairs; p += 32) {
        uint32_t c[4] = {(uint32_t)p, (uint32_t)r, 0x52415953u, 0u};
        philox4x32_10(c, k0, k1);
        const double u1 = unit_from_words(c[0], c[1]);
        const double u2 = unit_from_words(c[2], c[3]);
        const double rad = sqrt(-2.0 * log(u1));
        const double th = mul_rn(SB_TWO_PI, u2);
        const double x0 = mul_rn(rad, cos(th));
        ur[2 * p] = x0;
        ss += x0 * x0;
        if (2 * p + 1 < d) {
            const double x1 = mul_rn(rad, sin(th));
            ur[2 * p + 1] = x1;
            ss += x1 * x1;
        }
    }
    const double nrm = sqrt(warp_sum(ss));
    __syncwarp();
    for (int i = lane; i < d; i += 32) ur[i] = div_rn(ur[i], nrm);
    __syncwarp();
    const double tmin = warp_exit_min(lane, d, ur, half);
    if (lane == 0) texit[r] = tmin;
}

// The same rays for the mixed-precision path, generated in FP32 (the tensor-core
// operands carry fewer bits): the same Philox counters, uniforms from the top 24 bits
// of each 64-bit pair, Box-Muller with FP32 transcendentals, normalised in FP32 and
// widened to FP64; t_exit in FP64 for the widened direction, so the last sample of a
// ray lies on the box surface.
__global__ void __launch_bounds__(256) k_ray_dirs_f32(int d, int n_rays, uint32_t k0, uint32_t k1, const double *half,
                                                      double *u, double *texit) {
    const int lane = threadIdx.x & 31;
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= n_rays) return;
    double *ur = u + (size_t)r * d;
    const int npairs = (d + 1) / 2;
    constexpr int kPer = 16;  // pairs a lane keeps in registers before the norm is known
    float x[2 * kPer];
    float ss = 0.f;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int p = lane + 32 * q;
        x[2 * q] = x[2 * q + 1] = 0.f;
        if (p < npairs) {
            uint32_t c[4] = {(uint32_t)p, (uint32_t)r, 0x52415953u, 0u};
            philox4x32_10(c, k0, k1);
            const float u1 = ((float)(c[0] >> 8) + 0.5f) * (1.0f / 16777216.0f);
            const float u2 = ((float)(c[2] >> 8) + 0.5f) * (1.0f / 16777216.0f);
            const float rad = sqrtf(-2.0f * logf(u1));
            float sn, cs;
            sincospif(2.0f * u2, &sn, &cs);
            x[2 * q] = rad * cs;
            x[2 * q + 1] = 2 * p + 1 < d ? rad * sn : 0.f;
            ss += x[2 * q] * x[2 * q] + x[2 * q + 1] * x[2 * q + 1];
        }
    }
    // pairs beyond the register block (d > 1024) are stored unnormalised first
    for (int p = lane + 32 * kPer; p < npairs; p += 32) {
        uint32_t c[4] = {(uint32_t)p, (uint32_t)r, 0x52415953u, 0u};
        philox4x32_10(c, k0, k1);
        const float u1 = ((float)(c[0] >> 8) + 0.5f) * (1.0f / 16777216.0f);
        const float u2 = ((float)(c[2] >> 8) + 0.5f) * (1.0f / 16777216.0f);
        const float rad = sqrtf(-2.0f * logf(u1));
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        const float x0 = rad * cs;
        ur[2 * p] = x0;
        ss += x0 * x0;
        if (2 * p + 1 < d) {
            const float x1 = rad * sn;
            ur[2 * p + 1] = x1;
            ss += x1 * x1;
        }
    }
    const float inv = 1.0f / sqrtf(warp_sum(ss));
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int p = lane + 32 * q;
        if (p < npairs) {
            ur[2 * p] = (double)(x[2 * q] * inv);
            if (2 * p + 1 < d) ur[2 * p + 1] = (double)(x[2 * q + 1] * inv);
        }
    }
    for (int p = lane + 32 * kPer; p < npairs; p += 32) {
        ur[2 * p] = (double)((float)ur[2 * p] * inv);
        if (2 * p + 1 < d) ur[2 * p + 1] = (double)((float)ur[2 * p + 1] * inv);
    }
    __syncwarp();
    const double tmin = warp_exit_min(lane, d, ur, half);
    if (lane == 0) texit[r] = tmin;
}

// Tier and rank of every sample, histogram of buckets: a warp per ray, rays in turn, the
// histogram kept per CTA. l is compared as order-preserving integers (a rank is n_steps
// comparisons per sample: 2 n_steps FP64 instructions took 260 us for 16384 rays x 64
// samples together with a global atomic per sample, 40 us now); a NaN is never greater.
constexpr int RB_WARPS = 8;
__global__ void __launch_bounds__(32 * RB_WARPS) k_ray_bucket(const double *ell, int n_rays, int S, int32_t *bucket,
                                                              uint32_t *hist) {
    extern __shared__ uint64_t sh[];  // [RB_WARPS][S], then the histogram [2 S]
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    uint64_t *row = sh + (size_t)wl * S;
    uint32_t *h = reinterpret_cast<uint32_t *>(sh + (size_t)RB_WARPS * S);
    for (int b = threadIdx.x; b < 2 * S; b += blockDim.x) h[b] = 0;
    __syncthreads();
    for (int r = blockIdx.x * RB_WARPS + wl; r < n_rays; r += gridDim.x * RB_WARPS) {
        for (int j = lane; j < S; j += 32) {
            const double l = ell[(size_t)r * S + j];
            const uint64_t b = (uint64_t)__double_as_longlong(l);
            // 0: below every key of a number; -0 as +0
            row[j] = (b << 1) > 0xffe0000000000000ull ? 0ull : ordered_bits((b << 1) == 0 ? 0.0 : l);
        }
        __syncwarp();
        constexpr uint64_t kNegInf = 0x000fffffffffffffull;  // ordered_bits(-inf)
        for (int j = lane; j < S; j += 32) {
            const uint64_t l = row[j];
            const uint64_t left = j > 0 ? row[j - 1] : kNegInf;
            const uint64_t right = j + 1 < S ? row[j + 1] : kNegInf;
            const bool nan = l == 0;
            const int tier = (!nan && left != 0 && right != 0 && l > left && l >= right) ? 0 : 1;
            int rank = 0;
            if (!nan)
                for (int j2 = 0; j2 < S; ++j2) {
                    const uint64_t l2 = row[j2];
                    rank += (l2 > l || (l2 == l && j2 < j)) ? 1 : 0;
                }
            const int b = tier * S + rank;
            bucket[(size_t)r * S + j] = b;
            atomicAdd(&h[b], 1u);
        }
        __syncwarp();
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 2 * S; b += blockDim.x)
        if (h[b]) atomicAdd(&hist[b], h[b]);
}

__device__ __forceinline__ void sample_key(const double *ell, int64_t f, uint64_t &hi, uint32_t &lo) {
    hi = ~ordered_bits(ell[f]);  // ascending hi = descending l
    lo = (uint32_t)f;
}

// The bucket that holds the n_starts-th sample (state[0]), the rank of that sample inside it
// (state[1], from 1), and the list of the bucket's samples (one per ray at most of finite ones,
// but every NaN sample has tier 1, rank 0, so the list has room for all samples): every CTA
// finds the bucket from the histogram itself.
__global__ void __launch_bounds__(256) k_cut_gather(const int32_t *bucket, int64_t total, const uint32_t *hist,
                                                    int nbins, int n_starts, uint64_t *state, int32_t *list) {
    __shared__ uint32_t wsum[8];
    __shared__ int s_cut;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per = (nbins + 255) / 256, b0 = threadIdx.x * per;
    uint32_t own = 0;
    for (int b = b0; b < b0 + per && b < nbins; ++b) own += hist[b];
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    uint32_t before = incl - own;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    if (before < (uint32_t)n_starts && before + own >= (uint32_t)n_starts) {
        int b = b0;
        while (before + hist[b] < (uint32_t)n_starts) before += hist[b++];
        s_cut = b;
        if (blockIdx.x == 0) {
            state[0] = (uint64_t)b;
            state[1] = (uint64_t)n_starts - before;
        }
    }
    __syncthreads();
    const int cut = s_cut;
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(state + 4);
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < total; f += (int64_t)gridDim.x * blockDim.x)
        if (bucket[f] == cut) list[atomicAdd(cnt, 1ull)] = (int32_t)f;
}

// The 96-bit key of that sample (state[2], state[3]) by radix selection over the listed
// samples, 8 bits a pass, in one CTA; it stops as soon as one sample is left, or all that
// are left are selected. (Two launches a pass over every sample, the digit found by one
// thread: 24 launches, 150 us for 16384 samples.)
__global__ void __launch_bounds__(1024) k_cut_select(const double *ell, const int32_t *list, uint64_t *state) {
    __shared__ uint32_t h[256];
    __shared__ uint32_t s_digit, s_cum, s_left;
    const int n = (int)state[4];
    uint64_t phi = 0, need = state[1];
    uint32_t plo = 0;
    for (int pass = 0; pass < 12; ++pass) {
        if (threadIdx.x < 256) h[threadIdx.x] = 0;
        __syncthreads();
        const int sft = pass < 8 ? 56 - 8 * pass : 24 - 8 * (pass - 8);
        auto match = [&](int e, uint32_t &digit) {
            uint64_t hi;
            uint32_t lo;
            sample_key(ell, list[e], hi, lo);
            if (pass < 8) {
                digit = (uint32_t)(hi >> sft) & 0xffu;
                return pass == 0 || (hi >> (sft + 8)) == (phi >> (sft + 8));
            }
            digit = (lo >> sft) & 0xffu;
            return hi == phi && (pass == 8 || (lo >> (sft + 8)) == (plo >> (sft + 8)));
        };
        for (int e = threadIdx.x; e < n; e += blockDim.x) {
            uint32_t digit;
            if (match(e, digit)) atomicAdd(&h[digit], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 32) {  // the digit where the count reaches need: eight bins a lane
            const int lane = threadIdx.x;
            uint32_t own = 0;
            for (int q = 0; q < 8; ++q) own += h[8 * lane + q];
            uint32_t incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            uint32_t cum = incl - own;
            if (cum < need && incl >= need) {
                int q = 8 * lane;
                while (cum + h[q] < need) cum += h[q++];
                s_digit = (uint32_t)q;
                s_cum = cum;
                s_left = h[q];
            }
        }
        __syncthreads();
        const uint32_t dg = s_digit, left = s_left;
        need -= s_cum;
        if (pass < 8)
            phi |= (uint64_t)dg << sft;
        else
            plo |= dg << sft;
        if (need == left) {  // every sample with this prefix is selected: the largest such key
            if (pass < 8) {
                phi |= (1ull << sft) - 1ull;
                plo = 0xffffffffu;
            } else {
                plo |= (1u << sft) - 1u;
            }
            break;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        state[2] = phi;
        state[3] = (uint64_t)plo;
    }
}

__device__ __forceinline__ bool is_selected(const double *ell, const int32_t *bucket, int64_t f,
                                            const uint64_t *state) {
    const int64_t b = bucket[f];
    const int64_t cut = (int64_t)state[0];
    if (b < cut) return true;
    if (b > cut) return false;
    uint64_t hi;
    uint32_t lo;
    sample_key(ell, f, hi, lo);
    const uint64_t khi = state[2];
    const uint32_t klo = (uint32_t)state[3];
    return hi < khi || (hi == khi && lo <= klo);
}

constexpr int SEL_BLOCK = 1024;

__global__ void __launch_bounds__(SEL_BLOCK) k_sel_count(const double *ell, const int32_t *bucket, int64_t total,
                                                         const uint64_t *state, int32_t *blockcnt) {
    const int64_t f = (int64_t)blockIdx.x * SEL_BLOCK + threadIdx.x;
    const int sel = (f < total) && is_selected(ell, bucket, f, state);
    const int cnt = __syncthreads_count(sel);
    if (threadIdx.x == 0) blockcnt[blockIdx.x] = cnt;
}

__global__ void __launch_bounds__(SEL_BLOCK) k_sel_scatter(const double *ell, const int32_t *bucket, int64_t total,
                                                           const uint64_t *state, const int32_t *blockcnt,
                                                           int64_t *idx) {
    __shared__ int warp_tot[32];
    __shared__ long long s_base;
    // offset of this block = sum of the preceding block counts
    long long part = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += SEL_BLOCK) part += blockcnt[b];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_tot[wid] = (int)part;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long s = 0;
        for (int w = 0; w < SEL_BLOCK / 32; ++w) s += warp_tot[w];
        s_base = s;
    }
    __syncthreads();
    const int64_t f = (int64_t)blockIdx.x * SEL_BLOCK + threadIdx.x;
    const int sel = (f < total) && is_selected(ell, bucket, f, state);
    const unsigned bal = __ballot_sync(0xffffffffu, sel);
    const int in_warp = __popc(bal & ((1u << lane) - 1u));
    __syncthreads();
    if (lane == 0) warp_tot[wid] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < SEL_BLOCK / 32; ++w) {
            const int t = warp_tot[w];
            warp_tot[w] = s;
            s += t;
        }
    }
    __syncthreads();
    if (sel) idx[s_base + warp_tot[wid] + in_warp] = f;
}

__global__ void __launch_bounds__(256) k_gather_starts(int d, const double *c, const double *u, const double *texit,
                                                       int n_steps, const int64_t *idx, const double *ell_all,
                                                       int n_starts, double *starts, double *ell_starts) {
    const int lane = threadIdx.x & 31;
    const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= n_starts) return;
    const int64_t f = idx[s];
    const int r = (int)(f / n_steps), j = (int)(f % n_steps);
    const double scale = mul_rn(div_rn((double)(j + 1), (double)n_steps), texit[r]);
    for (int i = lane; i < d; i += 32)
        starts[(size_t)s * d + i] = add_rn(c[i], mul_rn(scale, u[(size_t)r * d + i]));
    if (lane == 0) ell_starts[s] = ell_all[f];
}

}  // namespace

size_t select_blocks(int64_t total) { return (size_t)((total + SEL_BLOCK - 1) / SEL_BLOCK); }

void launch_ray_dirs(int d, int n_rays, uint64_t seed, const ProbView &pv, double *u, double *texit, bool fp32,
                     cudaStream_t s) {
    const int warps_per_block = 8;
    const unsigned grid = (unsigned)((n_rays + warps_per_block - 1) / warps_per_block);
    note_launch();
    if (fp32)
        k_ray_dirs_f32<<<grid, 256, 0, s>>>(d, n_rays, (uint32_t)seed, (uint32_t)(seed >> 32), pv.half, u, texit);
    else
        k_ray_dirs<<<grid, 256, 0, s>>>(d, n_rays, (uint32_t)seed, (uint32_t)(seed >> 32), pv.half, u, texit);
}

void launch_select_starts(const double *ell_all, int n_rays, int n_steps, int n_starts, const SelectWs &w,
                          cudaStream_t s) {
    const int64_t total = (int64_t)n_rays * n_steps;
    const int nbins = 2 * n_steps;
    cudaMemsetAsync(w.hist, 0, sizeof(uint32_t) * (size_t)nbins, s);
    cudaMemsetAsync(w.state, 0, sizeof(uint64_t) * 8, s);
    const size_t sm = sizeof(uint64_t) * RB_WARPS * n_steps + sizeof(uint32_t) * nbins;
    if (sm > kFreeSmem) allow_smem(k_ray_bucket, (int)sm);
    const int rb = (n_rays + RB_WARPS - 1) / RB_WARPS;
    note_launch();
    k_ray_bucket<<<rb < 608 ? rb : 608, 32 * RB_WARPS, sm, s>>>(ell_all, n_rays, n_steps, w.bucket, w.hist);
    const int hb = (int)((total + 255) / 256 < 1184 ? (total + 255) / 256 : 1184);
    note_launch();
    k_cut_gather<<<hb, 256, 0, s>>>(w.bucket, total, w.hist, nbins, n_starts, w.state, w.list);
    note_launch();
    k_cut_select<<<1, 1024, 0, s>>>(ell_all, w.list, w.state);
    const int nb = (int)select_blocks(total);
    note_launch();
    k_sel_count<<<nb, SEL_BLOCK, 0, s>>>(ell_all, w.bucket, total, w.state, w.blockcnt);
    note_launch();
    k_sel_scatter<<<nb, SEL_BLOCK, 0, s>>>(ell_all, w.bucket, total, w.state, w.blockcnt, w.idx);
}

void launch_gather_starts(const ProbView &pv, const double *u, const double *texit, int n_steps, const int64_t *idx,
                          const double *ell_all, int n_starts, double *starts, double *ell_starts, cudaStream_t s) {
    note_launch();
    k_gather_starts<<<(n_starts + 7) / 8, 256, 0, s>>>(pv.d, pv.c, u, texit, n_steps, idx, ell_all, n_starts, starts,
                                                       ell_starts);
}

}  // namespace sb
