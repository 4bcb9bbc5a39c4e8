// sb_small_f64.cuh -- FP64 likelihood and L-BFGS of small problems, whole walkers in one
// launch (small_f64.cu).
#pragma once
#include "sb_internal.cuh"
#include "sb_lbfgs.cuh"

namespace sb {

// Whether the packed triangles of all L_k fit one SM's shared memory beside the walkers'
// buffers (d <= 128), so that the launchers below take the problem (m: history pairs).
bool small_f64_fits(int d, int K, int m);

// The whole refinement of the n walkers at starts: sb_refine's FP64 results (x, l, status,
// iters, the evaluation count added to *n_evals after it is cleared). a: knobs, S, Y and
// the walker counter a.n_act; Z: [n][K][d] scratch.
void launch_small_refine_f64(const ProbView &pv, const LbfgsArgs<double> &a, const double *starts, int n, double *Z,
                             double *x_out, double *ell_out, int8_t *status_out, int32_t *iters_out,
                             int64_t *n_evals, cudaStream_t s);

// l (and grad l when a.G is given, which takes a.Z as scratch) at gathered points, or at
// ray samples (rays): a's ell and G outputs; R and qpart are not written.
void launch_small_points_f64(const LikF64Args &a, bool rays, cudaStream_t s);

}  // namespace sb
