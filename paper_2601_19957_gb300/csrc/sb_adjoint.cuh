// sb_adjoint.cuh -- FP64 adjoint of log Z (adjoint.cu).
#pragma once
#include <vector>

#include "sb_internal.cuh"
#include "sb_laplace.cuh"

namespace sb {

constexpr int kMaxAdjModes = 1024;

struct AdjWs {
    // per mode of a group, but for P_k: H (its factor C), C^-1, merge scratch, C^-1 L_k, |X_k|^2 partials
    double *P, *H, *Ci, *T2, *X, *trp;
    double *Z, *R, *qpart, *gbar, *ell, *GK;
    double *V, *Y, *WV;  // [K + 1][d]: right-hand sides, C^-1 V, W V
    double *T, *eps, *gam, *U, *PY, *pi;
    int32_t *info, *count, *onehot, *p_done, *p_need;
    uint32_t *bar;  // grid-barrier state of the cooperative factorisation
};

void adjoint_carve(Carver &cv, AdjWs &w, int d, int K);
sb_status adjoint_run(const ProbView &pv, const AdjWs &w, const double *modes, const double *logZk, int n_modes,
                      double grad_logZ, double *dmu, double *dL, cudaStream_t s);

}  // namespace sb
