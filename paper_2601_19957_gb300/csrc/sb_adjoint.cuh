// sb_adjoint.cuh -- FP64 adjoint of log Z (adjoint.cu).
#pragma once
#include <vector>

#include "sb_internal.cuh"
#include "sb_laplace.cuh"

namespace sb {

constexpr int kMaxAdjModes = 1024;

struct AdjWs {
    int group;  // modes taken together
    // per mode of a group, but for P_k: H (its factor C), C^-1, X_k = W L_k (before that the
    // merge scratch of C^-1), tr(W P_k)
    double *P, *H, *Ci, *X, *trp;
    double *Z, *R, *qpart, *gbar, *ell, *GK;
    double *V, *Y;   // [K + 1][d]: right-hand sides, then W applied to them; C^-1 V, or L_k^T of a vector per component
    double *T, *eps;  // [d] t, then W t
    double *gam;      // [K][d] P_k (W gbar - W g_k) for t, then gam_k
    double *pi;
    int32_t *info, *count, *onehot, *p_done, *p_need;
    uint32_t *bar;  // grid-barrier state of the cooperative factorisation
};

// Modes a group holds where the workspace allows it: four matrices of each kind, fewer with
// many components (X_k).
int adjoint_group(int K);
// Scratch for groups of `group` modes. group 0: one mode at a time in the least room (C^-1 in
// P_k's place, which is formed again for every mode). The results do not depend on it.
void adjoint_carve(Carver &cv, AdjWs &w, int d, int K, int group);
sb_status adjoint_run(const ProbView &pv, const AdjWs &w, const double *modes, const double *logZk, int n_modes,
                      double grad_logZ, double *dmu, double *dL, cudaStream_t s);

}  // namespace sb
