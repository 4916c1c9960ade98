// nr_cofit.cuh -- the pull-back of the co-fit model's likelihood gradient to
// the unconstrained coordinates, shared by the HMC stages (nr_hmc.cu) and the
// variational step (nr_vi.cu).
#pragma once

#include <cmath>
#include <cstdint>

#include <cuda_runtime.h>

#include "nr_internal.h"

namespace nrimpl {
namespace {

// d log pi / d u_k of chain c: the packed gradient summed over the slots that
// copy parameter k, the chain rule through the sigmoid, and the prior term,
// whose logarithm is added to lp
__device__ __forceinline__ double cofit_pull_back(const CofitStageArgs &a, int c, int k, double uk, double &lp)
{
    const double *gpk = a.gpk + (int64_t)c * a.NS;
    const double s = 1.0 / (1.0 + exp(-uk));
    const double au = fabs(uk);
    lp += -au - 2.0 * log1p(exp(-au));
    double gt = 0.0;
    for (int t = a.tie_ptr[k]; t < a.tie_ptr[k + 1]; ++t) gt += gpk[a.tie_slot[t]];
    if (k == a.res_param) {
        // d loglik / d f = (d loglik / d ln f) / f, summed over the contrasts
        const double f = a.lo[k] + (a.hi[k] - a.lo[k]) * s;
        double gr = 0.0;
        for (int i = 0; i < a.n_contrast; ++i) gr += a.gres[(int64_t)c * a.n_contrast + i];
        gt += gr / f;
    }
    return gt * (a.hi[k] - a.lo[k]) * s * (1.0 - s) + (1.0 - 2.0 * s);
}

} // namespace
} // namespace nrimpl
