// nr_vi.cu -- variational inference for a co-fitted slab model on the GPU,
// many independent restarts at once (arXiv 2509.06924, Sec. 2.4; the LED
// co-fit of Sec. 4.2 runs 100 restarts of a multivariate normal q in an
// unconstrained space, optimised by Adam).
//
// phi of one restart: mu [P] and the lower triangle of the Cholesky factor L,
// packed row by row ((i, j <= i) at i (i + 1) / 2 + j) with log L_ii on the
// diagonal.  One iteration with a standard-normal draw e (an input) is three
// launches, each one block per restart around the likelihood's gradient:
//   vi_sample: u = mu + L e, the part of the ELBO estimate that does not
//              involve the likelihood, e^T e / 2 + sum_i log L_ii + P/2 log 2 pi,
//              and the packed parameters of the restart's stacks at u;
//   the gradient kernels on those stacks;
//   vi_adam:   log pi(u) and its gradient g (as cofit_stage), the gradient of
//              the single-sample negative ELBO (Eqs. 22-24, e held fixed:
//              d/d mu = -g, d/d L_ij = -g_i e_j, d/d log L_ii =
//              -g_i e_i L_ii - 1) and one Adam step of every entry of phi (the
//              moments and the step in FP32 arithmetic on FP64 storage); the
//              ELBO estimate log pi(u) + (the part above) per restart.
//
// What bounds them: latency, for the tens to hundreds of restarts of a fit
// (FP64 chains of exp, log1p and divisions, dependent loads), so the work of
// a restart is spread over a block: eight lanes share a row of L (coalesced),
// and theta is formed once per parameter, not once per packed slot.  100
// restarts of a 51-parameter co-fit: sample 24, gather 6, pull-back 16 and
// Adam 14 us as four launches of a warp per restart; the iteration fell from
// 193 to 172 us (176 with the present gradient kernel).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "nr_cofit.cuh"
#include "nr_internal.h"

namespace nrimpl {
namespace {

constexpr unsigned kMask = 0xffffffffu;
constexpr double kHalfLog2Pi = 0.91893853320467274178032973640562; // ln(2 pi) / 2

constexpr int kSampleBlock = 256;
constexpr int kSampleStageP = 2048; // parameters whose draw and theta are staged in shared memory

// sum over the block in a fixed order (result in thread 0); sh: one double per warp
__device__ __forceinline__ double block_sum(double v, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kMask, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)blockDim.x >> 5; ++w) s += sh[w];
    return s;
}

__global__ void __launch_bounds__(kSampleBlock)
vi_sample_kernel(const double *phi, const double *eps, int P, int64_t nphi, double *u, double *part, int32_t *t_dev,
                 double beta1, double beta2, double *bias, const CofitGatherArgs a)
{
    extern __shared__ double sh_eu[]; // staged: e_r, then theta_r [P]; u_r [P]
    __shared__ double sh_w[kSampleBlock / 32];
    const int r = blockIdx.x, tid = threadIdx.x;
    // the iteration counter lives on the device, so a captured iteration
    // advances it on every replay; vi_adam (later in the stream) reads the
    // Adam bias corrections 1 / (1 - beta^t) formed here once per iteration
    // (by the last warp, beside the others' work)
    if (r == 0 && tid == kSampleBlock - 1) {
        const int t = *t_dev + 1;
        *t_dev = t;
        bias[0] = 1.0 / (1.0 - pow(beta1, (double)t));
        bias[1] = 1.0 / (1.0 - pow(beta2, (double)t));
    }
    const bool staged = P <= kSampleStageP;
    const double *mu = phi + (int64_t)r * nphi;
    const double *tri = mu + P;
    const double *er = eps + (int64_t)r * P;
    double *ur = u + (int64_t)r * P;
    double *sh_e = sh_eu, *sh_u = sh_eu + P;
    // mu_i + L_ii e_i
    double acc = 0.0;
    for (int i = tid; i < P; i += kSampleBlock) {
        const double ei = er[i], lii = tri[(int64_t)i * (i + 1) / 2 + i];
        const double w = mu[i] + exp(lii) * ei;
        if (staged) {
            sh_e[i] = ei;
            sh_u[i] = w;
        } else {
            ur[i] = w;
        }
        acc += 0.5 * ei * ei + lii + kHalfLog2Pi;
    }
    acc = block_sum(acc, sh_w); // synchronises: the terms above are visible to the block
    if (tid == 0) part[r] = acc;
    // + sum_{j < i} L_ij e_j, eight lanes a row
    const double *e = staged ? sh_e : er;
    for (int i0 = 0; i0 < P; i0 += kSampleBlock / 8) {
        const int i = i0 + (tid >> 3);
        double s = 0.0;
        if (i < P) {
            const double *row = tri + (int64_t)i * (i + 1) / 2;
            for (int j = tid & 7; j < i; j += 8) s += row[j] * e[j];
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(kMask, s, o);
        if (i < P && (tid & 7) == 0) {
            s += staged ? sh_u[i] : ur[i];
            if (staged) sh_u[i] = s;
            ur[i] = s;
        }
    }
    __syncthreads();
    // theta, and the stacks' packed slots and resolution scales
    auto theta = [&](int k) {
        const double s = 1.0 / (1.0 + exp(-(staged ? sh_u[k] : ur[k])));
        return a.lo[k] + (a.hi[k] - a.lo[k]) * s;
    };
    if (staged) {
        for (int k = tid; k < P; k += kSampleBlock) sh_e[k] = theta(k);
        __syncthreads();
    }
    for (int slot = tid; slot < a.NS; slot += kSampleBlock) {
        const int k = a.src[slot];
        a.params[(int64_t)r * a.NS + slot] = k < 0 ? a.val[slot] : staged ? sh_e[k] : theta(k);
    }
    if (a.res_param >= 0)
        for (int c = tid; c < a.NC; c += kSampleBlock)
            a.dq_scale[(int64_t)r * a.NC + c] = staged ? sh_e[a.res_param] : theta(a.res_param);
}

// The restart's gradient and draw are staged as floats in shared memory (when
// P <= kAdamStageP; else the gradient goes through global memory), and the
// moments and the step are formed in FP32 arithmetic: phi, m and v keep their
// FP64 storage, so phi accumulates its updates at full precision, while the
// update itself (a heuristic scaling of the gradient, whose own error is
// ~1e-5) needs no more than FP32.  In FP64 the square root and division
// alone bound this kernel on GB300's FP64 rate.
constexpr int kAdamBlock = 256;
constexpr int kAdamStageP = 4096;

__global__ void __launch_bounds__(kAdamBlock)
vi_adam_kernel(double *phi, double *m, double *v, const double *eps, double *g, const double *part, int64_t nphi,
               const double *bias, float lr, float beta1, float beta2, float eps_adam, double *elbo,
               const CofitStageArgs a)
{
    extern __shared__ float sh_ge[]; // g_r [P], eps_r [P]
    __shared__ double sh_w[kAdamBlock / 32];
    const int r = blockIdx.x, tid = threadIdx.x, P = a.P;
    const bool stage = P <= kAdamStageP;
    const double *ur = a.u + (int64_t)r * P, *er = eps + (int64_t)r * P;
    double *gr = g + (int64_t)r * P;
    double lp = 0.0;
    for (int i = tid; i < a.n_contrast; i += kAdamBlock) lp += a.ll[(int64_t)r * a.n_contrast + i];
    for (int k = tid; k < P; k += kAdamBlock) {
        const double gk = cofit_pull_back(a, r, k, ur[k], lp);
        if (stage) {
            sh_ge[k] = (float)gk;
            sh_ge[P + k] = (float)er[k];
        } else {
            gr[k] = gk;
        }
    }
    lp = block_sum(lp, sh_w); // synchronises: the gradient is visible to the block
    if (tid == 0 && elbo) elbo[r] = lp + part[r];
    auto gi = [&](int i) { return stage ? sh_ge[i] : (float)gr[i]; };
    auto ej = [&](int j) { return stage ? sh_ge[P + j] : (float)er[j]; };
    const float c0 = (float)bias[0], c1 = (float)bias[1];
    double *phr = phi + (int64_t)r * nphi, *mr = m + (int64_t)r * nphi, *vr = v + (int64_t)r * nphi;
    for (int64_t p = tid; p < nphi; p += kAdamBlock) {
        float grad;
        if (p < P) {
            grad = -gi((int)p);
        } else {
            // packed triangle index -> (i, j): i (i + 1) / 2 <= q < (i + 1) (i + 2) / 2
            const int64_t q = p - P;
            int i = (int)((sqrtf(8.f * (float)q + 1.f) - 1.f) * 0.5f); // corrected below
            while ((int64_t)(i + 1) * (i + 2) / 2 <= q) ++i;
            while ((int64_t)i * (i + 1) / 2 > q) --i;
            const int j = (int)(q - (int64_t)i * (i + 1) / 2);
            grad = (i == j) ? -gi(i) * ej(i) * expf((float)phr[p]) - 1.f : -gi(i) * ej(j);
        }
        const float mm = fmaf(beta1, (float)mr[p], (1.f - beta1) * grad);
        const float vv = fmaf(beta2, (float)vr[p], (1.f - beta2) * grad * grad);
        mr[p] = mm;
        vr[p] = vv;
        phr[p] -= (double)(lr * (mm * c0) / (sqrtf(vv * c1) + eps_adam));
    }
}

} // namespace

cudaError_t launch_vi_sample(const double *phi, const double *eps, int R, int P, double *u, double *part,
                             int32_t *t_dev, double beta1, double beta2, double *bias, const CofitGatherArgs &a,
                             cudaStream_t st)
{
    if (R == 0) return cudaSuccess;
    const int64_t nphi = (int64_t)P + (int64_t)P * (P + 1) / 2;
    const size_t smem = P <= kSampleStageP ? sizeof(double) * 2 * (size_t)P : 0;
    vi_sample_kernel<<<R, kSampleBlock, smem, st>>>(phi, eps, P, nphi, u, part, t_dev, beta1, beta2, bias, a);
    return cudaGetLastError();
}

cudaError_t launch_vi_adam(double *phi, double *m, double *v, const double *eps, double *g, const double *part,
                           const double *bias, double lr, double beta1, double beta2, double eps_adam, double *elbo,
                           const CofitStageArgs &a, cudaStream_t st)
{
    const int64_t nphi = (int64_t)a.P + (int64_t)a.P * (a.P + 1) / 2;
    if (a.C == 0 || nphi == 0) return cudaSuccess;
    const size_t smem = a.P <= kAdamStageP ? sizeof(float) * 2 * (size_t)a.P : 0;
    vi_adam_kernel<<<a.C, kAdamBlock, smem, st>>>(phi, m, v, eps, g, part, nphi, bias, (float)lr, (float)beta1,
                                                  (float)beta2, (float)eps_adam, elbo, a);
    return cudaGetLastError();
}

} // namespace nrimpl
