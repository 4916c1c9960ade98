// nr_profile.cu -- SLD and absorption depth profiles of a batch of stacks.
//
// The paper's figures draw the scattering-length-density profile through
// the film with posterior bands (Sec. 4.1, quartz; Sec. 4.2, LED device):
// one profile per posterior sample, evaluated on a common depth grid.  With
// Gaussian interfacial roughness every interface is an error-function step,
//   rho(z) = rho_0 + sum_j (rho_{j+1} - rho_j) (1 + erf((z - z_j) / (sqrt(2) sigma_j))) / 2,
// z_j = d_1 + ... + d_j the depth of interface j (z_0 = 0), and the same for
// the absorption iota(z) (iota_0 = 0).  sigma_j = 0 is the sharp step, which
// takes the deeper medium's value at z = z_j.
//
// What bounds it.  Written plainly the kernel is a stream of error functions,
// n + 1 per depth, and far from the rate its outputs could be stored at.  But
// an interface whose error function is saturated over a whole run of depths
// (|z - z_j| >= 4 sqrt(2) sigma_j, where erff is exactly +-1) is a constant
// there, and a depth grid meets one to three interfaces per run that are not.
// So a warp takes runs of 64 depths (two a lane).  Its lanes first hold one
// interface each against the run's span: the deepest interface wholly above
// the run gives the run's base value, the SLD of the medium under it (exact),
// and only the interfaces that a ballot names are evaluated, each as its
// difference from what the base already counts.  That holds for any order of
// the depths (a run then just spans more).  16384 stacks of ten layers x 512
// depths, both curves: 165 -> 49 us a call (1.5 TB/s of its 67 MB output and
// 6 MB of parameters; stacks of one layer count upload no metadata either).
//
// A CTA stages 8 stacks at a time, one per warp: lane j forms interface j's
// depth (FP64, kept as a float pair), its steps and its reach;
// then the warps share out the 8 stacks' runs.  z - z_j is formed as
// (z - z_hi) - z_lo, exact near the interface (where the error function is
// steep) and FP32-accurate elsewhere.  Few stacks leave SMs idle that way, so
// the runs of a group are then shared out to several CTAs, each of which
// stages the group for itself, as long as every warp gets a run: 8 stacks x
// 65536 depths, ten layers, 409 -> 27 us (222 with a CTA per stack that
// evaluated every interface), one layer 483 -> 27 us (89).
#include <cuda_runtime.h>

#include <cstdint>

#include "nr_internal.h"

namespace nrimpl {
namespace {

constexpr int kProfileBlock = 256;
constexpr int kProfileWarps = kProfileBlock / 32; // stacks staged together
constexpr int kRun = 64;                          // depths of a run
constexpr int kIfMax = NR_MAX_LAYERS + 1;         // interfaces of a stack
constexpr int kRounds = (kIfMax + 31) / 32;
constexpr float kErfOne = 4.f;                    // erff(x) == +-1 from here on
constexpr unsigned kAll = 0xffffffffu;

struct ProfileStack {
    float4 at[kIfMax];   // interface j: depth (hi, lo), 1 / (sqrt(2) sigma_j) or 0 (sharp), SLD step
    float4 med[kIfMax];  // its absorption step, its reach (beyond it erff is +-1), SLD and absorption below it
    float rho0;
    int n;               // layers; -1: a non-finite parameter, every interface is evaluated everywhere
};

// order-preserving map of floats to signed integers
__device__ __forceinline__ int float_order(float x)
{
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// finite, by the exponent bits (an FP64 comparison of a warp takes 16 cycles of its SM)
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// below zero, by the bits (the float of a tiny negative number is -0)
__device__ __forceinline__ bool negative_bits(double v)
{
    const int h = __double2hiint(v);
    return h < 0 && ((h & 0x7fffffff) | __double2loint(v)) != 0;
}

// One warp stages stack parameters p (n layers) into st.
__device__ void stage_profile(ProfileStack &st, const double *p, int n, int lane, int32_t *status)
{
    double base = 0.0; // depth of the first interface of the round
    bool bad = false, sharp = false;
    for (int j = lane; j <= n; j += 32) sharp |= __double2hiint(p[3 * n + 3 + j]) < 0x38000000; // below 2^-127
    sharp = __any_sync(kAll, sharp);
    for (int j0 = 0; j0 <= n; j0 += 32) {
        const int j = j0 + lane;
        const bool on = j <= n;
        // the thicknesses above, added in FP64.  A stack with a sharp step adds
        // them from the top down, as a program forms the depths it puts such a
        // step's grid points on; the others by a scan (10 layers, 512 depths,
        // 16384 stacks: 2 of 53 us less than all from the top down).
        const double d = j < n ? p[j] : 0.0;
        const int last = min(31, n - j0);
        double depth = base;
        if (sharp) {
            for (int i = 0; i < last; ++i) {
                const double di = __shfl_sync(kAll, d, i);
                if (lane > i) depth += di;
            }
            base = __shfl_sync(kAll, depth + d, 31);
        } else {
            double sum = d; // of the thicknesses of this round down to layer j + 1
            for (int o = 1; o <= last; o <<= 1) {
                const double t = __shfl_up_sync(kAll, sum, o);
                if (lane >= o) sum += t;
            }
            const double above = __shfl_up_sync(kAll, sum, 1);
            if (lane > 0) depth += above;
            if (n - j0 >= 32) base += __shfl_sync(kAll, sum, 31);
        }
        const float h = (float)depth, l = (float)(depth - (double)h);
        if (on) {
            const double rj = p[n + j], rj1 = p[n + j + 1];
            const double ij = j >= 1 ? p[2 * n + 2 + j - 1] : 0.0, ij1 = p[2 * n + 2 + j];
            const double sgd = p[3 * n + 3 + j];
            const float sg = (float)sgd;
            st.at[j] = make_float4(h, l, sg > 0.f ? 1.f / (1.41421356237f * sg) : 0.f, (float)(rj1 - rj));
            // a little past 4 sqrt(2) sigma, and past the rounding of z - z_j
            const float reach = fmaf(1.41421356237f * 1.00001f * kErfOne, fmaxf(sg, 0.f), 1e-6f * fabsf(h) + 1e-30f);
            st.med[j] = make_float4((float)(ij1 - ij), reach, (float)rj1, (float)ij1);
            if (j == 0) st.rho0 = (float)rj;
            bad |= !finite_bits(depth) || !finite_bits(rj) || !finite_bits(rj1) || !finite_bits(ij) ||
                   !finite_bits(ij1) || !finite_bits(sgd) || negative_bits(sgd);
        }
    }
    bad = __any_sync(kAll, bad);
    if (lane == 0) {
        st.n = bad ? -1 - n : n;
        if (bad) atomicOr(status, NR_FLAG_NONFINITE_PARAM);
    }
}

__global__ void __launch_bounds__(kProfileBlock)
nr_profile_kernel(const double *params, const int64_t *par_off, const int32_t *n_layers, int n_same, int n_stacks,
                  int parts, const float *z, int nz, float *rho_out, float *iota_out, int32_t *status)
{
    __shared__ ProfileStack sh[kProfileWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int runs = (nz + kRun - 1) / kRun;
    const int groups = (n_stacks + kProfileWarps - 1) / kProfileWarps;
    // parts > 1: one (group, part) per CTA
    for (int g = blockIdx.x / parts; g < groups; g += gridDim.x / parts) {
        const int s0 = g * kProfileWarps, part = blockIdx.x - blockIdx.x / parts * parts;
        __syncthreads(); // the previous stacks' entries are no longer read
        if (const int s = s0 + warp; s < n_stacks) {
            const int64_t off = par_off ? par_off[s] : (4 * (int64_t)n_same + 6) * s;
            stage_profile(sh[warp], params + off, n_layers ? n_layers[s] : n_same, lane, status);
        }
        __syncthreads();
        const int here = min(kProfileWarps, n_stacks - s0);
        // the 8 stacks' runs, run by run, in equal shares: a warp forms a run's
        // span once for the stacks it takes it for
        const int total = here * runs, warps = kProfileWarps * parts, share = (total + warps - 1) / warps;
        int at = (part * kProfileWarps + warp) * share;
        const int end = min(at + share, total);
        int run = at / here, k = at - run * here;
        float z0 = 0.f, z1 = 0.f, zlo = 0.f, zhi = 0.f, slack = 0.f;
        for (bool fresh = true; at < end; ++at, ++k) {
            if (k == here) {
                k = 0;
                ++run;
                fresh = true;
            }
            const int i0 = run * kRun + lane, i1 = i0 + 32;
            if (fresh) {
                fresh = false;
                z0 = z[min(i0, nz - 1)];
                z1 = z[min(i1, nz - 1)];
                // the run's span; a NaN depth or parameter evaluates everything
                const int o0 = float_order(z0), o1 = float_order(z1);
                zlo = order_float(__reduce_min_sync(kAll, min(o0, o1)));
                zhi = order_float(__reduce_max_sync(kAll, max(o0, o1)));
                slack = 1e-6f * fmaxf(fabsf(zlo), fabsf(zhi)); // rounding of z - z_j
            }
            const ProfileStack &st = sh[k];
            const int n = st.n >= 0 ? st.n : -1 - st.n;
            const bool plain = st.n >= 0 && zhi - zlo >= 0.f;
            unsigned above[kRounds], eval[kRounds]; // interfaces wholly above the run; those to evaluate
            int m = 0;                              // the base counts interfaces 0 .. m-1 whole
#pragma unroll
            for (int r = 0; r < kRounds; ++r) {
                above[r] = eval[r] = 0;
                if (32 * r > n) continue;
                const int j = 32 * r + lane;
                bool up = false, in = false;
                if (j <= n) {
                    const float zj = st.at[j].x, reach = st.med[j].y + slack;
                    up = plain && zlo - zj >= reach;
                    in = !up && !(plain && zj - zhi >= reach);
                }
                above[r] = __ballot_sync(kAll, up);
                eval[r] = __ballot_sync(kAll, in);
                if (above[r]) m = 32 * r + 32 - __clz(above[r]);
            }
            float r0 = st.rho0, a0 = 0.f;
            if (m > 0) {
                const float4 b = st.med[m - 1];
                r0 = b.z;
                a0 = b.w;
            }
            float r1 = r0, a1 = a0;
#pragma unroll
            for (int r = 0; r < kRounds; ++r) {
                if (32 * r > n) continue;
                // counted whole by the base, but not wholly above the run
                const unsigned whole = m >= 32 * r + 32 ? kAll : m > 32 * r ? (1u << (m - 32 * r)) - 1u : 0u;
                for (unsigned todo = eval[r] | (whole & ~above[r]); todo; todo &= todo - 1) {
                    const int b = __ffs(todo) - 1, j = 32 * r + b;
                    const float4 f = st.at[j];
                    const float di = st.med[j].x, base = whole >> b & 1 ? 1.f : 0.f;
                    const float t0 = (z0 - f.x) - f.y, t1 = (z1 - f.x) - f.y;
                    float st0, st1;
                    if (f.z > 0.f) {
                        st0 = 0.5f * (1.f + erff(t0 * f.z));
                        st1 = 0.5f * (1.f + erff(t1 * f.z));
                    } else {
                        st0 = t0 >= 0.f ? 1.f : 0.f;
                        st1 = t1 >= 0.f ? 1.f : 0.f;
                    }
                    r0 = fmaf(f.w, st0 - base, r0);
                    r1 = fmaf(f.w, st1 - base, r1);
                    a0 = fmaf(di, st0 - base, a0);
                    a1 = fmaf(di, st1 - base, a1);
                }
            }
            const int64_t row = (int64_t)(s0 + k) * nz;
            if (rho_out) {
                if (i0 < nz) rho_out[row + i0] = r0;
                if (i1 < nz) rho_out[row + i1] = r1;
            }
            if (iota_out) {
                if (i0 < nz) iota_out[row + i0] = a0;
                if (i1 < nz) iota_out[row + i1] = a1;
            }
        }
    }
}

} // namespace

cudaError_t launch_profile(const double *params, const int64_t *par_off, const int32_t *n_layers, int n_same,
                           int n_stacks, const float *z, int nz, float *rho_out, float *iota_out, int32_t *status, int sms,
                           cudaStream_t st)
{
    if (n_stacks == 0 || nz == 0) return cudaSuccess;
    const int groups = (n_stacks + kProfileWarps - 1) / kProfileWarps;
    // fewer groups than the SMs take CTAs (4 each): share out their runs
    const int runs = (nz + kRun - 1) / kRun;
    const int here = n_stacks < kProfileWarps ? n_stacks : kProfileWarps;
    const int most = (here * runs + kProfileWarps - 1) / kProfileWarps; // a run per warp
    int parts = 4 * sms / groups;
    parts = parts > most ? most : parts < 1 ? 1 : parts;
    const int grid = parts > 1 ? groups * parts : groups < 8 * sms ? groups : 8 * sms;
    nr_profile_kernel<<<grid, kProfileBlock, 0, st>>>(params, par_off, n_layers, n_same, n_stacks, parts, z, nz,
                                                      rho_out, iota_out, status);
    return cudaGetLastError();
}

} // namespace nrimpl
