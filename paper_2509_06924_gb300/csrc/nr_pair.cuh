// nr_pair.cuh -- two evaluations per thread in paired FP32 arithmetic
// (sm_100-family add/mul/fma.rn.f32x2): the value types, the primitives with
// double-float guards and the pieces of the forward model that the kernels of
// nr_pair.cu and nr_roll.cu share.
#pragma once

#include "nr_device.cuh"

namespace nrimpl {
namespace {

// ---------------------------------------------------- paired FP32 values --
// f2 holds one FP32 value of each of the thread's two evaluations.
using f2 = float2;
struct b2 {
    bool x, y;
};

__device__ __forceinline__ f2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 pneg(f2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ f2 padd(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 psub(f2 a, f2 b) { return __fadd2_rn(a, pneg(b)); }
__device__ __forceinline__ f2 pmul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 pfma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 pabs(f2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ f2 pmax(f2 a, f2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ f2 psel(b2 c, f2 a, f2 b) { return make_float2(c.x ? a.x : b.x, c.y ? a.y : b.y); }
__device__ __forceinline__ f2 prcp(f2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }
__device__ __forceinline__ f2 prsqrt(f2 a) { return make_float2(rsqrt_approx(a.x), rsqrt_approx(a.y)); }
__device__ __forceinline__ f2 pex2(f2 a) { return make_float2(ex2_approx(a.x), ex2_approx(a.y)); }
__device__ __forceinline__ void psincos(f2 a, f2 &s, f2 &c)
{
    sincos_approx(a.x, s.x, c.x);
    sincos_approx(a.y, s.y, c.y);
}
__device__ __forceinline__ float half(f2 a, int h) { return h ? a.y : a.x; }
// cis_tab (nr_device.cuh) on both halves: (cos, sin) of ph + pl table steps
__device__ __forceinline__ void pcis_tab(f2 ph, f2 pl, const float *tab, f2 &cs, f2 &sn)
{
    const f2 t = padd(ph, bc(kRoundMagic));
    const f2 nt = padd(t, bc(-kRoundMagic));
    const int i0 = __float_as_int(t.x) & (kTabN - 1), i1 = __float_as_int(t.y) & (kTabN - 1);
    const f2 tc = make_float2(tab[i0], tab[i1]), ts = make_float2(tab[kTabN + i0], tab[kTabN + i1]);
    const f2 x = padd(psub(ph, nt), pl);
    const f2 z = pmul(x, x);
    const f2 sx = pmul(x, pfma(z, bc(kTabS3), bc(kTabS1)));
    const f2 cx = pfma(z, bc(kTabC2), bc(1.f));
    cs = pfma(tc, cx, pneg(pmul(ts, sx)));
    sn = pfma(ts, cx, pmul(tc, sx));
}
// (cos, sin) of |x| <= kNcSmall = 1/8 radians without reduction: minimax
// x (1 - d + b x^2) and 1 + x^2 (c + e x^2), within 1.6e-8 and 2e-10; five
// operations against the table's twelve and its four shared loads
__device__ __forceinline__ void pcis_small(f2 x, f2 &cs, f2 &sn)
{
    const f2 z = pmul(x, x);
    cs = pfma(z, pfma(z, bc(0.04163646f), bc(-0.49999985f)), bc(1.f));
    sn = pmul(x, pfma(z, bc(-0.16650396f), bc(0.99999936f)));
}

// error-free transformations on both halves (every paired add rounds once)
__device__ __forceinline__ void two_sum2(f2 a, f2 b, f2 &s, f2 &e)
{
    s = padd(a, b);
    const f2 bb = psub(s, a);
    e = padd(psub(a, psub(s, bb)), psub(b, bb));
}
__device__ __forceinline__ void fast_two_sum2(f2 a, f2 b, f2 &s, f2 &e)
{
    s = padd(a, b);
    e = psub(b, psub(s, a));
}

// complex numbers of both evaluations
struct c2 {
    f2 re, im;
};
__device__ __forceinline__ c2 czero() { return c2{bc(0.f), bc(0.f)}; }
__device__ __forceinline__ c2 cadd2(c2 a, c2 b) { return c2{padd(a.re, b.re), padd(a.im, b.im)}; }
__device__ __forceinline__ c2 cmul2(c2 a, c2 b)
{
    return c2{pfma(a.re, b.re, pneg(pmul(a.im, b.im))), pfma(a.re, b.im, pmul(a.im, b.re))};
}
// conj(a) * b
__device__ __forceinline__ c2 cmulc2(c2 a, c2 b)
{
    return c2{pfma(a.re, b.re, pmul(a.im, b.im)), pfma(a.re, b.im, pneg(pmul(a.im, b.re)))};
}
// 1 - a^2
__device__ __forceinline__ c2 one_minus_sq2(c2 a)
{
    return c2{pfma(pneg(a.re), a.re, pfma(a.im, a.im, bc(1.f))), pmul(bc(-2.f), pmul(a.re, a.im))};
}
// conj(a) * b + c
__device__ __forceinline__ c2 cfmac2(c2 a, c2 b, c2 c)
{
    return c2{pfma(a.re, b.re, pfma(a.im, b.im, c.re)), pfma(a.re, b.im, pfma(pneg(a.im), b.re, c.im))};
}

// wavevector of both evaluations (value + low word of Re k, as Kz) and
// 1 / |k|^2, a by-product of the root
struct Kz2 {
    f2 re, im, lo, y;
};
__device__ __forceinline__ c2 kc2(const Kz2 &k) { return c2{k.re, k.im}; }

// What is kept of a root's refinement.  kRootPlain: nothing (the backing, and
// adjoint factors).  kRootPhase: the correction of Re k as a low word, which
// only the phase takes (t, two approximate reciprocal roots, is up to three
// roundings off; the same t in both interfaces' k_a + k_b leaves most of it to
// cancel).  kRootFull: Re k itself rounded from the exact root too (two more
// additions, 0.5 % of the time): the deep gradients, where a waveguide
// resonance carries whatever does not cancel (1632 twelve-layer stacks, 99.9 %
// quantile of the scaled gradient's error 2.4e-5 with kRootPhase, 2.3e-5 with
// kRootFull; the worst stack 1.9e-4 and 1.3e-4).
enum : int { kRootPlain = 0, kRootPhase = 1, kRootFull = 2 };

// principal sqrt of u + i a (u = uh + ul, a >= 0 the stack's 4 pi iota,
// a2 = a^2), as kz_sqrt
template <int REFINE>
__device__ __forceinline__ Kz2 kz_sqrt2(f2 uh, f2 ul, float a, float a2)
{
    Kz2 k;
    const f2 au = pabs(uh);
    const f2 m2 = pfma(uh, uh, bc(a2));
    k.y = prsqrt(pmax(m2, bc(1e-37f)));
    const f2 H = pfma(m2, k.y, au);                          // |u| + |z| = 2 t^2
    const f2 i2t = prsqrt(pfma(H, bc(2.f), bc(4e-30f)));     // 1 / (2 t)
    const f2 t = pmul(H, i2t);
    const f2 small = pmul(bc(a), i2t);
    const b2 prop{uh.x >= 0.f, uh.y >= 0.f};
    if constexpr (REFINE != kRootPlain) {
        const f2 e = padd(pfma(pneg(t), t, au), pfma(small, small, psel(prop, ul, pneg(ul))));
        const f2 corr = pmul(e, i2t);
        const f2 s = padd(t, corr);
        k.re = psel(prop, REFINE == kRootFull ? s : t, small);
        k.im = psel(prop, small, s);
        k.lo = psel(prop, REFINE == kRootFull ? psub(corr, psub(s, t)) : corr, bc(0.f));
    } else {
        k.re = psel(prop, t, small);
        k.im = psel(prop, small, t);
        k.lo = bc(0.f);
    }
    return k;
}

// k_0^2 split by the quantum of magic number M
__device__ __forceinline__ void quantise2(f2 &p_hi, f2 &p_lo, float M)
{
    const f2 h = padd(padd(p_hi, bc(M)), bc(-M));
    p_lo = padd(psub(p_hi, h), p_lo);
    p_hi = h;
}

// k of medium j >= 1 from k_0^2 = (p_hi + p_lo) and the staged medium entry;
// QUANT: both split by a common quantum (split_media)
template <int REFINE, bool QUANT>
__device__ __forceinline__ Kz2 medium_kz2(f2 p_hi, f2 p_lo, float4 m)
{
    if constexpr (REFINE != kRootPlain) {
        f2 uh, ul;
        if constexpr (QUANT) {
            uh = padd(p_hi, bc(-m.x)); // exact
            ul = padd(p_lo, bc(-m.y));
        } else {
            two_sum2(p_hi, bc(-m.x), uh, ul);
            ul = padd(ul, padd(p_lo, bc(-m.y)));
        }
        fast_two_sum2(uh, ul, uh, ul);
        return kz_sqrt2<REFINE>(uh, ul, m.z, m.w);
    } else {
        const f2 u = padd(padd(p_hi, bc(-m.x)), padd(p_lo, bc(-m.y)));
        return kz_sqrt2<kRootPlain>(u, bc(0.f), m.z, m.w);
    }
}

// sin / cos of a factor: the special-function unit's, the table's, or the
// reduction-free polynomial of a small Nevot-Croce phase
enum : int { kTrigMufu = 0, kTrigTable = 1, kTrigSmall = 2 };

// E = exp(2 i k d), phase in double-float (as layer_phase).  TAB: the table
// sin / cos (NR_SINCOS_TABLE), else the special-function unit's.
template <bool TAB>
__device__ __forceinline__ c2 layer_phase2(const Kz2 &k, float4 L, const float *tab)
{
    const f2 ph = pmul(k.re, bc(L.x));
    f2 pl = pfma(k.re, bc(L.x), pneg(ph));
    pl = pfma(k.re, bc(L.y), pl);
    pl = pfma(k.lo, bc(L.x), pl);
    const f2 amp = pex2(pmul(k.im, bc(L.z)));
    f2 s, c;
    if constexpr (TAB && NR_SINCOS_TABLE) {
        pcis_tab(ph, pl, tab, c, s);
    } else {
        const f2 nt = padd(pfma(ph, bc(1.f / kTabN), bc(kRoundMagic)), bc(-kRoundMagic));
        const f2 red = pmul(padd(pfma(pneg(nt), bc((float)kTabN), ph), pl), bc(kTabStep));
        psincos(red, s, c);
    }
    return c2{pmul(amp, c), pmul(amp, s)};
}

// G = exp(s k_a k_b) / S^2, S = k_a + k_b: the Nevot-Croce Fresnel
// coefficient without its numerator, r = N G.  G = w (cos + i sin) conj(S^2)
// with w = exp(s Re) / |S^2|^2.  S is the sum itself: an error of k_j then
// enters the interfaces above and below it alike and mostly cancels, which
// S^2 = k_a^2 + k_b^2 + 2 k_a k_b from the known squares does not allow.  That
// form saves three operations (log-likelihoods 0-2 % faster) and left thick
// films a larger error of the gradient call's log-likelihood (99 % quantile of
// 1500: 6.3e-7 against 5.0e-7) and of the gradient (median 4.1e-7, 3.6e-7).
// REAL_A: k_a is real (the fronting medium).  A vanishing S (k_a = k_b = 0)
// gives a finite G whose numerator is 0.
template <bool REAL_A, int TRIG>
__device__ __forceinline__ c2 fresnel_g2(const Kz2 &ka, const Kz2 &kb, float4 I, const float *tab)
{
    const c2 kk = REAL_A ? c2{pmul(ka.re, kb.re), pmul(ka.re, kb.im)} : cmul2(kc2(ka), kc2(kb));
    const f2 Sx = padd(ka.re, kb.re), Sy = REAL_A ? kb.im : padd(ka.im, kb.im);
    const f2 A = pfma(Sx, Sx, pneg(pmul(Sy, Sy))); // Re S^2
    const f2 B = pmul(padd(Sx, Sx), Sy);           // Im S^2
    const f2 inv = prcp(pmax(pfma(A, A, pmul(B, B)), bc(1e-36f)));
    const f2 w = pmul(pex2(pmul(bc(I.w), kk.re)), inv);
    const f2 ph = pmul(bc(I.z), kk.im);
    f2 sn, cs;
    if constexpr (TRIG == kTrigSmall) pcis_small(ph, cs, sn);
    else if constexpr (TRIG == kTrigTable && NR_NC_TABLE) pcis_tab(pmul(ph, bc(kTabScale)), bc(0.f), tab, cs, sn);
    else psincos(ph, sn, cs);
    const f2 fc = pmul(w, cs), fs = pmul(w, sn);
    return c2{pfma(fc, A, pmul(fs, B)), pfma(fs, A, pneg(pmul(fc, B)))};
}

// The stack's recursion in projective form: X_j = B_j / A_j with A_n = 1,
// B_n = r_n and, from interface j + 1 up to j,
//   b = E_{j+1} B_{j+1},  A_j = A_{j+1} + r_j b,  B_j = r_j A_{j+1} + b.
// Against X_j = (r_j + Y) / (1 + r_j Y), Y = E_{j+1} X_{j+1}, it needs no
// division per interface (12 operations for 19 and two reciprocals) and its
// chain from one interface to the next is four dependent operations long.
// Stacks whose A would overflow (kNcGrows) divide by it after every interface.
// a b + c
__device__ __forceinline__ c2 cfma2(c2 a, c2 b, c2 c)
{
    return c2{pfma(a.re, b.re, pfma(pneg(a.im), b.im, c.re)), pfma(a.re, b.im, pfma(a.im, b.re, c.im))};
}
// c - a b
__device__ __forceinline__ c2 cfnma2(c2 a, c2 b, c2 c)
{
    return c2{pfma(pneg(a.re), b.re, pfma(a.im, b.im, c.re)), pfma(pneg(a.re), b.im, pfma(pneg(a.im), b.re, c.im))};
}
// a times the scalar complex (x, y)
__device__ __forceinline__ c2 cscl2(float x, float y, c2 a)
{
    return c2{pfma(bc(x), a.re, pneg(pmul(bc(y), a.im))), pfma(bc(x), a.im, pmul(bc(y), a.re))};
}
// (x, y) a + c
__device__ __forceinline__ c2 cscla2(float x, float y, c2 a, c2 c)
{
    return c2{pfma(bc(x), a.re, pfma(bc(-y), a.im, c.re)), pfma(bc(x), a.im, pfma(bc(y), a.re, c.im))};
}
// 1 / A, A scaled by its larger component first so that |A|^2 neither
// overflows nor underflows however deep the stack
__device__ __forceinline__ c2 cinv2(c2 A)
{
    const f2 s = prcp(pmax(pabs(A.re), pabs(A.im)));
    const f2 x = pmul(A.re, s), y = pmul(A.im, s);
    const f2 iv = pmul(prcp(pfma(x, x, pmul(y, y))), s);
    return c2{pmul(x, iv), pneg(pmul(y, iv))};
}

} // namespace
} // namespace nrimpl
