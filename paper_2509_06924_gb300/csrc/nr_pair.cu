// nr_pair.cu -- the gradient kernels of one- and two-layer stacks and the
// forward kernels (model, log-likelihood) of any depth, with two evaluations
// per thread in paired FP32 arithmetic (sm_100-family add/mul/fma.rn.f32x2).
//
// What bounds them.  The FP32 pipe: a paired instruction holds it two cycles
// for two operations a lane, scalar FP32 instructions hold it as long for
// one, and compares, selects and integer operations take part of a cycle
// each beside it (measured with one kind at a time mixed into a stream of
// paired FMAs), while special functions and shared-memory loads run along for
// free.  So every thread carries two (Q point, quadrature node) evaluations
// and the forward model, smearing seed and adjoint of both run as one stream
// of paired operations.  Per-stack constants enter as a scalar replicated to
// both halves (free on the hardware), negated operands are free as well;
// nothing is swapped between the halves, which would cost moves.
//
// The recursion runs in projective form (nr_pair.cuh), Nevot-Croce phases come
// from a polynomial where the stack's roughnesses allow it, and layer phases
// are staged in table steps.  Against the Moebius form with table phases, the
// later changes below included: 16384 one-layer stacks x 400 Q x 21 nodes,
// gradient 1.464 -> 1.310 ms, log-likelihood 0.820 -> 0.756 ms; 12288
// ten-layer stacks, model curves 1.779 -> 1.446 ms; 10000 stacks of 1-20
// layers, log-likelihood 1.623 -> 1.381 ms.
//
// The forward modes run the same code up to the smearing sum (model: write
// scale S + bkg; log-likelihood: the residual terms) and no adjoint.
// Everything else follows the one-evaluation-per-thread kernel (nr_mixed.cu)
// with the same double-float guards and the same interior critical-edge
// treatment: evaluations whose k_j falls in the edge band are queued per warp
// and drained by the scalar edge adjoint, one entry per lane.  A thread
// carries two adjacent evaluation slots of its tile.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "nr_internal.h"
#include "nr_pair.cuh"

// threads per CTA, and CTAs per SM asked of the compiler (register cap) for
// the 1- and the 2-layer kernels: the paired kernels are latency-bound at
// low occupancy, and the 2-layer kernel spills beyond 3 CTAs
#ifndef NR_PAIR_BLOCK
#define NR_PAIR_BLOCK 128
#endif
#ifndef NR_PAIR_MINB1
#define NR_PAIR_MINB1 5
#endif
#ifndef NR_PAIR_MINB2
#define NR_PAIR_MINB2 3
#endif
// 1: the runtime-n forward bucket (model / loglik of stacks with n != 1)
// runs the paired kernel too
#ifndef NR_PAIR_FWD_ANY
#define NR_PAIR_FWD_ANY 1
#endif
// CTAs per SM of the forward (model / loglik) kernels
#ifndef NR_PAIR_MINB_FWD
#define NR_PAIR_MINB_FWD 8
#endif
// 0: every bucket keeps the one-evaluation kernel
#ifndef NR_PAIR
#define NR_PAIR 1
#endif

namespace nrimpl {
namespace {

constexpr int kPairBlock = NR_PAIR_BLOCK;

// ---------------------------------------------------------------- traits --
// 1-2 layer gradients: unrolled sweeps, every forward intermediate and the
// partial gradients in registers.  Forward modes: the 1-layer kernel unrolled,
// the runtime-n ones (NMAX = 0: up to 20 layers; 64: deeper) rolled.
template <int MODE, int NMAX>
struct PairTraits {
    static constexpr bool GRAD = MODE == kGrad || MODE == kGradRes;
    static constexpr bool RFWD = !GRAD && NMAX != 1;
    static constexpr int NACC = 4 * NMAX + 3;
    static constexpr int MINB = !GRAD ? NR_PAIR_MINB_FWD : NMAX == 1 ? NR_PAIR_MINB1 : NR_PAIR_MINB2;
};

// ---------------------------------------------------------------- kernel --
template <int MODE, int NMAX, int KC>
__global__ void __launch_bounds__(kPairBlock, PairTraits<MODE, NMAX>::MINB)
nr_pair_kernel(const KernelArgs ka, const QuadConst qc)
{
    using PT = PairTraits<MODE, NMAX>;
    constexpr bool GRAD = PT::GRAD;
    constexpr bool LIK = MODE != kModel;
    // sin / cos by table for the model, the gradient and stacks deeper than 20
    // layers; the log-likelihood alone keeps the special-function unit's up to
    // there (its sum over Q points averages their error: within 5e-6 of the
    // oracle on every workload)
    constexpr bool TAB = MODE != kLoglik || NMAX > 20;
    static_assert(GRAD ? (NMAX == 1 || NMAX == 2) : (NMAX == 1 || NMAX == 0 || NMAX == 64),
                  "paired kernel: 1-2 layer gradients, 1-layer and runtime-n forward");
    constexpr int NM = NMAX > 0 ? NMAX : NR_MAX_LAYERS; // shared-memory capacity in layers
    constexpr int BLOCK = kPairBlock;
    constexpr int WARPS = BLOCK / 32;
    constexpr bool RES = MODE == kGradRes;
    constexpr bool QUANT = PT::RFWD; // wavevectors from a common quantum (split_media)
    constexpr int NACC = PT::NACC;
    constexpr int NRAW = 4 * NM + 7;
    constexpr int CAPQ = 256;
    // a warp's tile queues at most 64 n interior-edge entries and keeps fewer
    // than 32 between tiles
    constexpr int EQ = 64 * NM + 32;
    // k_{j-1}, k_j, k_{j+1}, Z, Xbar_{j-1} (+ k_0 dk_0/d ln f)
    constexpr int EQF = 5 + (RES ? 1 : 0);
    static_assert(CAPQ >= 2 * BLOCK / kSubLanes, "a super-tile holds at least one tile");

    __shared__ StackSmem<NM> sm;
    __shared__ float sh_cs[2 * kTabN]; // cos, sin at multiples of 2 pi / kTabN
    // w_k R per (Q slot, node), double-buffered: TQ KP <= 4 BLOCK for any K >= 3
    constexpr int WRN = 4 * BLOCK;
    __shared__ __align__(16) float sh_wR[2][WRN];
    __shared__ float4 sh_qd[CAPQ];                      // (Q/2, dQ/2, R_obs, 1/err) per staged Q point
    __shared__ float2 sh_rs[LIK ? CAPQ : 1];            // (residual, S) per staged Q point
    static_assert(WARPS == 4, "sum4 adds the warps' sums");
    __shared__ float sh_red[WARPS][32];
    __shared__ float sh_redd[WARPS][5]; // loglik (hi), d/dscale, d/dbkg, d/d ln f; loglik (lo)
    __shared__ double sh_raw[NRAW];
    __shared__ int sh_item;
    __shared__ int sh_last;
    __shared__ float2 sh_eq[GRAD ? WARPS : 1][EQF][GRAD ? EQ : 1];
    __shared__ int sh_eqj[GRAD ? WARPS : 1][GRAD ? EQ : 1];
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int K = KC > 0 ? KC : qc.K; // K >= 3 (the host's choice of this kernel)
    const int KP = (K + 3) & ~3;      // node stride of a Q slot in sh_wR (whole float4s)
    const int TQ = ka.tile_q;
    // Warp-local tiles: when every warp's 64 evaluation slots hold whole Q
    // points and the CTA tile is exactly those (TQ = warps x floor(64/K), no
    // slot lost against the CTA-wide layout, e.g. K = 21: 4 x 3 Q points),
    // each warp owns its Q slots and the smearing exchange needs only a warp
    // barrier.  Otherwise the thread carries tile slots 2 tid + h and the
    // exchange takes a CTA barrier.
    const int tqw = 64 / K;
    const bool wloc = TQ == WARPS * tqw;
    int qslot[2], kn[2];
    bool lane_on[2];
    f2 g_hi, g_lo, wk;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int e = wloc ? 2 * lane + h : 2 * tid + h;
        const int ls = e / K;
        kn[h] = e - ls * K;
        qslot[h] = wloc ? warp * tqw + ls : ls;
        lane_on[h] = wloc ? ls < tqw : ls < TQ;
        const float gh = lane_on[h] ? qc.g_hi[kn[h]] : 0.f;
        const float gl = lane_on[h] ? qc.g_lo[kn[h]] : 0.f;
        const float w = lane_on[h] ? qc.w[kn[h]] : 0.f;
        if (h == 0) { g_hi.x = gh; g_lo.x = gl; wk.x = w; }
        else { g_hi.y = gh; g_lo.y = gl; wk.y = w; }
    }
    // smearing sums: the warp's 64 evaluations touch Q slots qs0.. (at most
    // nslots of them; exactly tqw with warp-local tiles, and only those are
    // summed); sgl lanes per slot (depends on K only)
    const int qs0 = wloc ? warp * tqw : (warp * 64) / K;
    const int qs_end = wloc ? qs0 + tqw : TQ;
    const int nslots = (63 + K - 1) / K + 1;
    const int sgl = nslots <= 1 ? 32 : nslots <= 2 ? 16 : nslots <= 4 ? 8 : nslots <= 8 ? 4 : nslots <= 16 ? 2 : 1;
    // per-thread places of the tile: staged Q point, w R entry, whether it leads
    // its Q point, the row this lane adds up and the lanes that end with its sums
    const int sg = lane / sgl, part = lane - sg * sgl;
    const bool row_on = qs0 + sg < qs_end;
    const int row_at = row_on ? (qs0 + sg) * KP : 0;
    int slot_at[2], wr_at[2], from[2];
    bool lead[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        slot_at[h] = lane_on[h] ? qslot[h] : 0;
        wr_at[h] = qslot[h] * KP + kn[h];
        lead[h] = lane_on[h] && kn[h] == 0;
        from[h] = ((qslot[h] - qs0) * sgl) & 31;
    }
    const float g_max = fmaxf(fabsf(qc.g_hi[0]), fabsf(qc.g_hi[K - 1]));

    for (int i = tid; i < 2 * WRN; i += BLOCK) (&sh_wR[0][0])[i] = 0.f; // padding stays 0
    for (int i = tid; i < 2 * kTabN; i += BLOCK) sh_cs[i] = qc.cs_tab[i];  // read after the item barrier

    // The first item of a CTA is its own, the others come by ticket.  An item
    // takes five barriers: its staged stack, its first Q points, the end of
    // its tiles, the warps' sums, their total.  The next item's record is
    // loaded before the output, and the first Q points before the staging,
    // so that an item waits for memory about twice: 1024 one-layer stacks,
    // gradient 50.6 -> 48.9 us, against ten barriers and four waits in line.
    // (The rolled gradient kernels keep the plain order: the records held over
    // an item cost them registers inside their sweeps, 25.4 -> 26.3 ms.)
    int item = blockIdx.x, par = 0;
    if (tid < 2) sm.nc_big[tid] = 0;
    WorkItem wi{};
    if (item < ka.n_items) wi = ka.items[item];
    __syncthreads();
    for (; item < ka.n_items; par ^= 1) {
        if constexpr (NR_DEBUG) {
            if (!item_in_bounds(ka, wi, NMAX)) { // uniform over the block
                if (tid == 0) {
                    atomicOr(ka.status, NR_FLAG_DEBUG_BOUNDS);
                    sh_item = gridDim.x + atomicAdd(&ka.ticket[0], 1);
                }
                __syncthreads();
                item = sh_item;
                if (item < ka.n_items) wi = ka.items[item];
                __syncthreads(); // every thread has read sh_item
                continue;
            }
        }
        const StackInfo si = ka.stacks[wi.stack];
        const int n = (NMAX == 1 && NR_EXACT1) ? 1 : si.n;
        const double *p = ka.params + si.par_off;

        f2 accr[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) accr[i] = bc(0.f);
        constexpr int oD = 0, oUr = NM, oUi = 2 * NM + 1, oS = 3 * NM + 2;
        f2 gres_acc = bc(0.f);
        int eq_cnt = 0; // entries in this warp's interior-edge queue (warp-uniform)
        // drain `cnt` <= 32 queued entries, one per lane (scalar edge adjoint)
        auto eq_drain = [&](int cnt) {
            if (lane < cnt) {
                const int j = sh_eqj[warp][lane];
                const float2 ub = edge_ubar(sh_eq[warp][0][lane], sh_eq[warp][1][lane], sh_eq[warp][2][lane],
                                            sm.sig[j - 1], sm.sig[j], 0.5f * sm.adj[j - 1].w, sh_eq[warp][3][lane],
                                            j == n, sh_eq[warp][4][lane]);
                // conj(kbar)/k_j = 2 conj(ubar)
#pragma unroll
                for (int t = 1; t <= NM; ++t)
                    if (t == j) {
                        accr[oUr + t - 1].x += 2.f * ub.x;
                        accr[oUi + t - 1].x += -2.f * ub.y;
                    }
                if constexpr (RES) gres_acc.x = fmaf(2.f * ub.x, sh_eq[warp][EQF - 1][lane].x, gres_acc.x);
            }
            __syncwarp();
            const int rest = eq_cnt - cnt;
            for (int e = lane; e < rest; e += 32) {
                const int src = cnt + e;
#pragma unroll
                for (int f = 0; f < EQF; ++f) sh_eq[warp][f][e] = sh_eq[warp][f][src];
                sh_eqj[warp][e] = sh_eqj[warp][src];
            }
            __syncwarp();
            eq_cnt = rest;
        };

        // per-thread sums of the loglik terms, d/dscale, d/dbkg (per Q point)
        float ll_hi = 0.f, ll_lo = 0.f, gsc_acc = 0.f, gbk_acc = 0.f;
        const float *qp = ka.q + si.q_begin, *dqp = ka.dq + si.q_begin;
        const float fsc = ka.dq_scale ? (float)ka.dq_scale[wi.stack] : 1.f; // resolution scale of the stack
        const float *rop = ka.r_obs + si.q_begin, *rep = ka.r_err + si.q_begin;
        const int span = (CAPQ / TQ) * TQ;
        int sb = wi.q_lo, s_cnt = 0;
        auto consume = [&](int i) __attribute__((always_inline)) {
            if constexpr (LIK) {
                const float2 rs = sh_rs[i];
                const float Re = __ldg(rep + sb + i);
                if (!(Re > 0.f)) atomicOr(ka.status, NR_FLAG_BAD_ERR);
                float t1, t2;
                two_sum(ll_hi, fmaf(rs.x, rs.x, kLog2Pi + 2.f * logf(Re)), t1, t2);
                ll_hi = t1;
                ll_lo += t2;
                if constexpr (GRAD) {
                    const float dldm = -(rs.x * fabsf(sh_qd[i].w));
                    gsc_acc = fmaf(dldm, rs.y, gsc_acc);
                    gbk_acc += dldm;
                }
            }
        };
        // one Q point of the dataset (zeros past the item's end), and its staged form
        auto fetch = [&](int qa) __attribute__((always_inline)) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (qa < wi.q_hi) {
                v.x = __ldg(qp + qa);
                v.y = __ldg(dqp + qa);
                if constexpr (LIK) {
                    v.z = __ldg(rop + qa);
                    v.w = __ldg(rep + qa);
                }
            }
            return v;
        };
        int p_bits = 0; // largest k_0^2 (or |c_j|) this thread staged (QUANT)
        float magic = 0.f;
        auto place = [&](int i, int qa, float4 r) __attribute__((always_inline)) {
            float4 v = make_float4(0.05f, 0.f, 0.f, 0.f); // past the end: a harmless node, 1/err = 0
            if (qa < wi.q_hi) {
                v.x = 0.5f * r.x;
                v.y = 0.5f * fsc * r.y;
                if constexpr (QUANT) {
                    const float k = fabsf(v.x) + fabsf(v.y) * g_max;
                    p_bits = max(p_bits, quantum_bits(k * k));
                }
                if constexpr (LIK) {
                    v.z = r.z;
                    v.w = rcp_approx(r.w);
                }
                if constexpr (GRAD) {
                    // may a node of this Q point reach an interior-edge band,
                    // or (two layers) lie below an edge?  (negative 1/err: yes)
                    const float a = fabsf(v.y) * g_max;
                    const float lo = fmaxf(v.x - a, 0.f), hi = v.x + a;
                    const float k2lo = lo * lo * (1.f - 1.5f * kEdgeFrac);
                    const float k2hi = hi * hi * (1.f + 1.5f * kEdgeFrac);
                    bool e = false;
                    for (int j = 1; j <= n; ++j) {
                        const float c = sm.med[j].x;
                        e |= c > 0.f && (NMAX == 2 || c < k2hi) && c > k2lo;
                    }
                    if (e && v.w > 0.f) v.w = -v.w;
                }
            }
            sh_qd[i] = v;
        };
        static_assert(CAPQ <= 2 * BLOCK, "a super-tile's Q points: two a thread");
        // the forward kernels, at 64 registers, fetch after the staging
        float4 first0 = make_float4(0.f, 0.f, 0.f, 0.f), first1 = first0;
        if constexpr (GRAD) {
            first0 = fetch(wi.q_lo + tid);
            first1 = fetch(wi.q_lo + tid + BLOCK);
        }
        // one layer cannot grow (the fronting medium propagates); its log-likelihood takes no table
        constexpr int FLAGS = NMAX == 1 ? (TAB ? kNcBig : 0) : kNcBig | kNcGrows;
        stage_stack<NM, FLAGS>(sm, &sm.nc_big[par], p, n, tid, ka.status);
        if (QUANT && tid == 0) sm.p_max = 0;
        __syncthreads();
        if (tid == 0) sm.nc_big[par ^ 1] = 0;
        auto restage = [&](int q0) {
            if (!GRAD || q0 > wi.q_lo) {
                if (q0 > wi.q_lo) __syncthreads(); // the previous super-tile's reads and pairs are complete
                for (int i = tid; i < span; i += BLOCK) {
                    if (i < s_cnt) consume(i);
                    place(i, q0 + i, fetch(q0 + i));
                }
            } else {
                if (tid < span) place(tid, q0 + tid, first0);
                if (tid + BLOCK < span) place(tid + BLOCK, q0 + tid + BLOCK, first1);
            }
            sb = q0;
            s_cnt = min(span, wi.q_hi - q0);
            if constexpr (QUANT) {
                if (tid <= n) p_bits = max(p_bits, quantum_bits(fabsf(sm.med[tid + 1].x + sm.med[tid + 1].y)));
                p_bits = __reduce_max_sync(kFull, p_bits);
                if (lane == 0) atomicMax(&sm.p_max, p_bits);
                __syncthreads();
                magic = quantum_magic(sm.p_max);
                split_media(sm, n, tid, magic);
            }
            __syncthreads();
        };

        const float scale = sm.scale, bkg = sm.bkg;
        const f2 wks = pmul(wk, bc(scale));
        int buf = 0;
        // t0: the tile's first Q point within the staged super-tile.  Slots past
        // the last Q point are staged harmless (1/err = 0), so the tile needs no
        // test of its end; idle lanes repeat slot 0 with weight 0.
        for (int q0 = wi.q_lo; q0 < wi.q_hi; q0 += span) {
        restage(q0);
        for (int t0 = 0; t0 < s_cnt; t0 += TQ, buf ^= 1) {
            const float4 qd[2] = {sh_qd[t0 + slot_at[0]], sh_qd[t0 + slot_at[1]]};
            const f2 Qh = make_float2(qd[0].x, qd[1].x), dQh = make_float2(qd[0].y, qd[1].y);
            // a1: node position k_0 = q/2 in double-float, k_0^2
            f2 k0h, k0l;
            {
                const f2 th = pmul(dQh, g_hi);
                f2 tl = pfma(dQh, g_hi, pneg(th));
                tl = pfma(dQh, g_lo, tl);
                f2 s, e;
                two_sum2(Qh, th, s, e);
                e = padd(e, tl);
                fast_two_sum2(s, e, k0h, k0l);
            }
            const b2 qok{k0h.x > 0.f, k0h.y > 0.f};
            f2 p_hi = pmul(k0h, k0h);
            f2 p_lo = pfma(k0h, k0h, pneg(p_hi));
            p_lo = pfma(padd(k0h, k0h), k0l, p_lo);
            if constexpr (QUANT) quantise2(p_hi, p_lo, magic);

            // a3-a6 forward from the backing up, projective (X_j = B_j / A_j);
            // the gradient kernels keep every intermediate
            constexpr int NK = GRAD ? NM + 2 : 1;
            Kz2 kst[NK];
            c2 rst[NK], Gst[NK], Est[NK], bst[NK], Ast[NK];
            c2 A = c2{bc(1.f), bc(0.f)}, B = czero();
            Kz2 kbelow = medium_kz2<kRootPlain, QUANT>(p_hi, p_lo, sm.med[n + 1]);
            bool renorm = false; // divide by A at every interface
            auto fwd_step = [&](int j, auto TOP, auto BOT, auto TRIG) __attribute__((always_inline)) {
                const bool top = pos_flag(TOP, j == 0), bot = pos_flag(BOT, j == n);
                Kz2 kj;
                if (top) kj = Kz2{k0h, bc(0.f), k0l, bc(0.f)};
                else kj = medium_kz2<kRootPhase, QUANT>(p_hi, p_lo, sm.med[j]);
                const float4 Ij = sm.itf[j];
                const c2 Gj = top ? fresnel_g2<true, decltype(TRIG)::value>(kj, kbelow, Ij, sh_cs)
                                  : fresnel_g2<false, decltype(TRIG)::value>(kj, kbelow, Ij, sh_cs);
                const c2 rj = cscl2(Ij.x, Ij.y, Gj);
                if (bot) {
                    B = rj;
                    if constexpr (GRAD) kst[j + 1] = kbelow;
                } else {
                    const c2 Ej = layer_phase2<TAB>(kbelow, sm.lay[j + 1], sh_cs);
                    const c2 b = cmul2(B, Ej);
                    if constexpr (NMAX == 1) { // A_1 = 1
                        const c2 rb = cmul2(rj, b);
                        A = c2{padd(bc(1.f), rb.re), rb.im};
                        B = cadd2(rj, b);
                    } else {
                        const c2 An = A;
                        A = cfma2(rj, b, An);
                        B = cfma2(rj, An, b);
                        if constexpr (PT::RFWD && decltype(TRIG)::value == kTrigTable) {
                            if (renorm) {
                                B = cmul2(B, cinv2(A));
                                A = c2{bc(1.f), bc(0.f)};
                            }
                        }
                    }
                    if constexpr (GRAD) {
                        Est[j + 1] = Ej;
                        bst[j] = b;
                    }
                }
                if constexpr (GRAD) {
                    kst[j] = kj;
                    rst[j] = rj;
                    Gst[j] = Gj;
                    Ast[j] = A;
                }
                kbelow = kj;
            };
            auto forward = [&](auto TRIG) __attribute__((always_inline)) {
                if constexpr (PT::RFWD) {
                    fwd_step(n, Pos<kRt>{}, Pos<kYes>{}, TRIG);
#pragma unroll 1
                    for (int j = n - 1; j >= 1; --j) fwd_step(j, Pos<kNo>{}, Pos<kNo>{}, TRIG);
                    if (n >= 1) fwd_step(0, Pos<kYes>{}, Pos<kNo>{}, TRIG);
                } else {
#pragma unroll
                    for (int j = NM; j >= 0; --j)
                        if (j <= n) fwd_step(j, Pos<kRt>{}, Pos<kRt>{}, TRIG);
                }
            };
            const int nc = sm.nc_big[par];
            renorm = nc & kNcGrows;
            if constexpr (!TAB) {
                if (PT::RFWD && renorm) forward(Pos<kTrigTable>{});
                else forward(Pos<kTrigMufu>{});
            } else {
                if (nc) forward(Pos<kTrigTable>{});
                else forward(Pos<kTrigSmall>{});
            }
            // X_0 = B_0 / A_0 and R = |X_0|^2; |A_0| (kNcGrows) needs scaling in
            // the deepest bucket, and in the gradient of two layers that may grow
            c2 iA = czero(), X0 = czero();
            f2 R;
            if constexpr (GRAD || NMAX > 20) {
                if (NMAX > 20 || (NMAX == 2 && renorm)) {
                    iA = cinv2(A);
                } else {
                    const f2 iv = prcp(pfma(A.re, A.re, pmul(A.im, A.im)));
                    iA = c2{pmul(A.re, iv), pneg(pmul(A.im, iv))};
                }
                X0 = cmul2(B, iA);
                R = pfma(X0.re, X0.re, pmul(X0.im, X0.im));
            } else {
                R = pmul(pfma(B.re, B.re, pmul(B.im, B.im)), prcp(pfma(A.re, A.re, pmul(A.im, A.im))));
            }
            if (!(qok.x && qok.y)) {
                atomicOr(ka.status, NR_FLAG_BAD_Q);
                if (!qok.x) R.x = __int_as_float(0x7fffffff);
                if (!qok.y) R.y = __int_as_float(0x7fffffff);
            }

            // a8-a10: smearing sum, model, residual, adjoint seed
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (lane_on[h]) sh_wR[buf][wr_at[h]] = half(wk, h) * half(R, h);
            if (wloc) __syncwarp();
            else __syncthreads();
            f2 S;
            {
                float ps = 0.f;
                if (row_on) {
                    const float4 *row = reinterpret_cast<const float4 *>(&sh_wR[buf][row_at]);
                    auto add4 = [&](int c) __attribute__((always_inline)) {
                        const float4 v = row[c];
                        ps += (v.x + v.y) + (v.z + v.w);
                    };
                    if constexpr (KC > 0) {
                        constexpr int NSL = (63 + KC - 1) / KC + 1;
                        constexpr int SGL = NSL <= 1 ? 32 : NSL <= 2 ? 16 : NSL <= 4 ? 8 : NSL <= 8 ? 4
                                                                                : NSL <= 16 ? 2 : 1;
#pragma unroll
                        for (int i = 0; i < ((KC + 3) / 4 + SGL - 1) / SGL; ++i)
                            if (part + i * SGL < (KC + 3) / 4) add4(part + i * SGL);
                    } else {
                        for (int c = part; c < KP / 4; c += sgl) add4(c);
                    }
                }
                for (int o = 1; o < sgl; o <<= 1) ps += __shfl_xor_sync(kFull, ps, o);
                S.x = __shfl_sync(kFull, ps, from[0]);
                S.y = __shfl_sync(kFull, ps, from[1]);
            }
            if constexpr (MODE == kModel) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (lead[h] && t0 + slot_at[h] < s_cnt)
                        ka.r_out[si.out_off + sb + t0 + slot_at[h]] = fmaf(scale, half(S, h), bkg);
            } else {
                const f2 ie = make_float2(fabsf(qd[0].w), fabsf(qd[1].w));
                const f2 res = pmul(psub(pfma(bc(scale), S, bc(bkg)), make_float2(qd[0].z, qd[1].z)), ie);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (lead[h]) sh_rs[t0 + slot_at[h]] = make_float2(half(res, h), half(S, h));
                if constexpr (GRAD) {
                    const f2 Rb = pmul(wks, pneg(pmul(res, ie))); // w_k scale dl/dm (0 on idle slots)

                    // a7: adjoint sweep from the fronting down to the backing.
                    // With Xbar_0 = 2 Rbar X_0: Bbar_0 = Xbar_0 / conj(A_0) and
                    // Abar_0 = -conj(X_0) Bbar_0; every step then applies the
                    // conjugate transpose of the forward one.  Near an edge and
                    // below it two layers carry Z_j = Bbar_j / conj(A_j) in Bb
                    // instead (nr_roll.cu): 600 unsmeared points below an edge,
                    // 90 % within 3.2e-5 of the layers' gradient, 5.3e-5 with Abar.
                    const f2 Rb2 = padd(Rb, Rb);
                    c2 Bb = cmulc2(iA, X0);
                    Bb = c2{pmul(Bb.re, Rb2), pmul(Bb.im, Rb2)};
                    const f2 mR = pneg(pmul(Rb2, R));
                    c2 Ab = c2{pmul(iA.re, mR), pneg(pmul(iA.im, mR))};
                    c2 kbar = czero();
                    Kz2 kj = Kz2{k0h, bc(0.f), k0l, bc(0.f)};
                    c2 Xb_up = czero(); // Xbar_{j-1} (edge sweeps)
                    const bool reach[2] = {lane_on[0] && qd[0].w < 0.f, lane_on[1] && qd[1].w < 0.f};
                    Kz2 kjm1 = kj;
                    const f2 edge_u = pmul(bc(kEdgeFrac), pmul(k0h, k0h));
                    const f2 wres = RES ? pmul(dQh, g_hi) : bc(0.f);
                    f2 res_sum = bc(0.f), res_k0 = bc(0.f);
                    // acc += Im(conj(k) U) etc.: partial gradients in registers
                    auto adj_step = [&](int j, auto TOP, auto BOT, auto EDG) __attribute__((always_inline)) {
                        const bool top = pos_flag(TOP, j == 0), bot = pos_flag(BOT, j == n);
                        const float4 Ij = sm.itf[j], Cj = sm.adj[j];
                        const Kz2 kj1 = kst[j + 1];
                        const c2 rj = rst[j], Gj = Gst[j];
                        constexpr bool ZF = decltype(EDG)::value && NMAX == 2;
                        c2 Xb_in = decltype(EDG)::value ? cmulc2(Ast[j], Bb) : czero();
                        if constexpr (ZF) Xb_in = cmulc2(Ast[j], Xb_in);
                        c2 kbar1 = czero(), rb = Bb;
                        if (!bot) {
                            const c2 b = bst[j];
                            // adjoint of b; the phase enters through b = E B only: with
                            // U = conj(b) bbar the thickness sum takes Im(conj(k) U)
                            // and kbar_{j+1} gets -2 i d U
                            c2 bb;
                            if constexpr (ZF) {
                                const c2 A1 = Ast[j + 1];
                                rb = cmulc2(cmul2(cadd2(A1, b), c2{psub(A1.re, b.re), psub(A1.im, b.im)}), Bb);
                                const c2 t = cmulc2(one_minus_sq2(rj), Bb);
                                bb = cmulc2(A1, t);
                                Bb = cmulc2(Est[j + 1], t);
                            } else {
                                if constexpr (NMAX == 1) rb = cfmac2(b, Ab, Bb); // A_1 = 1
                                else rb = cfmac2(b, Ab, cmulc2(Ast[j + 1], Bb));
                                bb = cfmac2(rj, Ab, Bb);
                                if constexpr (NMAX > 1) Ab = cfmac2(rj, Bb, Ab);
                                Bb = cmulc2(Est[j + 1], bb);
                            }
                            const c2 U = cmulc2(b, bb);
                            accr[oD + j] = pfma(kj1.re, U.im, pfma(pneg(kj1.im), U.re, accr[oD + j]));
                            kbar1 = c2{pmul(bc(Cj.w), U.im), pneg(pmul(bc(Cj.w), U.re))};
                        }
                        // Fresnel: with g = conj(G) rbar and N the numerator,
                        // dr/dk_j and dr/dk_{j+1} give kbar_j += conj(k_{j+1}) g (s conj(N) + 2)
                        // and kbar_{j+1} += conj(k_j) g (s conj(N) - 2); the roughness sum
                        // takes Re(N conj(g) k_j k_{j+1})
                        const c2 gg = cmulc2(Gj, rb);
                        const c2 ga = cmulc2(kc2(kj1), gg);
                        const c2 gb = top ? c2{pmul(kj.re, gg.re), pmul(kj.re, gg.im)} : cmulc2(kc2(kj), gg);
                        kbar1 = cscla2(Cj.y, Cj.z, gb, kbar1);
                        const c2 t = top ? c2{pmul(ga.re, kj.re), pneg(pmul(ga.im, kj.re))} : cmulc2(ga, kc2(kj));
                        accr[oS + j] = pfma(bc(Ij.x), t.re, pfma(bc(-Ij.y), t.im, accr[oS + j]));
                        if (RES && top) res_k0 = pfma(bc(Cj.x), ga.re, pneg(pmul(bc(Cj.z), ga.im)));
                        if (!top) {
                            kbar = cscla2(Cj.x, Cj.z, ga, kbar);
                            // k_j complete: accumulate conj(kbar) / k_j, or queue the
                            // interior-edge evaluation
                            b2 edge{false, false};
                            if constexpr (decltype(EDG)::value) {
                                const f2 far = pmul(edge_u, kj.y); // |k_j|^2 < edge_u
                                edge = b2{reach[0] && far.x > 1.f, reach[1] && far.y > 1.f};
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const bool eh = h ? edge.y : edge.x;
                                    const unsigned em = __ballot_sync(kFull, eh);
                                    if (em) {
                                        if (eh) {
                                            const int slot =
                                                queue_slot<EQ>(eq_cnt + __popc(em & ((1u << lane) - 1u)), ka.status);
                                            // Z = E X of the layer below (0 at the bottom interface)
                                            float2 Z = make_float2(0.f, 0.f);
                                            if (!bot)
                                                Z = cdiv(make_float2(half(bst[j].re, h), half(bst[j].im, h)),
                                                         make_float2(half(Ast[j + 1].re, h), half(Ast[j + 1].im, h)));
                                            if constexpr (RES)
                                                sh_eq[warp][EQF - 1][slot] = make_float2(half(k0h, h) * half(wres, h), 0.f);
                                            sh_eq[warp][0][slot] = make_float2(half(kjm1.re, h), half(kjm1.im, h));
                                            sh_eq[warp][1][slot] = make_float2(half(kj.re, h), half(kj.im, h));
                                            sh_eq[warp][2][slot] = make_float2(half(kj1.re, h), half(kj1.im, h));
                                            sh_eq[warp][3][slot] = Z;
                                            sh_eq[warp][4][slot] = make_float2(half(Xb_up.re, h), half(Xb_up.im, h));
                                            sh_eqj[warp][slot] = j;
                                        }
                                        eq_cnt = queue_count<EQ>(eq_cnt + __popc(em));
                                    }
                                }
                            }
                            const c2 kq = cmul2(kbar, kc2(kj));
                            f2 inv = kj.y;
                            if constexpr (decltype(EDG)::value) inv = psel(edge, bc(0.f), inv);
                            const f2 ur = pmul(kq.re, inv);
                            accr[oUr + j - 1] = padd(accr[oUr + j - 1], ur);
                            accr[oUi + j - 1] = pfma(pneg(kq.im), inv, accr[oUi + j - 1]);
                            if constexpr (RES) res_sum = padd(res_sum, ur);
                        }
                        Xb_up = Xb_in;
                        kbar = kbar1;
                        kjm1 = kj;
                        kj = kj1;
                        if (bot) { // backing medium n+1
                            const c2 kk = cmul2(kbar, kc2(kj));
                            const f2 inv = kj.y;
                            const f2 ur = pmul(kk.re, inv);
                            accr[oUr + j] = padd(accr[oUr + j], ur);
                            accr[oUi + j] = pfma(pneg(kk.im), inv, accr[oUi + j]);
                            if constexpr (RES) res_sum = padd(res_sum, ur);
                        }
                    };
                    auto sweep = [&](auto EDG) __attribute__((always_inline)) {
                        if constexpr (decltype(EDG)::value && NMAX == 2) Bb = cmulc2(iA, Bb); // Z_0
#pragma unroll
                        for (int j = 0; j <= NM; ++j)
                            if (j <= n) adj_step(j, Pos<kRt>{}, Pos<kRt>{}, EDG);
                        if constexpr (decltype(EDG)::value) {
                            while (eq_cnt >= 32) {
                                __syncwarp();
                                eq_drain(32);
                            }
                        }
                    };
                    // the staged sign of 1/err marks Q points whose nodes may reach an
                    // interior-edge band or, with two layers, lie below an edge
                    // (warp-uniform choice)
                    if (__any_sync(kFull, reach[0] || reach[1]))
                        sweep(std::true_type{});
                    else
                        sweep(std::false_type{});
                    if constexpr (RES) gres_acc = pfma(wres, pfma(k0h, res_sum, res_k0), gres_acc);
                } // GRAD
            } // LIK
        }
        }

        if (tid == 0) sh_item = gridDim.x + atomicAdd(&ka.ticket[0], 1); // its latency overlaps the reductions

        if constexpr (LIK) {
            if constexpr (GRAD) {
                if (eq_cnt > 0) {
                    __syncwarp();
                    eq_drain(eq_cnt);
                }
            }
            // ---- CTA reduction of the item's partial sums into sh_raw ----
            __syncthreads();
            for (int i = tid; i < s_cnt; i += BLOCK) consume(i);
            static_assert(!GRAD || NACC <= 32, "register partials exceed one reduction batch");
            if constexpr (GRAD) {
#pragma unroll
                for (int t = 0; t < NACC; ++t) {
                    float v = accr[t].x + accr[t].y;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
                    if (lane == 0) sh_red[warp][t] = v;
                }
            }
            {   // loglik (float pair), d/dscale, d/dbkg, d/d ln(dQ scale)
                float h = ll_hi, l = ll_lo, a1 = gsc_acc, a2 = gbk_acc, a3 = gres_acc.x + gres_acc.y;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float h2 = __shfl_xor_sync(kFull, h, o), l2 = __shfl_xor_sync(kFull, l, o);
                    float s, e;
                    two_sum(h, h2, s, e);
                    h = s;
                    l = __fadd_rn(__fadd_rn(l, l2), e);
                    a1 += __shfl_xor_sync(kFull, a1, o);
                    a2 += __shfl_xor_sync(kFull, a2, o);
                    if constexpr (RES) a3 += __shfl_xor_sync(kFull, a3, o);
                }
                if (lane == 0) {
                    sh_redd[warp][0] = h;
                    sh_redd[warp][1] = a1;
                    sh_redd[warp][2] = a2;
                    sh_redd[warp][3] = a3;
                    sh_redd[warp][4] = l;
                }
            }
            __syncthreads();
            if constexpr (GRAD) {
                if (tid < NACC) {
                    const int t = tid;
                    // accumulator slot -> raw index for this stack's n (-1: unused)
                    const int i = t < NM ? (t < n ? t : -1)
                                  : t < 2 * NM + 1 ? (t - NM <= n ? n + (t - NM) : -1)
                                  : t < 3 * NM + 2 ? (t - 2 * NM - 1 <= n ? 2 * n + 1 + (t - 2 * NM - 1) : -1)
                                                   : (t - 3 * NM - 2 <= n ? 3 * n + 2 + (t - 3 * NM - 2) : -1);
                    if (i >= 0) sh_raw[i] = sum4(sh_red[0][t], sh_red[1][t], sh_red[2][t], sh_red[3][t], 0.f);
                }
            }
            // by another warp: the likelihood sums
            if (const int t = tid - 32; t >= 0 && t < (RES ? 4 : 3)) {
                const float lo = t == 0 ? (sh_redd[0][4] + sh_redd[1][4]) + (sh_redd[2][4] + sh_redd[3][4]) : 0.f;
                sh_raw[4 * n + 3 + t] = sum4(sh_redd[0][t], sh_redd[1][t], sh_redd[2][t], sh_redd[3][t], lo);
            }
            item = sh_item;
            const WorkItem done = wi;
            if (item < ka.n_items) wi = ka.items[item];
            __syncthreads();
            const int nout = GRAD ? 4 * n + (RES ? 7 : 6) : 1;
            const int off0 = GRAD ? 0 : 4 * n + 3; // loglik mode: llsum only
            if (si.n_chunks == 1) {
                finalize_stack<MODE>(sh_raw, n, p, done.stack, si.par_off, ka.ll_out, ka.grad_out, ka.res_out, tid,
                                     BLOCK);
            } else {
                double *slot = ka.partials + si.part_base + (int64_t)done.chunk * n_slot(n);
                for (int i = tid; i < nout; i += BLOCK) slot[off0 + i] = sh_raw[off0 + i];
                __syncthreads();
                if (tid == 0) {
                    __threadfence(); // after the barrier: covers the whole CTA's slot
                    const int prev = atomicAdd(&ka.stack_done[done.stack], 1);
                    sh_last = prev == si.n_chunks - 1;
                }
                __syncthreads();
                if (sh_last) {
                    __threadfence();
                    for (int i = tid; i < nout; i += BLOCK) {
                        double s = 0.0;
#pragma unroll 8
                        for (int c = 0; c < si.n_chunks; ++c)
                            s += __ldcg(ka.partials + si.part_base + (int64_t)c * n_slot(n) + off0 + i);
                        sh_raw[off0 + i] = s;
                    }
                    __syncthreads();
                    finalize_stack<MODE>(sh_raw, n, p, done.stack, si.par_off, ka.ll_out, ka.grad_out, ka.res_out,
                                         tid, BLOCK);
                    if (tid == 0) ka.stack_done[done.stack] = 0;
                }
            }
        } else {
            __syncthreads(); // the tiles' reads of sm and sh_qd are complete
            item = sh_item;
            if (item < ka.n_items) wi = ka.items[item];
        }
        // no barrier here: the next item writes sm and sh_qd, which nothing
        // reads any more, and its own barriers lie before its other writes
    }
    // last CTA out resets the queue for the next launch
    if (tid == 0) {
        __threadfence();
        const int done = atomicAdd(&ka.ticket[1], 1);
        if (done == (int)gridDim.x - 1) {
            ka.ticket[0] = 0;
            ka.ticket[1] = 0;
            __threadfence();
        }
    }
}

template <int MODE, int NMAX, int KC>
cudaError_t pair_launch_k(int grid, const KernelArgs &a, const QuadConst &qc, cudaStream_t st)
{
    nr_pair_kernel<MODE, NMAX, KC><<<grid, kPairBlock, 0, st>>>(a, qc);
    return cudaGetLastError();
}

template <int MODE, int NMAX, int KC>
cudaError_t pair_occupancy_k(int *blocks)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, nr_pair_kernel<MODE, NMAX, KC>, kPairBlock, 0);
}

// the 1-layer kernels are also compiled for the workloads' quadrature
// orders (17 and 21 nodes); for deeper stacks the fixed count gains about 1%
// and doubles the build time
template <int MODE, int NMAX>
cudaError_t pair_launch_one(int grid, const KernelArgs &a, const QuadConst &qc, cudaStream_t st)
{
    if constexpr (NMAX == 1) {
        if (qc.K == 21) return pair_launch_k<MODE, NMAX, 21>(grid, a, qc, st);
        if (qc.K == 17) return pair_launch_k<MODE, NMAX, 17>(grid, a, qc, st);
    }
    return pair_launch_k<MODE, NMAX, 0>(grid, a, qc, st);
}

template <int MODE, int NMAX>
cudaError_t pair_occupancy_one(int K, int *blocks)
{
    if constexpr (NMAX == 1) {
        if (K == 21) return pair_occupancy_k<MODE, NMAX, 21>(blocks);
        if (K == 17) return pair_occupancy_k<MODE, NMAX, 17>(blocks);
    }
    return pair_occupancy_k<MODE, NMAX, 0>(blocks);
}

} // namespace

bool pair_eligible(int mode, int nmax, int K)
{
    if (!NR_PAIR || K < 3) return false;
    if (!is_grad_mode(mode)) return nmax == 1 || (NR_PAIR_FWD_ANY && (nmax == 0 || nmax == 64));
    return nmax >= 1;
}

int pair_block_threads() { return kPairBlock; }

// (MODE, NMAX) of a launch: buckets of 1-2 layers and the forward ones here,
// the deeper gradient buckets in nr_roll.cu
#define NR_PAIR_DISPATCH(CALL)                                                  \
    switch (mode) {                                                             \
    case kModel: return nmax == 1 ? CALL(kModel, 1) : nmax == 0 ? CALL(kModel, 0) : CALL(kModel, 64);     \
    case kLoglik: return nmax == 1 ? CALL(kLoglik, 1) : nmax == 0 ? CALL(kLoglik, 0) : CALL(kLoglik, 64); \
    case kGradRes: return nmax == 1 ? CALL(kGradRes, 1) : CALL(kGradRes, 2);    \
    default: return nmax == 1 ? CALL(kGrad, 1) : CALL(kGrad, 2);                \
    }

cudaError_t pair_occupancy(int mode, int nmax, int K, int *blocks)
{
    if (is_grad_mode(mode) && nmax > 2) return roll_occupancy(mode, nmax, blocks);
#define NR_CALL(M, B) pair_occupancy_one<M, B>(K, blocks)
    NR_PAIR_DISPATCH(NR_CALL)
#undef NR_CALL
}

cudaError_t launch_pair(int mode, int nmax, int grid, const KernelArgs &a, const QuadConst &qc, cudaStream_t st)
{
    if (is_grad_mode(mode) && nmax > 2) return launch_roll(mode, nmax, grid, a, qc, st);
#define NR_CALL(M, B) pair_launch_one<M, B>(grid, a, qc, st)
    NR_PAIR_DISPATCH(NR_CALL)
#undef NR_CALL
}

} // namespace nrimpl
