// nr_roll.cu -- gradient kernels of stacks with more than two layers (3 to
// 64), two evaluations per thread in paired FP32 arithmetic, for sm_103a.
//
// What bounds it.  The gradient is a stream of FP32 operations: the forward
// sweep from the backing up (wavevector, Fresnel factor, phase, recursion)
// and the adjoint sweep back down, which needs the forward's factors again.
// A kernel that forms them a second time spends a third of its FP32
// operations on it.  Here every evaluation keeps them: per layer and pair of
// evaluations 32 bytes (G_j, E_{j+1}) in tensor memory, used as 256 KB of
// per-thread scratch per SM, and 16 bytes (b_j) in shared memory; only k_j,
// the cheapest, is formed again.  The recursion runs in projective form
// (nr_pair.cuh), without divisions and with short chains in both directions.
// Against forming the factors twice in the Moebius form, with everything in
// shared memory: 196608 twelve-layer stacks x 300 Q x 21 nodes 150.8 -> 104.5
// ms, 12288 ten-layer stacks (150-300 Q, 17 nodes) 5.03 -> 3.50 ms, 10000
// stacks of 1-20 layers 5.83 -> 3.96 ms; 1024 stacks of 21-64 layers, which
// ran one evaluation per thread, 3.69 -> 1.74 ms.  Storing 32 bytes a layer
// in TMEM and reading them back costs about 30 cycles per warp and layer (16
// warps an SM), forming them again 200.
//
// Layout.  Tensor memory belongs to one CTA of an SM, so one CTA fills the
// SM: TEAMS teams of 128 threads (4 warps, one per TMEM lane quarter), each
// team with its own queue ticket, shared-memory state and TMEM columns, and
// its own named barrier.  A thread owns 512 / TEAMS TMEM columns of its lane:
// up to 16 layers 4 teams (16 warps, 128 registers a thread), up to 20 layers
// 3, up to 32 layers 2, up to 64 layers 1.
//
// Partial gradients.  Each step adds four sums (thickness, roughness, Re and
// Im of conj(kbar) / k); a warp reduces them over quads of lanes while it
// distributes the four sums over the quad's lanes (two shuffle stages), so
// that every lane updates one float in shared memory.  All additions have a
// fixed order: results are bitwise reproducible.
//
// Everything else (node positions, smearing exchange, super-tiles, edge
// queue, chunked stacks) follows nr_pair.cu.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "nr_internal.h"
#include "nr_once.h"
#include "nr_pair.cuh"

namespace nrimpl {
namespace {

constexpr int kTeam = 128;            // threads of a team
constexpr int kTeamWarps = kTeam / 32;
constexpr int kTmemCols = 512;        // TMEM columns of an SM
constexpr int kSlotCols = 8;          // columns of one layer: G_j, E_{j+1} of both halves
constexpr int kEqCap = 32;            // interior-edge queue entries of a warp

__host__ __device__ constexpr int roll_teams(int nmax)
{
    return nmax <= 16 ? 4 : nmax <= 20 ? 3 : nmax <= 32 ? 2 : 1;
}

// Shared-memory state of one team
template <int NM, bool RES>
struct TeamSmem {
    static constexpr int CAPQ = 72;              // staged Q points (a super-tile)
    static constexpr int WRN = 416;              // TQ KP of any K >= 3 (408 at K = 5)
    float4 b[(NM + 1) * kTeam];                  // b_j of both halves, j < n; slot NM: G_n
    float acc[kTeamWarps][(NM + 2) * 32];        // partial gradients: 4 sums x 8 lane quads per step
    float wR[2][WRN];                            // w_k R per (Q slot, node), double-buffered
    float4 qd[CAPQ];                             // (Q/2, dQ/2, R_obs, 1/err) per staged Q point
    float2 rs[CAPQ];                             // (residual, S) per staged Q point
    float2 eq[kTeamWarps][3][kEqCap];            // edge queue: node k_0 (hi, lo), Z, Xbar_{j-1}
    float eqr[RES ? kTeamWarps : 1][RES ? kEqCap : 1]; // k_0 dk_0 / d ln f of an entry
    int eqj[kTeamWarps][kEqCap];                 // its medium
    float redd[kTeamWarps][5];                   // loglik (hi), d/dscale, d/dbkg, d/d ln f; loglik (lo)
    double raw[4 * NM + 7];
    StackSmem<NM> sm;
    int item, last;
};

template <int NMAX, bool RES>
struct RollTraits {
    static constexpr int TEAMS = roll_teams(NMAX);
    static constexpr int BLOCK = TEAMS * kTeam;
    static constexpr int COLS = kTmemCols / TEAMS / kSlotCols * kSlotCols; // columns a thread owns
    // sin / cos table, and the TMEM address the allocation returns
    static constexpr size_t TAB = 2 * kTabN * sizeof(float) + 16;
    static constexpr size_t DYN = TAB + TEAMS * sizeof(TeamSmem<NMAX, RES>);
    static_assert(NMAX * kSlotCols <= COLS, "the layers' slots fit the thread's columns");
    static_assert(DYN <= 227 * 1024, "shared memory of one CTA");
};

// ------------------------------------------------------- tensor memory ----
// 8 columns of the warp's own 32 lanes: one thread's 32 bytes each.  .sync:
// the whole warp executes them together.
__device__ __forceinline__ void tmem_store(uint32_t at, c2 u, c2 v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at),
                 "f"(u.re.x), "f"(u.re.y), "f"(u.im.x), "f"(u.im.y), "f"(v.re.x), "f"(v.re.y), "f"(v.im.x),
                 "f"(v.im.y));
}
struct Slot {
    f2 a, b, c, d;
};
__device__ __forceinline__ void tmem_load(uint32_t at, Slot &s)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(s.a.x), "=f"(s.a.y), "=f"(s.b.x), "=f"(s.b.y), "=f"(s.c.x), "=f"(s.c.y), "=f"(s.d.x),
                   "=f"(s.d.y)
                 : "r"(at));
}
__device__ __forceinline__ void tmem_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// the slot's registers are valid after this
__device__ __forceinline__ void tmem_wait_load(Slot &s)
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(s.a.x), "+f"(s.a.y), "+f"(s.b.x), "+f"(s.b.y), "+f"(s.c.x), "+f"(s.c.y), "+f"(s.d.x),
                   "+f"(s.d.y));
}

__device__ __forceinline__ void team_sync(int team)
{
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeam) : "memory");
}

// Drains the `cnt` <= 32 queued interior-edge entries of one warp, one per
// lane, into the warp's partials (acc: [step][32], sums 1 and 3 of a quad are
// Re and Im).  The four lanes of a quad share a slot and add in turn, so the
// order of the additions is fixed.  Kept out of line (rare).
template <bool RES>
__device__ __noinline__ float roll_drain(const float2 (*q)[kEqCap], const int *qj, const float *qr, const float4 *med,
                                         const float *sig, const float4 *adj, int n, int lane, int cnt, float *acc)
{
    float res = 0.f;
    const bool on = lane < cnt;
    int j = 1;
    float2 ub = make_float2(0.f, 0.f);
    __syncwarp();
    if (on) {
        j = qj[lane];
        ub = edge_entry_ubar(q[0][lane], q[1][lane], q[2][lane], j, n, med, sig, adj);
        if constexpr (RES) res = 2.f * ub.x * qr[lane];
    }
    for (int turn = 0; turn < 4; ++turn) {
        if (on && (lane & 3) == turn) {
            // conj(kbar)/k_j = 2 conj(ubar)
            acc[j * 32 + (lane & ~3) + 1] += 2.f * ub.x;
            acc[j * 32 + (lane & ~3) + 3] += -2.f * ub.y;
        }
        __syncwarp();
    }
    return res;
}

// ---------------------------------------------------------------- kernel --
template <int MODE, int NMAX>
__global__ void __launch_bounds__(RollTraits<NMAX, MODE == kGradRes>::BLOCK, 1)
nr_roll_kernel(const KernelArgs ka, const QuadConst qc, const int workers)
{
    constexpr bool RES = MODE == kGradRes;
    constexpr int NM = NMAX;
    using RT = RollTraits<NMAX, RES>;
    using TS = TeamSmem<NMAX, RES>;
    constexpr int WRN = TS::WRN;
    extern __shared__ __align__(16) unsigned char sh_dyn[];
    float *sh_cs = reinterpret_cast<float *>(sh_dyn); // cos, sin at multiples of 2 pi / kTabN

    uint32_t &sh_tmem = *reinterpret_cast<uint32_t *>(sh_dyn + RT::TAB - 16);

    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & (kTeamWarps - 1);
    const int team = threadIdx.x / kTeam;
    const int tid = threadIdx.x & (kTeam - 1);
    TS &ts = reinterpret_cast<TS *>(sh_dyn + RT::TAB)[team];
    StackSmem<NM> &sm = ts.sm;
    float *acc = ts.acc[warp];

    // all 512 columns: one CTA per SM holds them (an allocation waits until
    // an earlier CTA of the SM has freed its own, which every CTA does)
    if (threadIdx.x < 32) {
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(&sh_tmem);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(at), "n"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (int i = threadIdx.x; i < 2 * kTabN; i += RT::BLOCK) sh_cs[i] = qc.cs_tab[i];
    for (int i = tid; i < 2 * WRN; i += kTeam) (&ts.wR[0][0])[i] = 0.f; // padding stays 0
    __syncthreads();
    const uint32_t tmem_base = sh_tmem;
    // this warp's lane quarter, this team's columns
    const uint32_t tm = tmem_base + ((uint32_t)warp << 21) + (uint32_t)(team * RT::COLS);

    const int K = qc.K;          // K >= 3 (the host's choice of this kernel)
    const int KP = (K + 3) & ~3; // node stride of a Q slot in wR (whole float4s)
    const int TQ = ka.tile_q;
    // warp-local tiles where every warp's 64 slots hold whole Q points (as nr_pair.cu)
    const int tqw = 64 / K;
    const bool wloc = TQ == kTeamWarps * tqw;
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

    // `workers` teams take items (the launch's request; the others of the last
    // round of CTAs stay idle): the first ones go round the SMs, the rest by ticket
    int item = team * gridDim.x + blockIdx.x;
    if (item >= workers) item = ka.n_items;
    for (; item < ka.n_items;) {
        const WorkItem wi = ka.items[item];
        if (tid == 0) {
            sm.nc_big[0] = 0;
            sm.p_max = 0;
        }
        team_sync(team);
        if constexpr (NR_DEBUG) {
            if (!item_in_bounds(ka, wi, NMAX)) { // uniform over the team
                if (tid == 0) {
                    atomicOr(ka.status, NR_FLAG_DEBUG_BOUNDS);
                    ts.item = workers + atomicAdd(&ka.ticket[0], 1);
                }
                team_sync(team);
                item = ts.item;
                team_sync(team); // every thread has read ts.item
                continue;
            }
        }
        const StackInfo si = ka.stacks[wi.stack];
        const int n = si.n;
        const double *p = ka.params + si.par_off;
        stage_stack<NM, kNcBig | kNcGrows>(sm, &sm.nc_big[0], p, n, tid, ka.status);
        for (int i = lane; i < (n + 2) * 32; i += 32) acc[i] = 0.f;

        // step j's four sums: over the quad's lanes, one sum left in each lane
        // (lane bit 0: the first or second pair of sums, bit 1: which of the pair)
        const bool odd = lane & 1, high = lane & 2;
        auto add4 = [&](int j, f2 v0, f2 v1, f2 v2, f2 v3) __attribute__((always_inline)) {
            const float a0 = v0.x + v0.y, a1 = v1.x + v1.y, a2 = v2.x + v2.y, a3 = v3.x + v3.y;
            const float t0 = __shfl_xor_sync(kFull, odd ? a0 : a2, 1), t1 = __shfl_xor_sync(kFull, odd ? a1 : a3, 1);
            const f2 k = padd(make_float2(odd ? a2 : a0, odd ? a3 : a1), make_float2(t0, t1));
            const float u = __shfl_xor_sync(kFull, high ? k.x : k.y, 2);
            acc[j * 32 + lane] += (high ? k.y : k.x) + u;
        };
        f2 gres_acc = bc(0.f);
        int eq_cnt = 0; // entries in this warp's interior-edge queue (warp-uniform)
        auto eq_drain = [&]() {
            const float r = roll_drain<RES>(ts.eq[warp], ts.eqj[warp], RES ? ts.eqr[warp] : nullptr, sm.med, sm.sig,
                                            sm.adj, n, lane, eq_cnt, acc);
            if constexpr (RES) gres_acc.x += r;
            eq_cnt = 0;
        };

        // per-thread sums of the loglik terms, d/dscale, d/dbkg (per Q point)
        float ll_hi = 0.f, ll_lo = 0.f, gsc_acc = 0.f, gbk_acc = 0.f;
        const float *qp = ka.q + si.q_begin, *dqp = ka.dq + si.q_begin;
        const float fsc = ka.dq_scale ? (float)ka.dq_scale[wi.stack] : 1.f; // resolution scale of the stack
        const float *rop = ka.r_obs + si.q_begin, *rep = ka.r_err + si.q_begin;
        const int span = (TS::CAPQ / TQ) * TQ;
        int sb = wi.q_lo, s_cnt = 0;
        auto consume = [&](int i) __attribute__((always_inline)) {
            const float2 rs = ts.rs[i];
            const float Re = __ldg(rep + sb + i);
            if (!(Re > 0.f)) atomicOr(ka.status, NR_FLAG_BAD_ERR);
            float t1, t2;
            two_sum(ll_hi, fmaf(rs.x, rs.x, kLog2Pi + 2.f * logf(Re)), t1, t2);
            ll_hi = t1;
            ll_lo += t2;
            const float dldm = -(rs.x * fabsf(ts.qd[i].w));
            gsc_acc = fmaf(dldm, rs.y, gsc_acc);
            gbk_acc += dldm;
        };
        float magic = 0.f; // of the common quantum (split_media)
        auto restage = [&](int q0) {
            int p_bits = 0; // largest k_0^2 or |c_j| this thread sees
            team_sync(team); // the previous super-tile's reads and pairs are complete
            for (int i = tid; i < span; i += kTeam) {
                if (i < s_cnt) consume(i);
                const int qa = q0 + i;
                float4 v = make_float4(0.05f, 0.f, 0.f, 0.f); // past the end: a harmless node, 1/err = 0
                if (qa < wi.q_hi) {
                    v.x = 0.5f * __ldg(qp + qa);
                    v.y = 0.5f * fsc * __ldg(dqp + qa);
                    v.z = __ldg(rop + qa);
                    v.w = rcp_approx(__ldg(rep + qa));
                    // may a node of this Q point lie below an interior edge or
                    // reach its band?  (negative 1/err: yes)
                    const float a = fabsf(v.y) * g_max;
                    const float lo = fmaxf(v.x - a, 0.f), hi = v.x + a;
                    p_bits = max(p_bits, quantum_bits(hi * hi));
                    const float k2lo = lo * lo * (1.f - 1.5f * kEdgeFrac);
                    bool e = false;
                    for (int j = 1; j <= n; ++j) {
                        const float c = sm.med[j].x + sm.med[j].y;
                        e |= c > 0.f && c > k2lo;
                    }
                    if (e && v.w > 0.f) v.w = -v.w;
                }
                ts.qd[i] = v;
            }
            sb = q0;
            s_cnt = min(span, wi.q_hi - q0);
            if (tid <= n) p_bits = max(p_bits, quantum_bits(fabsf(sm.med[tid + 1].x + sm.med[tid + 1].y)));
            p_bits = __reduce_max_sync(kFull, p_bits);
            if (lane == 0) atomicMax(&sm.p_max, p_bits);
            team_sync(team);
            magic = quantum_magic(sm.p_max);
            split_media(sm, n, tid, magic);
            team_sync(team);
        };
        team_sync(team);

        const float scale = sm.scale, bkg = sm.bkg;
        const int nc = sm.nc_big[0];
        const bool renorm = nc & kNcGrows; // divide by A at every interface
        const f2 wks = pmul(wk, bc(scale));
        int buf = 0;
        // t0: the tile's first Q point within the staged super-tile.  Slots past
        // the last Q point are staged harmless (1/err = 0), so the tile needs no
        // test of its end; idle lanes repeat slot 0 with weight 0.
        for (int q0 = wi.q_lo; q0 < wi.q_hi; q0 += span) {
        restage(q0);
        for (int t0 = 0; t0 < s_cnt; t0 += TQ, buf ^= 1) {
            const float4 qd[2] = {ts.qd[t0 + slot_at[0]], ts.qd[t0 + slot_at[1]]};
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
            quantise2(p_hi, p_lo, magic);
            __syncwarp();

            // a3-a6 forward from the backing up (n >= 3: the top, middle and
            // bottom steps are distinct)
            c2 A = c2{bc(1.f), bc(0.f)}, B;
            auto forward = [&](auto TRIG) __attribute__((always_inline)) {
                constexpr int T = decltype(TRIG)::value;
                Kz2 kb = medium_kz2<kRootPlain, true>(p_hi, p_lo, sm.med[n + 1]);
                {
                    const Kz2 kj = medium_kz2<kRootFull, true>(p_hi, p_lo, sm.med[n]);
                    const float4 I = sm.itf[n];
                    const c2 G = fresnel_g2<false, T>(kj, kb, I, sh_cs);
                    B = cscl2(I.x, I.y, G);
                    ts.b[NM * kTeam + tid] = make_float4(G.re.x, G.re.y, G.im.x, G.im.y);
                    kb = kj;
                }
                auto step = [&](int j, auto TOP) __attribute__((always_inline)) {
                    constexpr bool top = decltype(TOP)::value;
                    Kz2 kj;
                    if constexpr (top) kj = Kz2{k0h, bc(0.f), k0l, bc(0.f)};
                    else kj = medium_kz2<kRootFull, true>(p_hi, p_lo, sm.med[j]);
                    const float4 I = sm.itf[j];
                    const float4 L = sm.lay[j + 1];
                    const c2 G = fresnel_g2<top, T>(kj, kb, I, sh_cs);
                    const c2 E = layer_phase2<true>(kb, L, sh_cs);
                    tmem_store(tm + j * kSlotCols, G, E);
                    const c2 r = cscl2(I.x, I.y, G);
                    const c2 b = cmul2(B, E);
                    ts.b[j * kTeam + tid] = make_float4(b.re.x, b.re.y, b.im.x, b.im.y);
                    B = cfma2(r, A, b);
                    A = cfma2(r, b, A);
                    if constexpr (T == kTrigTable) {
                        if (renorm) {
                            B = cmul2(B, cinv2(A));
                            A = c2{bc(1.f), bc(0.f)};
                        }
                    }
                    kb = kj;
                };
#pragma unroll 1
                for (int j = n - 1; j >= 1; --j) step(j, std::false_type{});
                step(0, std::true_type{});
            };
            if (nc) forward(Pos<kTrigTable>{});
            else forward(Pos<kTrigSmall>{});
            const c2 iA = cinv2(A); // 1 / A_0
            const c2 X0 = cmul2(B, iA);
            f2 R = pfma(X0.re, X0.re, pmul(X0.im, X0.im));
            if (!(qok.x && qok.y)) {
                atomicOr(ka.status, NR_FLAG_BAD_Q);
                if (!qok.x) R.x = __int_as_float(0x7fffffff);
                if (!qok.y) R.y = __int_as_float(0x7fffffff);
            }
            __syncwarp(); // the wait is .aligned: lanes with a bad Q point are back
            tmem_wait_store();

            // a8-a10: smearing sum, model, residual, adjoint seed
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (lane_on[h]) ts.wR[buf][wr_at[h]] = half(wk, h) * half(R, h);
            if (wloc) __syncwarp();
            else team_sync(team);
            f2 S;
            {
                float ps = 0.f;
                if (row_on) {
                    const float4 *row = reinterpret_cast<const float4 *>(&ts.wR[buf][row_at]);
                    for (int c = part; c < KP / 4; c += sgl) {
                        const float4 v = row[c];
                        ps += (v.x + v.y) + (v.z + v.w);
                    }
                }
                for (int o = 1; o < sgl; o <<= 1) ps += __shfl_xor_sync(kFull, ps, o);
                S.x = __shfl_sync(kFull, ps, from[0]);
                S.y = __shfl_sync(kFull, ps, from[1]);
            }
            const f2 ie = make_float2(fabsf(qd[0].w), fabsf(qd[1].w));
            const f2 res = pmul(psub(pfma(bc(scale), S, bc(bkg)), make_float2(qd[0].z, qd[1].z)), ie);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (lead[h]) ts.rs[t0 + slot_at[h]] = make_float2(half(res, h), half(S, h));
            const f2 Rb = pmul(wks, pneg(pmul(res, ie))); // w_k scale dl/dm (0 on idle slots)

            // a7: adjoint sweep from the fronting down to the backing.  With
            // Xbar_0 = 2 Rbar X_0: Bbar_0 = Xbar_0 / conj(A_0), Abar_0 =
            // -conj(X_0) Bbar_0; every step applies the conjugate transpose of
            // the forward one.  A_{j+1} = A_j - r_j b_j runs the forward's A back.
            // Abar and Bbar cancel where the reflectivity is near 1 (their common
            // scale is free, and roundings along it are amplified); there the sweep
            // carries Z_j = Bbar_j / conj(A_j) alone:
            //   rbar_j = conj(A_{j+1}^2 - b_j^2) Z_j,  bbar_j = conj(A_{j+1}) t_j,
            //   Z_{j+1} = conj(E_{j+1}) t_j,  t_j = conj(1 - r_j^2) Z_j,
            // eight operations a layer more, as accurate as the Moebius form.
            // Layers' gradients of 600 unsmeared points below an edge, 90 % within
            // 9.8e-5 (4 layers), 2.9e-4 (10), 1.3e-3 (40) with Abar and Bbar,
            // 2.9e-5, 4.4e-5, 5.6e-5 with Z.  On the tiles that need it it costs the
            // ten- and twelve-layer gradients 1 %.
            const f2 Rb2 = padd(Rb, Rb);
            c2 Bb = cmulc2(iA, X0);
            Bb = c2{pmul(Bb.re, Rb2), pmul(Bb.im, Rb2)};
            const f2 mR = pneg(pmul(Rb2, R));
            c2 Ab = c2{pmul(iA.re, mR), pneg(pmul(iA.im, mR))};
            c2 kbar = czero();
            c2 kj = c2{k0h, bc(0.f)};
            f2 yj = bc(0.f); // 1 / |k_j|^2
            c2 Xb_up = czero(); // Xbar_{j-1} (edge sweeps)
            const bool reach[2] = {lane_on[0] && qd[0].w < 0.f, lane_on[1] && qd[1].w < 0.f};
            const f2 edge_u = pmul(bc(kEdgeFrac), pmul(k0h, k0h));
            const f2 wres = RES ? pmul(dQh, g_hi) : bc(0.f);
            f2 res_sum = bc(0.f), res_k0 = bc(0.f);
            // EDG: Bb holds Z, Ab is not used; REN (stacks divided by A at every
            // interface): A_j = 1, Bb holds Xbar_j between the steps
            auto adj_step = [&](int j, auto TOP, auto BOT, auto EDG, auto REN) __attribute__((always_inline)) {
                constexpr bool top = decltype(TOP)::value, bot = decltype(BOT)::value, edg = decltype(EDG)::value;
                // G_j, E_{j+1}: the load runs while k_{j+1} is formed (never across a
                // loop iteration: its registers may not be copied before the wait)
                Slot sl;
                if constexpr (!bot) tmem_load(tm + j * kSlotCols, sl);
                const float4 I = sm.itf[j], C = sm.adj[j];
                const Kz2 kz1 = medium_kz2<kRootPlain, true>(p_hi, p_lo, sm.med[j + 1]);
                const c2 kj1 = kc2(kz1);
                const float4 bv = ts.b[(bot ? NM : j) * kTeam + tid];
                c2 G, b = czero(), kbar1 = czero(), rb = Bb, Xb_in = czero();
                f2 accD = bc(0.f);
                float2 Z[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if constexpr (bot) {
                    G = c2{make_float2(bv.x, bv.y), make_float2(bv.z, bv.w)};
                } else {
                    tmem_wait_load(sl);
                    G = c2{sl.a, sl.b};
                    const c2 E = c2{sl.c, sl.d};
                    b = c2{make_float2(bv.x, bv.y), make_float2(bv.z, bv.w)};
                    const c2 r = cscl2(I.x, I.y, G);
                    if constexpr (decltype(REN)::value) {
                        const c2 rb1 = cmul2(r, b), iD = cinv2(c2{padd(bc(1.f), rb1.re), rb1.im});
                        Xb_in = Bb;
                        Bb = cmulc2(iD, cmulc2(iD, Bb));
                        A = c2{bc(1.f), bc(0.f)};
                    } else {
                        if constexpr (edg) Xb_in = cmulc2(A, cmulc2(A, Bb));
                        A = cfnma2(r, b, A); // A_{j+1}
                    }
                    // adjoint of b = E B: with U = conj(b) bbar the thickness sum
                    // takes Im(conj(k) U) and kbar_{j+1} gets -2 i d U
                    c2 bb;
                    if constexpr (edg) {
                        const c2 s = cadd2(A, b), d = c2{psub(A.re, b.re), psub(A.im, b.im)};
                        rb = cmulc2(cmul2(s, d), Bb);
                        const c2 t = cmulc2(one_minus_sq2(r), Bb);
                        bb = cmulc2(A, t);
                        Bb = cmulc2(E, t);
                    } else {
                        rb = cfmac2(b, Ab, cmulc2(A, Bb));
                        bb = cfmac2(r, Ab, Bb);
                        Ab = cfmac2(r, Bb, Ab);
                        Bb = cmulc2(E, bb);
                    }
                    const c2 U = cmulc2(b, bb);
                    accD = pfma(kj1.re, U.im, pneg(pmul(kj1.im, U.re)));
                    kbar1 = c2{pmul(bc(C.w), U.im), pneg(pmul(bc(C.w), U.re))};
                }
                // Fresnel: with g = conj(G) rbar and N the numerator, kbar_j +=
                // conj(k_{j+1}) g (s conj(N) + 2), kbar_{j+1} += conj(k_j) g
                // (s conj(N) - 2); the roughness sum takes Re(N conj(g) k_j k_{j+1})
                const c2 gg = cmulc2(G, rb);
                const c2 ga = cmulc2(kj1, gg);
                const c2 gb = top ? c2{pmul(kj.re, gg.re), pmul(kj.re, gg.im)} : cmulc2(kj, gg);
                kbar1 = cscla2(C.y, C.z, gb, kbar1);
                const c2 t = top ? c2{pmul(ga.re, kj.re), pneg(pmul(ga.im, kj.re))} : cmulc2(ga, kj);
                const f2 accS = pfma(bc(I.x), t.re, pneg(pmul(bc(I.y), t.im)));
                f2 ur = bc(0.f), ui = bc(0.f);
                if constexpr (top) {
                    if constexpr (RES) res_k0 = pfma(bc(C.x), ga.re, pneg(pmul(bc(C.z), ga.im)));
                } else {
                    kbar = cscla2(C.x, C.z, ga, kbar);
                    // k_j complete: accumulate conj(kbar) / k_j, or queue the
                    // interior-edge evaluation
                    f2 inv = yj;
                    if constexpr (edg) {
                        const f2 far = pmul(edge_u, yj); // |k_j|^2 < edge_u
                        const b2 edge{reach[0] && far.x > 1.f, reach[1] && far.y > 1.f};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const bool eh = h ? edge.y : edge.x;
                            const unsigned em = __ballot_sync(kFull, eh);
                            if (em) {
                                if (eq_cnt + __popc(em) > kEqCap) eq_drain();
                                if (eh) {
                                    const int slot =
                                        queue_slot<kEqCap>(eq_cnt + __popc(em & ((1u << lane) - 1u)), ka.status);
                                    // Z = E X of the layer below (0 at the bottom interface)
                                    if (!bot)
                                        Z[h] = cdiv(make_float2(half(b.re, h), half(b.im, h)),
                                                    make_float2(half(A.re, h), half(A.im, h)));
                                    if constexpr (RES) ts.eqr[warp][slot] = half(k0h, h) * half(wres, h);
                                    ts.eq[warp][0][slot] = make_float2(half(k0h, h), half(k0l, h));
                                    ts.eq[warp][1][slot] = Z[h];
                                    ts.eq[warp][2][slot] = make_float2(half(Xb_up.re, h), half(Xb_up.im, h));
                                    ts.eqj[warp][slot] = j;
                                }
                                __syncwarp();
                                eq_cnt = queue_count<kEqCap>(eq_cnt + __popc(em));
                            }
                        }
                        inv = psel(edge, bc(0.f), inv);
                    }
                    const c2 kq = cmul2(kbar, kj);
                    ur = pmul(kq.re, inv);
                    ui = pneg(pmul(kq.im, inv));
                    if constexpr (RES) res_sum = padd(res_sum, ur);
                }
                add4(j, accD, accS, ur, ui);
                if constexpr (edg) Xb_up = Xb_in;
                kbar = kbar1;
                kj = kj1;
                yj = kz1.y;
                if constexpr (bot) { // backing medium n+1
                    const c2 kq = cmul2(kbar, kj);
                    ur = pmul(kq.re, yj);
                    ui = pneg(pmul(kq.im, yj));
                    add4(n + 1, bc(0.f), bc(0.f), ur, ui);
                    if constexpr (RES) res_sum = padd(res_sum, ur);
                }
            };
            auto sweep = [&](auto EDG, auto REN) __attribute__((always_inline)) {
                if constexpr (decltype(EDG)::value) Bb = cmulc2(iA, Bb); // Z_0 (Xbar_0 where A_0 = 1)
                adj_step(0, std::true_type{}, std::false_type{}, EDG, REN);
#pragma unroll 1
                for (int j = 1; j <= n - 1; ++j) adj_step(j, std::false_type{}, std::false_type{}, EDG, REN);
                adj_step(n, std::false_type{}, std::true_type{}, EDG, REN);
            };
            // the staged sign of 1/err marks Q points whose nodes may lie below an
            // interior edge or in its band (warp-uniform choice)
            __syncwarp(); // the sweeps begin with an .aligned load, whichever lanes stored above
            if (renorm) sweep(std::true_type{}, std::true_type{});
            else if (__any_sync(kFull, reach[0] || reach[1])) sweep(std::true_type{}, std::false_type{});
            else sweep(std::false_type{}, std::false_type{});
            if constexpr (RES) gres_acc = pfma(wres, pfma(k0h, res_sum, res_k0), gres_acc);
        }
        }
        if (tid == 0) ts.item = workers + atomicAdd(&ka.ticket[0], 1); // its latency overlaps the reductions
        if (eq_cnt > 0) eq_drain();

        // ---- team reduction of the item's partial sums into raw ----
        team_sync(team);
        for (int i = tid; i < s_cnt; i += kTeam) consume(i);
        for (int i = tid; i < 4 * n + 3; i += kTeam) {
            // raw layout: accD [n] | accUr [n+1] | accUi [n+1] | accS [n+1];
            // step of the sum, and which lane of the quads holds it
            const int step = i < n ? i : i < 2 * n + 1 ? i - n + 1 : i < 3 * n + 2 ? i - 2 * n : i - 3 * n - 2;
            const int of = i < n ? 0 : i < 2 * n + 1 ? 1 : i < 3 * n + 2 ? 3 : 2;
            float w4[kTeamWarps];
#pragma unroll
            for (int w = 0; w < kTeamWarps; ++w) {
                const float *v = ts.acc[w] + step * 32 + of;
                w4[w] = ((v[0] + v[4]) + (v[8] + v[12])) + ((v[16] + v[20]) + (v[24] + v[28]));
            }
            ts.raw[i] = sum4(w4[0], w4[1], w4[2], w4[3], 0.f);
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
                ts.redd[warp][0] = h;
                ts.redd[warp][1] = a1;
                ts.redd[warp][2] = a2;
                ts.redd[warp][3] = a3;
                ts.redd[warp][4] = l;
            }
        }
        team_sync(team);
        if (tid < (RES ? 4 : 3)) {
            const float lo = tid == 0 ? (ts.redd[0][4] + ts.redd[1][4]) + (ts.redd[2][4] + ts.redd[3][4]) : 0.f;
            ts.raw[4 * n + 3 + tid] = sum4(ts.redd[0][tid], ts.redd[1][tid], ts.redd[2][tid], ts.redd[3][tid], lo);
        }
        item = ts.item; // the next item, before its slot is written again
        team_sync(team);
        const int nout = 4 * n + (RES ? 7 : 6);
        if (si.n_chunks == 1) {
            finalize_stack<MODE>(ts.raw, n, p, wi.stack, si.par_off, ka.ll_out, ka.grad_out, ka.res_out, tid, kTeam);
        } else {
            double *slot = ka.partials + si.part_base + (int64_t)wi.chunk * n_slot(n);
            for (int i = tid; i < nout; i += kTeam) slot[i] = ts.raw[i];
            team_sync(team);
            if (tid == 0) {
                __threadfence(); // after the barrier: covers the whole team's slot
                const int prev = atomicAdd(&ka.stack_done[wi.stack], 1);
                ts.last = prev == si.n_chunks - 1;
            }
            team_sync(team);
            if (ts.last) {
                __threadfence();
                for (int i = tid; i < nout; i += kTeam) {
                    double s = 0.0;
#pragma unroll 8
                    for (int c = 0; c < si.n_chunks; ++c)
                        s += __ldcg(ka.partials + si.part_base + (int64_t)c * n_slot(n) + i);
                    ts.raw[i] = s;
                }
                team_sync(team);
                finalize_stack<MODE>(ts.raw, n, p, wi.stack, si.par_off, ka.ll_out, ka.grad_out, ka.res_out, tid,
                                     kTeam);
                if (tid == 0) ka.stack_done[wi.stack] = 0;
            }
        }
        team_sync(team); // sm / raw / item / wR reused by the next item
    }
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols));
    // last CTA out resets the queue for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        const int done = atomicAdd(&ka.ticket[1], 1);
        if (done == (int)gridDim.x - 1) {
            ka.ticket[0] = 0;
            ka.ticket[1] = 0;
            __threadfence();
        }
    }
}

template <int MODE, int NMAX>
cudaError_t roll_attr()
{
    return cudaFuncSetAttribute(nr_roll_kernel<MODE, NMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)RollTraits<NMAX, MODE == kGradRes>::DYN);
}

// `workers` teams: as many CTAs as there are SMs before a second team of one is used
template <int MODE, int NMAX>
cudaError_t roll_launch_one(int workers, const KernelArgs &a, const QuadConst &qc, cudaStream_t st)
{
    using RT = RollTraits<NMAX, MODE == kGradRes>;
    static OncePerDevice attr;
    int dev = 0, sms = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = attr.run(dev, roll_attr<MODE, NMAX>);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int full = (workers + RT::TEAMS - 1) / RT::TEAMS;
    const int grid = full > sms ? full : workers < sms ? workers : sms;
    nr_roll_kernel<MODE, NMAX><<<grid, RT::BLOCK, RT::DYN, st>>>(a, qc, workers);
    return cudaGetLastError();
}

} // namespace

#define NR_ROLL_BUCKETS(X) X(4) X(8) X(12) X(16) X(20) X(32) X(64)

// resident teams per SM (the work queue's consumers)
cudaError_t roll_occupancy(int mode, int nmax, int *teams)
{
    (void)mode;
    *teams = roll_teams(nmax);
    return cudaSuccess;
}

cudaError_t launch_roll(int mode, int nmax, int workers, const KernelArgs &a, const QuadConst &qc, cudaStream_t st)
{
    if (mode == kGradRes) {
#define X(B) if (nmax == B) return roll_launch_one<kGradRes, B>(workers, a, qc, st);
        NR_ROLL_BUCKETS(X)
#undef X
    } else {
#define X(B) if (nmax == B) return roll_launch_one<kGrad, B>(workers, a, qc, st);
        NR_ROLL_BUCKETS(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

} // namespace nrimpl
