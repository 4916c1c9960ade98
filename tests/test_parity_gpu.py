"""GPU parity: the CUDA path (through the C ABI) against the CPU oracle on the
same seeded inputs, element by element.

Tolerances (per stack):
  smeared model m:   max |log m - log m_ref|              <= 2e-5
  log-likelihood:    |l - l_ref| / |l_ref|                <= 1e-5
  gradient:          ||(g - g_ref) * typ||_inf / ||g_ref * typ||_inf <= 1e-4
with typ = (1 A, 1e-6 A^-2, 1e-8 A^-2, 1 A, 1, 1e-7) per parameter class
(the pre-scaling advice of Sec. 2.3.1).  The model bound is twice the
log-likelihood's: a quadrature node within about 0.1 % (in k^2) of an
interior layer's critical edge loses digits to the cancellation of the
Parratt step above that layer (relative error ~ u k_0 / |k_j|), which the
smeared value keeps in part while the sum over Q points of the likelihood
averages it away.  A stack whose exact results move
by more than these bounds / 8 when its inputs are perturbed by one FP32
unit roundoff (oracle.perturbation_floor: an ill-conditioned stack, e.g.
a waveguide resonance sampled at its peak) is held to 8 times that response
instead: an FP32 evaluation cannot land closer than its own roundings allow.
The plain FP64 path is held to 1e-12 (log-likelihood; 1e-10 on films of up
to 5000 A), FP32 rounding of its float output (model) and 1e-5 (its
central-difference gradient).
"""
import ctypes
import os

import numpy as np
import pytest

import oracle
import paper_2509_06924_gb300 as nr
from paper_2509_06924_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL_M, TOL_LL, TOL_G = 2e-5, 1e-5, 1e-4
COND = 8.0  # headroom over the oracle's own response to FP32-size input perturbations


def run_gpu(wl, precision="mixed", modes=("model", "loglik", "grad"), **kw):
    ctx = nr.Context(n_quad=wl.n_quad, precision=precision, **kw)
    b = nr.Batch.from_workload(wl)
    out = {}
    if "model" in modes:
        out["m"] = ctx.reflectivity(b).cpu().numpy().astype(np.float64)
    if "loglik" in modes:
        out["ll"] = ctx.loglik(b).cpu().numpy()
    if "grad" in modes:
        ll, g = ctx.loglik_grad(b)
        out["ll_g"], out["g"] = ll.cpu().numpy(), g.cpu().numpy()
    out["flags"] = ctx.device_status()
    ctx.close()
    return out


def run_oracle(wl, modes=("model", "grad")):
    out = {}
    if "model" in modes:
        out["m"] = oracle.batch("model", wl.n_layers, wl.params, wl.dataset, wl.q_off, wl.q, wl.dq, None, None,
                                wl.n_quad)
    if "grad" in modes:
        out["ll"], out["g"] = oracle.batch("grad", wl.n_layers, wl.params, wl.dataset, wl.q_off, wl.q, wl.dq,
                                           wl.r_obs, wl.r_err, wl.n_quad)
    return out


def grad_err(wl, g, g_ref, stacks=None):
    po = wl.par_off
    worst = 0.0
    for s in (range(wl.n_stacks) if stacks is None else stacks):
        typ = W.typical_scale(int(wl.n_layers[s]))
        a, b = g[po[s]:po[s + 1]] * typ, g_ref[po[s]:po[s + 1]] * typ
        den = np.max(np.abs(b))
        worst = max(worst, float(np.max(np.abs(a - b)) / den) if den > 0 else float(np.max(np.abs(a))))
    return worst


def stack_errors(wl, gpu, ref):
    """Per-stack errors of the outputs present in both gpu and ref:
    'model' max |log m - log m_ref|, 'loglik' and 'loglik_g' (the gradient
    call's) |l - l_ref| / |l_ref|, 'grad' the scaled gradient error."""
    S = wl.n_stacks
    out = {}
    if "m" in gpu and "m" in ref:
        assert np.all(np.isfinite(gpu["m"]))
        e = np.abs(np.log(gpu["m"]) - np.log(ref["m"]))
        oo = wl.out_off
        out["model"] = np.array([e[oo[s]:oo[s + 1]].max() if oo[s + 1] > oo[s] else 0.0 for s in range(S)])
    if "ll" in gpu and "ll" in ref:
        out["loglik"] = np.abs(gpu["ll"] - ref["ll"]) / np.maximum(np.abs(ref["ll"]), 1e-300)
    if "g" in gpu and "g" in ref:
        out["loglik_g"] = np.abs(gpu["ll_g"] - ref["ll"]) / np.maximum(np.abs(ref["ll"]), 1e-300)
        out["grad"] = np.array([grad_err(wl, gpu["g"], ref["g"], [s]) for s in range(S)])
    return out


FLOOR_OF = {"model": "model", "loglik": "loglik", "loglik_g": "loglik", "grad": "grad"}


def check_bounds(wl, errs, tol):
    """Every stack within its base bound tol[kind], or, where the stack is
    ill-conditioned, within COND times the oracle's response to FP32-size
    input perturbations (computed for the stacks over the base bound only)."""
    over = sorted({s for k, e in errs.items() for s in np.flatnonzero(e > tol[k])})
    if not over:
        return
    sub = wl.subset(over)
    typ = np.concatenate([W.typical_scale(int(n)) for n in sub.n_layers])
    fl = oracle.perturbation_floor(sub.n_layers, sub.params, sub.dataset, sub.q_off, sub.q, sub.dq, sub.r_obs,
                                   sub.r_err, sub.n_quad, typ)
    for i, s in enumerate(over):
        for k, e in errs.items():
            bound = max(tol[k], COND * fl[FLOOR_OF[k]][i])
            assert e[s] <= bound, (f"stack {s} {k}: error {e[s]:.3e} above {tol[k]:.0e} and above {COND:g} x its "
                                   f"FP32 perturbation floor {fl[FLOOR_OF[k]][i]:.3e}")


def assert_parity(wl, gpu, ref, tol_m=TOL_M, tol_ll=TOL_LL, tol_g=TOL_G):
    assert gpu["flags"] == 0
    errs = stack_errors(wl, gpu, ref)
    check_bounds(wl, errs, {"model": tol_m, "loglik": tol_ll, "loglik_g": tol_ll, "grad": tol_g})


# ------------------------------------------------------------ workloads ----
# sizes the oracle finishes in seconds, spanning several CTA tiles and a
# ragged last tile (400 = 33 x 12 + 4 for K = 21, 200 = 13 x 15 + 5 for K = 17)
SMALL = [("film_1l", 96), ("thick_oxide", 128), ("oled_cofit", 8), ("uneven", 48), ("vi_step", 4)]


@pytest.mark.parametrize("name,S", SMALL)
def test_mixed_parity_small(name, S):
    wl = W.make_workload(name, n_stacks=S)
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


@pytest.mark.parametrize("name,S", [("film_1l", 8), ("thick_oxide", 8), ("oled_cofit", 2), ("uneven", 10)])
def test_fp64_plain_parity(name, S):
    wl = W.make_workload(name, n_stacks=S)
    gpu = run_gpu(wl, precision="fp64")
    ref = run_oracle(wl)
    assert gpu["flags"] == 0
    # model output is float32: its rounding only
    np.testing.assert_allclose(gpu["m"], ref["m"], rtol=1.2e-7, atol=0)
    np.testing.assert_allclose(gpu["ll"], ref["ll"], rtol=1e-12)
    np.testing.assert_array_equal(gpu["ll"], gpu["ll_g"])
    # central differences with h = eps^(1/3) typ: truncation error
    assert grad_err(wl, gpu["g"], ref["g"]) <= 1e-5


# full-size workloads in the launch configuration the benchmark times;
# sampled stacks are compared with the oracle one by one
FULL = [("thick_oxide", 64), ("film_1l", 48), ("oled_cofit", 12), ("uneven", 12), ("vi_step", 6)]


@pytest.mark.parametrize("name,samples", FULL)
def test_mixed_parity_full_size_sampled(name, samples):
    wl = W.make_workload(name)
    gpu = run_gpu(wl, modes=("loglik", "grad"))
    assert gpu["flags"] == 0
    assert np.all(np.isfinite(gpu["g"])) and np.all(np.isfinite(gpu["ll_g"])) and np.all(np.isfinite(gpu["ll"]))
    rng = np.random.default_rng(20250906)
    stacks = np.sort(rng.choice(wl.n_stacks, size=min(samples, wl.n_stacks), replace=False))
    sub = wl.subset(stacks)
    ref = run_oracle(sub, modes=("model", "grad"))
    po, oo = wl.par_off, wl.out_off
    # the smeared model of the whole batch (nr_reflectivity), the sampled
    # stacks' slices taken on the device
    ctx = nr.Context(n_quad=wl.n_quad)
    m_all = ctx.reflectivity(nr.Batch.from_workload(wl))
    idx = torch.as_tensor(np.concatenate([np.arange(oo[s], oo[s + 1]) for s in stacks]), device=m_all.device)
    m = m_all[idx].cpu().numpy().astype(np.float64)
    assert ctx.device_status() == 0
    ctx.close()
    del m_all
    sel = {"m": m, "ll": gpu["ll"][stacks], "ll_g": gpu["ll_g"][stacks],
           "g": np.concatenate([gpu["g"][po[s]:po[s + 1]] for s in stacks])}
    check_bounds(sub, stack_errors(sub, sel, ref), {"model": TOL_M, "loglik": TOL_LL, "loglik_g": TOL_LL,
                                                   "grad": TOL_G})
    # a property that holds for every stack: only SLD differences matter,
    # so d/d rho_0 = -sum_j d/d rho_j
    for s in range(0, wl.n_stacks, max(1, wl.n_stacks // 4096)):
        n = int(wl.n_layers[s])
        gr = gpu["g"][po[s]:po[s + 1]][W.layout(n)["rho"]]
        assert abs(gr[0] + gr[1:].sum()) <= 1e-9 * np.abs(gr).max() + 1e-300


def test_full_size_is_deterministic():
    wl = W.make_workload("thick_oxide")
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    ll1, g1 = ctx.loglik_grad(b)
    ll2, g2 = ctx.loglik_grad(b)
    assert torch.equal(ll1, ll2) and torch.equal(g1, g2)
    assert ctx.device_status() == 0


# ----------------------------------------------------------- edge cases ----
def custom_workload(stacks, datasets, K=17, data_from_oracle=True):
    """stacks: list of (n, packed params, dataset index); datasets: list of
    (Q, dQ) arrays.  Data: oracle model of the first stack on each dataset
    x 1.03, e = 5 %."""
    q_off = np.concatenate([[0], np.cumsum([len(q) for q, _ in datasets])]).astype(np.int64)
    q = np.concatenate([np.asarray(q, np.float32) for q, _ in datasets]) if datasets else np.zeros(0, np.float32)
    dq = np.concatenate([np.asarray(d, np.float32) for _, d in datasets]) if datasets else np.zeros(0, np.float32)
    r_obs = np.ones_like(q)
    r_err = np.full_like(q, 0.05)
    if data_from_oracle:
        for di in range(len(datasets)):
            a, b = int(q_off[di]), int(q_off[di + 1])
            owner = [s for s in stacks if s[2] == di]
            if owner and b > a:
                m = oracle.model(owner[0][0], owner[0][1], q[a:b], dq[a:b], K)
                r_obs[a:b] = (1.03 * m).astype(np.float32)
                r_err[a:b] = (0.05 * m).astype(np.float32)
    return W.Workload("custom", np.array([s[0] for s in stacks], np.int32),
                      np.concatenate([s[1] for s in stacks]), np.array([s[2] for s in stacks], np.int32),
                      q_off, q, dq, r_obs, r_err, K)


def rand_stack(rng, n, front=0.0, back=2.07e-6, d_range=(20, 400), absorbing=True):
    d = rng.uniform(*d_range, n)
    rho = rng.uniform(-0.5e-6, 6.5e-6, n)
    iota = rng.uniform(0, 1e-8, n) if absorbing else np.zeros(n)
    sig = rng.uniform(0, 15, n + 1)
    return W.pack(d, np.concatenate([[front], rho, [back]]), np.concatenate([iota, [0.0]]), sig,
                  rng.uniform(0.9, 1.1), rng.uniform(1e-8, 1e-6))


def edge_points(n, lo, hi, S=600):
    """S stacks of n layers, each on its own unsmeared Q point with k_j^2 / k_0^2
    of one layer uniform in [lo, hi)."""
    rng = np.random.default_rng(n)
    stacks, datasets = [], []
    while len(stacks) < S:
        st = rand_stack(rng, n)
        c = 4 * np.pi * (st[W.layout(n)["rho"]][rng.integers(1, n + 1)] - st[W.layout(n)["rho"]][0])
        f = rng.uniform(lo, hi)
        if c > 1e-6:
            q = np.array([2 * np.sqrt(c / (1 - f))], np.float32)
            stacks.append((n, st, len(datasets)))
            datasets.append((q, 0 * q))
    return custom_workload(stacks, datasets, K=5)


def layer_grad_err(wl, n):
    """Scaled gradient errors of n-layer stacks, scale and background left out."""
    g, ref = run_gpu(wl, modes=("grad",))["g"], run_oracle(wl, modes=("grad",))["g"]
    g, ref = ((v.reshape(wl.n_stacks, -1) * W.typical_scale(n))[:, :4 * n + 4] for v in (g, ref))
    return np.max(np.abs(g - ref), 1) / np.max(np.abs(ref), 1)


def test_bare_substrates_mixed_with_films():
    rng = np.random.default_rng(1)
    grid = (W.log_grid(123, 0.004, 0.3), 0.04 * W.log_grid(123, 0.004, 0.3))
    stacks = [(0, W.pack([], [0.0, 2.07e-6], [0.0], [4.0], 1.0, 1e-7), 0),
              (1, rand_stack(rng, 1), 0),
              (0, W.pack([], [6.35e-6, 2.07e-6], [1e-9], [0.0], 1.0, 5e-7), 0)]
    wl = custom_workload(stacks, [grid])
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_deep_stacks_every_bucket():
    rng = np.random.default_rng(2)
    grid = (W.log_grid(77, 0.005, 0.25), 0.05 * W.log_grid(77, 0.005, 0.25))
    ns = [2, 3, 5, 9, 13, 17, 20]           # one stack in every register bucket up to 20 layers
    stacks = [(n, rand_stack(rng, n), 0) for n in ns]
    wl = custom_workload(stacks, [grid])
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_stacks_deeper_than_the_workloads():
    """21..64 layers (beyond every workload), under the same bounds."""
    rng = np.random.default_rng(4)
    grid = (W.log_grid(77, 0.005, 0.25), 0.05 * W.log_grid(77, 0.005, 0.25))
    ns = [21, 33, 64]
    stacks = [(n, rand_stack(rng, n, d_range=(5, 60)), 0) for n in ns]
    wl = custom_workload(stacks, [grid])
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_empty_and_ragged_datasets():
    rng = np.random.default_rng(3)
    grids = [(np.zeros(0), np.zeros(0)),
             (W.log_grid(1, 0.05, 0.05), np.array([0.002])),
             (W.log_grid(253, 0.005, 0.3), 0.03 * W.log_grid(253, 0.005, 0.3)),
             (W.log_grid(13, 0.01, 0.2), 0.08 * W.log_grid(13, 0.01, 0.2))]
    stacks = [(1, rand_stack(rng, 1), 0), (2, rand_stack(rng, 2), 1), (3, rand_stack(rng, 3), 2),
              (1, rand_stack(rng, 1), 3), (4, rand_stack(rng, 4), 0)]
    wl = custom_workload(stacks, grids)
    gpu = run_gpu(wl)
    ref = run_oracle(wl)
    assert gpu["flags"] == 0
    # stacks on the empty dataset: loglik 0 and a zero gradient
    for s in (0, 4):
        assert gpu["ll_g"][s] == 0.0 and ref["ll"][s] == 0.0
        po = wl.par_off
        assert np.all(gpu["g"][po[s]:po[s + 1]] == 0.0)
    keep = [1, 2, 3]
    sub = wl.subset(keep)
    po = wl.par_off
    g = np.concatenate([gpu["g"][po[s]:po[s + 1]] for s in keep])
    assert grad_err(sub, g, run_oracle(sub, modes=("grad",))["g"]) <= TOL_G
    assert gpu["m"].size == int(wl.out_off[-1])
    e = np.max(np.abs(np.log(gpu["m"]) - np.log(ref["m"])))
    assert e <= TOL_M


@pytest.mark.parametrize("K", [1, 2, 32])
def test_quadrature_orders(K):
    wl = W.make_workload("film_1l", n_stacks=40)
    wl.n_quad = K
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


# The 1- and 2-layer gradient buckets (n = 0, 1, 2) run two evaluations per
# thread when K >= 3; a warp's 64 evaluations straddle Q slots differently
# for every K.  Stacks with films denser than the substrate put nodes in the
# interior critical-edge band (the per-warp queue); the second dataset is
# dense around those edges.
@pytest.mark.parametrize("K", [3, 4, 5, 7, 13, 31])
def test_paired_gradient_kernel_orders_and_buckets(K):
    rng = np.random.default_rng(100 + K)
    q1, q2 = W.log_grid(61, 0.004, 0.3), W.log_grid(29, 0.008, 0.03)
    datasets = [(q1, 0.05 * q1), (q2, 0.06 * q2)]
    stacks = [(1, rand_stack(rng, 1), 0), (2, rand_stack(rng, 2), 1),
              (0, W.pack([], [0.0, 2.07e-6], [0.0], [3.0], 1.0, 1e-7), 0),
              (2, W.pack([300.0, 150.0], [0.0, 6.0e-6, 4.5e-6, 2.07e-6], [0.0, 0.0, 0.0], [3.0, 5.0, 4.0],
                         1.0, 1e-7), 1),
              (1, W.pack([900.0], [0.0, 5.0e-6, 2.07e-6], [2e-9, 0.0], [4.0, 6.0], 1.0, 1e-7), 1),
              (1, rand_stack(rng, 1), 1)]
    wl = custom_workload(stacks, datasets, K=K)
    ref_ll, ref_g, ref_r = oracle.batch("grad_res", wl.n_layers, wl.params, wl.dataset, wl.q_off, wl.q, wl.dq,
                                        wl.r_obs, wl.r_err, K)
    ref = {"ll": ref_ll, "g": ref_g, "m": run_oracle(wl, modes=("model",))["m"]}
    # model and log-likelihood run the paired forward kernels (the 1-layer
    # bucket and the runtime-n bucket with n = 0 and 2)
    assert_parity(wl, run_gpu(wl), ref)
    # several items per stack and a tile shorter than the widest, with the
    # resolution derivative through the same kernel
    ctx = nr.Context(n_quad=K, chunk_q=9, tile_q=5)
    ll, g, gr = (t.cpu().numpy() for t in ctx.loglik_grad_res(nr.Batch.from_workload(wl)))
    assert ctx.device_status() == 0
    ctx.close()
    assert np.max(np.abs(ll - ref_ll) / np.abs(ref_ll)) <= TOL_LL
    assert res_err(wl, g, gr, ref_g, ref_r) <= TOL_G


# Gradients of more than two layers keep their factors in tensor memory, with
# a different number of teams per SM and columns per thread from bucket to
# bucket (edges at 4, 8, 12, 16, 20, 32, 64 layers).  Beside random stacks:
# adjoining equal media without roughness (r = 0), and roughnesses whose
# Nevot-Croce phase needs the reduced sin / cos instead of the polynomial.
# The bounds are the module's, which hold at every depth.
@pytest.mark.parametrize("K", [3, 17, 21, 32])
def test_rolled_gradient_kernel_bucket_edges(K):
    rng = np.random.default_rng(300 + K)
    q1, q2 = W.log_grid(53, 0.005, 0.25), W.log_grid(23, 0.008, 0.03)
    datasets = [(q1, 0.04 * q1), (q2, 0.05 * q2)]
    stacks = [(n, rand_stack(rng, n, d_range=(5, 60)) if n > 20 else rand_stack(rng, n), n % 2)
              for n in (3, 4, 5, 8, 9, 12, 13, 16, 17, 20, 21, 32, 33, 64)]
    rho = [0.0, 4e-6, 4e-6, 4e-6, 1e-6, 2.07e-6]
    stacks.append((4, W.pack([120.0, 80.0, 0.0, 200.0], rho, np.zeros(5), [4.0, 0.0, 0.0, 3.0, 0.0], 1.0, 1e-7), 0))
    for n in (3, 7, 14):
        st = rand_stack(rng, n, d_range=(200, 600))
        L = W.layout(n)
        st[L["sigma"]] = rng.uniform(40, 80, n + 1)
        stacks.append((n, st, n % 2))
    wl = custom_workload(stacks, datasets, K=K)
    ref_ll, ref_g, ref_r = oracle.batch("grad_res", wl.n_layers, wl.params, wl.dataset, wl.q_off, wl.q, wl.dq,
                                        wl.r_obs, wl.r_err, K)
    ref = {"ll": ref_ll, "g": ref_g, "m": run_oracle(wl, modes=("model",))["m"]}
    assert_parity(wl, run_gpu(wl), ref)
    # several items per stack, more teams than items, and the resolution derivative
    ctx = nr.Context(n_quad=K, chunk_q=9, tile_q=5)
    ll, g, gr = (t.cpu().numpy() for t in ctx.loglik_grad_res(nr.Batch.from_workload(wl)))
    assert ctx.device_status() == 0
    ctx.close()
    po = wl.par_off
    e_res = [res_err(wl.subset([i]), g[po[i]:po[i + 1]], gr[i:i + 1], ref_g[po[i]:po[i + 1]], ref_r[i:i + 1])
             for i in range(wl.n_stacks)]
    check_bounds(wl, {"loglik": np.abs(ll - ref_ll) / np.abs(ref_ll), "grad": np.array(e_res)},
                 {"loglik": TOL_LL, "grad": TOL_G})


# Sweeps over more than two layers (and the forward ones) take k_0^2 - c_j from
# a common quantum that grows with the Q points staged so far: several
# super-tiles in ascending and in shuffled order, Q up to 1.2 (the quantum far
# above the low-Q nodes' own rounding), fronting media denser than the layers
# (negative c_j), equal SLDs (c_j = 0) and a dense metal.  The bounds are the
# module's.
@pytest.mark.parametrize("order", ["up", "shuffled"])
def test_common_quantum(order):
    rng = np.random.default_rng(17)
    q = np.concatenate([W.log_grid(180, 0.004, 1.2), W.log_grid(120, 0.008, 0.03)])
    q = np.sort(q) if order == "up" else rng.permutation(q)
    datasets = [(q, 0.04 * q.astype(np.float64))]
    stacks = []
    for n in (0, 3, 4, 9, 20, 33):
        for front in (0.0, 6.35e-6):
            st = rand_stack(rng, n, front=front, d_range=(10, 80) if n > 10 else (20, 400))
            if n >= 3:
                st[W.layout(n)["rho"]][1:3] = (front, 1.2e-5)
            stacks.append((n, st, 0))
    wl = custom_workload(stacks, datasets)
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_gradient_on_a_waveguide_resonance():
    """One quadrature node near a guided mode carries most of a gradient
    component.  In a 64-bit evaluation of this stack a relative change of
    6e-8 (one FP32 rounding) of the wavevectors inside the Fresnel factors
    moves the scaled gradient by up to 1.1e-4, of r or the recursion's b by
    7e-5 and 4e-5, of the phases by 8e-5: together 1.6e-4; 2e-4 with the
    approximate special functions' share.  Wavevectors off by three roundings
    exceed it."""
    wl = W.make_workload("vi_step").subset([86])
    gpu, ref = run_gpu(wl, modes=("grad",)), run_oracle(wl, modes=("grad",))
    assert gpu["flags"] == 0 and grad_err(wl, gpu["g"], ref["g"]) < 2e-4


def test_fresnel_factor_keeps_shared_errors_correlated():
    """An error of k_j that enters the interfaces above and below it alike
    mostly cancels.  Bounds: the errors of 1500 thick films of a kernel whose
    (k_a + k_b)^2 is formed from the sum (gradient median 3.56e-7, 99 %
    quantile of its log-likelihood 4.28e-7), and their own spread over 1500
    draws, 8 % and 25 %.  From the known squares, 4.0e-7 and 6.3e-7."""
    wl = W.make_workload("thick_oxide", n_stacks=1500)
    err = stack_errors(wl, run_gpu(wl, modes=("grad",)), run_oracle(wl, modes=("grad",)))
    assert np.median(err["grad"]) <= 1.08 * 3.56e-7
    assert np.quantile(err["loglik_g"], 0.99) <= 1.25 * 4.28e-7


def test_gradient_errors_around_a_waveguide_resonance():
    """The error on one resonant stack is one draw; over 96 copies of it (and of a
    second one) with parameters varied by 1e-6 the gradient's errors are no
    larger than those of a kernel that differentiates the division and forms the
    factors twice: rms 2.07e-4 and 4.33e-5, with 15 % for the spread of an rms
    over 96 draws."""
    for name, i, rms in (("vi_step", 86, 2.07e-4), ("uneven", 429, 4.33e-5)):
        wl = W.make_workload(name).subset([i] * 96)
        wl.params = wl.params * (1 + 1e-6 * np.random.default_rng(i).normal(size=wl.params.size))
        err = stack_errors(wl, run_gpu(wl, modes=("grad",)), run_oracle(wl, modes=("grad",)))["grad"]
        assert np.sqrt(np.mean(err ** 2)) <= 1.15 * rms


# One unsmeared Q point per stack, k_j^2 of one layer at 1 to 4 % of k_0^2: the
# plain adjoint loses up to k_0^2 / |k_j|^2 = 100 roundings there.  The error is
# taken against the layers' own components (d/dscale, of order 1 in total
# reflection, hides them).  Nine stacks of ten meet the module's gradient bound;
# the others are ill-conditioned (total reflection, whose gradient is the small
# remainder of large terms).
@pytest.mark.parametrize("n", [1, 2, 4])
def test_unsmeared_points_near_an_interior_edge(n):
    wl = edge_points(n, 0.0102, 0.0398)
    assert np.quantile(layer_grad_err(wl, n), 0.9) <= TOL_G


# The same for deeper stacks, and for points below an edge (k_j^2 down to
# -k_0^2): near total reflection the adjoint of a recursion without divisions
# cancels from layer to layer unless it carries the one combination that does
# not.  Bounds: nine of ten stacks within the errors of a kernel that
# differentiates the division itself (`q90`), with 30 % for the spread of that
# quantile over 600 stacks.
@pytest.mark.parametrize("n,lo,hi,q90", [(10, 0.0102, 0.0398, 5.62e-5), (20, 0.0102, 0.0398, 8.15e-5),
                                         (2, -1.0, -0.05, 3.40e-5), (4, -1.0, -0.05, 3.83e-5),
                                         (10, -1.0, -0.05, 5.09e-5), (40, -1.0, -0.05, 6.66e-5)])
def test_unsmeared_points_in_total_reflection(n, lo, hi, q90):
    assert np.quantile(layer_grad_err(edge_points(n, lo, hi), n), 0.9) <= 1.3 * q90


# Between two evanescent media the Nevot-Croce factor exp(-2 sigma^2 k_a k_b)
# grows; products of it over the layers must not overflow as long as each
# reflection stays finite.  Roughnesses from where the recursion is first
# divided at every layer to where the products of 64 layers pass 1e90; thin and
# thick layers, an absorbing stack.  Every output is finite, and the median
# stack meets the module's bounds (guided modes behind such interfaces are
# ill-conditioned beyond what input perturbations show: factors of e^20 carry
# the roundings of their exponents).
@pytest.mark.parametrize("n", [2, 3, 10, 20, 32, 64])
def test_very_rough_evanescent_layers(n):
    rng = np.random.default_rng(70 + n)
    q = W.log_grid(40, 0.004, 0.02)
    datasets, stacks = [], []
    for sigma in (60.0, 120.0, 180.0, 220.0, 260.0, 320.0):
        for d, iota in ((100.0, 0.0), (300.0, 0.0), (40.0, 1e-8)):
            rho = np.where(np.arange(n) % 2, 6.3e-6, 3.5e-6) * rng.uniform(0.97, 1.03, n)
            p = W.pack(np.full(n, d), np.concatenate([[0.0], rho, [6.3e-6]]), np.full(n + 1, iota),
                       sigma * rng.uniform(0.95, 1.05, n + 1), 1.0, 1e-7)
            stacks.append((n, p, len(datasets)))
            datasets.append((q, 0.03 * q.astype(np.float64)))
    wl = custom_workload(stacks, datasets)
    gpu = run_gpu(wl)
    assert gpu["flags"] == 0 and all(np.all(np.isfinite(gpu[k])) for k in ("m", "ll", "ll_g", "g"))
    err = stack_errors(wl, gpu, run_oracle(wl))
    for kind, tol in (("model", TOL_M), ("loglik", TOL_LL), ("loglik_g", TOL_LL), ("grad", TOL_G)):
        assert np.median(err[kind]) <= tol
    ctx = nr.Context(n_quad=wl.n_quad)
    assert all(torch.isfinite(t).all() for t in ctx.loglik_grad_res(nr.Batch.from_workload(wl)))
    ctx.close()


@pytest.mark.parametrize("n", [1, 2, 4])
def test_absorption_steps_between_nearly_equal_media(n):
    """Equal SLDs and absorptions that differ by 1 part in 10^4, only in the last
    interface, behind a surface too rough to reflect: what is measured is that
    difference, which FP32 absorptions do not hold to better than 4e-4.  The
    parameters are FP64: the module's bounds, without its allowance for FP32
    roundings of the inputs."""
    rho, iota = np.zeros(n + 2), np.full(n + 1, 1e-6)
    iota[-1] *= 1.0001
    sigma = np.concatenate([[70.0], np.full(n - 1, 5.0), [3.0]])
    q = W.log_grid(60, 0.08, 0.12)
    wl = custom_workload([(n, W.pack(np.full(n, 40.0), rho, iota, sigma, 1.0, 0.0), 0)],
                         [(q, 0.02 * q.astype(np.float64))])
    err = stack_errors(wl, run_gpu(wl), run_oracle(wl))
    assert err["model"] <= TOL_M and max(err["loglik"], err["loglik_g"]) <= TOL_LL and err["grad"] <= TOL_G


def test_a_bad_q_point_leaves_the_others():
    """A non-positive or NaN Q point raises the flag and spoils its own model
    value only."""
    rng = np.random.default_rng(18)
    q = W.log_grid(90, 0.01, 0.2)
    wl = custom_workload([(n, rand_stack(rng, n), 0) for n in (1, 2, 6, 24)], [(q, 0.03 * q.astype(np.float64))])
    good = run_gpu(wl, modes=("model",))["m"].reshape(4, -1)
    wl.q = wl.q.copy()
    wl.q[[7, 40]] = (-0.01, np.nan)
    ctx = nr.Context(n_quad=wl.n_quad)
    m = ctx.reflectivity(nr.Batch.from_workload(wl)).cpu().numpy().astype(np.float64).reshape(4, -1)
    assert ctx.device_status() & nr.NR_FLAG_BAD_Q
    ctx.close()
    keep = np.setdiff1d(np.arange(q.size), [7, 40])
    assert np.all(np.isnan(m[:, [7, 40]])) and np.all(np.isfinite(m[:, keep]))
    # the quantum may differ by the spoiled points: within the model bound
    assert np.max(np.abs(np.log(m[:, keep]) - np.log(good[:, keep]))) <= TOL_M


@pytest.mark.parametrize("n", [1, 2, 3, 12, 24, 40])
def test_a_bad_q_point_in_a_gradient_spoils_its_own_stacks(n):
    """Two stacks on two curves, one with a non-positive and a NaN point: the flag
    is raised, that stack's gradient is NaN, the other's within the bounds."""
    rng = np.random.default_rng(20 + n)
    q = W.log_grid(90, 0.01, 0.2)
    wl = custom_workload([(n, rand_stack(rng, n, d_range=(20, 100)), i) for i in (0, 1)],
                         [(q, 0.03 * q.astype(np.float64))] * 2)
    good = wl.subset([1])
    ref_ll, ref_g, ref_r = oracle.batch("grad_res", good.n_layers, good.params, good.dataset, good.q_off, good.q,
                                        good.dq, good.r_obs, good.r_err, good.n_quad)
    wl.q = wl.q.copy()
    wl.q[[7, 40]] = (-0.01, np.nan)
    for res in (False, True):
        ctx = nr.Context(n_quad=wl.n_quad)
        b = nr.Batch.from_workload(wl)
        out = ctx.loglik_grad_res(b) if res else ctx.loglik_grad(b)
        ll, g = (t.cpu().numpy() for t in out[:2])
        assert ctx.device_status() & nr.NR_FLAG_BAD_Q
        ctx.close()
        g = g.reshape(2, -1)
        assert np.isnan(ll[0]) and np.isnan(g[0, 4 * n + 4]) and (n < 1 or np.isnan(g[0, 0]))
        assert abs(ll[1] - ref_ll[0]) <= TOL_LL * abs(ref_ll[0])
        assert grad_err(good, g[1], ref_g) <= TOL_G
        if res:
            assert res_err(good, g[1], out[2].cpu().numpy()[1:], ref_g, ref_r) <= TOL_G


def test_zero_resolution_is_unsmeared():
    wl = W.make_workload("thick_oxide", n_stacks=16)
    wl.dq = np.zeros_like(wl.dq)
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_quartz_posterior_stack_from_table1():
    vals = {}
    for line in open(os.path.join(ROOT, "tests", "golden", "quartz_table1.txt")):
        if line.strip() and not line.startswith("#"):
            k, v = line.split()
            vals[k] = float(v)
    p = W.pack([vals["thick_quartz"], vals["thick_oxide"]],
               [vals["sld_air"], vals["sld_quartz"], vals["sld_oxide"], vals["sld_si"]], [0.0, 0.0, 0.0],
               [vals["rough_air_quartz"], vals["rough_quartz_oxide"], vals["rough_oxide_si"]],
               vals["scale"], vals["bkg"])
    q = W.log_grid(300, 0.006, 0.2)
    wl = custom_workload([(2, p, 0)], [(q, 0.02 * q.astype(np.float64))], K=21)
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


def test_chunked_matches_unchunked():
    wl = W.make_workload("oled_cofit", n_stacks=4)
    a = run_gpu(wl)
    b = run_gpu(wl, chunk_q=24, tile_q=5)
    np.testing.assert_array_equal(a["m"], b["m"])
    np.testing.assert_allclose(b["ll_g"], a["ll_g"], rtol=1e-12)
    assert grad_err(wl, b["g"], a["g"]) <= 1e-6
    assert_parity(wl, b, run_oracle(wl))


def test_chunk_choice_follows_the_makespan_estimate():
    """Whole stacks where one wave of them nearly fills the GPU (the
    one-layer film: 1024 stacks, 760 resident CTAs; a chunk's fixed cost
    outweighs the shorter tail), Q-range chunks where a few deep stacks
    would leave most CTAs idle; every Q point is covered exactly once
    either way, so the chunked plan keeps parity."""
    film = W.make_workload("film_1l")
    ctx = nr.Context(n_quad=film.n_quad)
    bf = nr.Batch.from_workload(film)
    groups = ctx.plan_groups(bf, grad=True)
    assert sum(g["items"] for g in groups) == film.n_stacks
    wl = W.make_workload("vi_step", n_stacks=4)             # 12 stacks of 12 layers x 300 Q
    ctx2 = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    groups = ctx2.plan_groups(b, grad=True)
    assert sum(g["items"] for g in groups) > 4 * wl.n_stacks
    ctx.close()
    ctx2.close()
    assert_parity(wl, run_gpu(wl), run_oracle(wl))


@pytest.mark.parametrize("n,S,whole", [(1, 300, True), (1, 1, False), (10, 100, False), (10, 608, True)])
def test_chunk_choice_of_small_batches(n, S, whole):
    """A few hundred short stacks stay whole (one or two per SM are fast
    enough), a single one or long stacks that leave SMs idle are cut, long
    ones that fill the SMs are not; the first stacks keep parity."""
    rng = np.random.default_rng(n * 1000 + S)
    q = W.log_grid(225 if n > 1 else 200, 0.005, 0.3)
    wl = custom_workload([(n, rand_stack(rng, n), 0) for _ in range(S)], [(q, 0.05 * q.astype(np.float64))])
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    items = sum(g["items"] for g in ctx.plan_groups(b, grad=True))
    assert (items == S) == whole
    ll, g = (t.cpu().numpy() for t in ctx.loglik_grad(b))
    assert ctx.device_status() == 0
    ctx.close()
    k = min(S, 4)
    sub = wl.subset(np.arange(k))
    ref = run_oracle(sub, modes=("grad",))
    errs = stack_errors(sub, {"ll_g": ll[:k], "g": g[:sub.params.size]}, ref)
    check_bounds(sub, errs, {"loglik_g": TOL_LL, "grad": TOL_G})


def test_requested_consumers_are_the_ones_that_run():
    """grid_ctas counts the teams of the multi-layer gradients: one per SM leaves
    three quarters of an SM's warps out (measured: a little over half its rate).
    Results do not depend on it."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(12)
    q = W.log_grid(100, 0.005, 0.25)
    wl = custom_workload([(10, rand_stack(rng, 10), 0) for _ in range(8 * sms)], [(q, 0.04 * q.astype(np.float64))])
    ms, res = {}, []
    for teams in (sms, 4 * sms):
        ctx, b = nr.Context(n_quad=wl.n_quad, grid_ctas=teams), nr.Batch.from_workload(wl)
        assert ctx.plan_info(b)["grid_ctas"] >= 1
        assert [g["grid"] for g in ctx.plan_groups(b, grad=True)] == [teams]
        t = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            torch.cuda.synchronize()
            e0.record()
            out = ctx.loglik_grad(b)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        ms[teams] = min(t)
        res.append(out)
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*res))
    assert ms[sms] >= 1.35 * ms[4 * sms]


def test_host_memory_calls_match_device_calls():
    wl = W.make_workload("uneven", n_stacks=20)
    ctx = nr.Context(n_quad=wl.n_quad)
    bd = nr.Batch.from_workload(wl)
    bh = nr.Batch.from_workload(wl, device="cpu", pin=True)
    lld, gd = ctx.loglik_grad(bd)
    llh, gh = ctx.loglik_grad(bh)
    assert not llh.is_cuda
    assert torch.equal(lld.cpu(), llh) and torch.equal(gd.cpu(), gh)
    assert torch.equal(ctx.reflectivity(bd).cpu(), ctx.reflectivity(bh))
    assert torch.equal(ctx.loglik(bd).cpu(), ctx.loglik(bh))


def test_autograd_backward_of_mixed_layer_counts():
    """Stacks of different layer counts take the general form of backward,
    stacks of one count the broadcast; both weight every stack's gradient by
    its own factor, expanded (stride 0) or not."""
    for S in ("uneven", "oled_cofit"):
        wl = W.make_workload(S, n_stacks=5)
        ctx = nr.Context(n_quad=wl.n_quad)
        b = nr.Batch.from_workload(wl)
        _, g = ctx.loglik_grad(b)
        per = torch.as_tensor(4 * wl.n_layers.astype(np.int64) + 6, device=g.device)
        for w in (torch.linspace(0.5, 2.0, wl.n_stacks, dtype=torch.float64, device=g.device),
                  torch.full((1,), 0.3, dtype=torch.float64, device=g.device).expand(wl.n_stacks)):
            params = b.params.clone().requires_grad_(True)
            (got,) = torch.autograd.grad(nr.loglik_autograd(params, ctx, b), params, grad_outputs=w)
            torch.testing.assert_close(got, g * torch.repeat_interleave(w, per), rtol=0, atol=0)
        ctx.close()


def test_autograd_function_backward_is_the_exact_gradient():
    wl = W.make_workload("film_1l", n_stacks=12)
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    params = b.params.clone().requires_grad_(True)
    ll = nr.loglik_autograd(params, ctx, b)
    w = torch.linspace(0.5, 2.0, wl.n_stacks, dtype=torch.float64, device=ll.device)
    (ll * w).sum().backward()
    _, g = ctx.loglik_grad(b)
    per = torch.as_tensor(4 * wl.n_layers.astype(np.int64) + 6, device=g.device)
    torch.testing.assert_close(params.grad, g * torch.repeat_interleave(w, per), rtol=0, atol=0)


def test_device_data_errors_raise_flags_not_faults():
    wl = W.make_workload("film_1l", n_stacks=3)
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    bad_err = b.r_err.clone()
    bad_err[5] = 0.0
    ll = ctx.loglik(nr.Batch(b.n_layers, b.dataset, b.q_off, b.params, b.q, b.dq, b.r_obs, bad_err))
    assert ctx.device_status() & nr.NR_FLAG_BAD_ERR
    assert not torch.isfinite(ll).all()
    bad_p = b.params.clone()
    bad_p[3] = float("nan")
    ctx.loglik_grad(b.with_params(bad_p))
    assert ctx.device_status() & nr.NR_FLAG_NONFINITE_PARAM
    bad_q = b.dq.clone()
    bad_q[0] = 10.0    # nodes at q <= 0
    m = ctx.reflectivity(nr.Batch(b.n_layers, b.dataset, b.q_off, b.params, b.q, bad_q))
    assert ctx.device_status() & nr.NR_FLAG_BAD_Q
    assert not torch.isfinite(m[0])
    # the context stays usable and clean afterwards
    ll2, _ = ctx.loglik_grad(b)
    assert ctx.device_status() == 0 and torch.isfinite(ll2).all()


def test_metadata_validation():
    wl = W.make_workload("film_1l", n_stacks=2)
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    for bad in (dict(n_layers=np.array([1, 65], np.int32)), dict(dataset=np.array([0, 1], np.int32)),
                dict(q_off=np.array([0, -1], np.int64))):
        fields = dict(n_layers=b.n_layers, dataset=b.dataset, q_off=b.q_off)
        fields.update(bad)
        bb = nr.Batch(fields["n_layers"], fields["dataset"], fields["q_off"], b.params, b.q, b.dq, b.r_obs, b.r_err)
        with pytest.raises(nr.NRError) as ei:
            ctx.loglik(bb)
        assert ei.value.status == nr.NR_EINVAL
    with pytest.raises(nr.NRError):
        ctx.loglik(nr.Batch(b.n_layers, b.dataset, b.q_off, b.params, b.q, b.dq))  # no data
    # an empty batch is fine
    e = nr.Batch(np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(1, np.int64), b.params[:0], b.q[:0], b.dq[:0],
                 b.r_obs[:0], b.r_err[:0])
    ll, g = ctx.loglik_grad(e)
    assert ll.numel() == 0 and g.numel() == 0


def test_plan_before_capture_and_graph_replay():
    wl = W.make_workload("thick_oxide", n_stacks=64)
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    ctx.plan(b)
    ll = torch.empty(wl.n_stacks, dtype=torch.float64, device="cuda")
    g = torch.empty(b.params.numel(), dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx.loglik_grad(b, ll_out=ll, grad_out=g, stream=s)
    torch.cuda.synchronize()
    ref_ll, ref_g = ll.clone(), g.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        ctx.loglik_grad(b, ll_out=ll, grad_out=g, stream=s)
    ll.zero_()
    g.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(ll, ref_ll) and torch.equal(g, ref_g)


# ---------------------------------------------- resolution-scale derivative
def res_err(wl, g, gr, g_ref, gr_ref):
    """The resolution derivative as one more gradient component (typical
    scale 1, like the model scale): max over stacks of the scaled error over
    the stack's largest scaled component."""
    po = wl.par_off
    worst = 0.0
    for s in range(wl.n_stacks):
        typ = W.typical_scale(int(wl.n_layers[s]))
        ref = np.append(g_ref[po[s]:po[s + 1]] * typ, gr_ref[s])
        got = np.append(g[po[s]:po[s + 1]] * typ, gr[s])
        worst = max(worst, float(np.max(np.abs(got - ref)) / np.max(np.abs(ref))))
    return worst


@pytest.mark.parametrize("name,S,kw", [("thick_oxide", 48, {}), ("film_1l", 40, {}), ("oled_cofit", 4, {}),
                                       ("uneven", 24, {}), ("vi_step", 2, {}),
                                       ("oled_cofit", 3, {"chunk_q": 40, "tile_q": 3})])
def test_resolution_derivative_parity(name, S, kw):
    wl = W.make_workload(name, n_stacks=S)
    ctx = nr.Context(n_quad=wl.n_quad, **kw)
    b = nr.Batch.from_workload(wl)
    ll, g, gr = (t.cpu().numpy() for t in ctx.loglik_grad_res(b))
    ll0, g0 = (t.cpu().numpy() for t in ctx.loglik_grad(b))
    assert ctx.device_status() == 0
    ctx.close()
    ref_ll, ref_g, ref_r = oracle.batch("grad_res", wl.n_layers, wl.params, wl.dataset, wl.q_off, wl.q, wl.dq,
                                        wl.r_obs, wl.r_err, wl.n_quad)
    assert np.all(np.isfinite(gr))
    assert np.max(np.abs(ll - ref_ll) / np.abs(ref_ll)) <= TOL_LL
    assert res_err(wl, g, gr, ref_g, ref_r) <= TOL_G
    # the log-likelihood and parameter gradient are those of nr_loglik_grad
    assert np.max(np.abs(ll - ll0) / np.abs(ll0)) <= 1e-6
    assert grad_err(wl, g, g0) <= 1e-5


def test_resolution_derivative_host_batch_and_fp64_refusal():
    wl = W.make_workload("thick_oxide", n_stacks=6)
    ctx = nr.Context(n_quad=wl.n_quad)
    lld, gd, rd = ctx.loglik_grad_res(nr.Batch.from_workload(wl))
    llh, gh, rh = ctx.loglik_grad_res(nr.Batch.from_workload(wl, device="cpu", pin=True))
    assert not rh.is_cuda
    assert torch.equal(rd.cpu(), rh) and torch.equal(gd.cpu(), gh)
    ctx.close()
    ctx64 = nr.Context(n_quad=wl.n_quad, precision="fp64")
    with pytest.raises(nr.NRError):
        ctx64.loglik_grad_res(nr.Batch.from_workload(wl))
    ctx64.close()


# ------------------------------------------------------------- SLD profiles
def profile_ref(wl, z):
    po = wl.par_off
    rho = np.zeros((wl.n_stacks, z.size))
    iota = np.zeros((wl.n_stacks, z.size))
    for s in range(wl.n_stacks):
        rho[s], iota[s] = oracle.sld_profile(int(wl.n_layers[s]), wl.params[po[s]:po[s + 1]], z.astype(np.float64))
    return rho, iota


@pytest.mark.parametrize("name,S", [("thick_oxide", 16), ("oled_cofit", 9), ("uneven", 40), ("vi_step", 6)])
def test_sld_profile_parity(name, S):
    wl = W.make_workload(name, n_stacks=S)
    depth = max(float(np.sum(wl.stack_params(s)[:int(wl.n_layers[s])])) for s in range(S))
    z = np.linspace(-60.0, depth + 60.0, 1037).astype(np.float32)   # ragged against the 256-thread sweep
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    rho, iota = ctx.sld_profile(b, torch.as_tensor(z, device="cuda"))
    assert ctx.device_status() == 0
    rho, iota = rho.cpu().numpy(), iota.cpu().numpy()
    ref_r, ref_i = profile_ref(wl, z)
    for s in range(S):
        scale_r = np.max(np.abs(ref_r[s]))
        scale_i = max(np.max(np.abs(ref_i[s])), 1e-12)
        assert np.max(np.abs(rho[s] - ref_r[s])) <= 2e-6 * scale_r
        assert np.max(np.abs(iota[s] - ref_i[s])) <= 2e-6 * scale_i
    ctx.close()


# Runs of 64 depths skip the error functions that are saturated over the whole
# run: depths in any order (sorted, reversed, shuffled), fewer than one run
# and one more than a whole number of them, more interfaces than a warp has
# lanes, neighbouring roughnesses of very different width (a narrow interface
# is passed while a wide one above it still counts), sharp steps and
# zero-thickness layers.  Bound as for the workloads: FP32 rounding of the sum.
@pytest.mark.parametrize("nz,order", [(1, "up"), (63, "down"), (65, "shuffled"), (640, "up"), (641, "shuffled")])
def test_sld_profile_runs(nz, order):
    rng = np.random.default_rng(nz)
    stacks = []
    for n in (0, 1, 5, 31, 32, 40, 64, 5, 12):
        st = rand_stack(rng, n)
        L = W.layout(n)
        st[L["sigma"]] = rng.choice([0.0, 0.5, 3.0, 25.0, 80.0], n + 1)
        if n >= 5:
            st[L["d"]][2] = 0.0
        stacks.append((n, st, 0))
    q = W.log_grid(10, 0.01, 0.2)
    wl = custom_workload(stacks, [(q, 0.05 * q.astype(np.float64))])
    z = np.sort(rng.uniform(-300.0, 14000.0 if nz > 100 else 900.0, nz)).astype(np.float32)
    z = z[::-1].copy() if order == "down" else rng.permutation(z) if order == "shuffled" else z
    ctx = nr.Context(n_quad=wl.n_quad)
    for sub in (wl, wl.subset([2, 7])):  # different layer counts, and one count
        rho, iota = ctx.sld_profile(nr.Batch.from_workload(sub), torch.as_tensor(z, device="cuda"))
        assert ctx.device_status() == 0
        ref_r, ref_i = profile_ref(sub, z)
        for s in range(sub.n_stacks):
            assert np.max(np.abs(rho[s].cpu().numpy() - ref_r[s])) <= 2e-6 * max(np.max(np.abs(ref_r[s])), 1e-6)
            assert np.max(np.abs(iota[s].cpu().numpy() - ref_i[s])) <= 2e-6 * max(np.max(np.abs(ref_i[s])), 1e-8)
    ctx.close()


@pytest.mark.parametrize("sigma,flagged", [(-1e-60, True), (-5e-324, True), (-3.0, True), (-0.0, False), (1e-60, False)])
def test_sld_profile_flags_any_negative_roughness(sigma, flagged):
    wl = custom_workload([(1, W.pack([50.0], [0.0, 4e-6, 2e-6], [0.0, 0.0], [sigma, 3.0], 1.0, 0.0), 0)],
                         [(W.log_grid(10, 0.01, 0.2), np.zeros(10))])
    ctx = nr.Context(n_quad=wl.n_quad)
    ctx.sld_profile(nr.Batch.from_workload(wl), torch.linspace(-10, 90, 41, device="cuda"))
    assert bool(ctx.device_status() & nr.NR_FLAG_NONFINITE_PARAM) == flagged
    ctx.close()


@pytest.mark.parametrize("S,n,nz", [(1, 3, 100000), (1, 0, 1), (3, 33, 70), (8, 10, 65536), (9, 2, 4097),
                                    (60, 5, 1000), (2000, 1, 129)])
def test_sld_profile_shares_out_the_runs_of_few_stacks(S, n, nz):
    """Few stacks are spread over the device by runs of depths; every output is
    written, whatever the remainders.  Bound as for the workloads."""
    rng = np.random.default_rng(S)
    q = W.log_grid(10, 0.01, 0.2)
    wl = custom_workload([(n, rand_stack(rng, n), 0) for _ in range(S)], [(q, 0.05 * q.astype(np.float64))])
    z = np.linspace(-50.0, 200.0 * n + 60.0, nz).astype(np.float32)
    ctx = nr.Context(n_quad=wl.n_quad)
    out = [torch.full((S * nz,), float("nan"), device="cuda") for _ in range(2)]
    rho, iota = ctx.sld_profile(nr.Batch.from_workload(wl), torch.as_tensor(z, device="cuda"), *out)
    ctx.close()
    at = rng.permutation(nz)[:2000]
    assert torch.isfinite(rho).all() and torch.isfinite(iota).all()
    for s in range(0, S, max(1, S // 20)):
        ref_r, ref_i = (v[0] for v in profile_ref(wl.subset([s]), z[at]))
        got_r, got_i = (v.reshape(S, nz)[s].cpu().numpy()[at] for v in (rho, iota))
        assert np.max(np.abs(got_r - ref_r)) <= 2e-6 * max(np.max(np.abs(ref_r)), 1e-6)
        assert np.max(np.abs(got_i - ref_i)) <= 2e-6 * max(np.max(np.abs(ref_i)), 1e-8)


def test_sld_profile_of_few_stacks_fills_the_device():
    """8 stacks x 65536 depths take no longer than three times 512 stacks x 1024
    depths (as many outputs, every SM busy)."""
    rng = np.random.default_rng(4)
    q = W.log_grid(10, 0.01, 0.2)
    ms = []
    for S, nz in ((8, 65536), (512, 1024)):
        wl = custom_workload([(5, rand_stack(rng, 5), 0) for _ in range(S)], [(q, 0.05 * q.astype(np.float64))])
        ctx, b = nr.Context(n_quad=wl.n_quad), nr.Batch.from_workload(wl)
        z = torch.linspace(-50.0, 1100.0, nz, device="cuda")
        out = [torch.empty(S * nz, device="cuda") for _ in range(2)]
        t = []
        for _ in range(12):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            torch.cuda.synchronize()
            e0.record()
            ctx.sld_profile(b, z, *out)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        ms.append(min(t))
        ctx.close()
    assert ms[0] <= 3.0 * ms[1]


def test_sld_profile_sharp_steps_on_grid_depths():
    """Sharp steps whose depths, added up in FP64 from thicknesses in tenths, lie
    on float grid points take the deeper medium's value there, in stacks of more
    interfaces than a warp has lanes too."""
    rng = np.random.default_rng(3)
    stacks, zs = [], set()
    for n in np.repeat([2, 5, 8, 40], 60):
        st = rand_stack(rng, int(n))
        L = W.layout(int(n))
        st[L["d"]] = np.round(rng.uniform(5, 300, n), 1)
        st[L["sigma"]] = 0.0
        stacks.append((int(n), st, 0))
        depth = 0.0
        for d in st[L["d"]]:
            depth += d
            if float(np.float32(depth)) == depth:
                zs.add(depth)
    z = np.array(sorted(zs), np.float32)
    q = W.log_grid(10, 0.01, 0.2)
    wl = custom_workload(stacks, [(q, 0.05 * q.astype(np.float64))])
    ctx = nr.Context(n_quad=wl.n_quad)
    rho = ctx.sld_profile(nr.Batch.from_workload(wl), torch.as_tensor(z, device="cuda"))[0]
    ctx.close()
    for (n, st, _), got in zip(stacks, rho):
        depth = np.cumsum(st[W.layout(n)["d"]])  # sequential, as the library adds
        want = st[W.layout(n)["rho"]][np.searchsorted(np.concatenate([[0.0], depth]), z.astype(np.float64), "right")]
        got = got.cpu().numpy()
        assert np.max(np.abs(got - want)) <= 2e-6 * np.max(np.abs(want))


def test_sld_profile_sharp_steps_host_batch_and_flags():
    d = [120.0, 35.0]
    rho = [0.0, 4.1e-6, -0.4e-6, 2.07e-6]
    stacks = [(2, W.pack(d, rho, [1e-8, 0.0, 0.0], [0.0, 0.0, 0.0], 1.0, 0.0), 0),
              (0, W.pack([], [0.0, 2.07e-6], [0.0], [3.0], 1.0, 0.0), 0)]
    q = W.log_grid(10, 0.01, 0.2)
    wl = custom_workload(stacks, [(q, 0.05 * q.astype(np.float64))])
    z = np.array([-10.0, 0.0, 119.0, 120.0, 154.0, 155.0, 400.0], np.float32)
    ctx = nr.Context(n_quad=wl.n_quad)
    rho_d, iota_d = ctx.sld_profile(nr.Batch.from_workload(wl), torch.as_tensor(z, device="cuda"))
    rho_h, iota_h = ctx.sld_profile(nr.Batch.from_workload(wl, device="cpu", pin=True), torch.as_tensor(z))
    assert torch.equal(rho_d.cpu(), rho_h) and torch.equal(iota_d.cpu(), iota_h)
    # sharp steps: the deeper medium's value from the interface depth on
    np.testing.assert_allclose(rho_h[0].numpy(), [0.0, 4.1e-6, 4.1e-6, -0.4e-6, -0.4e-6, 2.07e-6, 2.07e-6],
                               rtol=0, atol=2e-12)
    assert abs(float(rho_h[1, 1]) - 2.07e-6 / 2) < 1e-12
    assert ctx.device_status() == 0
    bad = wl.params.copy()
    bad[0] = np.nan
    wl_bad = custom_workload([(2, bad[:14], 0)], [(q, 0.05 * q.astype(np.float64))], data_from_oracle=False)
    ctx.sld_profile(nr.Batch.from_workload(wl_bad), torch.as_tensor(z, device="cuda"))
    assert ctx.device_status() & nr.NR_FLAG_NONFINITE_PARAM
    ctx.close()


# ------------------------------------------------------- on-device HMC step
def sampler_setup(C=8, seed=7, res=False):
    """A two-contrast co-fit sampler and its CPU reference; res: one more
    free parameter, the resolution scale f of every dQ (prior [0.6, 1.4])."""
    import sys
    sys.path.insert(0, os.path.dirname(__file__))
    from test_oracle_hmc import small_model, with_resolution
    from oracle import hmc
    model, u_t = small_model(seed)
    if res:
        model = with_resolution(model)
        u_t = np.append(u_t, 0.4)
    # the device holds the data as float32: the reference uses the same values
    f32 = lambda a: np.asarray(a, np.float32)
    ref = hmc.Model(model.n_layers, model.dataset, model.slot_src, model.slot_val, model.lo, model.hi,
                    model.q_off, f32(model.Q), f32(model.dQ), f32(model.Robs), f32(model.err), model.K,
                    res_param=model.res_param)
    ctx = nr.Context(n_quad=model.K)
    dev = lambda a: torch.as_tensor(f32(a), device="cuda")
    smp = nr.Sampler(ctx, C, model.n_layers, model.dataset, model.q_off, dev(model.Q), dev(model.dQ),
                     dev(model.Robs), dev(model.err), model.slot_src, model.slot_val, model.lo, model.hi,
                     res_param=model.res_param)
    rng = np.random.default_rng(seed + 1)
    u = u_t[None, :] + 0.2 * rng.normal(size=(C, model.P))
    return ctx, smp, ref, u, rng


@pytest.mark.parametrize("res", [False, True])
def test_sampler_logp_grad_parity(res):
    ctx, smp, ref, u, _ = sampler_setup(res=res)
    lp, g = smp.logp_grad(torch.as_tensor(u, device="cuda"))
    lp, g = lp.cpu().numpy(), g.cpu().numpy()
    for c in range(u.shape[0]):
        lr, gr = ref.logp_grad(u[c])
        assert abs(lp[c] - lr) <= 1e-5 * abs(lr)
        assert np.max(np.abs(g[c] - gr)) <= 1e-4 * np.max(np.abs(gr))
    smp.close()
    ctx.close()


@pytest.mark.parametrize("res", [False, True])
def test_hmc_step_parity_and_graph_replay(res):
    C, P_eps, L = 8, 4e-4, 6
    ctx, smp, ref, u, rng = sampler_setup(C, res=res)
    z = rng.normal(size=(C, ref.P))
    inv_mass = np.full(ref.P, 1.0)
    # first half of the chains must accept, the rest reject: decisions that
    # do not hinge on rounding; both branches of every kernel path run
    log_u = np.where(np.arange(C) < C // 2, -np.inf, np.inf)
    ud = torch.as_tensor(u, device="cuda")
    lp, acc = smp.hmc_step(ud, torch.as_tensor(z, device="cuda"), torch.as_tensor(log_u, device="cuda"),
                           torch.as_tensor(inv_mass, device="cuda"), P_eps, L)
    assert ctx.device_status() == 0
    ug, lp, acc = ud.cpu().numpy(), lp.cpu().numpy(), acc.cpu().numpy()
    from oracle import hmc
    for c in range(C):
        ur, lr, ar, H0, H1 = hmc.hmc_step(ref.logp_grad, u[c], z[c], log_u[c], inv_mass, P_eps, L)
        assert bool(acc[c]) == ar
        assert abs(lp[c] - lr) <= 1e-5 * abs(lr)
        # L leapfrog steps amplify the gradient's relative error by ~eps^2 L^2 |d2 log pi|
        assert np.max(np.abs(ug[c] - ur)) <= 1e-6 + 1e-6 * np.max(np.abs(ur))
    # the same step as a captured CUDA graph reproduces the eager result
    u2 = torch.as_tensor(u, device="cuda")
    zt, lt, mt = (torch.as_tensor(a, device="cuda") for a in (z, log_u, inv_mass))
    lp2 = torch.empty(C, dtype=torch.float64, device="cuda")
    acc2 = torch.empty(C, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        smp.hmc_step(u2, zt, lt, mt, P_eps, L, lp2, acc2, stream=s)    # warm-up (plans stay cached)
    torch.cuda.synchronize()
    u2.copy_(torch.as_tensor(u, device="cuda"))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        smp.hmc_step(u2, zt, lt, mt, P_eps, L, lp2, acc2, stream=s)
    u2.copy_(torch.as_tensor(u, device="cuda"))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(u2.cpu(), torch.as_tensor(ug)) and torch.equal(acc2.cpu(), torch.as_tensor(acc))
    smp.close()
    ctx.close()


def test_sampler_rejects_bad_models():
    ctx = nr.Context(n_quad=17)
    q = torch.ones(4, device="cuda")
    with pytest.raises(nr.NRError):      # slot source out of range
        nr.Sampler(ctx, 2, [0], [0], [0, 4], q, q, q, q, [5, -1, -1, -1, -1, -1], [0.0] * 6, [0.0], [1.0])
    with pytest.raises(nr.NRError):      # empty prior box
        nr.Sampler(ctx, 2, [0], [0], [0, 4], q, q, q, q, [0, -1, -1, -1, -1, -1], [0.0] * 6, [1.0], [1.0])
    ctx.close()


# ---------------------------------------------- variational-inference step
def test_vi_step_parity_and_graph_replay():
    from oracle import vi
    R = 6
    ctx, smp, ref, u_c, rng = sampler_setup(R, seed=11)
    P = ref.P
    nphi = nr.vi_phi_size(P)
    phi = np.zeros((R, nphi))
    phi[:, :P] = u_c                                   # mu: the chains' starting points
    for r in range(R):                                 # L = 0.1 I plus a little correlation
        idx = P
        for i in range(P):
            for j in range(i + 1):
                phi[r, idx] = np.log(0.1) if i == j else 0.02 * rng.normal()
                idx += 1
    m0 = 0.01 * np.abs(rng.normal(size=(R, nphi)))
    v0 = 0.001 * np.abs(rng.normal(size=(R, nphi)))
    eps = rng.normal(size=(R, P))
    t0 = 4                                             # iterations already done
    dev = lambda a: torch.as_tensor(a, device="cuda")
    ph, m, v, t = dev(phi), dev(m0), dev(v0), dev(np.array([t0], np.int32))
    elbo = smp.vi_step(ph, m, v, t, dev(eps), lr=0.05)
    assert ctx.device_status() == 0 and int(t.item()) == t0 + 1
    ph, m, v, elbo = ph.cpu().numpy(), m.cpu().numpy(), v.cpu().numpy(), elbo.cpu().numpy()
    for r in range(R):
        mu_r, tri_r, m_r, v_r, el_r = vi.vi_step(ref.logp_grad, phi[r, :P], phi[r, P:], m0[r], v0[r], t0 + 1,
                                                 eps[r], 0.05)
        assert abs(elbo[r] - el_r) <= 1e-5 * abs(el_r)
        # the gradient carries the mixed path's ~1e-5 relative error; Adam's
        # step is lr * mhat / sqrt(vhat): its error stays a small fraction of lr
        np.testing.assert_allclose(ph[r], np.concatenate([mu_r, tri_r]), rtol=0, atol=2e-3 * 0.05)
        # Adam's first moment carries the gradient's error: held to the
        # gradient bound, 1e-4 of the largest gradient term (1 - beta1) g
        assert np.max(np.abs(m[r] - m_r)) <= 1e-4 * np.max(np.abs(m_r - 0.9 * m0[r]))
    # a captured iteration replays with the device counter advancing
    ph2, m2, v2, t2, e2 = dev(phi), dev(m0), dev(v0), dev(np.array([t0], np.int32)), dev(eps)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        smp.vi_step(ph2, m2, v2, t2, e2, stream=s)
    torch.cuda.synchronize()
    ph2.copy_(dev(phi)); m2.copy_(dev(m0)); v2.copy_(dev(v0)); t2.fill_(t0)
    graph = torch.cuda.CUDAGraph()
    el2 = torch.empty(R, dtype=torch.float64, device="cuda")
    with torch.cuda.graph(graph, stream=s):
        smp.vi_step(ph2, m2, v2, t2, e2, elbo_out=el2, stream=s)
    ph2.copy_(dev(phi)); m2.copy_(dev(m0)); v2.copy_(dev(v0)); t2.fill_(t0)
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert int(t2.item()) == t0 + 2
    smp.close()
    ctx.close()


# A restart is one block: the number of free parameters against its threads
# (rows of L in passes of 32, eight lanes a row), the sampled resolution
# scale, and more parameters than the block stages in shared memory (2048).
# Bounds as in the test above.
@pytest.mark.parametrize("case", ["res", "many"])
def test_vi_step_blocks(case):
    from oracle import hmc
    R = 3
    if case == "res":
        ctx, smp, ref, u_c, rng = sampler_setup(R, seed=5, res=True)
    else:
        rng = np.random.default_rng(8)
        n, NC = 12, 40
        q = W.log_grid(10, 0.01, 0.2)
        val = np.concatenate([rand_stack(rng, n, d_range=(20, 60)) for _ in range(NC)])
        L = W.layout(n)
        half = np.empty(4 * n + 6)
        for k, w in (("d", 5.0), ("rho", 2e-7), ("iota", 0.0), ("sigma", 0.0), ("scale", 0.05), ("bkg", 1e-8)):
            half[L[k]] = w
        v = val.reshape(NC, -1)
        half = np.where(half > 0, half, 0.2 * np.abs(v))         # iota, sigma stay positive
        lo, hi = (v - half).ravel(), (v + half + np.where(half > 0, 0.0, 1e-9)).ravel()
        m = oracle.model(n, v[0], q, (0.05 * q).astype(np.float32), 5)
        f32 = lambda a: np.asarray(a, np.float32)
        ref = hmc.Model([n] * NC, [0] * NC, np.arange(val.size), val, lo, hi, [0, q.size], q, f32(0.05 * q),
                        f32(1.03 * m), f32(0.05 * m), 5)
        ctx = nr.Context(n_quad=5)
        dev32 = lambda a: torch.as_tensor(f32(a), device="cuda")
        smp = nr.Sampler(ctx, R, ref.n_layers, ref.dataset, ref.q_off, dev32(ref.Q), dev32(ref.dQ), dev32(ref.Robs),
                         dev32(ref.err), ref.slot_src, val, lo, hi)
        u_c = 0.2 * rng.normal(size=(R, ref.P))
    P = ref.P
    assert case == "res" or P > 2048
    i, j = np.tril_indices(P)
    tri = np.where(i == j, np.log(0.1), 0.02 / np.sqrt(P) * rng.normal(size=(R, i.size)))
    phi = np.concatenate([u_c, tri], axis=1)
    eps = rng.normal(size=(R, P))
    dev = lambda a: torch.as_tensor(a, device="cuda")
    ph, m, v, t = dev(phi), dev(0.0 * phi), dev(0.0 * phi), dev(np.array([0], np.int32))
    elbo = smp.vi_step(ph, m, v, t, dev(eps), lr=0.05).cpu().numpy()
    assert ctx.device_status() == 0
    m = m.cpu().numpy()
    for r in range(R):
        u = u_c[r] + np.bincount(i, np.where(i == j, np.exp(tri[r]), tri[r]) * eps[r][j], P)
        lp, g = ref.logp_grad(u)
        el = lp + 0.5 * eps[r] @ eps[r] + tri[r][i == j].sum() + 0.5 * P * np.log(2 * np.pi)
        assert abs(elbo[r] - el) <= 1e-5 * abs(el)
        grad = np.concatenate([-g, np.where(i == j, -g[i] * eps[r][i] * np.exp(tri[r]) - 1.0, -g[i] * eps[r][j])])
        assert np.max(np.abs(m[r] - 0.1 * grad)) <= 1e-4 * np.max(np.abs(0.1 * grad))
    smp.close()
    ctx.close()


@pytest.mark.parametrize("name,S", [("uneven", 40), ("thick_oxide", 64), ("oled_cofit", 6), ("film_1l", 48)])
def test_autotuned_plan_keeps_parity(name, S):
    """nr_plan with autotune = 1 times the candidate launch shapes (paired or
    one-evaluation kernel, widest tile or half) per register bucket and keeps
    the fastest; whatever it picks matches the oracle."""
    wl = W.make_workload(name, n_stacks=S)
    ctx = nr.Context(n_quad=wl.n_quad, autotune=True)
    b = nr.Batch.from_workload(wl)
    ctx.plan(b)
    info = ctx.plan_info(b)
    assert info["tile_q"] >= 1 and info["grid_ctas"] >= 1 and info["launches"] >= 1
    gpu = {"m": ctx.reflectivity(b).cpu().numpy().astype(np.float64), "ll": ctx.loglik(b).cpu().numpy()}
    ll, g = ctx.loglik_grad(b)
    gpu["ll_g"], gpu["g"] = ll.cpu().numpy(), g.cpu().numpy()
    gpu["flags"] = ctx.device_status()
    ctx.close()
    assert_parity(wl, gpu, run_oracle(wl))


# ------------------------------------------------- failure injection ------
def test_alloc_failure_leaves_context_usable():
    """An allocation failure (injected on the host: nr_debug_fail_allocs,
    no cudaMalloc is called) surfaces as NR_ENOMEM, and the same context
    completes the plan and the call afterwards."""
    wl = W.make_workload("oled_cofit", n_stacks=4)
    try:
        nr.debug_fail_allocs(1)                # the context's status word
        with pytest.raises(nr.NRError) as err:
            nr.Context(n_quad=wl.n_quad)
        assert err.value.status == nr.NR_ENOMEM
        nr.debug_fail_allocs(0)
        ctx = nr.Context(n_quad=wl.n_quad)
        b = nr.Batch.from_workload(wl)
        nr.debug_fail_allocs(2)                # the new plan's work-list buffers
        with pytest.raises(nr.NRError) as err:
            ctx.loglik_grad(b)
        assert err.value.status == nr.NR_ENOMEM
    finally:
        nr.debug_fail_allocs(0)
    ll, g = ctx.loglik_grad(b)
    assert ctx.device_status() == 0
    ref = run_oracle(wl, modes=("grad",))
    assert np.max(np.abs(ll.cpu().numpy() - ref["ll"]) / np.abs(ref["ll"])) <= TOL_LL
    assert grad_err(wl, g.cpu().numpy(), ref["g"]) <= TOL_G
    ctx.close()


DEBUG_CASES = (("thick_oxide", 64), ("oled_cofit", 8), ("uneven", 40))
DEBUG_CHILD = r"""
import sys
import numpy as np
import paper_2509_06924_gb300 as nr
from paper_2509_06924_gb300 import _build, workloads as W
assert nr.debug_build_selected() and nr.library_path() == _build.DEBUG_LIB
out = {}
for name, S in %r:
    wl = W.make_workload(name, n_stacks=S)
    ctx = nr.Context(n_quad=wl.n_quad)
    b = nr.Batch.from_workload(wl)
    out[name + "_m"] = ctx.reflectivity(b).cpu().numpy().astype(np.float64)
    ll, g = ctx.loglik_grad(b)
    f0 = ctx.device_status()
    ctx.debug_poison_plan(b, True)
    ctx.loglik_grad(b)
    f1 = ctx.device_status()
    ctx.debug_poison_plan(b, False)
    ll2, g2 = ctx.loglik_grad(b)
    f2 = ctx.device_status()
    ctx.close()
    out[name + "_ll"], out[name + "_g"] = ll.cpu().numpy(), g.cpu().numpy()
    out[name + "_ll2"], out[name + "_g2"] = ll2.cpu().numpy(), g2.cpu().numpy()
    out[name + "_flags"] = np.array([f0, f1, f2])
np.savez(sys.argv[1], **out)
""" % (DEBUG_CASES,)


def test_debug_build_reports_a_corrupted_plan(tmp_path):
    """The NR_DEBUG library (device bounds checks that set a status flag and
    skip the access instead of trapping), run in a child process with
    NR_DEBUG=1: on clean batches of the one-layer, rolled and per-bucket
    kernels it raises no flag and keeps parity with the oracle; a plan whose
    first work item names a stack one past the batch (nr_debug_poison_plan)
    gives NR_FLAG_DEBUG_BOUNDS and no fault; restored, the same plan
    reproduces the clean results."""
    import subprocess
    import sys
    from paper_2509_06924_gb300 import _build
    _build.build_debug()
    out = str(tmp_path / "debug.npz")
    r = subprocess.run([sys.executable, "-c", DEBUG_CHILD, out], cwd=ROOT, capture_output=True, text=True,
                       timeout=900, env={**os.environ, "NR_DEBUG": "1"})
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    d = np.load(out)
    for name, S in DEBUG_CASES:
        assert list(d[name + "_flags"]) == [0, nr.NR_FLAG_DEBUG_BOUNDS, 0], name
        wl = W.make_workload(name, n_stacks=S)
        gpu = {"m": d[name + "_m"], "ll_g": d[name + "_ll"], "g": d[name + "_g"], "flags": 0}
        assert_parity(wl, gpu, run_oracle(wl))
        np.testing.assert_allclose(d[name + "_ll2"], d[name + "_ll"], rtol=1e-12, atol=0)
        np.testing.assert_allclose(d[name + "_g2"], d[name + "_g"], rtol=1e-12, atol=1e-300)


def test_strong_absorbers_thick_layers_and_total_reflection():
    """Outside the workloads' ranges: absorption up to 1e-6 A^-2 (a strong
    neutron absorber; the workloads stop at 1e-8), layers up to 5000 A
    (layer phases up to 1500 rad at the top of the Q range, deep into the
    sin/cos table's reduction), Q from well below the backing's critical
    edge (total reflection, evanescent layers) and roughness up to 25 A.
    The same conditioning-aware bounds."""
    rng = np.random.default_rng(77)
    q = W.log_grid(240, 0.004, 0.3)
    stacks = []
    for t in range(12):
        n = 1 + t % 4
        d = rng.uniform(500.0, 5000.0, n)
        rho = np.concatenate([[0.0], rng.uniform(-0.5e-6, 7e-6, n), [(2.07e-6, 6.36e-6)[t % 2]]])
        iota = np.concatenate([rng.choice([0.0, 1e-7, 1e-6], n), [0.0]])
        sig = rng.uniform(0.0, 25.0, n + 1)
        stacks.append((n, W.pack(d, rho, iota, sig, 1.0, 1e-7), 0))
    wl = custom_workload(stacks, [(q, 0.03 * q)], K=17)
    gpu, ref = run_gpu(wl), run_oracle(wl)
    assert_parity(wl, gpu, ref)
    # the plain FP64 path (Parratt, against the oracle's Abeles product):
    # phases of 1e3 rad carry ~1e-13 relative rounding, amplified by the
    # fringes of thick films
    fp = run_gpu(wl, precision="fp64", modes=("loglik",))
    np.testing.assert_allclose(fp["ll"], ref["ll"], rtol=1e-10)


def test_waveguide_resonance_stacks():
    """A 520-700 A low-SLD layer between two 300 A high-SLD layers guides
    neutrons between the critical edges of its neighbours: sharp resonances
    whose gradient is most sensitive to rounding (the first stack's exact
    gradient moves by 7e-5 of its largest component under one-unit-roundoff
    input perturbations).  Dense Q over the guided range, 21 nodes; the
    scaled gradient error must stay within 5e-5 here, half the general bound."""
    q = W.log_grid(160, 0.006, 0.03)
    stacks = []
    for d_core, rho_hi in ((600.0, 6.0e-6), (600.0, 5.3e-6), (520.0, 6.3e-6), (700.0, 5.8e-6)):
        stacks.append((3, W.pack([300.0, d_core, 300.0], [0.0, rho_hi, 1.0e-6, rho_hi, 2.07e-6],
                                 [1e-9, 2e-10, 1e-9, 0.0], [4.0, 3.0, 3.0, 5.0], 1.0, 1e-7), 0))
    wl = custom_workload(stacks, [(q, 0.05 * q)], K=21)
    gpu, ref = run_gpu(wl), run_oracle(wl)
    assert_parity(wl, gpu, ref)
    assert grad_err(wl, gpu["g"], ref["g"]) <= 5e-5
