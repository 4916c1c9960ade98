"""The calls that a program using this package makes, with the sizes it makes
them at: gradients and log-likelihoods for samplers and optimisers, model
curves and SLD profiles for posterior bands, a variational iteration and a
torch optimiser's step.

Every number comes from the package's own workloads (one-layer films, thick
oxides, the ten-layer co-fit, the uneven batch, the twelve-layer variational
step) or from the sizes its tests cover (up to 64 layers, 5 to 32 nodes).

The programs around the library hold their chains, curves and optimiser state
in single precision, as torch programs do: the library computes the
likelihood and its gradient in FP32 and hands them over in FP64 storage, and
the program takes them from there as float32.  That conversion is part of a
pass.
"""
import functools
import math

import numpy as np
import torch

import paper_2509_06924_gb300 as nr

#: fronting and backing SLD of the contrasts of a co-fit (air / Si, D2O / Si, air / quartz-like)
CONTRASTS = ((0.0, 2.07e-6), (6.35e-6, 2.07e-6), (0.0, 4.2e-6))
FOUR_PI = 4.0 * math.pi
#: layer evaluations (nodes x (layers + 1)) above which exact() would take too long
EXACT_MOST = 4e9


def _case(name, kind, stacks, **more):
    c = {"name": name, "kind": kind, "stacks": stacks, "contrasts": 1, "n_lo": 1, "n_hi": 1, "pts_lo": 200,
         "pts_hi": 200, "own": False, "q_max": 0.3, "res_lo": 0.05, "res_hi": 0.05, "nodes": 17, "d_lo": 50.0,
         "d_hi": 600.0, "sig_lo": 3.0, "sig_hi": 20.0, "spread": 1.0, "depths": 0}
    assert set(more) <= set(c)
    return {**c, **more}


def listed():
    co = {"contrasts": 3, "spread": 0.2}
    return [
        # one step of a torch optimiser fitting one measured curve of a two-layer film: all latency
        _case("point_fit", "fit", 1, n_lo=2, n_hi=2, pts_lo=400, pts_hi=400, q_max=0.25, res_lo=0.03, res_hi=0.03,
              nodes=21, spread=0.05),
        # a thousand chains on a thin film: a short gradient call
        _case("film_grad", "grad", 1024, d_lo=10.0, d_hi=300.0, sig_lo=1.0, sig_hi=10.0),
        # the thick oxide film: many samples of one layer, gradient (samplers, optimisers) ...
        _case("oxide_grad", "grad", 16384, pts_lo=400, pts_hi=400, q_max=0.25, res_lo=0.03, res_hi=0.03, nodes=21,
              d_lo=1000.0, d_hi=3000.0, sig_lo=2.0, sig_hi=15.0),
        # ... and the likelihood alone (importance weights, gradient-free samplers)
        _case("oxide_loglik", "loglik", 16384, pts_lo=400, pts_hi=400, q_max=0.25, res_lo=0.03, res_hi=0.03,
              nodes=21, d_lo=1000.0, d_hi=3000.0, sig_lo=2.0, sig_hi=15.0),
        # chains of a ten-layer device co-fitted to three contrasts: the gradient of a sampler's step
        _case("oled_grad", "grad", 4096, n_lo=10, n_hi=10, pts_lo=150, pts_hi=300, **co),
        # the same device's model curves: posterior predictive bands
        _case("oled_model", "model", 4096, n_lo=10, n_hi=10, pts_lo=150, pts_hi=300, **co),
        # candidate models of 1 to 20 layers, each on its own measured curve
        _case("uneven_grad", "grad", 10000, n_lo=1, n_hi=20, pts_lo=50, pts_hi=500, own=True, res_lo=0.02,
              res_hi=0.08),
        _case("uneven_loglik", "loglik", 10000, n_lo=1, n_hi=20, pts_lo=50, pts_hi=500, own=True, res_lo=0.02,
              res_hi=0.08),
        # periodic multilayers (mirrors, superlattices) of 21 to 64 layers
        _case("deep_grad", "grad", 1024, n_lo=21, n_hi=64, d_lo=20.0, d_hi=200.0, sig_lo=2.0, sig_hi=8.0),
        # one gradient of a large variational step: reparameterised samples of a twelve-layer co-fit
        _case("vi_grad", "grad", 65536, n_lo=12, n_hi=12, pts_lo=300, pts_hi=300, nodes=21, **co),
        # one whole variational iteration of a few restarts that also infer the smearing scale
        _case("vi_restarts", "vi", 100, n_lo=10, n_hi=10, pts_lo=150, pts_hi=300, **co),
        # SLD profiles of posterior samples (bands over depth)
        _case("sld_bands", "profile", 16384, n_lo=10, n_hi=10, depths=512),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["grad", "grad", "grad", "grad", "loglik", "loglik", "model", "grad_res", "fit", "vi",
                       "profile"])
    own = kind in ("grad", "loglik", "model") and rng.random() < 0.35
    contrasts = 3 if kind == "vi" or (not own and rng.random() < 0.4) else 1
    n_lo = log_int(1, 24 if kind in ("vi", "fit") else 56)
    n_hi = min(64, n_lo + rng.randint(0, 19)) if own else n_lo
    pts_lo = log_int(50, 400)
    pts_hi = pts_lo + rng.randint(0, 200) if own or contrasts > 1 else pts_lo
    nodes = rng.choice([5, 9, 11, 13, 16, 17, 17, 17, 19, 21, 21, 21, 25, 32])
    res = rng.uniform(0.02, 0.08)
    thick = n_hi <= 2 and rng.random() < 0.4
    deep = n_hi > 20
    # stacks: logarithmic, at most a few milliseconds' worth
    per = contrasts * nodes * 0.5 * (pts_lo + pts_hi) * (0.5 * (n_lo + n_hi) + 1.0)
    most = {"fit": 16, "vi": 256, "profile": 40000}.get(kind, 40000)
    if kind in ("fit", "vi"):
        stacks = log_int(1, max(2, min(most, int(6e7 / per))))
    else:
        stacks = log_int(16, max(17, min(most, int(1.5e9 / per))))
    c = _case("", kind, stacks, contrasts=contrasts, n_lo=n_lo, n_hi=n_hi, pts_lo=pts_lo, pts_hi=pts_hi, own=own,
              q_max=rng.choice([0.2, 0.25, 0.3]), res_lo=res, res_hi=min(0.08, res + 0.03) if own else res,
              nodes=nodes, d_lo=1000.0 if thick else 20.0 if deep else 50.0,
              d_hi=3000.0 if thick else 200.0 if deep else 600.0, sig_lo=2.0 if deep else 3.0,
              sig_hi=8.0 if deep else rng.choice([10.0, 15.0, 20.0]),
              spread=0.05 if kind == "fit" else 0.2 if contrasts > 1 else rng.choice([0.2, 1.0]),
              depths=rng.choice([200, 333, 512, 1000]) if kind == "profile" else 0)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs --
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


@functools.lru_cache(maxsize=64)
def _nodes(K):
    x, w = np.polynomial.hermite.hermgauss(K)
    return x / (2.0 * math.sqrt(math.log(2.0))), w / math.sqrt(math.pi)


def _draw_stacks(c, g, chains, n):
    """Packed parameters [chains, contrasts, 4 n + 6] of `chains` draws of n layers."""
    dev = _device()

    def uniform(lo, hi, k):
        return lo + (hi - lo) * torch.rand((chains, k), generator=g, dtype=torch.float64, device=dev)

    if c["d_lo"] >= 1000.0:  # oxide-like films
        rho = 4.2e-6 + 1e-7 * torch.randn((chains, n), generator=g, dtype=torch.float64, device=dev)
    elif n == 1:
        rho = uniform(1e-6, 6e-6, n)
    else:
        rho = uniform(-0.5e-6, 6e-6, n)
    d, iota = uniform(c["d_lo"], c["d_hi"], n), uniform(0.0, 1e-8 if n > 1 else 0.0, n)
    sig = uniform(c["sig_lo"], c["sig_hi"], n + 1)
    one = torch.ones((chains, 1), dtype=torch.float64, device=dev)
    return torch.stack([torch.cat([d, front * one, rho, back * one, iota, 0.0 * one, sig, one, 1e-7 * one], 1)
                        for front, back in CONTRASTS[:c["contrasts"]]], 1)


def _inputs(c, seed):
    """Everything one call is made of, on the device: metadata (numpy), packed
    parameters, and measured curves: a true stack's smeared reflectivity
    with 5 % noise.  The stacks lie `spread` of the prior's width around it."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 11)
    chains, nc = c["stacks"], c["contrasts"]
    # layer counts and curve lengths belong to the case, every value to the seed
    h = np.random.default_rng([chains, nc, c["n_lo"], c["n_hi"], c["pts_lo"], c["pts_hi"], c["nodes"]])
    if c["own"]:
        n_chain = h.integers(c["n_lo"], c["n_hi"] + 1, chains)
        lens = h.integers(c["pts_lo"], c["pts_hi"] + 1, chains)
        rel = h.uniform(c["res_lo"], c["res_hi"], chains)
        dataset = np.arange(chains)
    else:
        n_chain = h.integers(c["n_lo"], c["n_hi"] + 1, chains) if c["n_lo"] < c["n_hi"] else np.full(chains, c["n_lo"])
        lens = np.linspace(c["pts_lo"], c["pts_hi"], nc).round().astype(np.int64)
        rel = np.full(nc, c["res_lo"])
        dataset = np.tile(np.arange(nc), chains)
    n_layers = np.repeat(n_chain, nc)
    par_off = np.concatenate([[0], np.cumsum(4 * n_layers + 6)])
    params = torch.empty(int(par_off[-1]), dtype=torch.float64, device=dev)
    truth = {}
    for n in sorted(set(int(v) for v in n_chain)):
        at = np.flatnonzero(n_chain == n)
        t = _draw_stacks(c, g, 1, n)
        p = _draw_stacks(c, g, len(at), n)
        truth[n] = t[0]
        rows = torch.as_tensor(par_off[:-1].reshape(chains, nc)[at], device=dev).reshape(-1)
        cols = torch.arange(4 * n + 6, device=dev)
        params[rows[:, None] + cols] = (t + c["spread"] * (p - t)).reshape(-1, 4 * n + 6)
    q_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    sets = torch.as_tensor(np.repeat(np.arange(len(lens)), lens), device=dev)
    step = torch.arange(int(q_off[-1]), device=dev) - torch.as_tensor(q_off[:-1], device=dev)[sets]
    length = torch.as_tensor(lens, device=dev)[sets].double()
    lo, hi = math.log(0.005), math.log(c["q_max"])
    q = torch.exp(lo + (hi - lo) * step / (length - 1.0)).float()
    dq = (torch.as_tensor(rel, device=dev)[sets] * q.double()).float()
    x = {"n_layers": n_layers.astype(np.int32), "dataset": dataset.astype(np.int32), "q_off": q_off,
         "par_off": par_off, "params": params, "q": q, "dq": dq, "truth": truth, "gen": g}
    if c["kind"] == "profile":
        return x
    # the measured curves: of the one true stack, or (own curves) of a true
    # stack with as many layers, at its nodes' weighted positions
    r = torch.empty(q.numel(), dtype=torch.float64, device=dev)
    with torch.no_grad():
        if c["own"]:
            n_of = torch.as_tensor(n_layers, device=dev)[sets]
            for n, t in truth.items():
                at = torch.nonzero(n_of == n).reshape(-1)
                r[at] = _model64(t[:1], n, q[at].double()[None], 0.0 * q[at].double()[None], 1)[0]
        else:
            n = int(n_chain[0])
            for k in range(nc):
                s = slice(int(q_off[k]), int(q_off[k + 1]))
                r[s] = _model64(truth[n][k:k + 1], n, q[s].double()[None], dq[s].double()[None], c["nodes"])[0]
    noise = torch.randn(r.numel(), generator=g, dtype=torch.float64, device=dev)
    x["r_obs"], x["r_err"] = (r * torch.exp(0.05 * noise)).float(), (0.05 * r).float()
    return x


def _cofit(c, x, seed):
    """The sampler's model of a co-fit: layers shared by the contrasts, a free
    scale and background for each, and a free scale of every resolution."""
    n, nc = c["n_lo"], c["contrasts"]
    stacks = x["truth"][n].cpu().numpy()
    t = stacks[0]
    lo, hi, mid = [], [], []

    def free(a, b, v):
        lo.append(a), hi.append(b), mid.append(v)
        return len(lo) - 1

    shared = {}
    for j in range(n):
        shared[j] = free(0.6 * t[j], 1.4 * t[j], t[j])
        shared[n + 1 + j] = free(t[n + 1 + j] - 1.5e-6, t[n + 1 + j] + 1.5e-6, t[n + 1 + j])
        shared[2 * n + 2 + j] = free(0.0, 2e-8, min(max(t[2 * n + 2 + j], 1e-9), 1.9e-8))
    for j in range(n + 1):
        shared[3 * n + 3 + j] = free(1.0, 30.0, t[3 * n + 3 + j])
    src, val = [], []
    for k in range(nc):
        s = -np.ones(4 * n + 6, np.int32)
        for slot, i in shared.items():
            s[slot] = i
        s[4 * n + 4], s[4 * n + 5] = free(0.8, 1.2, 1.0), free(1e-8, 1e-6, 1e-7)
        src.append(s)
        val.append(stacks[k])
    res = free(0.7, 1.3, 1.0)
    lo, hi, mid = (np.array(v) for v in (lo, hi, mid))
    P, R, dev = lo.size, c["stacks"], _device()
    u = torch.as_tensor(np.log((mid - lo) / (hi - mid)), device=dev)
    mu = u + 0.05 * torch.randn((R, P), generator=x["gen"], dtype=torch.float64, device=dev)
    low = torch.zeros((R, P * (P + 1) // 2), dtype=torch.float64, device=dev)
    low[:, torch.arange(P, device=dev) * (torch.arange(P, device=dev) + 3) // 2] = math.log(0.01)
    eps = torch.randn((R, P), generator=x["gen"], dtype=torch.float64, device=dev)
    return {"src": np.concatenate(src), "val": np.concatenate(val), "lo": lo, "hi": hi, "res": res,
            "phi": torch.cat([mu, low], 1), "eps": eps}


def prepare(case, seed):
    x = _inputs(case, seed)
    dev = x["params"].device
    ctx = nr.Context(n_quad=case["nodes"])
    s = {"kind": case["kind"], "ctx": ctx}
    if case["kind"] == "vi":
        m = _cofit(case, x, seed)
        nc = case["contrasts"]
        s["sampler"] = nr.Sampler(ctx, case["stacks"], x["n_layers"][:nc], x["dataset"][:nc], x["q_off"], x["q"],
                                  x["dq"], x["r_obs"], x["r_err"], m["src"], m["val"], m["lo"], m["hi"],
                                  res_param=m["res"])
        s["phi"], s["eps"] = m["phi"], m["eps"]
        s["m"], s["v"] = torch.zeros_like(m["phi"]), torch.zeros_like(m["phi"])
        s["t"] = torch.zeros(1, dtype=torch.int32, device=dev)
        s["elbo"] = torch.empty(case["stacks"], dtype=torch.float64, device=dev)
        return s
    batch = nr.Batch(x["n_layers"], x["dataset"], x["q_off"], x["params"], x["q"], x["dq"], x.get("r_obs"),
                     x.get("r_err"))
    s["batch"] = batch
    if case["kind"] == "profile":
        s["z"] = torch.linspace(-100.0, float(case["d_hi"] * case["n_hi"] * 0.6 + 100.0), case["depths"], device=dev)
        s["rho"] = torch.empty(batch.n_stacks * case["depths"], device=dev)
        s["iota"] = torch.empty_like(s["rho"])
        return s
    if case["kind"] == "fit":
        s["theta"] = x["params"].float().requires_grad_()
    elif case["kind"] == "model":
        s["m"] = torch.empty(batch.total_out, device=dev)
    else:
        s["ll"] = torch.empty(batch.n_stacks, dtype=torch.float64, device=dev)
        s["g"] = torch.empty(batch.params.numel(), dtype=torch.float64, device=dev)
        s["res"] = torch.empty(batch.n_stacks, dtype=torch.float64, device=dev)
    ctx.plan(batch)
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "grad":
        ll, g = s["ctx"].loglik_grad(s["batch"], s["ll"], s["g"])
        return {"loglik": ll.float(), "grad": g.float()}
    if kind == "loglik":
        return {"loglik": s["ctx"].loglik(s["batch"], s["ll"]).float()}
    if kind == "model":
        return {"model": s["ctx"].reflectivity(s["batch"], s["m"])}
    if kind == "grad_res":
        ll, g, r = s["ctx"].loglik_grad_res(s["batch"], s["ll"], s["g"], s["res"])
        return {"loglik": ll.float(), "grad": g.float(), "res": r.float()}
    if kind == "fit":
        ll = nr.loglik_autograd(s["theta"].double(), s["ctx"], s["batch"])
        (g,) = torch.autograd.grad(ll.sum(), s["theta"])
        return {"loglik": ll.detach().float(), "grad": g}
    if kind == "vi":
        elbo = s["sampler"].vi_step(s["phi"], s["m"], s["v"], s["t"], s["eps"], lr=1e-3, elbo_out=s["elbo"])
        return {"elbo": elbo.float(), "phi": s["phi"].float(), "m": s["m"].float(), "v": s["v"].float()}
    rho, iota = s["ctx"].sld_profile(s["batch"], s["z"], s["rho"], s["iota"])
    return {"rho": rho, "iota": iota}


# -------------------------------------------------------------------- work --
def work(case):
    c = case
    n = 0.5 * (c["n_lo"] + c["n_hi"])
    stacks = c["stacks"] * c["contrasts"]
    pts = 0.5 * (c["pts_lo"] + c["pts_hi"])
    par = 4.0 * n + 6.0
    if c["kind"] == "profile":
        # an error function (about 20 operations) and two sums per interface and depth
        return {"bytes": stacks * (8.0 * par + 8.0 * c["depths"]) + 4.0 * c["depths"],
                "flops": stacks * c["depths"] * (n + 1.0) * 26.0}
    evals = stacks * pts * c["nodes"]
    curves = c["stacks"] if c["own"] else c["contrasts"]
    data = curves * pts * (8.0 if c["kind"] == "model" else 16.0)
    # operations per node: the wavevector, Fresnel factor, phase and Parratt
    # step of every layer; the adjoint of each once more (nothing recomputed)
    flops = evals * (83.0 + 135.0 * n)
    if c["kind"] == "model":
        return {"bytes": 8.0 * par * stacks + data + 4.0 * stacks * pts, "flops": flops}
    if c["kind"] == "loglik":
        return {"bytes": 8.0 * par * stacks + data + 4.0 * stacks, "flops": flops}
    flops += evals * (50.0 + 109.0 * n)
    if c["kind"] == "vi":
        P = 4.0 * n + 2.0 + 2.0 * c["contrasts"]
        phi = c["stacks"] * (P + P * (P + 1.0) / 2.0)
        return {"bytes": data + 8.0 * c["stacks"] * P + 8.0 * 6.0 * phi + 4.0 * 3.0 * phi, "flops": flops}
    return {"bytes": (8.0 + 4.0) * par * stacks + data + 4.0 * stacks, "flops": flops}


# ----------------------------------------------------- the same in 64 bits --
def _model64(p, n, q, dq, K, f=None):
    """scale * (smeared reflectivity) + background of packed stacks p [M, 4n+6]
    at q, dq [M, Q] (Parratt recursion, Nevot-Croce roughness)."""
    x, w = (torch.as_tensor(v, device=p.device) for v in _nodes(K))
    if f is not None:
        dq = dq * f[:, None]
    k0 = 0.5 * (q[..., None] + dq[..., None] * x)

    def col(i):
        return p[:, i, None, None]

    def wave(j):
        if j == 0:
            return torch.complex(k0, torch.zeros_like(k0))
        u = k0 * k0 - FOUR_PI * (col(n + j) - col(n))
        return torch.sqrt(torch.complex(u, (FOUR_PI * col(2 * n + 1 + j)).expand_as(u)))

    below, X = wave(n + 1), None
    for j in range(n, -1, -1):
        k = wave(j)
        # k^2 differences without the cancellation of k_j - k_{j+1}
        num = torch.complex(FOUR_PI * (col(n + j + 1) - col(n + j)),
                            FOUR_PI * ((col(2 * n + 1 + j) if j else 0.0 * col(0)) - col(2 * n + 2 + j)))
        S = k + below
        r = num / (S * S) * torch.exp(-2.0 * k * below * col(3 * n + 3 + j) ** 2)
        if X is None:
            X = r
        else:
            Y = X * torch.exp(2j * below * col(j))
            X = (r + Y) / (1.0 + r * Y)
        below = k
    R = X.real * X.real + X.imag * X.imag
    return p[:, 4 * n + 4, None] * (R @ w) + p[:, 4 * n + 5, None]


def _pieces(c, x):
    """The batch in pieces of stacks with one layer count, their curves padded
    to one length: (n, stacks, q, dq, r_obs, r_err, mask)."""
    dev = x["q"].device
    lens = np.diff(x["q_off"])
    for n in sorted(set(int(v) for v in x["n_layers"])):
        at = np.flatnonzero(x["n_layers"] == n)
        at = at[np.argsort(lens[x["dataset"][at]], kind="stable")]
        i = 0
        while i < len(at):
            most = lens[x["dataset"][at[i]]]
            step = max(1, int(6e6 / (most * c["nodes"] * (n + 1))))
            s = at[i:i + step]
            i += len(s)
            ds = x["dataset"][s]
            pts = np.arange(int(lens[ds].max()))
            mask = pts[None] < lens[ds][:, None]
            idx = torch.as_tensor(np.where(mask, x["q_off"][ds][:, None] + pts, x["q_off"][ds][:, None]), device=dev)
            got = [x[k][idx].double() if k in x else None for k in ("q", "dq", "r_obs", "r_err")]
            yield n, s, got, torch.as_tensor(mask, device=dev)


def _rows(x, s, n):
    first = torch.as_tensor(x["par_off"][s], device=x["params"].device)
    return first[:, None] + torch.arange(4 * n + 6, device=first.device)


def _loglik64(p, n, K, data, mask, f=None):
    q, dq, r, e = data
    m = _model64(p, n, q, dq, K, f)
    return -0.5 * (torch.where(mask, ((m - r) / e) ** 2 + torch.log(2.0 * math.pi * e * e), 0.0)).sum(1)


def _vi64(c, x, seed):
    """One variational iteration: reparameterised draw, -ELBO gradient, Adam (step 1)."""
    m = _cofit(c, x, seed)
    n, nc, R = c["n_lo"], c["contrasts"], c["stacks"]
    P, dev = m["lo"].size, x["q"].device
    phi = m["phi"].clone().requires_grad_()
    i, j = torch.tril_indices(P, P, device=dev)
    L = torch.zeros((R, P, P), dtype=torch.float64, device=dev)
    L = L.index_put((torch.arange(R, device=dev)[:, None], i, j), torch.where(i == j, torch.exp(phi[:, P:]), phi[:, P:]))
    u = phi[:, :P] + (L @ m["eps"][..., None])[..., 0]
    lo, hi = (torch.as_tensor(m[k], device=dev) for k in ("lo", "hi"))
    th = lo + (hi - lo) * torch.sigmoid(u)
    src = torch.as_tensor(m["src"].astype(np.int64), device=dev)
    packed = torch.where(src >= 0, th[:, src.clamp(min=0)], torch.as_tensor(m["val"], device=dev))
    logp = (torch.nn.functional.logsigmoid(u) + torch.nn.functional.logsigmoid(-u)).sum(1)
    for k in range(nc):
        s = slice(int(x["q_off"][k]), int(x["q_off"][k + 1]))
        data = [x[v][s].double().expand(R, -1) for v in ("q", "dq", "r_obs", "r_err")]
        mask = torch.ones_like(data[0], dtype=torch.bool)
        logp = logp + _loglik64(packed[:, k * (4 * n + 6):(k + 1) * (4 * n + 6)], n, c["nodes"], data, mask,
                                th[:, m["res"]])
    diag = torch.arange(P, device=dev) * (torch.arange(P, device=dev) + 3) // 2 + P
    elbo = logp + 0.5 * (m["eps"] ** 2).sum(1) + phi[:, diag].sum(1) + 0.5 * P * math.log(2.0 * math.pi)
    (g,) = torch.autograd.grad(-elbo.sum(), phi)
    new = m["phi"] - 1e-3 * g / (g.abs() + 1e-8)
    return {"elbo": elbo.detach(), "phi": new, "m": 0.1 * g, "v": 1e-3 * g * g}


def exact(case, seed):
    c = case
    lay = c["stacks"] * c["contrasts"] * 0.5 * (c["pts_lo"] + c["pts_hi"]) * c["nodes"] * (0.5 * (c["n_lo"] + c["n_hi"]) + 1.0)
    if c["kind"] != "profile" and lay > EXACT_MOST:
        return None
    x = _inputs(c, seed)
    dev, kind = x["q"].device, c["kind"]
    S = len(x["n_layers"])
    if kind == "vi":
        return _vi64(c, x, seed)
    if kind == "fit":
        x["params"] = x["params"].float().double()
    if kind == "profile":
        z = torch.linspace(-100.0, float(c["d_hi"] * c["n_hi"] * 0.6 + 100.0), c["depths"], device=dev).double()
        out = {k: torch.zeros((S, c["depths"]), dtype=torch.float64, device=dev) for k in ("rho", "iota")}
        for n in sorted(set(int(v) for v in x["n_layers"])):
            s = np.flatnonzero(x["n_layers"] == n)
            p, at = x["params"][_rows(x, s, n)], torch.as_tensor(s, device=dev)
            depth, rho, iota = torch.zeros_like(p[:, :1]), p[:, n, None] + 0.0 * z, 0.0 * p[:, :1] + 0.0 * z
            for j in range(n + 1):
                step = 0.5 * (1.0 + torch.erf((z - depth) / (math.sqrt(2.0) * p[:, 3 * n + 3 + j, None])))
                rho = rho + (p[:, n + j + 1] - p[:, n + j])[:, None] * step
                iota = iota + (p[:, 2 * n + 2 + j] - (p[:, 2 * n + 1 + j] if j else 0.0))[:, None] * step
                depth = depth + p[:, j, None] if j < n else depth
            out["rho"][at], out["iota"][at] = rho, iota
        return out
    ll = torch.zeros(S, dtype=torch.float64, device=dev)
    res, g = torch.zeros_like(ll), torch.zeros_like(x["params"])
    lens = np.diff(x["q_off"])[x["dataset"]]
    out_off = np.concatenate([[0], np.cumsum(lens)])
    model = torch.zeros(int(out_off[-1]), dtype=torch.float64, device=dev) if kind == "model" else None
    for n, s, data, mask in _pieces(c, x):
        rows, at = _rows(x, s, n), torch.as_tensor(s, device=dev)
        p = x["params"][rows]
        if kind == "model":
            with torch.no_grad():
                m = _model64(p, n, data[0], data[1], c["nodes"])
            to = torch.as_tensor(out_off[s], device=dev)[:, None] + torch.arange(mask.shape[1], device=dev)
            model[to[mask]] = m[mask]
        elif kind == "loglik":
            with torch.no_grad():
                ll[at] = _loglik64(p, n, c["nodes"], data, mask)
        else:
            p.requires_grad_()
            f = torch.ones_like(p[:, 0].detach()).requires_grad_()
            v = _loglik64(p, n, c["nodes"], data, mask, f)
            gp, gf = torch.autograd.grad(v.sum(), (p, f))
            ll[at], g[rows], res[at] = v.detach(), gp, gf
    if kind == "model":
        return {"model": model}
    if kind == "loglik":
        return {"loglik": ll}
    return {"loglik": ll, "grad": g, "res": res} if kind == "grad_res" else {"loglik": ll, "grad": g}
