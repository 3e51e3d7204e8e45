"""The calls that a user of this library has it do, for timing and for comparing results.

Every case is one pass through the public entry points of paper_1704_08919_gb300 at sizes
of the workloads in inputs.py, of the tests or between them.  Results of the paths that
hold their state in FP32 are good to FP32 however they are stored, and a program keeps
them so (the network's targets, the densities of a population): they are handed on as
FP32.  Results of the FP64 paths stay FP64.
"""
import math

import numpy as np
import torch

import paper_1704_08919_gb300 as pp
from paper_1704_08919_gb300 import inputs

BAND = 2.0  # every pulse model here has its modes on [0, 2]
DE = inputs.DE_BATCH
BIG = inputs.LARGE_SCALE
LOCAL = inputs.LOCAL_SEARCH
NET = inputs.SURROGATE_DE


def listed():
    return [
        # The library's default precision and scheme on a small grid, as a first look at a few
        # pulses: launches and the serial chain over the steps count.
        dict(name="score-defaults-small", kind="score", precision="fp32", scheme="rk4", cands=8, nx=12, ny=10,
             nz=5, ext=2.0, dt=0.05, n_steps=800, uneven=False, densities=False),
        # A screened generation of a small search: network, proposals, synthesis, scoring.
        dict(name="screened-small", kind="screened", precision="fp32fast", scheme="magnus4", NP=16, R=8, K=8,
             nx=16, ny=16, nz=8, ext=2.0, T=50.0, n_steps=2048),
        # One given field on the parity path, with the densities: the rotating Gaussian pulse.
        dict(name="single-field-fp64", kind="gaussian", precision="fp64", scheme="rk4", nx=32, ny=32, nz=16,
             ext=1.5, n_steps=4000),
        # Reference scores of a population's best pulses on the parity path.
        dict(name="population-fp64", kind="score", precision="fp64", scheme="rk4", cands=2, nx=64, ny=64, nz=32,
             ext=2.0, dt=200.0 / 8192, n_steps=8192, uneven=False, densities=False),
        # The final pulses of a search, with the densities.
        dict(name="densities-fp32fast", kind="score", precision="fp32fast", scheme="magnus4", cands=2, nx=64,
             ny=64, nz=32, ext=2.0, dt=200.0 / 8192, n_steps=8192, uneven=False, densities=True),
        # Pulses of unlike lengths in compensated FP32 on an odd grid, with the densities.
        dict(name="compensated-uneven", kind="score", precision="fp32", scheme="magnus4", cands=8, nx=47, ny=45,
             nz=23, ext=2.0, dt=0.02, n_steps=9001, uneven=True, densities=True),
        # The paper's own integrator.
        dict(name="split-operator", kind="score", precision="fp32fast", scheme="split2", cands=4, nx=40, ny=40,
             nz=20, ext=2.0, dt=0.02, n_steps=5000, uneven=False, densities=False),
        # One generation of the DE batch, the benchmark's step.
        dict(name="generation", kind="generation", precision="fp32fast", scheme="magnus4", NP=64, K=8, nx=64,
             ny=64, nz=32, ext=2.0, T=200.0, n_steps=8192),
        # One generation of the uneven batch, captured in a graph.
        dict(name="uneven-batch", kind="batch", precision="fp32fast", scheme="magnus4", NP=128, K=8, n_min=2500,
             n_max=20000, sides=96, generations=1),
        # A few pulses of the large-scale search: the longest pulses on the finest grid.
        dict(name="large-grid", kind="score", precision="fp32fast", scheme="magnus4", cands=4, nx=128, ny=128,
             nz=64, ext=2.5, dt=0.02, n_steps=20000, uneven=False, densities=True),
        # One objective evaluation of the multistart local search.
        dict(name="local-search-gradient", kind="gradient", precision="fp32", starts=16, K=8, nx=32, ny=32, nz=16,
             ext=2.0, T=50.0, n_steps=16384),
        # One mini-batch of the surrogate's training.
        dict(name="network-gradient", kind="network", rows=256, d_in=32, grad=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_sizes(rng, lo, hi):
    return dict(nx=_log(rng, lo, hi), ny=_log(rng, lo, hi), nz=max(1, _log(rng, lo, hi) // 2))


def draw(rng):
    """One more case: any of the kinds, sizes over their ranges."""
    kind = rng.choice(["score", "score", "score", "score", "generation", "screened", "batch", "gradient", "gaussian",
                       "network"])
    if kind == "score":
        precision, scheme, most = rng.choice([("fp32fast", "magnus4", 5e10), ("fp32fast", "magnus4", 5e9),
                                              ("fp32", "magnus4", 5e9), ("fp32", "rk4", 5e9),
                                              ("fp32fast", "rk4", 5e9), ("fp64", "rk4", 1e9),
                                              ("fp32fast", "split2", 5e9)])
        c = dict(kind=kind, precision=precision, scheme=scheme, cands=_log(rng, 1, 32), **_grid_sizes(rng, 5, 128),
                 ext=rng.choice([1.5, 2.0, 2.5]), dt=rng.choice([0.02, 0.02, 200.0 / 8192, 0.05]),
                 n_steps=_log(rng, 300, 20000), uneven=rng.random() < 0.3, densities=rng.random() < 0.5)
        while c["cands"] * c["nx"] * c["ny"] * c["nz"] * c["n_steps"] > most:
            k = rng.choice(["cands", "nx", "ny", "nz", "n_steps"])
            c[k] = max(1, int(c[k] * 0.7))
        return c
    if kind == "gaussian":
        return dict(kind=kind, precision="fp64", scheme="rk4", **_grid_sizes(rng, 8, 48), ext=1.5,
                    n_steps=_log(rng, 2000, 8000))
    if kind == "generation":
        n = _log(rng, 1000, 8192)
        return dict(kind=kind, precision="fp32fast", scheme="magnus4", NP=_log(rng, 8, 64), K=rng.choice([8, 16]),
                    **_grid_sizes(rng, 12, 64), ext=2.0, T=n * 0.02, n_steps=n)
    if kind == "screened":
        n = _log(rng, 1000, 8192)
        return dict(kind=kind, precision="fp32fast", scheme="magnus4", NP=_log(rng, 8, 128), R=rng.choice([4, 8]),
                    K=rng.choice([8, 16]), **_grid_sizes(rng, 12, 32), ext=2.0, T=n * 0.02, n_steps=n)
    if kind == "batch":
        return dict(kind=kind, precision="fp32fast", scheme="magnus4", NP=_log(rng, 8, 96), K=8,
                    n_min=_log(rng, 500, 2500), n_max=_log(rng, 3000, 16000), sides=rng.choice([32, 48, 64, 96]),
                    generations=rng.choice([1, 2]))
    if kind == "gradient":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "fp64"]), starts=_log(rng, 1, 8), K=8,
                    **_grid_sizes(rng, 6, 20), ext=2.0, T=20.0, n_steps=_log(rng, 2000, 5000))
    return dict(kind="network", rows=_log(rng, 64, 8192), d_in=rng.choice([32, 64]), grad=rng.random() < 0.5)


# ---------------------------------------------------------------------------------- inputs


def _grid(c):
    return dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], x0=-c["ext"], x1=c["ext"], y0=-c["ext"], y1=c["ext"], z0=0.0,
                z1=c["ext"] if c["nz"] > 1 else 0.0, mirror_z=1)


def _one_axis(g):
    """A grid axis of one node has equal bounds."""
    for a, n in (("x", "nx"), ("y", "ny")):
        if g[n] == 1:
            g[a + "0"] = g[a + "1"] = 0.3
    return g


def _potential(n_steps, dt, ld, seed, device, fluence=2.0, K=8):
    """A [2][ld] on the half-step grid: a pulse with modes on (0, BAND], amplitudes and phases
    interpolated from K random control points, A(-T/2) = 0, int E^2 dt = fluence."""
    rng = np.random.default_rng(seed)
    T = n_steps * dt
    w = 2.0 * math.pi / T * np.arange(1, max(1, int(BAND * T / (2.0 * math.pi))) + 1)
    knots = np.linspace(0.0, BAND, K)
    amp = np.stack([np.interp(w, knots, rng.random(K)) for _ in range(2)])
    phi = np.stack([np.interp(w, knots, 2.0 * math.pi * rng.random(K)) for _ in range(2)])
    amp *= math.sqrt(fluence / (0.5 * T * np.sum(amp ** 2)))
    t = -0.5 * T + 0.5 * dt * torch.arange(2 * n_steps + 1, dtype=torch.float64, device=device)
    W, P, Q = (torch.tensor(v, device=device) for v in (w, phi, amp / w))
    A = torch.zeros((2, ld), dtype=torch.float64, device=device)
    for a in range(2):
        s = torch.zeros_like(t)
        for j in range(0, len(w), 32):
            s -= (Q[a, j:j + 32, None] * torch.sin(W[j:j + 32, None] * t + P[a, j:j + 32, None])).sum(0)
        A[a, :2 * n_steps + 1] = s - s[0]
    return A


def _score_inputs(c, seed, device):
    """(A [cands][2][ld], n_steps of each) of a "score" or "gaussian" case."""
    n = c["n_steps"]
    if c["kind"] == "gaussian":
        rng = np.random.default_rng([seed, 5])
        g = dict(inputs.ROTATING_GAUSSIAN, n_steps=n)
        g["E0"] *= 0.8 + 0.4 * rng.random()
        g["w"] *= 0.9 + 0.2 * rng.random()
        return torch.tensor(inputs.rotating_gaussian_potential(g, 2 * n + 1)[None], device=device), [n]
    rng = np.random.default_rng([seed, 1])
    steps = [n] * c["cands"]
    if c["uneven"]:
        steps = [int(x) for x in rng.integers(max(1, n // 4), n + 1, size=c["cands"])]
        steps[0] = n
    A = torch.stack([_potential(s, c["dt"], 2 * n + 1, [seed, 2, i], device) for i, s in enumerate(steps)])
    return A.contiguous(), steps


def _dt(c):
    return 80.0 / c["n_steps"] if c["kind"] == "gaussian" else c["dt"]


def _search(c, seed):
    """Population, bounds and pulse model of a DE case."""
    lo, hi, per = (torch.tensor(v, device="cuda") for v in inputs.param_bounds(c["K"]))
    pop = torch.tensor(inputs.random_population(c["NP"], c["K"], [seed, 3]), device="cuda")
    return dict(pop=pop, lo=lo, hi=hi, per=per, seed=seed, generation=0)


def _spec(c):
    return dict(K=c["K"], order=4, w_min=0.0, w_max=BAND, T=c["T"], fluence=2.0, n_steps=c["n_steps"])


def _network_size(d_in, H=256):
    return H * d_in + H + 2 * (H * H + H) + H + 1


def _network_inputs(c, seed, device):
    rng = np.random.default_rng([seed, 4])
    d, H = c["d_in"], NET["hidden"]
    p = [rng.normal(0.0, math.sqrt(2.0 / f), s) for s, f in (((H, d), d), ((H,), 1e4), ((H, H), H), ((H,), 1e4),
                                                           ((H, H), H), ((H,), 1e4), ((H,), H), ((1,), 1e4))]
    flat = np.concatenate([v.ravel() for v in p]).astype(np.float32)
    X = (rng.random((c["rows"], d)) - 0.5).astype(np.float32)
    t = rng.normal(size=c["rows"]).astype(np.float32)
    return [torch.tensor(v, device=device) for v in (flat, X, t)]


def _starts(c, seed):
    """Starts uniform in the bounds, the amplitudes scaled to the search's fluence (a mode's
    spectrum is linear in them)."""
    X = inputs.random_population(c["starts"], c["K"], [seed, 6])
    P = torch.tensor(X, device="cuda")
    _, _, U, _ = pp.qke_gradient(P, dict(_spec(c), n_steps=8), _grid(dict(c, nx=2, ny=2, nz=2)), c["precision"],
                                 want_grad=False)
    s = (LOCAL["U_const"] / U).sqrt()[:, None]
    for blk in (0, 2):
        P[:, blk * c["K"]:(blk + 1) * c["K"]] *= s
    return P


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("score", "gaussian"):
        A, steps = _score_inputs(c, seed, "cuda")
        return dict(c=c, A=A, steps=steps if c.get("uneven") else None, grid=_one_axis(_grid(c)))
    if kind == "network":
        flat, X, t = _network_inputs(c, seed, "cuda")
        net = pp.Surrogate(c["d_in"], hidden=NET["hidden"], max_batch=max(4096, c["rows"]))
        net.set_params(flat)
        return dict(c=c, net=net, X=X, t=t)
    if kind == "gradient":
        return dict(c=c, X=_starts(c, seed), spec=_spec(c), grid=_grid(c))
    s = dict(c=c, **_search(c, seed))
    if kind == "batch":
        U = inputs.UNEVEN_BATCH
        rng = np.random.default_rng([seed, 7])
        steps = rng.integers(c["n_min"], c["n_max"] + 1, size=c["NP"])
        specs = inputs.uneven_specs(U, steps)
        peaks = []
        for i, sp in enumerate(specs):
            # the peak field on a coarse time grid
            _, E, _ = pp.synth_field(s["pop"][i:i + 1], dict(sp, n_steps=1024), want_E=True)
            peaks.append((E[0] ** 2).sum(0).max())
        sides = tuple(max(8, c["sides"] * k // 6) for k in (2, 3, 4, 5, 6))
        grids = inputs.grids_by_rank(dict(U, sides=sides), torch.stack(peaks).cpu().numpy())
        s["batch"] = pp.Batch(specs, grids, U["dt"], precision=c["precision"], scheme=c["scheme"])
        s["fit"] = s["batch"].pair_number(s["batch"].synth(s["pop"]))[0]
        s["batch"].set_generation(0)
        return s
    s["spec"], s["grid"] = _spec(c), _grid(c)
    A = pp.synth_field(s["pop"], s["spec"])[0]
    s["fit"] = pp.pair_number(A, c["T"] / c["n_steps"], s["grid"], precision=c["precision"], scheme=c["scheme"])[0]
    s["trial"], s["trial_fit"] = torch.empty_like(s["pop"]), torch.empty_like(s["fit"])
    if kind == "screened":
        s["net"] = pp.Surrogate(4 * c["K"], hidden=NET["hidden"], max_batch=max(4096, c["NP"] * c["R"]))
        s["net"].init(seed + 1)
        s["pred"] = torch.empty(c["NP"] * c["R"], dtype=torch.float32, device="cuda")
        s["kept"] = torch.empty(c["NP"], dtype=torch.int32, device="cuda")
    return s


def _kept(x, c):
    """A result as the caller keeps it: FP32 for the paths that hold their state in FP32."""
    return x if x is None or c["precision"] == "fp64" else x.float()


def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind in ("score", "gaussian"):
        N, n = pp.pair_number(s["A"], _dt(c), s["grid"], precision=c["precision"], n_steps=s["steps"],
                              want_n=c.get("densities", True), scheme=c["scheme"])
        return [_kept(N, c)] + ([] if n is None else [_kept(n, c)])
    if kind == "network":
        if c["grad"]:
            return list(s["net"].loss_grad(s["X"], s["t"]))
        return [s["net"].forward(s["X"])]
    if kind == "gradient":
        J, gJ, U, dU = pp.qke_gradient(s["X"], s["spec"], s["grid"], precision=c["precision"])
        return [_kept(J, c), _kept(gJ, c), U, dU]
    if kind == "batch":
        s["batch"].de_run(s["pop"], s["fit"], s["lo"], s["hi"], s["per"], DE["F"], DE["CR"], s["seed"],
                          c["generations"])
        return [s["pop"], _kept(s["fit"], c)]
    g = s["generation"]
    s["generation"] += 1
    args = (s["pop"], s["fit"], s["spec"], s["grid"], s["lo"], s["hi"], s["per"], DE["F"], DE["CR"], s["seed"], g)
    if kind == "screened":
        pp.de_screened_step(*args, c["R"], s["net"], precision=c["precision"], scheme=c["scheme"], mode="global",
                            trial_out=s["trial"], trial_fit_out=s["trial_fit"], pred_out=s["pred"],
                            kept_out=s["kept"])
        return [s["pop"], _kept(s["fit"], c), s["trial"], _kept(s["trial_fit"], c), s["pred"], s["kept"]]
    pp.de_step(*args, precision=c["precision"], scheme=c["scheme"], trial_out=s["trial"],
               trial_fit_out=s["trial_fit"])
    return [s["pop"], _kept(s["fit"], c), s["trial"], _kept(s["trial_fit"], c)]


# ---------------------------------------------------------------------------------- work

# Flops of one mode over one step, both spin channels: the 2 x 2 unitary applied to each channel's
# two-component state (16 multiply-adds less the 4 of a unit diagonal: 12, 24 flops), for the two
# channels.  Everything else (forming the step) is the algorithm's own business.
STEP_FLOPS = 48.0
# The kinetic equation: a real 6-component state through a step matrix with 12 nonzero entries in
# four stages, forward, and its transpose with the sample sensitivities, backward.
GRADIENT_FLOPS = 2 * 4 * 2 * 12.0 + 4 * 7 * 2


def work(case):
    c, kind = case, case["kind"]
    if kind == "network":
        H, d, B = NET["hidden"], c["d_in"], c["rows"]
        mm = 2.0 * B * (H * d + 2 * H * H + H)
        P = 4.0 * _network_size(d, H)
        return dict(bytes=P * (2 if c["grad"] else 1) + 4.0 * B * (d + 1), flops=mm * (3 if c["grad"] else 1))
    if kind == "batch":
        mean = (c["n_min"] + c["n_max"]) / 2
        modes = c["NP"] * sum((max(8, c["sides"] * k // 6) ** 3) / 2 for k in (2, 3, 4, 5, 6)) / 5
        return dict(bytes=8.0 * c["NP"] * (8 * c["K"] + 2) * c["generations"],
                    flops=STEP_FLOPS * modes * mean * c["generations"])
    modes, n = float(c["nx"] * c["ny"] * c["nz"]), c["n_steps"]
    if kind == "gradient":
        return dict(bytes=8.0 * c["starts"] * (12 * c["K"] + 2), flops=GRADIENT_FLOPS * modes * n * c["starts"])
    if kind in ("score", "gaussian"):
        cands = c.get("cands", 1)
        size = 8 if c["precision"] == "fp64" else 4
        out = cands * (1.0 + (modes if c.get("densities", True) else 0.0)) * size
        share = 0.625 if c.get("uneven") else 1.0
        return dict(bytes=16.0 * cands * (2 * n + 1) * share + out, flops=STEP_FLOPS * modes * n * cands * share)
    return dict(bytes=8.0 * c["NP"] * (8 * c["K"] + 2), flops=STEP_FLOPS * modes * n * c["NP"])


# ---------------------------------------------------------------------------------- 64-bit values


def _qmul(a, b):
    """Products of quaternions (w, x, y, z) stacked in the first dimension; 1, -i sigma_x,
    -i sigma_y, -i sigma_z multiply as 1, i, j, k."""
    return torch.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                        a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                        a[0] * b[2] + a[2] * b[0] + a[3] * b[1] - a[1] * b[3],
                        a[0] * b[3] + a[3] * b[0] + a[1] * b[2] - a[2] * b[1]])


def _one_plus(s, q):
    r = s * q
    r[0] += 1.0
    return r


def _expq(h):
    """exp(-i h.sigma) of pure quaternions h."""
    th = (h[1] ** 2 + h[2] ** 2 + h[3] ** 2).sqrt()
    r = h * torch.where(th > 0, torch.sin(th) / th, torch.ones_like(th))
    r[0] = torch.cos(th)
    return r


def _step(scheme, dt, h0, hm, h1):
    """One step's 2 x 2 propagator as a quaternion, from h at the step's start, middle and end."""
    if scheme == "rk4":
        k2 = _qmul(hm, _one_plus(0.5 * dt, h0))
        k3 = _qmul(hm, _one_plus(0.5 * dt, k2))
        k4 = _qmul(h1, _one_plus(dt, k3))
        return _one_plus(dt / 6.0, h0 + 2 * k2 + 2 * k3 + k4)
    cross = torch.stack([torch.zeros_like(h0[0]), h0[2] * h1[3] - h0[3] * h1[2], h0[3] * h1[1] - h0[1] * h1[3],
                         h0[1] * h1[2] - h0[2] * h1[1]])
    return _expq(dt * ((h0 + 4 * hm + h1) / 6.0 - dt / 6.0 * cross))


def _densities(A, n, dt, grid, scheme):
    """n(p) [nz][ny][nx] of one field A [2][2n+1]: the scheme's own step for each spin channel
    h = (p_x - A_x, +-(p_y - A_y), sqrt(1 + p_z^2)), the steps of a span multiplied as a tree."""
    dev = A.device
    ax = [torch.tensor(v, device=dev) for v in inputs.grid_axes(grid)]
    Z, Y, X = (v.reshape(-1) for v in torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij"))
    eps = (1.0 + Z * Z).sqrt()
    M = len(X)
    span = max(1, min(1024, int(6e6) // M))
    total = torch.zeros(M, dtype=torch.float64, device=dev)
    for s in (1.0, -1.0):
        def h(k):  # samples k [m] -> [4][m][M]
            a = A[:, k]
            P = X - a[0][:, None]
            return torch.stack([torch.zeros_like(P), P, s * (Y - a[1][:, None]), eps.expand_as(P)])
        U = torch.zeros((4, M), dtype=torch.float64, device=dev)
        U[0] = 1.0
        for lo in range(0, n, span):
            k = 2 * torch.arange(lo, min(n, lo + span), device=dev)
            if scheme == "split2":
                hm = h(k + 1)
                free = torch.stack([torch.zeros_like(X), X, s * Y, eps])[:, None]
                half = _expq(0.5 * dt * free)
                R = _qmul(half, _qmul(_expq(dt * (hm - free)), half))
            else:
                R = _step(scheme, dt, h(k), h(k + 1), h(k + 2))
            while R.shape[1] > 1:
                m = R.shape[1] // 2
                P = _qmul(R[:, 1:2 * m:2], R[:, 0:2 * m:2])
                R = torch.cat([P, R[:, 2 * m:]], 1) if R.shape[1] % 2 else P
            U = _qmul(R[:, 0], U)
        a = A[:, [0, 2 * n]]
        x, y = X - a[0, 0], s * (Y - a[1, 0])
        w = (x * x + y * y + eps * eps).sqrt()
        v = torch.stack([torch.complex(-x, y), torch.complex(w + eps, torch.zeros_like(w))]) / (2 * w * (w + eps)).sqrt()
        # (U0 - i (U.sigma)) v
        p0 = U[0] * v[0] - 1j * (U[3] * v[0] + torch.complex(U[1], -U[2]) * v[1])
        p1 = U[0] * v[1] - 1j * (torch.complex(U[1], U[2]) * v[0] - U[3] * v[1])
        x, y = X - a[0, 1], s * (Y - a[1, 1])
        w = (x * x + y * y + eps * eps).sqrt()
        amp = ((w + eps) * p0 + torch.complex(x, -y) * p1) / (2 * w * (w + eps)).sqrt()
        total += amp.real ** 2 + amp.imag ** 2
    return total.reshape(grid["nz"], grid["ny"], grid["nx"])


def _weights(v, mirror, dev):
    if len(v) == 1:
        return torch.ones(1, dtype=torch.float64, device=dev)
    w = torch.full((len(v),), float(v[-1] - v[0]) / (len(v) - 1), dtype=torch.float64, device=dev)
    w[0] *= 0.5
    w[-1] *= 0.5
    return 2.0 * w if mirror else w


def _network_exact(c, seed, dev):
    flat, X, t = (v.double() for v in _network_inputs(c, seed, dev))
    flat.requires_grad_(c["grad"])
    d, H, at, a = c["d_in"], NET["hidden"], 0, X
    for fan in (d, H, H):
        W = flat[at:at + H * fan].reshape(H, fan)
        b = flat[at + H * fan:at + H * fan + H]
        a = torch.nn.functional.gelu(a @ W.T + b)
        at += H * fan + H
    y = a @ flat[at:at + H] + flat[at + H]
    if not c["grad"]:
        return [y]
    loss = ((y - t) ** 2).mean()
    g, = torch.autograd.grad(loss, flat)
    return [loss.detach().reshape(1), g]


def exact(case, seed):
    """run()'s values in 64 bits; None for the kinds that select (a search's state) and for the
    kinetic equation's gradient, and where the scheme's steps would take too long."""
    c = case
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "network":
        return _network_exact(c, seed, dev)
    if c["kind"] not in ("score", "gaussian"):
        return None
    if c.get("cands", 1) * c["nx"] * c["ny"] * c["nz"] * c["n_steps"] > 5e9:
        return None
    A, steps = _score_inputs(c, seed, dev)
    grid = _one_axis(_grid(c))
    ax = inputs.grid_axes(grid)
    W = (_weights(ax[2], True, dev)[:, None, None] * _weights(ax[1], False, dev)[:, None]
         * _weights(ax[0], False, dev))
    n = torch.stack([_densities(A[i], m, _dt(c), grid, c["scheme"]) for i, m in enumerate(steps)])
    N = (n * W).sum((1, 2, 3))
    return [N, n] if c.get("densities", True) else [N]
