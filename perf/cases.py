"""The work that users of this library have it do, as cases that can be timed.

A case is a dict of plain values; ``prepare`` makes what a program has in hand
before the call (training data, scene, controller, device buffers) from a seed,
``run`` makes one pass through the public entry points, ``work`` counts what a
pass cannot do without, and ``exact`` evaluates the same definition in 64 bits
with plain torch.

Keys: call (step, host, refit, predict, grad, batch), precision (fp32, fp16,
bf16, bf16x3: the arithmetic of the GP variance), K samples, T steps, N
training points, O obstacles, path (eight, sine, straight), terrains (number of
terrain GPs mixed by Eq. 3; 1 = the single GP), nominal (variance mode of
Alg. 1 Step 2), lam (MPPI temperature), M (queries), B (controllers), shapes
(what a batch's sizes are drawn from).
"""
import math

import numpy as np
import torch

import paper_2411_03289_gb300 as gp

PRECISION = {"fp32": gp.GPMPPI_FP32, "bf16": gp.GPMPPI_BF16_SPLIT, "fp16": gp.GPMPPI_FP16_SPLIT,
             "bf16x3": gp.GPMPPI_BF16_SPLIT3}

# the robot's operating box: (v, omega, v_cmd, omega_cmd)
BOX_LO = np.array([0.0, -1.5, 0.0, -1.5])
BOX_HI = np.array([2.0, 1.5, 2.0, 1.5])
TERRAIN = ((0.10, 0.20, 0.00), (0.15, 0.30, 0.05), (0.05, 0.10, 0.00), (0.10, 0.15, 0.02))
TERRAIN_ELL = (0.5, 0.6, 0.45, 0.55)
TERRAIN_SF2 = (0.1, 0.08, 0.12, 0.1)
TERRAIN_W = (0.4, 0.3, 0.2, 0.1)
SLOPE = 20.0


def _step(name, **kw):
    c = dict(name=name, call="step", precision="fp32", K=1024, T=20, N=200, O=8, path="eight", terrains=1,
             nominal=False)
    c.update(kw)
    c["lam"] = c["T"] / 10.0      # the costs add up over the horizon, the temperature goes with them
    return c


def listed():
    return [
        # a small robot's control loop: few samples, few training points; latency
        _step("step_small", K=256, T=20, N=50, O=4, path="straight"),
        # the paper's workload (Sec. V sizes) in the library's default arithmetic
        _step("step_fp32", K=4096, T=50, N=500, O=16),
        # the same on the tensor cores: the benchmark's headline
        _step("step_fp16", K=4096, T=50, N=500, O=16, precision="fp16"),
        # a long horizon over a large training set and a crowded scene
        _step("step_fp16_large", K=16384, T=100, N=2048, O=64, precision="fp16"),
        # Alg. 1 with its Step 2 (the covariance along the update tightens the next call)
        _step("step_nominal", K=2500, T=45, N=350, O=11, path="sine", precision="fp16", nominal=True),
        # a receding-horizon loop with its arrays on the host; odd sizes, the 24-bit split
        _step("step_host", call="host", K=1500, T=37, N=777, O=9, path="sine", precision="bf16x3"),
        # terrain ensembles (Eq. 3) in the default arithmetic and on the tensor cores
        _step("terrain_fp32", K=2048, T=40, N=400, O=12, terrains=3),
        _step("terrain_fp16", K=4096, T=50, N=500, O=16, terrains=3, precision="fp16"),
        # learning through the rollout: the smoothed cost with both of its gradients
        _step("grad", call="grad", K=4096, T=50, N=1000, O=16),
        # a fleet: eight unequal controllers a step, through the replayed graph
        dict(name="batch", call="batch", B=8, shapes=7),
        # a refit on new data, and its posterior over the last steps' inputs
        dict(name="refit", call="refit", N=1500, M=200),
        # the posterior over a large set of queries (maps, Eq. 4's regressors)
        dict(name="predict", call="predict", N=1000, M=20000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "host", "terrain", "grad", "batch", "refit", "predict"])
    if call == "refit":
        return dict(call="refit", N=_log_int(rng, 40, 2500), M=_log_int(rng, 1, 2000))
    if call == "predict":
        return dict(call="predict", N=_log_int(rng, 30, 3000), M=_log_int(rng, 1, 30000))
    if call == "batch":
        return dict(call="batch", B=rng.randint(2, 8), shapes=rng.randint(0, 99999))
    while True:
        c = _step("", K=_log_int(rng, 64, 16384), T=rng.randint(5, 100), N=_log_int(rng, 20, 2500),
                  O=rng.randint(0, 64), path=rng.choice(["eight", "sine", "straight"]))
        del c["name"]
        c["precision"] = rng.choice(["fp32", "fp16", "fp16", "bf16x3"])
        if call == "host":
            c["call"] = "host"
        elif call == "terrain":
            c["terrains"] = rng.randint(2, 4)
            c["N"] = min(c["N"], 1500 // c["terrains"])      # their sets share one CTA's memory
        elif call == "grad":
            c.update(call="grad", precision="fp32", N=min(c["N"], 1500))
        else:
            c["nominal"] = rng.random() < 0.2
        # no more than the largest listed case: the FP32 path and the adjoint do
        # the same contraction at a fraction of the tensor cores' rate
        slow = 16.0 if c["precision"] == "fp32" else 2.0 if c["precision"] == "bf16x3" else 1.0
        if c["call"] == "grad":
            slow *= 3.0
        if slow * c["K"] * c["T"] * c["terrains"] * float(c["N"]) ** 2 <= 16384 * 100 * 2048.0 ** 2:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class Hyper:
    def __init__(self, ell, sf2):
        self.lengthscale, self.signal_var, self.noise_var = (ell,) * 4, sf2, 1e-4


class Params:
    """gpmppi_params of one controller."""

    def __init__(self, c, seed):
        self.K, self.T = c["K"], c["T"]
        self.dt, self.tau_v, self.tau_w = 0.05, 0.3, 0.2
        self.sigma = (0.5, 0.8)
        self.lam, self.p_x = c["lam"], 0.95
        self.u_min, self.u_max = (0.0, -1.5), (2.0, 1.5)
        self.alpha, self.beta = (1.0, 1.0, 0.0, 1.0, 0.5), (0.0, 1.0, 0.0, 0.0)
        self.P_lane, self.P_coll = 100.0, 1000.0
        # a corridor of six metres: its edge is where few of the samples that count go
        self.lane_half_width, self.v_desired = 3.0, 1.5
        self.seed = seed
        self.variance_mode = gp.GPMPPI_VAR_NOMINAL if c["nominal"] else gp.GPMPPI_VAR_PER_SAMPLE
        self.precision = PRECISION[c["precision"]]
        self.goal, self.goal_radius, self.P_goal = (0.0, 0.0), 0.5, 100.0


def _training_set(rng, N, terrain):
    """Noisy velocity residuals of one terrain over the operating box."""
    a, b, d = TERRAIN[terrain]
    X = BOX_LO + (BOX_HI - BOX_LO) * rng.random((N, 4))
    Y = np.stack([-a * X[:, 0] * np.abs(X[:, 1]) - d * X[:, 0], -b * X[:, 1] * X[:, 0]], axis=1)
    return X, Y + 0.01 * rng.standard_normal((N, 2)), (Hyper(TERRAIN_ELL[terrain], TERRAIN_SF2[terrain]),) * 2


def _path(kind):
    if kind == "straight":
        return np.array([[0.0, 0.0], [20.0, 0.0]])
    if kind == "eight":
        t = np.linspace(0.0, 2.0 * np.pi, 512)
        p = 5.0 * np.stack([np.sin(t), np.sin(t) * np.cos(t)], axis=1)
        p[-1] = p[0]
        return p
    x = np.linspace(0.0, 40.0, 512)
    return np.stack([x, 2.0 * np.sin(0.2 * np.pi * x)], axis=1)


def _inputs(c, seed):
    """Everything of one controller, on the host: training sets, scene, state, controls."""
    rng = np.random.Generator(np.random.PCG64(seed))
    sets = [_training_set(rng, c["N"], t) for t in range(c["terrains"])]
    path = _path(c["path"])
    i = int(rng.integers(0, max(1, len(path) // 2)))
    d = path[i + 1] - path[i]
    x0 = np.array([path[i, 0], path[i, 1], math.atan2(d[1], d[0]) + 0.1 * rng.standard_normal(),
                   0.7 + 0.8 * rng.random(), 0.2 * rng.standard_normal()])
    dense = path if len(path) > 2 else np.stack([np.linspace(0.0, 20.0, 201), np.zeros(201)], axis=1)
    obst = []
    while len(obst) < c["O"]:                # circles beside the lane, away from the robot
        o = path[i] + rng.uniform(-9.0, 9.0, 2)
        if np.min(np.hypot(*(dense - o).T)) > 0.7:
            obst.append([o[0], o[1], 0.2 + 0.4 * rng.random()])
    U = np.stack([1.5 + 0.1 * rng.standard_normal(c["T"]),
                  0.3 * np.sin(0.1 * np.arange(c["T"]) + 6.28 * rng.random())], axis=1)
    w = np.array(TERRAIN_W[:c["terrains"]])
    return dict(sets=sets, path=path.astype(np.float32), x0=x0.astype(np.float32),
                obst=np.array(obst, dtype=np.float32).reshape(-1, 3), U=U.astype(np.float32),
                w=(w / w.sum()).astype(np.float32), params=Params(c, int(rng.integers(0, 2 ** 62))),
                it=int(rng.integers(0, 2 ** 40)))


def _controller(i):
    gps = [gp.gp_fit(*s) for s in i["sets"]]
    if len(gps) > 1:
        ctrl = gp.mppi_create_ensemble(i["params"], i["obst"], i["path"], gps, i["w"])
    else:
        ctrl = gp.mppi_create(i["params"], i["obst"], i["path"], gps[0])
    gp.mppi_set_iteration(ctrl, i["it"])
    return ctrl


def _fleet(c):
    """The controllers of a batch: sizes from the case, alternating paths, the
    arithmetics in the proportions of a mixed fleet."""
    rng = np.random.Generator(np.random.PCG64(c["shapes"]))
    out = []
    for b in range(c["B"]):
        out.append(_step("", K=int(rng.integers(256, 6000)), T=int(rng.integers(20, 80)),
                         N=int(math.exp(rng.uniform(math.log(100.0), math.log(2500.0)))),
                         O=int(rng.integers(4, 65)), path="sine" if b % 2 == 0 else "eight",
                         precision=("fp16", "fp16", "bf16x3", "fp32")[b % 4]))
    return out


def prepare(case, seed):
    c, s = case, {"call": case["call"]}
    if c["call"] in ("refit", "predict"):
        rng = np.random.Generator(np.random.PCG64(seed))
        s["set"] = _training_set(rng, c["N"], 0)
        Z = (BOX_LO + (BOX_HI - BOX_LO) * rng.random((c["M"], 4))).astype(np.float32)
        s["Z"] = torch.tensor(Z, device="cuda")
        s["mean"] = torch.empty(c["M"], 2, device="cuda")
        s["var"] = torch.empty(c["M"], 2, device="cuda")
        if c["call"] == "predict":
            s["gp"] = gp.gp_fit(*s["set"])
        return s
    if c["call"] == "batch":
        ins = [_inputs(m, seed * 64 + b) for b, m in enumerate(_fleet(c))]
        s["batch"] = gp.mppi_batch_create([_controller(i) for i in ins])
        for b, i in enumerate(ins):
            s["batch"].state[b].copy_(torch.tensor(i["x0"]))
            s["batch"].U_nom[b].copy_(torch.tensor(i["U"]))
        s["stream"] = torch.cuda.Stream()
        gp.mppi_batch_autotune(s["batch"], s["stream"])
        torch.cuda.synchronize()
        return s
    i = _inputs(c, seed)
    s["ctrl"], s["x0"], K, T = _controller(i), i["x0"], c["K"], c["T"]
    if c["call"] == "host":
        s["U"] = torch.tensor(i["U"]).pin_memory()
        s["U_new"], s["weights"] = torch.empty(T, 2).pin_memory(), torch.empty(K).pin_memory()
        return s
    s["U"] = torch.tensor(i["U"], device="cuda")
    if c["call"] == "grad":
        s["J"] = torch.empty(1, device="cuda")
        s["dU"], s["dl"] = torch.empty(T, 2, device="cuda"), torch.empty(2, 4, device="cuda")
        return s
    s["U_new"], s["weights"] = torch.empty(T, 2, device="cuda"), torch.empty(K, device="cuda")
    s["sxy"] = torch.empty(T, 3, device="cuda") if c["nominal"] else None
    return s


def run(state):
    s = state
    if s["call"] == "step":
        gp.mppi_step(s["ctrl"], s["x0"], s["U"], s["U_new"], s["weights"])
        if s["sxy"] is None:
            return s["U_new"], s["weights"]
        gp.mppi_nominal_sxy(s["ctrl"], s["sxy"])
        return s["U_new"], s["weights"], s["sxy"]
    if s["call"] == "host":
        gp.mppi_step_host(s["ctrl"], s["x0"], s["U"], s["U_new"], s["weights"])
        return s["U_new"], s["weights"]
    if s["call"] == "grad":
        return gp.mppi_grad(s["ctrl"], s["x0"], s["U"], SLOPE, None, s["J"], s["dU"], s["dl"])
    if s["call"] == "batch":
        gp.mppi_batch_graph(s["batch"], s["stream"])
        # the results live in the batch's buffers, which go with it: take them out
        # behind the step, as a program does before it writes the next controls
        with torch.cuda.stream(s["stream"]):
            return [u.clone() for u in s["batch"].U_new], [w.clone() for w in s["batch"].weights]
    g = gp.gp_fit(*s["set"]) if s["call"] == "refit" else s["gp"]
    gp.gp_predict(g, s["Z"], s["mean"], s["var"])
    return s["mean"], s["var"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _rollout_work(c):
    q, N, M = c["K"] * c["T"], c["N"], c["terrains"]
    per = M * (N * (N + 1.0) + 16.0 * N) + 15.0 * c["O"] + 10.0 * (1 if c["path"] == "straight" else 25) + 150.0
    byts = M * 4.0 * (N * (N + 1) / 2 + 6 * N) + 4.0 * (2 * 2 * c["T"] + c["K"])
    return byts, q * per


def work(case):
    c = case
    if c["call"] == "refit":
        N, M = float(c["N"]), c["M"]
        return {"bytes": 8.0 * 6 * N + 4.0 * 8 * M, "flops": 2.0 * N ** 3 / 3 + 40.0 * N * N + M * (N * (N + 1) + 16 * N)}
    if c["call"] == "predict":
        N, M = float(c["N"]), c["M"]
        return {"bytes": 4.0 * (N * (N + 1) / 2 + 6 * N) + 4.0 * 8 * M, "flops": M * (N * (N + 1) + 16 * N)}
    if c["call"] == "batch":
        w = [_rollout_work(m) for m in _fleet(c)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    byts, flops = _rollout_work(c)
    if c["call"] == "grad":
        # the second triangular product, the adjoint row, and the symmetric Gram
        # sums of the lengthscale gradient (one triangle for each output)
        q, N = c["K"] * c["T"], c["N"]
        flops += q * (N * (N + 1.0) + 60.0 * N + 2.0 * N * (N + 1.0) + 400.0)
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same definitions in 64 bits (Eq. 1-16 and Alg. 1), plain torch
# ---------------------------------------------------------------------------

def _d(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda")


def _f(x):
    return float(np.float32(x))


class _Posterior:
    """One output's GP: k, alpha = K^-1 y and L^-1, differentiable in the lengthscales."""

    def __init__(self, X, y, ell, sf2, sn2):
        self.X, self.ell, self.sf2 = X, ell, sf2
        K = self.k(X) + sn2 * torch.eye(len(X), dtype=torch.float64, device=X.device)
        L = torch.linalg.cholesky(K)
        eye = torch.eye(len(X), dtype=torch.float64, device=X.device)
        self.Linv = torch.linalg.solve_triangular(L, eye, upper=False)
        self.alpha = self.Linv.T @ (self.Linv @ y)

    def k(self, Z):
        return self.sf2 * torch.exp(-0.5 * sum(((Z[:, None, d] - self.X[None, :, d]) / self.ell[d]) ** 2
                                               for d in range(4)))

    def __call__(self, Z):
        k = self.k(Z)
        return k @ self.alpha, (self.sf2 - ((k @ self.Linv.T) ** 2).sum(1)).clamp(min=0.0)


def _fit(data, ell=None):
    X, Y, h = data
    X, Y = _d(X), _d(Y)
    same = ell is None                       # both outputs share their hyper-parameters
    a = _Posterior(X, Y[:, 0] if not same else Y, _d(h[0].lengthscale) if same else ell[0], h[0].signal_var,
                   h[0].noise_var)
    return (a, None) if same else (a, _Posterior(X, Y[:, 1], ell[1], h[1].signal_var, h[1].noise_var))


def _predict(fit, Z):
    """(mean (Q, 2), variance (Q, 2))."""
    if fit[1] is None:
        m, v = fit[0](Z)
        return m, torch.stack([v, v], 1)
    a, b = fit[0](Z), fit[1](Z)
    return torch.stack([a[0], b[0]], 1), torch.stack([a[1], b[1]], 1)


def _noise(P, k, it):
    """Philox4x32-10 (Salmon et al., SC'11) at counters (k, s, it), then Box-Muller."""
    m32 = 0xFFFFFFFF
    full = lambda v: torch.full((P.K,), v, dtype=torch.int64, device="cuda")  # noqa: E731

    def mul(a, b):                            # (high, low) words of a 32 x 32-bit product
        lo = (a & 0xFFFF) * b
        hi = (a >> 16) * b
        s = (lo >> 16) + (hi & 0xFFFF)
        return (hi >> 16) + (s >> 16), ((s << 16) | (lo & 0xFFFF)) & m32

    c = [full(k), torch.arange(P.K, device="cuda"), full(it & m32), full(it >> 32)]
    k0, k1 = P.seed & m32, P.seed >> 32
    for r in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u = [(w.double() + 0.5) * 2.0 ** -32 for w in c[:2]]
    r = torch.sqrt(-2.0 * torch.log(u[0]))
    return torch.stack([_f(P.sigma[0]) * r * torch.cos(2 * math.pi * u[1]),
                        _f(P.sigma[1]) * r * torch.sin(2 * math.pi * u[1])], 1)


def _sqrt(x):
    """sqrt with derivative zero at zero."""
    pos = x > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, x, torch.ones_like(x))), torch.zeros_like(x))


def _lane_distance(p, path):
    a, ab = path[:-1], path[1:] - path[:-1]
    ap = p[:, None, :] - a[None]
    t = ((ap * ab).sum(-1) / (ab * ab).sum(-1)).clamp(0.0, 1.0)
    with torch.no_grad():
        j = ((ap - t[..., None] * ab) ** 2).sum(-1).argmin(1)
    r = torch.arange(len(p), device=p.device)
    return _sqrt(((ap[r, j] - t[r, j][:, None] * ab[j]) ** 2).sum(-1))


def _rollout(i, fits, U, samples=True, slope=None, sxy=None):
    """Costs (K,) and clamped controls (T, K, 2) of the sampled rollouts, and
    Sigma_XY (T, 3) of the first trajectory.  samples False: the one noise-free
    trajectory; slope: sigmoids for the indicators; sxy (T, 3): tightening
    covariance in place of each sample's own."""
    P = i["params"]
    n = P.K if samples else 1
    dt, tv, tw = _f(P.dt), _f(P.tau_v), _f(P.tau_w)
    p_x, r, vd = _f(P.p_x), _f(P.lane_half_width), _f(P.v_desired)
    chi = math.sqrt(-2.0 * math.log1p(-p_x))
    phi = float(torch.special.ndtri(torch.tensor(p_x, dtype=torch.float64)))
    path, obst, w = _d(i["path"]), _d(i["obst"]), _d(i["w"])
    lo, hi = _d(np.float32(P.u_min)), _d(np.float32(P.u_max))
    ind = (lambda m: (m > 0).double()) if slope is None else (lambda m: torch.sigmoid(slope * m))
    X, Y, th, v, om = (torch.full((n,), float(x), dtype=torch.float64, device="cuda") for x in i["x0"])
    S = torch.zeros(n, 5, 5, dtype=torch.float64, device="cuda")
    cost, uts, rec = torch.zeros(n, dtype=torch.float64, device="cuda"), [], []
    for k in range(P.T):
        u = U[k][None].expand(n, 2)
        u = torch.minimum(torch.maximum(u + _noise(P, k, i["it"]) if samples else u, lo), hi)
        uts.append(u)
        z = torch.stack([v, om, u[:, 0], u[:, 1]], 1)
        got = [_predict(f, z) for f in fits]
        m = sum(wt * g[0] for wt, g in zip(w, got)) if len(got) > 1 else got[0][0]
        var = sum(wt * wt * g[1] for wt, g in zip(w, got)) if len(got) > 1 else got[0][1]
        cs, sn, one, zero = torch.cos(th), torch.sin(th), torch.ones_like(v), torch.zeros_like(v)
        A = torch.stack([torch.stack(row, -1) for row in (
            (one, zero, -dt * v * sn, dt * cs, zero), (zero, one, dt * v * cs, dt * sn, zero),
            (zero, zero, one, zero, dt * one), (zero, zero, zero, (1 - dt / tv) * one, zero),
            (zero, zero, zero, zero, (1 - dt / tw) * one))], -2)
        X, Y, th, v, om = (X + dt * v * cs, Y + dt * v * sn, th + dt * om, v + dt / tv * (u[:, 0] - v) + m[:, 0],
                           om + dt / tw * (u[:, 1] - om) + m[:, 1])
        S = A @ S @ A.transpose(-1, -2) + torch.diag_embed(torch.stack([zero, zero, zero, var[:, 0], var[:, 1]], -1))
        xx, xy, yy = (S[:, 0, 0], S[:, 0, 1], S[:, 1, 1]) if sxy is None else (sxy[k, j] * one for j in range(3))
        rec.append(torch.stack([S[0, 0, 0], S[0, 0, 1], S[0, 1, 1]]))
        lam = _sqrt((0.5 * (xx + yy) + _sqrt((0.5 * (xx - yy)) ** 2 + xy ** 2)).clamp(min=0.0))
        p = torch.stack([X, Y], 1)
        e = _lane_distance(p, path)
        c = P.alpha[0] * var.sum(1) + P.alpha[1] * e / r + P.alpha[4] * (vd - v) ** 2
        c = c + P.alpha[3] * P.P_lane * 0.9 ** k * ind(e - (r - chi * lam))
        if len(obst):
            d = p[:, None, :] - obst[None, :, :2]
            rho = torch.sqrt((d * d).sum(-1)).clamp(min=1e-9)
            nx, ny = d[..., 0] / rho, d[..., 1] / rho
            sp = _sqrt((nx * nx * xx[:, None] + 2 * nx * ny * xy[:, None] + ny * ny * yy[:, None]).clamp(min=0.0))
            c = c + P.beta[1] * P.P_coll * ind(-(rho - obst[:, 2] - phi * sp).min(1).values)
        cost = cost + c
    return cost, torch.stack(uts), torch.stack(rec)


def exact(case, seed):
    c = case
    if c["call"] in ("refit", "predict"):
        rng = np.random.Generator(np.random.PCG64(seed))
        data = _training_set(rng, c["N"], 0)
        Z = (BOX_LO + (BOX_HI - BOX_LO) * rng.random((c["M"], 4))).astype(np.float32)
        fit = _fit(data)
        return tuple(torch.cat(x) for x in zip(*(_predict(fit, q) for q in _d(Z).split(4096))))
    # 64-bit products over the largest cases and over a whole fleet take minutes
    if c["call"] == "batch" or c["K"] * c["T"] * c["terrains"] * float(c["N"]) ** 2 > 1.5e12:
        return None
    i = _inputs(c, seed)
    U = _d(i["U"])
    if c["call"] == "grad":
        U.requires_grad_(True)
        ell = [_d(h.lengthscale).requires_grad_(True) for h in i["sets"][0][2]]
        J = _rollout(i, [_fit(i["sets"][0], ell)], U, slope=SLOPE)[0].mean()
        J.backward()
        return J.detach().reshape(1), U.grad, torch.stack([ell[0].grad, ell[1].grad])
    with torch.no_grad():
        fits = [_fit(s) for s in i["sets"]]
        zero = torch.zeros(c["T"], 3, dtype=torch.float64, device="cuda")
        cost, ut, _ = _rollout(i, fits, U, sxy=zero if c["nominal"] else None)
        w = torch.softmax(-cost / _f(c["lam"]), 0)
        U_new = U + (w[None, :, None] * (ut - U[:, None, :])).sum(1)
        if c["nominal"]:
            return U_new, w, _rollout(i, fits, U_new, samples=False)[2]
        return U_new, w
