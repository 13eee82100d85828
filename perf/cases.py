"""The analyses whose speed is measured, each through the public entry points.

One case is one analysis (mean and perturbation update) of one ensemble and one
observation network, one batched call over many of them, or one training step
of the learned preconditioner.  The sizes are those of the workload generators
(``paper_2503_00253_gb300.workloads``), the tests and the benchmark; ``draw``
spreads them over the ranges between.

The caller is a cycling data-assimilation program: it keeps its options, its
workspace and output buffers, asks for no statistics (so a call returns
once its work is queued), and hands the analysis back to its forecast model.
A program that asks for the single-precision or BF16 solver runs that model in
single precision, so those analyses are returned as float32; the FP64 solver's
are returned as they are.

Families (``kind``):
  gauss1d   Gaussian forecast on a circle, every ``stride``-th point observed
  layered   layered Lorenz-96 forecast, random observations
  gauss2d   Gaussian forecast on a torus, observations on a lattice (BF16 path)
  batch     uneven 1-D problems in one call
  channels  weighted-sum observations (CSR) on a circle
  train     loss and gradient of the learned preconditioner's network
"""
import math

import numpy as np
import torch

from paper_2503_00253_gb300 import binding as B
from paper_2503_00253_gb300 import learned, workloads

DEV = "cuda"
PRECISION = {"fp64": B.PRECISION_FP64, "fp32": B.PRECISION_FP32, "bf16": B.PRECISION_BF16}
SOLVER = {"pcg": B.SOLVER_PCG, "multishift": B.SOLVER_MULTISHIFT}


def gauss1d(n, members, stride, length, r2, half_width, nodes, tol, precision, solver="pcg", model=False, offset=0):
    return dict(kind="gauss1d", n=n, members=members, stride=stride, length=length, r2=r2, half_width=half_width,
                nodes=nodes, tol=tol, precision=precision, solver=solver, model=model, offset=offset)


def layered(nx, nz, members, fraction, cx, cz, nodes, tol, precision):
    return dict(kind="layered", nx=nx, nz=nz, members=members, fraction=fraction, r2=1.0, cx=cx, cz=cz, nodes=nodes,
                tol=tol, precision=precision, solver="pcg")


def gauss2d(nx, ny, members, stride, length, half_width, nodes, tol):
    return dict(kind="gauss2d", nx=nx, ny=ny, members=members, stride=stride, length=length, r2=0.5,
                half_width=half_width, nodes=nodes, tol=tol, precision="bf16", solver="pcg")


def batch(count, n_min, n_max, sizes, tol, precision):
    return dict(kind="batch", count=count, n_min=n_min, n_max=n_max, sizes=sizes, tol=tol, precision=precision,
                solver="pcg")


def channels(n, d, members, bandwidth, length, nodes, tol, precision):
    return dict(kind="channels", n=n, d=d, members=members, bandwidth=bandwidth, length=length, nodes=nodes, tol=tol,
                precision=precision, solver="pcg")


def train(samples, d):
    return dict(kind="train", samples=samples, d=d)


def listed():
    cases = [
        # The smallest: a toy-model cycle in FP64; launches and dependent steps are all of its time.
        ("gauss1d_240_fp64", gauss1d(240, 20, 4, 10.0, 0.5, 20.0, 16, 1e-12, "fp64")),
        # The benchmark's network with the paper's preconditioner, single precision.
        ("gauss1d_8192_fp32", gauss1d(8192, 40, 8, 64.0, 0.25, 256.0, 32, 1e-6, "fp32")),
        # The same with the trained correction: the benchmark's own analysis.
        ("gauss1d_8192_learned", gauss1d(8192, 40, 8, 64.0, 0.25, 256.0, 32, 1e-6, "fp32", model=True)),
        # The same by multi-shift CG, the solver for well-conditioned networks.
        ("gauss1d_8192_multishift", gauss1d(8192, 40, 8, 64.0, 0.25, 256.0, 32, 1e-6, "fp32", "multishift")),
        # The same in double precision to its own tolerance: the reference run of a precision study.
        ("gauss1d_8192_fp64", gauss1d(8192, 40, 8, 64.0, 0.25, 256.0, 32, 1e-12, "fp64")),
        # One cycle of the layered Lorenz-96 experiment with 25 % random observations, single precision.
        ("layered_7680_fp32", layered(960, 8, 40, 0.25, 60.0, 2.0, 24, 1e-6, "fp32")),
        # The same on the BF16 tensor-core path.
        ("layered_7680_bf16", layered(960, 8, 40, 0.25, 60.0, 2.0, 24, 1e-6, "bf16")),
        # A small 2-D grid: few systems, so each iteration's latency counts.
        ("gauss2d_128_bf16", gauss2d(128, 128, 16, 2, 8.0, 12.0, 8, 1e-6)),
        # A regional 2-D grid, the largest state here: the tensor-core products are most of its time.
        ("gauss2d_512_bf16", gauss2d(512, 512, 80, 2, 32.0, 48.0, 8, 1e-6)),
        # Serving: 64 uneven problems (1k to 65k points) in one call.
        ("batch_64_fp32", batch(64, 1024, 65536, 4, 1e-6, "fp32")),
        # The single-cycle experiment: Gaussian channel sums observed, dense covariances.
        ("channels_2000_fp64", channels(2000, 100, 20, 10.0, 12.0, 8, 1e-12, "fp64")),
        # One training step on the samples of one training problem of the benchmark (12 x 3 x 32).
        ("train_1152", train(1152, 1024)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["gauss1d", "gauss1d", "gauss1d", "layered", "layered", "gauss2d", "batch", "channels", "train"])
    if kind == "gauss1d":
        form = rng.choice(["fp64", "fp32", "learned", "multishift", "multishift64"])
        n = int(_log(rng, 240, 12000))
        stride = rng.randint(4, 16)
        reach = _log(rng, 16.0, 256.0) if n >= 2048 else rng.uniform(10.0, 30.0)   # half-width in grid points
        fp64 = form.endswith("64")
        return gauss1d(n, rng.choice([20, 33, 40, 64, 80]), stride, reach / 4.0, rng.choice([0.25, 0.5, 1.0]), reach,
                       rng.randint(16, 48), 1e-12 if fp64 else 1e-6, "fp64" if fp64 else "fp32",
                       "multishift" if form.startswith("multishift") else "pcg", form == "learned",
                       rng.randrange(stride))
    if kind == "layered":
        return layered(int(_log(rng, 90, 960)), rng.randint(2, 8), rng.choice([20, 31, 40]), rng.uniform(0.1, 0.3),
                       rng.uniform(10.0, 60.0), 2.0, rng.randint(8, 24), 1e-6, rng.choice(["fp32", "bf16"]))
    if kind == "gauss2d":
        nx, ny = (2 * int(_log(rng, 32, 192)) for _ in "xy")
        return gauss2d(nx, ny, rng.choice([16, 20, 40, 80]), 2, min(nx, ny) / 16.0, min(nx, ny) / 10.7,
                       rng.randint(6, 16), 1e-6)
    if kind == "batch":
        return batch(rng.randint(3, 40), 1024, int(_log(rng, 4096, 65536)), rng.randrange(1 << 20), 1e-6,
                     rng.choice(["fp32", "fp32", "fp64"]))
    if kind == "channels":
        n = int(_log(rng, 400, 2000))
        return channels(n, max(20, n // rng.randint(15, 25)), rng.choice([20, 27, 40]), rng.uniform(5.0, 10.0), 12.0,
                        rng.randint(8, 24), 1e-12, "fp64")
    return train(12 * rng.randint(8, 200), int(_log(rng, 240, 2048)))


# ---------------------------------------------------------------------------
# Inputs: Gaussian forecasts by FFT, the layered model by RK4, all on the GPU
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _chordal(delta, n):
    return (n / math.pi) * torch.sin(math.pi * delta.abs() / n)


def _forecast1d(n, members, length, g):
    row = torch.exp(-_chordal(torch.arange(n, device=DEV, dtype=torch.float64), n) ** 2 / (2.0 * length ** 2))
    row[0] += 1e-4
    lam = torch.fft.fft(row).real.clamp_min(0.0)
    xi = torch.randn(members + 1, n, device=DEV, dtype=torch.float64, generator=g)
    return torch.fft.ifft(lam.sqrt() * torch.fft.fft(xi), dim=1).real.contiguous()


def _forecast2d(nx, ny, members, length, g):
    cx = _chordal(torch.arange(nx, device=DEV, dtype=torch.float64), nx)
    cy = _chordal(torch.arange(ny, device=DEV, dtype=torch.float64), ny)
    row = torch.exp(-(cy[:, None] ** 2 + cx[None, :] ** 2) / (2.0 * length ** 2))
    row[0, 0] += 1e-4
    root = torch.fft.fft2(row).real.clamp_min(0.0).sqrt()
    out = torch.empty(members + 1, ny * nx, device=DEV, dtype=torch.float64)
    for k in range(members + 1):
        xi = torch.randn(ny, nx, device=DEV, dtype=torch.float64, generator=g)
        out[k] = torch.fft.ifft2(root * torch.fft.fft2(xi)).real.reshape(-1)
    return out


def _layered_forecast(nx, nz, members, g, steps=300, dt=0.01, force=8.0):
    def tendency(x):
        dx = torch.roll(x, 1, -1) * (torch.roll(x, -1, -1) - torch.roll(x, 2, -1)) - x + force
        dz = x[:, 1:] - x[:, :-1]
        dx[:, :-1] += dz
        dx[:, 1:] -= dz
        return dx

    x = force + torch.randn(members + 1, nz, nx, device=DEV, dtype=torch.float64, generator=g)
    for _ in range(steps):
        k1 = tendency(x)
        k2 = tendency(x + 0.5 * dt * k1)
        k3 = tendency(x + 0.5 * dt * k2)
        k4 = tendency(x + dt * k3)
        x = x + (dt / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return x.reshape(members + 1, nz * nx).contiguous()


def _problem(grid, draws, obs, r2, nodes, tol, g):
    """Forecast members, and observations of one more draw (the truth) with variance r2."""
    R = torch.full((obs.numel(),), float(r2), device=DEV, dtype=torch.float64)
    y = draws[-1][obs] + math.sqrt(r2) * torch.randn(obs.numel(), device=DEV, dtype=torch.float64, generator=g)
    return dict(grid=grid, X=draws[:-1].contiguous(), obs_idx=obs, y=y, R=R, Q=nodes, tol=tol)


def _problem1d(n, members, stride, length, r2, half_width, nodes, tol, offset, seed):
    g = _gen(seed)
    obs = torch.arange(offset % stride, n, stride, device=DEV, dtype=torch.int64)
    grid = workloads.Grid((n, 1, 1), (True, False, False), (half_width, 1.0, 1.0), True)
    return _problem(grid, _forecast1d(n, members, length, g), obs, r2, nodes, tol, g)


def _sizes(case):
    """The (n, members, stride, nodes) of a batch's problems: fixed by the case, not by the seed."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        out.append((n, int(rng.choice([20, 40, 80])), int(rng.integers(4, 17)), int(rng.integers(16, 49))))
    return out


def _problems(case, seed):
    kind = case["kind"]
    if kind == "gauss1d":
        return [_problem1d(case["n"], case["members"], case["stride"], case["length"], case["r2"], case["half_width"],
                           case["nodes"], case["tol"], case["offset"], seed)]
    if kind == "batch":
        return [_problem1d(n, N, stride, 16.0, 0.5, 64.0, Q, case["tol"], 0, 1000003 * int(seed) + i)
                for i, (n, N, stride, Q) in enumerate(_sizes(case))]
    g = _gen(seed)
    if kind == "layered":
        nx, nz = case["nx"], case["nz"]
        draws = _layered_forecast(nx, nz, case["members"], g)
        d = max(1, int(round(case["fraction"] * nx * nz)))
        obs = torch.randperm(nx * nz, device=DEV, generator=g)[:d].sort().values
        grid = workloads.Grid((nx, 1, nz), (True, False, False), (case["cx"], 1.0, case["cz"]), True)
        return [_problem(grid, draws, obs, case["r2"], case["nodes"], case["tol"], g)]
    if kind == "gauss2d":
        nx, ny, s = case["nx"], case["ny"], case["stride"]
        draws = _forecast2d(nx, ny, case["members"], case["length"], g)
        obs = (torch.arange(0, ny, s, device=DEV)[:, None] * nx + torch.arange(0, nx, s, device=DEV)).reshape(-1)
        grid = workloads.Grid((nx, ny, 1), (True, True, False), (case["half_width"], case["half_width"], 1.0), True)
        return [_problem(grid, draws, obs, case["r2"], case["nodes"], case["tol"], g)]
    # channels: Gaussian-weighted sums around evenly spaced centres, r^2 a tenth of the mean observable variance
    n, d = case["n"], case["d"]
    dense, (rowptr, col, val) = workloads.gaussian_channel_operator(n, d, case["bandwidth"])
    H = torch.tensor(dense, device=DEV)
    draws = _forecast1d(n, case["members"], case["length"] / 1.2, g)
    hx = draws @ H.T
    r2 = 0.1 * float((H @ H.T).diagonal().mean()) * case["length"]
    R = torch.full((d,), r2, device=DEV, dtype=torch.float64)
    y = hx[-1] + math.sqrt(r2) * torch.randn(d, device=DEV, dtype=torch.float64, generator=g)
    grid = workloads.Grid((n, 1, 1), (True, False, False), (math.sqrt(10.0 / 3.0) * case["length"], 1.0, 1.0), True)
    return [dict(grid=grid, X=draws[:-1].contiguous(), H=tuple(torch.tensor(a, device=DEV) for a in (rowptr, col, val)),
                 y=y, R=R, Q=case["nodes"], tol=case["tol"], dense_H=H)]


def _train_inputs(case, seed):
    """Samples as training sees them: normalized vectors v of the Krylov spaces of shifted localized covariances,
    their images y = (sigma + C) v and z = P^-1 y with the leading eigenvectors deflated; features; a fresh network."""
    S, d = case["samples"], case["d"]
    g = _gen(seed)
    members, width = 40, 12
    Z = _forecast1d(8 * d, members, 64.0, g)[:members, ::8]
    Z = (Z - Z.mean(0)) / math.sqrt(members - 1)
    lag = _chordal(torch.arange(d, device=DEV, dtype=torch.float64)[:, None] - torch.arange(d, device=DEV), d) * 8.0
    C = 4.0 * _gaspari_cohn(lag / 256.0) * (Z.T @ Z)
    lam, Q = torch.linalg.eigh(C)
    lam, Q = lam[-10:], Q[:, -10:]
    chains = S // width
    sigma = torch.exp(torch.linspace(0.0, math.log(1000.0), chains, device=DEV, dtype=torch.float64))
    v = torch.randn(chains, d, device=DEV, dtype=torch.float64, generator=g)
    V, Y, W = [], [], []
    for _ in range(width):
        v = v / v.norm(dim=1, keepdim=True)
        y = v @ C + sigma[:, None] * v
        z = y / sigma[:, None] + ((y @ Q) * (1.0 / (lam + sigma[:, None]) - 1.0 / sigma[:, None])) @ Q.T
        V.append(v)
        Y.append(y)
        W.append(z)
        v = y - (y * v).sum(1, keepdim=True) * v
    ls = torch.log(sigma) / 5.0
    feat = torch.stack([ls, ls * ls, torch.full_like(ls, math.log(float(C.diagonal().mean())) / 5.0),
                        torch.full_like(ls, math.log(float(C.abs().sum(1).max())) / 10.0)], dim=1)
    flat = lambda parts: torch.stack(parts, 1).reshape(chains * width, -1).float().contiguous()  # noqa: E731
    feat = feat.repeat_interleave(width, 0).float().contiguous()
    return dict(theta=learned.init_params(int(seed) % 9973, device=DEV), feat=feat, V=flat(V), Y=flat(Y), Z=flat(W))


_MODEL = []


def _model():
    """The network a user's program loads: trained once per process with the repository's recipe on the
    benchmark's training problems, whatever the case's seed."""
    if not _MODEL:
        theta, cutoff, _ = learned.fit([workloads.config2(tol=1e-6, seed=s) for s in (11, 12)], K=12,
                                       members_per_q=3, steps=300)
        _MODEL.append((theta, cutoff))
    return _MODEL[0]


def prepare(case, seed):
    if case["kind"] == "train":
        return dict(kind="train", **_train_inputs(case, seed))
    probs = _problems(case, seed)
    kw = dict(precision=PRECISION[case["precision"]], solver=SOLVER[case["solver"]])
    if case.get("model"):
        kw["learned_model"], kw["learned_max_shift"] = _model()
    options = B.make_options(**kw)
    # one output buffer for all problems of a call, each problem's part on a 256-byte boundary
    pad = lambda v: (v + 31) // 32 * 32  # noqa: E731
    n = [p["X"].shape[1] for p in probs]
    mu = torch.zeros(sum(pad(m) for m in n), device=DEV, dtype=torch.float64)
    A = torch.zeros(sum(pad(p["X"].numel()) for p in probs), device=DEV, dtype=torch.float64)
    at = ak = 0
    for p, m in zip(probs, n):
        k = p["X"].numel()
        p["mu_a"], p["A_a"] = mu[at:at + m], A[ak:ak + k].view(p["X"].shape)
        at, ak = at + pad(m), ak + pad(k)
    state = dict(kind=case["kind"], options=options, probs=probs, mu=mu, A=A, single=case["precision"] != "fp64")
    if case["kind"] not in ("batch", "channels"):   # the batched call takes its workspace from torch's pool
        p = probs[0]
        state["ws"] = B.workspace(B.workspace_size(p["grid"], p["X"].shape[0], p["obs_idx"].numel(), p["Q"], options))
    return state


def run(state):
    if state["kind"] == "train":
        loss, grad = B.learn_loss_grad(state["theta"], state["feat"], state["V"], state["Y"], state["Z"])
        return {"loss": loss, "grad": grad}
    if state["kind"] in ("batch", "channels"):
        B.info_esrf_analysis_batched(state["probs"], state["options"], stats=False)
    else:
        p = state["probs"][0]
        B.info_esrf_analysis(p["grid"], p["X"], p["obs_idx"], p["y"], p["R"], p["Q"], p["tol"], state["options"],
                             ws=state["ws"], mu_a=p["mu_a"], A_a=p["A_a"], stats=False)
    if state["single"]:
        return {"mean": state["mu"].float(), "anomalies": state["A"].float()}
    return {"mean": state["mu"], "anomalies": state["A"]}


# ---------------------------------------------------------------------------
# Work and exact values
# ---------------------------------------------------------------------------

def _gaspari_cohn(r):
    r = r.abs()
    lo = (((-0.25 * r + 0.5) * r + 0.625) * r - 5.0 / 3.0) * r * r + 1.0
    hi = ((((r / 12.0 - 0.5) * r + 0.625) * r + 5.0 / 3.0) * r - 5.0) * r + 4.0 - 2.0 / (3.0 * r.clamp_min(1e-30))
    return torch.where(r <= 1.0, lo, torch.where(r < 2.0, hi, torch.zeros_like(r)))


def work(case):
    """What one pass cannot do without: the ensemble, observations and results once; one weighted product of members
    for every pair inside the localization's support, one product with C for every shifted system (how many
    iterations follow depends on the data), and the state update's product."""
    kind = case["kind"]
    if kind == "train":
        S, d = case["samples"], case["d"]
        net = 2 * (4 * 32 + 32 * 32 + 32 * 18)
        return {"bytes": 4.0 * (3 * S * d + 4 * S + 2 * 1810), "flops": float(S) * (6 * 2 * 17 * d + 8 * d + 3 * net)}
    out = {"bytes": 0.0, "flops": 0.0}
    if kind == "batch":
        parts = [(n, N, (n + s - 1) // s, Q, 256.0 / s, 256.0 / s) for n, N, s, Q in _sizes(case)]
    else:
        N, Q = case["members"], case["nodes"]
        if kind == "gauss1d":
            n, d = case["n"], (case["n"] - case["offset"] + case["stride"] - 1) // case["stride"]
            near = 4.0 * case["half_width"] / case["stride"]
        elif kind == "layered":
            n = case["nx"] * case["nz"]
            d = int(round(case["fraction"] * n))
            near = case["fraction"] * 4.0 * case["cx"] * min(case["nz"], math.pi * case["cz"])
        elif kind == "gauss2d":
            n, d = case["nx"] * case["ny"], (case["nx"] // case["stride"]) * (case["ny"] // case["stride"])
            near = math.pi * (2.0 * case["half_width"] / case["stride"]) ** 2
        else:
            n, d = case["n"], case["d"]
            near = float(d)
        parts = [(n, N, d, Q, min(near, d), min(near, d))]
    size = 8.0 if case["precision"] == "fp64" else 4.0
    for n, N, d, Q, oo, xo in parts:
        out["bytes"] += 8.0 * n * N + 24.0 * d + size * n * (N + 1)
        out["flops"] += 2.0 * N * (d * oo + n * xo) + 2.0 * d * oo * (N * Q + 1) + 2.0 * n * xo * (N + 1)
    return out


def _elliptic(Q, ell):
    """Nodes and weights of the elliptic rule: s = sc^2(u | k), p = (2 K / (pi Q)) dn(u | k), k^2 = ell / (1 + ell), by
    the arithmetic-geometric mean, with u above K / 2 taken from the complementary argument."""
    kc = 1.0 / math.sqrt(1.0 + ell)
    a, c = [1.0], [math.sqrt(ell / (1.0 + ell))]
    b = kc
    while abs(c[-1]) > 1e-17 and len(a) < 20:
        a0 = a[-1]
        a.append(0.5 * (a0 + b))
        c.append(0.5 * (a0 - b))
        b = math.sqrt(a0 * b)
    K = math.pi / (2.0 * a[-1])
    s, p = [], []
    for q in range(Q):
        t = (q + 0.5) / Q
        v = min(t, 1.0 - t) * K
        phi = (1 << (len(a) - 1)) * a[-1] * v
        for i in range(len(a) - 1, 0, -1):
            phi = 0.5 * (phi + math.asin(c[i] / a[i] * math.sin(phi)))
        sn, cn = math.sin(phi), math.cos(phi)
        dn = math.sqrt(cn * cn + kc * kc * sn * sn)
        if t > 0.5:
            sc, dn = cn / (sn * kc), kc / dn
        else:
            sc = sn / cn
        s.append(sc * sc)
        p.append(2.0 * K / (math.pi * Q) * dn)
    return (torch.tensor(v, device=DEV, dtype=torch.float64) for v in (s, p))


def _radius(grid, ia, ib):
    """Localization argument between the flat indices ia [m][1] and ib [1][k]."""
    r2, div = 0.0, 1
    for ext, per, c in zip(grid.shape, grid.periodic, grid.half_width):
        if ext > 1:
            delta = ((ia // div) % ext - (ib // div) % ext).abs().double()
            r2 = r2 + ((_chordal(delta, ext) if per else delta) / c) ** 2
        div *= ext
    return r2.sqrt()


def _solve(apply, B0, sigma, limit=600):
    """CG on every column of (C + sigma_j) U = B0 in 64 bits, to rounding."""
    U, r = torch.zeros_like(B0), B0.clone()
    p, rr = r.clone(), (r * r).sum(0)
    stop = 1e-28 * rr
    for it in range(limit):
        live = rr > stop
        if it % 8 == 0 and not bool(live.any()):
            break
        Cp = apply(p) + sigma * p
        alpha = torch.where(live, rr / (p * Cp).sum(0).clamp_min(1e-300), torch.zeros_like(rr))
        U += alpha * p
        r -= alpha * Cp
        new = (r * r).sum(0)
        p = r + torch.where(live, new / rr.clamp_min(1e-300), torch.zeros_like(rr)) * p
        rr = torch.where(live, new, rr)
    return U


def _exact_problem(p):
    grid, X, y, R, Q = p["grid"], p["X"], p["y"], p["R"], p["Q"]
    N, n = X.shape
    mu = X.mean(0)
    Z = (X - mu) / math.sqrt(N - 1)
    ri = R.rsqrt()
    H = p.get("dense_H")
    rows = torch.arange(n, device=DEV)[:, None]
    if H is not None:
        Sxh = (_gaspari_cohn(_radius(grid, rows, rows.T)) * (Z.T @ Z)) @ H.T
        C = ri[:, None] * (H @ Sxh) * ri
        Wt, innov = H @ Z.T, y - H @ mu
    else:
        obs = p["obs_idx"]
        Wt, innov = Z[:, obs].T.contiguous(), y - mu[obs]
        d = obs.numel()
        reach = d
        if grid.shape[1] == 1 and grid.shape[2] == 1:   # observations in support are neighbours by number
            gap = int((obs[1:] - obs[:-1]).min()) if d > 1 else 1
            c = grid.half_width[0]
            far = n / math.pi * math.asin(min(1.0, 2.0 * c * math.pi / n)) if 2.0 * c * math.pi < n else n
            reach = int(far / gap) + 1
        if 2 * reach + 1 < d and d > 512:
            idx = torch.arange(d, device=DEV)
            diags = []
            for k in range(-reach, reach + 1):
                j = (idx + k) % d
                L = _gaspari_cohn(_radius(grid, obs, obs[j]))
                diags.append(L * (Wt * Wt[j]).sum(1) * ri * ri[j])
            C = torch.stack(diags)
        else:
            C = _gaspari_cohn(_radius(grid, obs[:, None], obs[None, :])) * (Wt @ Wt.T) * ri[:, None] * ri
    if C.shape[0] == C.shape[1]:
        apply, gersh = (lambda P: C @ P), float(C.abs().sum(1).max())
    else:
        w = C.shape[0] // 2

        def apply(P):
            P = torch.cat([P[-w:], P, P[:w]])
            out = torch.zeros_like(P[w:-w])
            for k in range(2 * w + 1):
                out.addcmul_(C[k][:, None], P[k:k + out.shape[0]])
            return out

        gersh = float(C.abs().sum(0).max())
    ell = 10.0 ** (math.floor(math.log10(max(gersh, 1.0))) + 1)
    s, wq = _elliptic(Q, ell)
    rhs = ri[:, None] * Wt
    U = _solve(apply, rhs.repeat(1, Q), (s + 1.0).repeat_interleave(N)[None, :])
    V = (U.view(-1, Q, N) * wq[None, :, None]).sum(1)
    um = _solve(apply, (ri * innov)[:, None], torch.ones(1, 1, device=DEV, dtype=torch.float64))
    V = ri[:, None] * torch.cat([V, um], 1)
    if H is not None:
        inc = Sxh @ V
    else:
        inc = torch.empty(n, N + 1, device=DEV, dtype=torch.float64)
        step = max(128, int(4e7 / d))
        for x in range(0, n, step):
            at = rows[x:x + step]
            inc[x:x + step] = (_gaspari_cohn(_radius(grid, at, obs[None, :])) * (Z[:, x:x + step].T @ Wt.T)) @ V
    return mu + inc[:, N], math.sqrt(N - 1) * (Z - inc[:, :N].T)


def _exact_train(t):
    """Loss mean_s ||a z + S^T S y - v||^2 / ||v||^2 and its gradient by autograd in 64 bits."""
    theta = t["theta"].double().requires_grad_(True)
    V, Y, Z, feat = (t[k].double() for k in ("V", "Y", "Z", "feat"))
    parts, at = [], 0
    for shape in ((32, 4), (32,), (32, 32), (32,), (18, 32), (18,)):
        size = math.prod(shape)
        parts.append(theta[at:at + size].view(shape))
        at += size
    W1, b1, W2, b2, W3, b3 = parts
    out = torch.tanh(torch.tanh(feat @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    sigma = torch.exp(5.0 * feat[:, :1])
    a, w = torch.exp(out[:, :1]) / sigma, out[:, 1:] / sigma.sqrt()
    Sy = sum(w[:, j:j + 1] * torch.roll(Y, 8 - j, 1) for j in range(17))
    e = a * Z - V + sum(w[:, j:j + 1] * torch.roll(Sy, j - 8, 1) for j in range(17))
    loss = ((e * e).sum(1) / (V * V).sum(1)).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": theta.grad}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(_train_inputs(case, seed))
    probs = _problems(case, seed)
    for p in probs:   # dense CG in 64 bits: about 100 iterations at a TFLOP/s
        d = p["R"].numel()
        if case["kind"] in ("layered", "gauss2d") and 200.0 * d * d * (p["Q"] * p["X"].shape[0] + 1) > 8e12:
            return None
    pad = lambda v: (v + 31) // 32 * 32  # noqa: E731
    mu = torch.zeros(sum(pad(p["X"].shape[1]) for p in probs), device=DEV, dtype=torch.float64)
    A = torch.zeros(sum(pad(p["X"].numel()) for p in probs), device=DEV, dtype=torch.float64)
    at = ak = 0
    for p in probs:
        N, n = p["X"].shape
        m, a = _exact_problem(p)
        mu[at:at + n], A[ak:ak + N * n] = m, a.reshape(-1)
        at, ak = at + pad(n), ak + pad(N * n)
    return {"mean": mu, "anomalies": A}
