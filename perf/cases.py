"""The work a user of the solver has it do, as cases that can be timed and checked.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (grid,
medium, state, network), ``run`` makes one pass through the public entry points, ``work`` counts
what the pass cannot do without and ``exact`` evaluates the same pass in FP64 with plain torch.

Kinds of case:
  steps     n Runge-Kutta steps of one block (or of a batch of states on one mesh)
  gradient  misfit and material gradient through torch autograd (forward run and discrete adjoint)
  energy    the discrete energy (the health check of a long run)
  setup     metric terms and coefficients of a new mesh and medium
  train     one training iteration of the surrogate network
  forward   the surrogate's traces for a batch of sources
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

FREE, ABSORB = ("free",), ("char", 0.0)
BC = (ABSORB, ABSORB, ABSORB, ABSORB, ABSORB, FREE)   # absorbing but for the free top surface
EXTENT = {"cube": (1000.0, 1000.0, 1000.0), "hill": (20000.0, 20000.0, 15000.0),
          "sines": (60000.0, 60000.0, 24000.0), "curved": (20000.0, 18000.0, 15000.0)}
CFL = 0.5
V_SCALE, S_SCALE = 1.0e-2, 1.2e5   # m/s and Pa of a passing wave
M0 = 1.0e14                        # N m


def _steps(name, nodes, order, precision, geometry, medium, steps, batch=1, operator="upwind", source=True, side=4):
    return dict(name=name, kind="steps", nq=nodes[0], nr=nodes[1], ns=nodes[2], order=order, operator=operator,
                precision=precision, geometry=geometry, medium=medium, steps=steps, batch=batch, source=source,
                side=side)


def listed():
    return [
        # the smallest run: a Cartesian FP64 cube in one wavefield, launches and latency count
        _steps("cube33_o4_fp64", (33, 33, 33), 4, 64, "cube", "homogeneous", 10, source=False, side=2),
        # the ordinary run: a topography block with a point source and surface stations
        _steps("hill129_o6_fp32", (129, 129, 97), 6, 32, "hill", "layered", 10),
        # the same block in double precision
        _steps("hill129_o6_fp64", (129, 129, 97), 6, 64, "hill", "layered", 2),
        # a production-size topography block, far beyond the caches
        _steps("topo769_o6_fp32", (769, 769, 257), 6, 32, "sines", "gradient", 1, source=False),
        # a fully curvilinear block (all nine metric terms), ragged along every axis
        _steps("curved257_o6_fp32", (257, 241, 161), 6, 32, "curved", "gradient", 2),
        # an odd-order operator of the accuracy comparison on the ordinary block
        _steps("hill129_o5_fp32", (129, 129, 97), 5, 32, "hill", "layered", 5),
        # generation of training data: 64 sources advance together on one mesh
        _steps("batch64_97_o4_fp32", (97, 97, 97), 4, 32, "hill", "layered", 2, batch=64, side=8),
        # inversion: misfit and gradient of eight sources, forward run, recomputation and adjoint
        dict(name="gradient129_o4_fp32", kind="gradient", nq=129, nr=129, ns=97, order=4, precision=32,
             geometry="hill", steps=16, sources=8, side=8),
        # the check of a long run
        dict(name="energy385_o6_fp32", kind="energy", nq=385, nr=385, ns=193, order=6, precision=32,
             geometry="hill"),
        # a new mesh and medium
        dict(name="setup257_o6_fp32", kind="setup", nq=257, nr=257, ns=129, order=6, precision=32, geometry="hill",
             medium="layered"),
        # the surrogate network at its full size: one training iteration, and traces for 64 sources
        dict(name="train_b32", kind="train", hidden=512, C=128, T0=32, n_up=5, receivers=64, batch=32),
        dict(name="forward_b64", kind="forward", hidden=512, C=128, T0=32, n_up=5, receivers=64, batch=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["gradient", "energy", "setup", "train", "forward"])
    if kind in ("train", "forward"):
        return dict(kind=kind, hidden=rng.choice([256, 512]), C=rng.choice([64, 128]), T0=32, n_up=rng.randint(3, 5),
                    receivers=rng.choice([16, 25, 36, 64]), batch=_log(rng, 5, 32 if kind == "train" else 64))
    if kind == "gradient":
        return dict(kind=kind, nq=rng.randint(33, 131), nr=rng.randint(33, 131), ns=rng.randint(33, 97),
                    order=rng.choice([2, 4, 4, 6]), precision=rng.choice([32, 32, 64]),
                    geometry=rng.choice(["hill", "curved"]), steps=rng.randint(4, 14), sources=rng.randint(1, 6),
                    side=rng.randint(2, 8))
    if kind in ("energy", "setup"):
        c = dict(kind=kind, nq=_log(rng, 33, 320), nr=_log(rng, 33, 320), ns=_log(rng, 33, 180),
                 order=rng.choice([2, 4, 5, 6]), precision=rng.choice([32, 64]),
                 geometry=rng.choice(["hill", "curved"]))
        return c if kind == "energy" else dict(c, medium=rng.choice(["layered", "gradient"]))
    operator = rng.choice(["upwind"] * 4 + ["traditional"])
    order = rng.choice([2, 4, 6] if operator == "traditional" else [2, 3, 4, 4, 5, 6, 6, 6, 7])
    precision = rng.choice([32, 32, 32, 64])
    nodes = [_log(rng, 33, 500) for _ in range(2)] + [_log(rng, 33, 260)]
    if rng.random() < 0.3:
        nodes = [min(n, 110) for n in nodes]
        batch = rng.randint(2, 24)
    else:
        batch = 1
    total = nodes[0] * nodes[1] * nodes[2] * batch * (10 if precision == 64 else 1)
    most = max(1, min(10, int(1.2e8 / total)))
    c = _steps("", nodes, order, precision, rng.choice(["hill", "hill", "sines", "curved"]),
               rng.choice(["layered", "gradient"]), rng.randint(1, most), batch=batch, operator=operator,
               source=rng.random() < 0.7, side=rng.randint(2, 8))
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _nodes(case):
    return case["nq"], case["nr"], case["ns"]


def _axes(case):
    nq, nr, ns = _nodes(case)
    f = lambda n: torch.arange(n, dtype=torch.float64, device=_device()) / (n - 1)  # noqa: E731
    return f(nq).view(1, 1, nq), f(nr).view(1, nr, 1), f(ns).view(ns, 1, 1)


def _mesh(case, rng):
    """Node coordinates (3, ns, nr, nq), FP64."""
    Lx, Ly, Lz = EXTENT[case["geometry"]]
    nq, nr, ns = _nodes(case)
    q, r, s = _axes(case)
    X = torch.empty(3, ns, nr, nq, dtype=torch.float64, device=_device())
    if case["geometry"] == "curved":
        e = rng.uniform(0.04, 0.08)
        X[0] = Lx * (q + e * torch.sin(math.pi * r + 0.3) * torch.cos(math.pi * s) + 0.5 * e * q * r)
        X[1] = Ly * (r + e * torch.sin(math.pi * q + 0.5) * torch.sin(math.pi * s + 0.2))
        X[2] = Lz * (s - 1 + e * torch.sin(math.pi * q) * torch.cos(math.pi * r + 0.1) + 0.5 * e * s * q)
        return X
    top = 0 * q + 0 * r
    if case["geometry"] == "hill":
        top = rng.uniform(1000.0, 1500.0) * torch.exp(-((Lx * q - Lx / 2) ** 2 + (Ly * r - Ly / 2) ** 2) / 4000.0 ** 2)
    elif case["geometry"] == "sines":
        for _ in range(8):
            lam, th, ph = rng.uniform(3000.0, 20000.0), rng.uniform(0, 2 * math.pi), rng.uniform(0, 2 * math.pi)
            k = 2 * math.pi / lam
            top = top + 75.0 * torch.sin(k * math.cos(th) * Lx * q + k * math.sin(th) * Ly * r + ph)
    X[0], X[1], X[2] = Lx * q, Ly * r, -Lz + s * (Lz + top)
    return X


def _medium(case, X, rng):
    """rho, lambda, mu (3, ns, nr, nq), FP64: vp = sqrt(3) vs (homogeneous: 6000, 3464 m/s)."""
    name = case.get("medium", "gradient")
    out = torch.empty_like(X)
    if name == "homogeneous":
        out[0], out[1], out[2] = 2700.0, 2700.0 * (6000.0 ** 2 - 2 * 3464.0 ** 2), 2700.0 * 3464.0 ** 2
        return out
    if name == "layered":
        d = -X[2]
        vs = torch.where(d < 1000.0, 1000.0, torch.where(d < 5000.0, 2000.0, 3500.0)).double()
        out[0] = torch.where(d < 1000.0, 2000.0, torch.where(d < 5000.0, 2400.0, 2700.0)).double()
    else:
        t = torch.clip(-X[2] / EXTENT[case["geometry"]][2], 0.0, 1.0)
        vs, out[0] = 2000.0 + 2000.0 * t, 2200.0 + 700.0 * t
    for _ in range(4):   # a smooth random perturbation of a few per cent
        k = rng.normal(size=3) * 2 * math.pi / 5000.0
        vs = vs * (1.0 + 0.02 * torch.cos(k[0] * X[0] + k[1] * X[1] + k[2] * X[2] + rng.uniform(0, 2 * math.pi)))
    out[2] = out[0] * vs ** 2
    out[1] = out[2]      # lambda = rho (vp^2 - 2 vs^2) with vp^2 = 3 vs^2
    return out


def _time_step(X, rlm):
    h2 = min(float(torch.diff(X, dim=d).square().sum(0).min()) for d in (1, 2, 3))
    return CFL * math.sqrt(h2 / float(((rlm[1] + 2 * rlm[2]) / rlm[0]).max()))


def _wavefield(case, rng, dtype):
    """A smooth random state (9 B, ns, nr, nq): products of waves along the three axes."""
    nq, nr, ns = _nodes(case)
    q, r, s = _axes(case)
    nf = 9 * case.get("batch", 1)
    Q = torch.empty(nf, ns, nr, nq, dtype=dtype, device=_device())
    for f in range(nf):
        acc = 0
        for _ in range(2):
            k, ph = rng.integers(1, 6, 3), rng.uniform(0, 2 * math.pi, 3)
            acc = acc + (torch.sin(2 * math.pi * k[0] * q + ph[0]) * torch.sin(2 * math.pi * k[1] * r + ph[1]) *
                         torch.sin(2 * math.pi * k[2] * s + ph[2]))
        Q[f] = acc * (V_SCALE if f % 9 < 3 else S_SCALE)
    return Q


def _double_couple(rng, moment):
    """Voigt (xx, yy, zz, xy, xz, yz) of M0 (n d^T + d n^T) with random normal n and slip d."""
    n = rng.normal(size=3)
    n /= np.linalg.norm(n)
    d = np.cross(n, rng.normal(size=3))
    d /= np.linalg.norm(d)
    M = moment * (np.outer(n, d) + np.outer(d, n))
    return [float(M[i, j]) for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]


def _stations(case):
    nq, nr, ns = _nodes(case)
    at = np.linspace(0.2, 0.8, case["side"])
    return [(int(round(a * (nq - 1))), int(round(b * (nr - 1))), ns - 1) for b in at for a in at]


def _inputs(case, seed):
    """Everything of a solver case but the solver: mesh, medium, time step, state, sources."""
    rng = np.random.default_rng([int(seed), 20])
    X = _mesh(case, rng)
    rlm = _medium(case, X, rng)
    d = dict(X=X, rlm=rlm, dt=_time_step(X, rlm), rng=rng)
    if case["kind"] in ("steps", "energy"):
        d["Q"] = _wavefield(case, rng, torch.float32 if case["precision"] == 32 else torch.float64)
    if case["kind"] == "steps" and case["source"]:
        d["f0"], d["t0"] = 2.0, 0.5 * case["steps"] * d["dt"]
        d["sources"] = [dict(ref=tuple(float(x) for x in rng.uniform((0.3, 0.3, 0.67), (0.7, 0.7, 0.85))),
                             moment=_double_couple(rng, M0)) for _ in range(case["batch"])]
    if case["kind"] == "gradient":
        # shallow sources under the stations and a short pulse, so that waves arrive within the run
        d["f0"] = 1.2 / (0.4 * case["steps"] * d["dt"])
        d["t0"] = 1.2 / d["f0"]
        moment = 3e5 * d["f0"] * S_SCALE * math.prod(EXTENT[case["geometry"]]) / X[0].numel()
        d["sources"] = [dict(ref=tuple(float(x) for x in rng.uniform((0.3, 0.3, 0.9), (0.7, 0.7, 0.96))),
                             moment=_double_couple(rng, moment)) for _ in range(case["sources"])]
        n = len(_stations(case))
        t = torch.arange(case["steps"], dtype=torch.float64) * d["dt"]
        # observed traces: a pulse of its own arrival time, width and amplitude per station and component
        arr = torch.from_numpy(rng.uniform(0, float(t[-1]), (case["sources"], n, 3, 1)))
        amp = torch.from_numpy(rng.normal(size=(case["sources"], n, 3, 1))) * V_SCALE
        d["data"] = (amp * torch.exp(-((t - arr) * 1.5 * d["f0"]) ** 2)).to(_device())
        d["norm"] = 1.0 / float(0.5 * d["dt"] * d["data"].square().sum())
    return d


def _network_inputs(case, seed):
    g = torch.Generator().manual_seed(int(seed))
    B, n_out, T = case["batch"], 3 * case["receivers"], case["T0"] * 2 ** case["n_up"]
    u = lambda *s: torch.rand(*s, generator=g)    # noqa: E731
    x = (2 * u(3, B) - 1).to(torch.bfloat16)
    m = torch.randn(6, B, generator=g) * 0.7
    y = torch.randn(n_out, B, 1, generator=g) * torch.sin(20 * u(n_out, B, 1) * torch.linspace(0, 1, T) + 6 * u(n_out, B, 1))
    return [t.to(_device()) for t in (x, m, y.reshape(n_out, B * T).contiguous())]


# ---- the calls ----------------------------------------------------------------------------------

def _solver(case, d, batch=1, keep=False):
    from paper_2011_02600_gb300 import ElasticSolver
    s = ElasticSolver(_nodes(case), case["order"], precision=case["precision"], bc=list(BC), batch=batch,
                      operator=case.get("operator", "upwind"))
    s.setup(d["X"], d["rlm"], keep_metrics=keep)
    return s


def prepare(case, seed):
    if case["kind"] in ("train", "forward"):
        return _prepare_network(case, seed)
    d = _inputs(case, seed)
    st = dict(kind=case["kind"])
    if case["kind"] == "setup":
        from paper_2011_02600_gb300 import ElasticSolver
        st["s"] = ElasticSolver(_nodes(case), case["order"], precision=case["precision"], bc=list(BC))
        st["X"], st["rlm"] = d["X"], d["rlm"]
    elif case["kind"] == "gradient":
        from paper_2011_02600_gb300.adjoint import MisfitProblem
        s = _solver(case, d, batch=case["sources"], keep=True)
        dtype = torch.float32 if case["precision"] == 32 else torch.float64
        st["m"] = [d["rlm"][f].to(dtype).requires_grad_() for f in range(3)]
        data = d["data"] if case["sources"] > 1 else d["data"][0]
        st["p"] = MisfitProblem(s, _stations(case), data, d["dt"], case["steps"], sources=d["sources"], f0=d["f0"])
        st["norm"] = d["norm"]
    else:
        s = st["s"] = _solver(case, d, batch=case.get("batch", 1), keep=bool(case.get("source")))
        s.view(s.qbuf[s.current], d["Q"].shape[0]).copy_(d["Q"])
        if case["kind"] == "steps":
            st["steps"], st["dt"] = case["steps"], d["dt"]
            st["traces"] = s.set_receivers(_stations(case), case["steps"])
            if case["source"]:
                s.set_sources(d["sources"], f0=d["f0"], t0=d["t0"])
    return st


def _prepare_network(case, seed):
    from paper_2011_02600_gb300.surrogate import SurrogateNet
    net = SurrogateNet(hidden=case["hidden"], C=case["C"], T0=case["T0"], n_up=case["n_up"],
                       n_out=3 * case["receivers"], seed=int(seed) % 1000003)
    x, m, y = _network_inputs(case, seed)
    _mid_training(net.names, net.b, net.vw, net.vb, seed)
    return dict(kind=case["kind"], net=net, x=x, m=m, target=y)


def _mid_training(names, b, vw, vb, seed):
    """Biases and second moments as they are some way into a training run."""
    g = torch.Generator().manual_seed(int(seed) + 1)
    for n in names:
        b[n].copy_((0.02 * torch.randn(b[n].shape, generator=g)).to(b[n].device))
        for v in (vw[n], vb[n]):
            v.copy_((1e-6 * (0.5 + torch.rand(v.shape, generator=g))).to(v.device))


LR = 1e-3


def run(state):
    kind = state["kind"]
    if kind == "steps":
        s = state["s"]
        s.set_time(0.0, 0)
        s.step(state["steps"], state["dt"])
        return [s.view(s.qbuf[s.current], 9 * s.batch), state["traces"]]
    if kind == "gradient":
        from paper_2011_02600_gb300.adjoint import ElasticMisfit
        rho, lam, mu = state["m"]
        # the misfit relative to the data's energy, in the model's precision
        loss = (ElasticMisfit.apply(rho, lam, mu, state["p"]) * state["norm"]).to(rho.dtype)
        return [loss.detach(), *torch.autograd.grad(loss, (rho, lam, mu))]
    if kind == "energy":
        return [state["s"].energy()]
    if kind == "setup":
        s = state["s"]
        jmet = s.setup(state["X"], state["rlm"], keep_metrics=True)
        return [s.view(jmet, 10), s.view(s.met, 9), s.view(s.mat, 3)]
    net = state["net"]
    if kind == "forward":
        return [net.forward(state["x"], state["m"])]
    from paper_2011_02600_gb300.surrogate import mse
    y = net.forward(state["x"], state["m"], keep=True)
    _, dy = mse(y, state["target"])
    net.backward(dy)
    net.adam(LR)
    return [y, *(d[n] for d in (net.gw, net.gb, net.w, net.b, net.wb) for n in net.names)]


# ---- what a pass cannot do without --------------------------------------------------------------

def work(case):
    if case["kind"] in ("train", "forward"):
        return _network_work(case)
    n = case["nq"] * case["nr"] * case["ns"]
    e = case["precision"] // 8
    taps = len(_interior(case["order"], case.get("operator", "upwind"))[0])
    flops = 190 + 36 * taps                      # per node and stage: fluxes, strains, rows, update
    metrics = 9 if case["geometry"] == "curved" else 4
    if case["kind"] == "energy":
        return dict(bytes=12 * e * n, flops=60 * n)
    if case["kind"] == "setup":
        return dict(bytes=(24 + 24 + 80 + 12 * e) * n, flops=(9 * 4 * taps + 80) * n)
    B = case["batch"] if case["kind"] == "steps" else case["sources"]
    # a step is five stages; a stage needs the whole of the one before it, so where the state does
    # not stay on the chip each stage reads and writes the state and the register (stage 0 reads
    # no register) and reads the metric terms and coefficients, which a batch shares
    stages = 5 * case["steps"]
    held = ((18 * B + metrics + 3) * e * n) <= 100e6
    state = 18 * e * n * B if held else stages * (36 - 9 / 5) * e * n * B
    shared = (metrics + 3) * e * n * (1 if held else stages)
    if case["kind"] == "steps":
        return dict(bytes=state + shared, flops=stages * flops * n * B)
    # gradient: the forward stages twice over again (segment, stage inputs), then per stage of the
    # adjoint the stage input, yhat read and written, both adjoint registers, and the gradient
    adjoint = stages * ((9 + 18 + 36) * e * n * B + (metrics + 3) * e * n) + 48 * n
    return dict(bytes=3 * (state + shared) + adjoint, flops=stages * n * B * (3 * flops + 2 * flops))


def _network_work(case):
    B, C, T0, H, n_up = case["batch"], case["C"], case["T0"], case["hidden"], case["n_up"]
    n_out, T = 3 * case["receivers"], T0 * 2 ** n_up
    gemms = [(H, 3, B), (H, H, B), (C * T0, H, B)]
    gemms += [(C, 5 * C, B * T0 * 2 ** (i + 1)) for i in range(n_up)] + [(6 * n_out, 5 * C, B * T)]
    flops = sum(2 * m * k * n for m, k, n in gemms)
    params = sum(m * (k + 1) for m, k, n in gemms)
    if case["kind"] == "forward":
        return dict(bytes=2 * params + 4 * n_out * B * T, flops=flops)
    # weights, their moments and gradients; the traces read against their target
    return dict(bytes=(2 + 7 * 4 + 2) * params + 3 * 4 * n_out * B * T, flops=3 * flops)


# ---- the same in FP64, from the definitions alone -----------------------------------------------

UPWIND = {2: (0, (-3 / 2, 2, -1 / 2)), 3: (1, (-1 / 3, -1 / 2, 1, -1 / 6)),
          4: (1, (-1 / 4, -5 / 6, 3 / 2, -1 / 2, 1 / 12)), 5: (2, (1 / 20, -1 / 2, -1 / 3, 1, -1 / 4, 1 / 30)),
          6: (2, (1 / 30, -2 / 5, -7 / 12, 4 / 3, -1 / 2, 2 / 15, -1 / 60)),
          7: (3, (-1 / 105, 1 / 10, -3 / 5, -1 / 4, 1, -3 / 10, 1 / 15, -1 / 140))}
CENTRAL = {2: (1 / 2,), 4: (2 / 3, -1 / 12), 6: (3 / 4, -3 / 20, 1 / 60)}
WIDTH = {("upwind", 2): 2, ("upwind", 3): 2, ("upwind", 4): 4, ("upwind", 5): 4, ("upwind", 6): 6, ("upwind", 7): 6,
         ("traditional", 2): 1, ("traditional", 4): 4, ("traditional", 6): 6}
# entries of the corner block that accuracy leaves open
OPEN = {("upwind", 4): {(3, 3): -4 / 5}, ("upwind", 5): {(3, 3): -3 / 8},
        ("upwind", 6): {(4, 4): -17 / 25, (4, 5): 131 / 100, (5, 4): -29 / 100, (5, 5): -3 / 5},
        ("upwind", 7): {(4, 4): -1 / 4, (4, 5): 47 / 50, (5, 4): -27 / 50, (5, 5): -1 / 4},
        ("traditional", 6): {(4, 2): -1 / 10}}


def _interior(order, operator):
    """(alpha_-r..alpha_q, r) of D+."""
    if operator == "upwind":
        r, a = UPWIND[order]
        return a, r
    g = CENTRAL[order]
    return tuple(-x for x in reversed(g)) + (0.0,) + g, len(g)


def _operator(order, operator):
    """D+ and D- on unit spacing as (interior coefficients, first offset, closure rows), and the norm
    weights: P = H D+ is the Toeplitz stencil but for a corner block, fixed with the weights by the
    accuracy of D+ and D- = H^-1 (B - P^T) in the closure rows (and P + P^T = B for a central one)."""
    alpha, r = _interior(order, operator)
    b, q = WIDTH[operator, order], len(alpha) - 1 - r
    p = order // 2
    cw = b + max(q, r)
    toeplitz = lambda i, c: alpha[c - i + r] if -r <= c - i <= q else 0.0   # noqa: E731
    rows, rhs = [], []
    for i in range(b):
        for m in range(p + 1):
            for minus in (False, True):
                row, known = np.zeros(b * b + b), 0.0
                for c in range(cw):
                    x = float((c - i) ** m) if m else 1.0     # moments about the row's own node
                    if c < b:
                        row[(c * b + i) if minus else (i * b + c)] += -x if minus else x
                    else:
                        known += (-toeplitz(c, i) if minus else toeplitz(i, c)) * x
                    if minus and i == 0 and c == 0:
                        known += -x
                row[b * b + i] = -1.0 if m == 1 else 0.0
                rows.append(row)
                rhs.append(-known)
    if operator == "traditional":
        for i in range(b):
            for c in range(i + 1):
                row = np.zeros(b * b + b)
                row[i * b + c] += 1.0
                row[c * b + i] += 1.0
                rows.append(row)
                rhs.append(-1.0 if i == c == 0 else 0.0)
    for (i, c), v in OPEN.get((operator, order), {}).items():
        row = np.zeros(b * b + b)
        row[i * b + c] = 1.0
        rows.append(row)
        rhs.append(v)
    u = np.linalg.lstsq(np.array(rows), np.array(rhs), rcond=None)[0]
    P, w = u[:b * b].reshape(b, b), u[b * b:]
    plus, minus = np.zeros((b, cw)), np.zeros((b, cw))
    for i in range(b):
        for c in range(cw):
            plus[i, c] = P[i, c] if c < b else toeplitz(i, c)
            minus[i, c] = -P[c, i] if c < b else -toeplitz(c, i)
    minus[0, 0] -= 1.0
    return dict(b=b, cw=cw, w=w, plus=(alpha, -r, plus / w[:, None], minus / w[:, None]),
                minus=(tuple(-a for a in reversed(alpha)), -q, minus / w[:, None], plus / w[:, None]))


def _apply(row, f, dim, b, cw):
    """D f along dim on unit spacing; the far end by D+[N-1-i][N-1-j] = -D-[i][j]."""
    alpha, j0, near, far = row
    n = f.shape[dim]
    mid = 0
    for k, a in enumerate(alpha):
        if a:
            mid = mid + a * f.narrow(dim, b + j0 + k, n - 2 * b)
    ends = []
    for rows, part in ((near, f.narrow(dim, 0, cw)), (-far[::-1, ::-1], f.narrow(dim, n - cw, cw))):
        w = torch.as_tensor(rows.copy(), dtype=f.dtype, device=f.device)
        ends.append(torch.tensordot(part.movedim(dim, -1), w.t(), dims=1).movedim(-1, dim))
    return torch.cat([ends[0], mid, ends[1]], dim)


class _Plain:
    """The scheme on one block: dQ/dt and the Runge-Kutta step, for states (B, 9, ns, nr, nq)."""

    def __init__(self, case, X):
        self.N = _nodes(case)
        self.op = _operator(case["order"], case.get("operator", "upwind"))
        up = _operator(case["order"], "upwind")
        der = []
        for xi in range(3):
            d = [0.5 * (self.N[xi] - 1) * (_apply(up["plus"], X[c], 2 - xi, up["b"], up["cw"]) +
                                           _apply(up["minus"], X[c], 2 - xi, up["b"], up["cw"])) for c in range(3)]
            der.append(d)
        cross = lambda u, v: [u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]]  # noqa: E731
        self.a = [cross(der[(xi + 1) % 3], der[(xi + 2) % 3]) for xi in range(3)]
        self.J = sum(der[0][c] * self.a[0][c] for c in range(3))

    def coefficients(self, rlm):
        return 1.0 / (rlm[0] * self.J), rlm[1] / self.J, rlm[2] / self.J

    def weights(self, xi):
        w = np.ones(self.N[xi])
        b = self.op["b"]
        w[:b], w[-b:] = self.op["w"], self.op["w"][::-1]
        return torch.as_tensor(w / (self.N[xi] - 1), dtype=torch.float64, device=self.J.device)

    def rate(self, Q, mat):
        v, s = [Q[:, c] for c in range(3)], [Q[:, 3 + c] for c in range(6)]
        sym = ((0, 3, 4), (3, 1, 5), (4, 5, 2))
        b, cw = self.op["b"], self.op["cw"]
        rv, e = [0] * 3, [0] * 6
        strain = lambda a, u: (a[0] * u[0], a[1] * u[1], a[2] * u[2], a[1] * u[0] + a[0] * u[1],  # noqa: E731
                               a[2] * u[0] + a[0] * u[2], a[2] * u[1] + a[1] * u[2])
        for xi in range(3):
            a, h = self.a[xi], float(self.N[xi] - 1)
            for c in range(3):
                F = a[0] * s[sym[c][0]] + a[1] * s[sym[c][1]] + a[2] * s[sym[c][2]]
                rv[c] = rv[c] + h * _apply(self.op["minus"], F, 3 - xi, b, cw)
            dv = [h * _apply(self.op["plus"], v[c], 3 - xi, b, cw) for c in range(3)]
            e = [x + y for x, y in zip(e, strain(a, dv))]
        for face, kind in enumerate(BC):
            xi, side = face // 2, face % 2
            at = lambda f: f.select(f.dim() - 1 - xi, self.N[xi] - 1 if side else 0)  # noqa: E731
            h0 = (self.N[xi] - 1) / float(self.op["w"][0])
            a = [at(x) for x in self.a[xi]]
            sig, vel = [at(x) for x in s], [at(x) for x in v]
            T = [sum(a[k] * sig[sym[c][k]] for k in range(3)) for c in range(3)]
            if kind[0] == "free":
                for c in range(3):
                    at(rv[c]).add_(T[c], alpha=-h0 if side else h0)
                continue
            gamma = kind[1]
            an = torch.sqrt(a[0] ** 2 + a[1] ** 2 + a[2] ** 2)
            n = [x / an for x in a]
            T = [x / an for x in T]
            ir, l, m = (at(x) for x in mat)
            Zp, Zs = torch.sqrt((l + 2 * m) / ir), torch.sqrt(m / ir)
            vn, Tn = sum(x * y for x, y in zip(vel, n)), sum(x * y for x, y in zip(T, n))
            cv, cT = 0.5 * (1 - gamma), 0.5 * (1 + gamma) * (1 if side else -1)
            Gn = cv * Zp * vn + cT * Tn
            gt = [cv * Zs * (vel[c] - vn * n[c]) + cT * (T[c] - Tn * n[c]) for c in range(3)]
            for c in range(3):
                at(rv[c]).sub_(an * h0 * (Gn * n[c] + gt[c]))
            for x, y in zip(e, strain(n, [(-h0 if side else h0) * an * (Gn / Zp * n[c] + gt[c] / Zs) for c in range(3)])):
                at(x).add_(y)
        ir, l, m = mat
        tr = l * (e[0] + e[1] + e[2])
        return torch.stack([ir * x for x in rv] + [tr + 2 * m * x for x in e[:3]] + [m * x for x in e[3:]], 1)

    def source(self, sources, order):
        """(index of member, node offsets, -M delta_h) per source: moment conditions to degree order + 1."""
        out = []
        for sc in sources:
            line = []
            for xi in range(3):
                n, m = self.N[xi], order + 1
                c = int(math.floor(sc["ref"][xi] * (n - 1))) - (m - 1) // 2
                c = max(0, min(n - 1 - m, c))
                xs = np.arange(c, c + m + 1) - sc["ref"][xi] * (n - 1)
                phi = np.linalg.solve(np.vander(xs, m + 1, increasing=True).T, np.eye(m + 1)[0])
                line.append((slice(c, c + m + 1),
                             torch.as_tensor(phi, device=self.J.device) / self.weights(xi)[c:c + m + 1]))
            (iq, pq), (jr, pr), (ks, ps) = line
            box = (ks, jr, iq)
            d = ps.view(-1, 1, 1) * pr.view(1, -1, 1) * pq.view(1, 1, -1) / self.J[box]
            out.append((box, -torch.tensor(sc["moment"], dtype=torch.float64, device=d.device).view(6, 1, 1, 1) * d))
        return out

    def step(self, Q, mat, t, dt, src, f0, t0):
        """One step of Carpenter and Kennedy's five-stage 2N-storage scheme."""
        c = _stage_times()
        W = torch.zeros_like(Q)
        for k in range(5):
            R = self.rate(Q, mat)
            if src:
                x = (math.pi * f0 * (t + c[k] * dt - t0)) ** 2
                for i, (box, d) in enumerate(src):
                    R[(i, slice(3, 9)) + box] += (1 - 2 * x) * math.exp(-x) * d
            W = RK_A[k] * W + dt * R
            Q = Q + RK_B[k] * W
        return Q


RK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
        -1275806237668 / 842570457699)
RK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
        3134564353537 / 4481467310338, 2277821191437 / 14882151754819)


def _stage_times():
    reg, acc, c = [0.0] * 5, [0.0] * 5, []
    for k in range(5):
        c.append(sum(acc))
        reg = [RK_A[k] * x + (j == k) for j, x in enumerate(reg)]
        acc = [x + RK_B[k] * y for x, y in zip(acc, reg)]
    return c


def exact(case, seed):
    if case["kind"] in ("train", "forward"):
        return _exact_network(case, seed)
    d = _inputs(case, seed)
    P = _Plain(case, d["X"])
    if case["kind"] == "setup":
        a = [x for xi in range(3) for x in P.a[xi]]
        return [torch.stack([P.J] + a), torch.stack(a), torch.stack(P.coefficients(d["rlm"]))]
    if case["kind"] == "energy":
        r, l, m = P.coefficients(d["rlm"])
        Q = d["Q"]
        dens = (Q[0].double() ** 2 + Q[1].double() ** 2 + Q[2].double() ** 2) / r
        tr = Q[3].double() + Q[4] + Q[5]
        sq = sum((1 if f < 6 else 2) * Q[f].double() ** 2 for f in range(3, 9))
        dens = dens + (sq - l / (3 * l + 2 * m) * tr ** 2) / (2 * m)
        w = P.weights(2).view(-1, 1, 1) * P.weights(1).view(1, -1, 1) * P.weights(0)
        return [float(0.5 * (w * dens).sum())]
    if case["kind"] == "gradient":
        return _exact_gradient(case, d, P)
    B = case["batch"]
    if B * case["nq"] * case["nr"] * case["ns"] > 2e8:
        return None
    mat = P.coefficients(d["rlm"])
    src = P.source(d["sources"], case["order"]) if case["source"] else []
    Q = d["Q"].double().unflatten(0, (B, 9))
    rec = _stations(case)
    traces = []
    for n in range(case["steps"]):
        Q = P.step(Q, mat, n * d["dt"], d["dt"], src, d.get("f0", 1.0), d.get("t0", 0.0))
        traces.append(torch.stack([Q[:, :3, k, j, i] for i, j, k in rec], 1))
    tr = torch.stack(traces, -1)
    return [Q.flatten(0, 1), tr if B > 1 else tr[0]]


def _exact_gradient(case, d, P):
    model = [d["rlm"][f].to(torch.float32 if case["precision"] == 32 else torch.float64).double().requires_grad_()
             for f in range(3)]
    src = P.source(d["sources"], case["order"])
    nq, nr, ns = _nodes(case)
    Q = torch.zeros(case["sources"], 9, ns, nr, nq, dtype=torch.float64, device=model[0].device)
    rec = _stations(case)
    i, j, k = (torch.tensor(x, device=Q.device) for x in zip(*rec))
    phi = 0
    for n in range(case["steps"]):
        Q = checkpoint(lambda Q, *m, n=n: P.step(Q, P.coefficients(m), n * d["dt"], d["dt"], src, d["f0"], d["t0"]),
                       Q, *model, use_reentrant=False)
        v = Q[:, :3, k, j, i].transpose(1, 2)
        phi = phi + 0.5 * d["dt"] * (v - d["data"][..., n]).square().sum()
    loss = phi * d["norm"]
    return [loss.detach(), *torch.autograd.grad(loss, model)]


def _exact_network(case, seed):
    """The network without any rounding of activations or gradients to 16 bits."""
    C, T0, H, n_up, B = case["C"], case["T0"], case["hidden"], case["n_up"], case["batch"]
    n_out = 3 * case["receivers"]
    g = torch.Generator(device="cpu").manual_seed(int(seed) % 1000003)
    shapes = [("fc1", H, 3), ("fc2", H, H), ("fc3", C * T0, H)] + [(f"conv{i}", C, 5 * C) for i in range(n_up)]
    shapes += [("out", 6 * n_out, 5 * C)]
    names = [s[0] for s in shapes]
    w32, w, b, vw, vb = {}, {}, {}, {}, {}
    for n, o, i in shapes:
        std = math.sqrt((1.0 if n == "out" else 2.0) / i)
        w32[n] = (torch.randn(o, i, generator=g, dtype=torch.float64) * std).float().to(_device())
        b[n] = torch.zeros(o, device=_device())
        vw[n], vb[n] = torch.zeros_like(w32[n]), torch.zeros_like(b[n])
    x, m, target = _network_inputs(case, seed)
    _mid_training(names, b, vw, vb, seed)
    for n in names:   # the products take the weights in 16 bits
        w[n] = w32[n].to(torch.bfloat16).double().requires_grad_()
        b[n] = b[n].double().requires_grad_()
    h = x.double()
    for n in names[:3]:
        h = torch.relu(w[n] @ h + b[n][:, None])
    h = h.view(C, T0, B).permute(2, 0, 1)
    conv = lambda n, h: torch.nn.functional.conv1d(h, w[n].view(-1, C, 5), b[n], padding=2)  # noqa: E731
    for n in names[3:-1]:
        h = torch.relu(conv(n, h.repeat_interleave(2, dim=2)))
    G = conv("out", h).view(B, 6, n_out, -1)
    y = torch.einsum("cb,bcot->obt", m.double(), G).reshape(n_out, -1)
    if case["kind"] == "forward":
        return [y.detach()]
    loss = (y - target.double()).square().mean()
    gw = dict(zip(names, torch.autograd.grad(loss, [w[n] for n in names], retain_graph=True)))
    gb = dict(zip(names, torch.autograd.grad(loss, [b[n] for n in names])))

    def adam(p, g, v):
        v = 0.999 * v.double() + 0.001 * g * g
        return p.detach().double() - LR * (0.1 * g / (1 - 0.9)) / (torch.sqrt(v / (1 - 0.999)) + 1e-8)
    nw = [adam(w32[n], gw[n], vw[n]) for n in names]
    return [y.detach(), *gw.values(), *gb.values(), *nw, *(adam(b[n], gb[n], vb[n]) for n in names), *nw]
