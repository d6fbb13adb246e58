"""The work that this solver is measured on: single calls through its public
entry points, from one QP of the 30-bus grid to batches of load scenarios, and
the warm-start network's training and prediction.

A case is a dict of plain values.  ``prepare`` makes what a user's program
holds before the call (grids, a handle, a network, device arrays), ``run`` is
one pass, ``work`` the bytes and operations the pass cannot do without, and
``exact`` the same results in 64 bits by plain torch and numpy.

Kinds:
  qp       one QP at the flat start of every instance of a handle (build, a
           fixed budget of ADMM iterations, step and multipliers read back)
  solve    complete SQP solves to 1e-4 under new loads, solution read back
  project  network predictions projected onto the linear constraints
  train    mini-batch Adam steps of the warm-start network, weights read back
  predict  the network's outputs for load scenarios on the device
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2310_13143_gb300 import binding, gridgen, warmstart

RHO = 2e4  # penalty of every ADMM here (the published large-case setting)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one small QP on a handle as it is created: the smallest call, all latency
        dict(name="qp_30bus", kind="qp", buses=30, scenarios=1, precision="mixed", shape="default", iters=50),
        # the plain path on the smallest grid: FP64, default ADMM settings
        dict(name="solve_30bus_fp64", kind="solve", buses=30, scenarios=1, precision="fp64", shape="cluster"),
        # the benchmark's headline: one 2,000-bus solve, mixed precision, tuned launch shape
        dict(name="solve_2000bus", kind="solve", buses=2000, scenarios=1, precision="mixed", shape="cluster"),
        # the same on the plain FP64 path
        dict(name="solve_2000bus_fp64", kind="solve", buses=2000, scenarios=1, precision="fp64", shape="resident"),
        # a batch of load scenarios in one handle, SQP loop from a CUDA graph
        dict(name="solve_2000bus_x128", kind="solve", buses=2000, scenarios=128, precision="mixed", shape="default"),
        # grids of uneven size (118 to 10,000 buses) in one launch
        dict(name="qp_uneven_x64", kind="qp", buses=118, buses_to=10000, grids=64, topology=1, precision="mixed",
             shape="default", iters=100),
        # the largest grid, 8 scenarios: a working set beyond the L2 cache
        dict(name="qp_70000bus_x8", kind="qp", buses=70000, scenarios=8, precision="mixed", shape="default",
             iters=100),
        # predicted starts of 128 scenarios made feasible before a solve
        dict(name="project_2000bus_x128", kind="project", buses=2000, scenarios=128),
        # training for the 2,000-bus grid, batch 256
        dict(name="train_2000bus", kind="train", buses=2000, rows=1024, batch=256, steps=128),
        # training for a small grid with a ragged batch: many small kernels
        dict(name="train_30bus", kind="train", buses=30, rows=700, batch=100, steps=64),
        # warm starts predicted for the held-out scenarios of the 2,000-bus grid
        dict(name="predict_2000bus_x512", kind="predict", buses=2000, rows=512),
        # one scenario that has just come in
        dict(name="predict_2000bus", kind="predict", buses=2000, rows=1),
    ]


def draw(rng):
    def log_int(a, b):
        return max(a, min(b, int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))))

    kind = rng.choice(("qp", "qp", "solve", "project", "train", "predict"))
    if kind == "qp":
        iters, precision = rng.randint(20, 100), rng.choice(("mixed", "fp64"))
        topology = rng.randint(2, 10000)
        if rng.random() < 0.3:
            return dict(kind="qp", buses=118, buses_to=10000, grids=rng.randint(3, 63), topology=topology,
                        precision=precision, shape="default", iters=iters)
        buses = log_int(30, 10000)
        most = max(1, min(128, (250000 if precision == "mixed" else 60000) // buses))
        scenarios = log_int(1, most)
        shape = "cluster" if buses <= 2000 and scenarios <= 16 and rng.random() < 0.5 else "default"
        return dict(kind="qp", buses=buses, topology=topology, scenarios=scenarios, precision=precision, shape=shape,
                    iters=iters)
    if kind == "solve":
        which = rng.choice(("30", "2000", "2000"))
        if which == "30":
            return dict(kind="solve", buses=30, scenarios=log_int(2, 24), precision="fp64",
                        shape=rng.choice(("default", "cluster")), check=rng.randint(1, 4))
        return dict(kind="solve", buses=2000, scenarios=log_int(2, 100), precision="mixed", shape="default",
                    check=rng.randint(1, 4))
    buses = log_int(30, 2000)
    topology = rng.randint(2, 10000)
    if kind == "project":
        return dict(kind="project", buses=buses, topology=topology,
                    scenarios=log_int(1, max(2, min(128, 200000 // buses))))
    rows = log_int(1, 1024)
    if kind == "predict":
        return dict(kind="predict", buses=buses, topology=topology, rows=rows)
    return dict(kind="train", buses=buses, topology=topology, rows=rng.randint(256, 1024),
                batch=rng.randint(24, 256), steps=rng.randint(24, 100))


# ------------------------------------------------------------------- inputs
@lru_cache(maxsize=128)
def _grid(buses, topology):
    if topology == 0 and buses == 30:
        return gridgen.grid_30bus()
    if topology == 0 and buses == 2000:
        return gridgen.grid_2000bus()
    if topology == 0 and buses == 70000:
        return gridgen.grid_70k()
    return gridgen.geometric_grid(buses, seed=1000 + topology)


def _bases(case):
    """The grids of the case's instances, before their loads are drawn."""
    topology = case.get("topology", 0)
    if "grids" in case:
        r = np.random.default_rng(topology)
        sizes = np.exp(r.uniform(math.log(case["buses"]), math.log(case["buses_to"]), case["grids"]))
        return [_grid(int(round(n)), 100 * topology + k) for k, n in enumerate(sizes)]
    return [_grid(case["buses"], topology)] * case["scenarios"]


def _scenario(grid, rng, sigma=0.05, length=0.1, features=64):
    """The grid under loads scaled by 1 + e, e a spatially correlated Gaussian
    field (random Fourier features)."""
    w = rng.standard_normal((2, features)) / length
    f = np.cos(grid.xy @ w + rng.uniform(0, 2 * math.pi, features)) if grid.xy is not None else \
        rng.standard_normal((grid.nbus, features))
    e = sigma * math.sqrt(2.0 / features) * (f @ rng.standard_normal(features))
    return grid.with_loads(grid.pd * (1 + e), grid.qd * (1 + e))


def _scenarios(case, seed):
    rng = np.random.default_rng(seed)
    return [_scenario(g, rng) for g in _bases(case)]


def _handle(case, grids):
    s = binding.Solver(grids, precision=case["precision"])
    if case["shape"] == "cluster":  # what the autotuner picks for one instance of these sizes
        s.tune(224 if case["buses"] > 100 else 64, 0, 4)
    elif case["shape"] == "resident":
        s.tune(64, 0, 3)
    return s


def _predictions(grids, seed):
    """Network outputs near an operating point, one row per scenario (only the
    NLP point is used): dispatch inside its box, voltages near 1, small angles."""
    width = warmstart.pad8(warmstart.output_width(grids[0]))
    rng = np.random.default_rng(seed + 1)
    out = np.zeros((len(grids), width), dtype=np.float32)
    for k, g in enumerate(grids):
        v, th = 1 + rng.uniform(-0.03, 0.03, g.nbus), rng.uniform(-0.05, 0.05, g.nbus)
        th[g.bus_type == gridgen.REF] = 0.0
        a, m = th[g.f] - th[g.t], v[g.f] * v[g.t]
        x = np.concatenate([g.pmin + (g.pmax - g.pmin) * rng.uniform(0.3, 0.7, g.ngen),
                            rng.uniform(-0.2, 0.2, g.ngen), v * v, th,
                            m * np.cos(a) + rng.uniform(-1e-3, 1e-3, g.nbranch),
                            m * np.sin(a) + rng.uniform(-1e-3, 1e-3, g.nbranch)])
        out[k, :x.size] = x
    return out


def _network_data(case, seed):
    """Grid, widths and device arrays: loads X and targets T, a smooth function
    of the loads plus noise, in columns of different scale."""
    g = _grid(case["buses"], case.get("topology", 0))
    dims = warmstart.dims_for(g)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, device="cuda", generator=gen)

    base = torch.zeros(dims[0], device="cuda")
    base[:2 * g.nbus] = torch.from_numpy(np.concatenate([g.pd, g.qd])).float()
    n = max(case["rows"], 256)  # the standardiser is fitted to at least 256 scenarios
    modes = normal(n, 12)
    X = (base * (1 + 0.05 * modes @ normal(12, dims[0]) / math.sqrt(12))).contiguous()
    scale = torch.exp(normal(dims[-1]))
    T = ((torch.tanh(modes @ normal(12, dims[-1]) / 3) + 0.1 * normal(n, dims[-1])) * scale + scale)
    return g, dims, X, T.contiguous()


def prepare(case, seed):
    if case["kind"] in ("qp", "solve"):
        grids = _scenarios(case, seed)
        s = _handle(case, grids)
        if case["kind"] == "qp":
            opts = binding.default_admm(rho=RHO, eps=0.0, max_iter=case["iters"], warm=0)
        elif case["buses"] == 30:
            opts = binding.default_sqp(tol=1e-4, max_sqp=30)
        else:
            mixed = case["precision"] == "mixed"
            opts = binding.default_sqp(tol=1e-4, max_sqp=20, soc=int(len(grids) > 1), restore=int(len(grids) > 1),
                                       admm=dict(rho=RHO, max_iter=1000, eps=1e-3, eps_dual=5e-3 if mixed else 0.0))
        return dict(case=case, grids=grids, solver=s, opts=opts)
    if case["kind"] == "project":
        grids = _scenarios(case, seed)
        pred = torch.from_numpy(_predictions(grids, seed)).cuda()
        return dict(case=case, grids=grids, pred=pred, solver=binding.Solver(grids, precision="mixed"))
    _, dims, X, T = _network_data(case, seed)
    net = binding.Mlp(dims, case.get("batch", 256))
    net.set_params(gridgen.mlp_init(dims, seed))
    net.fit_standardiser(X.data_ptr(), T.data_ptr(), X.shape[0])
    return dict(case=case, net=net, X=X, T=T, seed=seed, Y=torch.zeros(case["rows"], dims[-1], device="cuda"))


# -------------------------------------------------------------------- a pass
def _in_precision(case, arrays):
    """The mixed path computes its steps in FP32: its results in that type."""
    t = np.float32 if case["precision"] == "mixed" else np.float64
    return {k: np.concatenate([np.ravel(v) for v in vs]).astype(t) for k, vs in arrays.items()}


def run(state):
    case = state["case"]
    if case["kind"] == "qp":
        s = state["solver"]
        s.admm_solve_qp(1.0, state["opts"])
        steps = [s.get_step(k) for k in range(len(state["grids"]))]
        return _in_precision(case, dict(d=[d for d, _ in steps], pi=[p for _, p in steps]))
    if case["kind"] == "solve":
        s = state["solver"]
        if len(state["grids"]) == 1:
            g = state["grids"][0]
            s.set_loads(0, g.pd, g.qd)
            s.sqp_solve(state["opts"])
        else:
            s.sqp_solve_graph(state["opts"], check_every=case.get("check", 2))
        sols = [s.get_solution(k) for k in range(len(state["grids"]))]
        return _in_precision(case, {k: [x[k] for x in sols] for k in sols[0]})
    if case["kind"] == "project":
        s, pred = state["solver"], state["pred"]
        s.set_warm_start_device(pred.data_ptr(), pred.shape[1], use_x=True, use_pi=False, use_lambda=False,
                                use_rho=False)
        s.project_linear(rho=0.5, eps=1e-4)
        return np.concatenate([s.get_iterate(k)[0] for k in range(len(state["grids"]))])
    net, X, T, Y = state["net"], state["X"], state["T"], state["Y"]
    if case["kind"] == "predict":
        net.forward(X.data_ptr(), case["rows"], Y.data_ptr())
        return Y
    losses = warmstart.train(net, X, T, case["rows"], case["steps"], case["batch"], 1e-3, state["seed"], "cos")
    return dict(losses=losses, params=net.get_params())


# ---------------------------------------------------------------------- work
def _qp_bytes(B, L, G, w):
    """One ADMM iteration: 8 words per coupling (the component side reads z and
    lambda and writes x; the bus side reads x, lambda and z and writes z and
    lambda), 40 words of QP data per branch, 8 per generator, 4 per bus and a
    4-byte index per branch end and generator."""
    return (8 * (8 * L + 2 * G) + 40 * L + 8 * G + 4 * B) * w + 4 * (2 * L + G)


def work(case):
    if case["kind"] in ("qp", "solve", "project"):
        grids = _bases(case)
        B, L, G = (sum(getattr(g, n) for g in grids) for n in ("nbus", "nbranch", "ngen"))
        w = 4 if case.get("precision") == "mixed" else 8
        if case["kind"] == "project":
            # about 500 iterations; per iteration 6 words per end and side, 10 of data per branch
            return dict(bytes=500.0 * 8 * (2 * L * 3 * 8 + 2 * G * 8 + 10 * L + 4 * B), flops=500.0 * (250 * L + 40 * B))
        # a solve: 8 QPs of 1,000 iterations, or 28,000 iterations on the 30-bus grid
        n = case["iters"] if case["kind"] == "qp" else 28000 if case["buses"] == 30 else 8000
        return dict(bytes=float(n) * _qp_bytes(B, L, G, w), flops=float(n) * (400 * L + 60 * (2 * L + G) + 30 * B))
    dims = warmstart.dims_for(_grid(case["buses"], case.get("topology", 0)))
    p = sum(a * b + b for a, b in zip(dims, dims[1:]))
    if case["kind"] == "predict":
        return dict(bytes=2.0 * p + 4.0 * case["rows"] * (dims[0] + dims[-1]), flops=2.0 * p * case["rows"])
    # per step: bfloat16 weights read, FP32 weights and moments read and written, bfloat16 weights written
    return dict(bytes=case["steps"] * (28.0 * p + 4.0 * case["batch"] * (dims[0] + dims[-1])),
                flops=6.0 * p * case["batch"] * case["steps"])


# ----------------------------------------------------- the results in 64 bits
def exact(case, seed):
    if case["kind"] == "qp":
        if sum(g.nbranch for g in _bases(case)) * case["iters"] > 25e6:
            return None  # too long
        return _exact_qp(case, _scenarios(case, seed))
    if case["kind"] == "project":
        grids = _scenarios(case, seed)
        return _exact_projection(grids, _predictions(grids, seed))
    if case["kind"] in ("train", "predict"):
        return _exact_network(case, seed)
    return None  # a whole solve: thousands of QP iterations, too long


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _cat(grids, name):
    return np.concatenate([np.asarray(getattr(g, name), dtype=np.float64) for g in grids])


class _Model:
    """The instances' components concatenated, and the flow maps of the pi
    model: p_ij, q_ij, p_ji, q_ji linear in (w_i, w_j, wR, wI)."""

    def __init__(self, grids):
        off = np.cumsum([0] + [g.nbus for g in grids])
        self.f = _t(np.concatenate([g.f + o for g, o in zip(grids, off)]), torch.int64)
        self.t = _t(np.concatenate([g.t + o for g, o in zip(grids, off)]), torch.int64)
        self.gbus = _t(np.concatenate([g.gbus + o for g, o in zip(grids, off)]), torch.int64)
        self.B, self.L, self.G = int(off[-1]), self.f.numel(), self.gbus.numel()
        self.ref = _t(np.concatenate([g.bus_type == gridgen.REF for g in grids]), torch.bool)
        for n in ("pd", "qd", "gs", "bs", "pmin", "pmax", "qmin", "qmax", "rate", "angmin", "angmax"):
            setattr(self, n, _t(_cat(grids, n)))
        self.wmin, self.wmax = _t(_cat(grids, "vmin")) ** 2, _t(_cat(grids, "vmax")) ** 2
        base = np.concatenate([np.full(g.ngen, g.base_mva) for g in grids])
        self.c2, self.c1 = _t(_cat(grids, "c2") * base ** 2), _t(_cat(grids, "c1") * base)
        y = 1.0 / (_cat(grids, "r") + 1j * _cat(grids, "x"))
        ysh, tap = y + 0.5j * _cat(grids, "b"), _cat(grids, "tap")
        rot = np.exp(1j * _cat(grids, "shift"))
        ff, ft, tf, tt = ysh / tap ** 2, -y / tap * rot, -y / tap / rot, ysh
        J = np.zeros((self.L, 4, 4))  # columns w_i, w_j, wR, wI
        J[:, 0, 0], J[:, 0, 2], J[:, 0, 3] = ff.real, ft.real, ft.imag
        J[:, 1, 0], J[:, 1, 2], J[:, 1, 3] = -ff.imag, -ft.imag, ft.real
        J[:, 2, 1], J[:, 2, 2], J[:, 2, 3] = tt.real, tf.real, -tf.imag
        J[:, 3, 1], J[:, 3, 2], J[:, 3, 3] = -tt.imag, -tf.imag, -tf.real
        self.J = _t(J)

    def at_buses(self, ends, gens=None):
        """Sums over each bus of per-end values [L, 2, n] (and per-generator values [G, n])."""
        out = torch.zeros(self.B, ends.shape[2], dtype=torch.float64, device="cuda")
        out.index_add_(0, self.f, ends[:, 0])
        out.index_add_(0, self.t, ends[:, 1])
        if gens is not None:
            out.index_add_(0, self.gbus, gens)
        return out

    def split(self, grids, blocks):
        """Concatenated component arrays, [pg | qg | w | theta | wR | wI] per instance."""
        pg, qg, w, th, wr, wi = (b.cpu().numpy() for b in blocks)
        out, b, g0, l0 = [], 0, 0, 0
        for g in grids:
            G, B, L = slice(g0, g0 + g.ngen), slice(b, b + g.nbus), slice(l0, l0 + g.nbranch)
            out += [pg[G], qg[G], w[B], th[B], wr[L], wi[L]]
            g0, b, l0 = g0 + g.ngen, b + g.nbus, l0 + g.nbranch
        return np.concatenate(out)


def _bus_system(m, s_inv, v1, v2, qw, cw):
    """d_w and the two multipliers of every bus's balance rows: the 2 x 2 system with shunts."""
    m11, m22, m12 = s_inv + m.gs ** 2 / qw, s_inv + m.bs ** 2 / qw, -m.gs * m.bs / qw
    r1, r2 = v1 - m.gs * cw / qw, v2 + m.bs * cw / qw
    det = m11 * m22 - m12 ** 2
    n1, n2 = (m22 * r1 - m12 * r2) / det, (m11 * r2 - m12 * r1) / det
    return n1, n2, (cw + m.gs * n1 - m.bs * n2) / qw


def _kkt(Q, c, lo, hi, N, b, on, fx, up, act):
    """Stationary point on the given active set of min 1/2 x'Qx + c'x, lo <= x
    <= hi, N x <= b: bounds held (fx; at hi where up) and rows held (act).
    Returns x, the rows' multipliers and the changes to the set that the KKT
    conditions ask for, with their sizes."""
    n, dev = Q.shape[0], Q.device
    A = torch.zeros(n, 8, 8, dtype=torch.float64, device=dev)
    rhs = torch.zeros(n, 8, dtype=torch.float64, device=dev)
    s = Q.abs().amax((1, 2))[:, None]  # rows scaled alike
    eye = torch.eye(4, dtype=torch.float64, device=dev).expand(n, 4, 4)
    A[:, :4, :4] = torch.where(fx[:, :, None], eye, Q / s[:, :, None])
    A[:, :4, 4:] = torch.where(fx[:, :, None], 0.0, N.transpose(1, 2))
    rhs[:, :4] = torch.where(fx, torch.where(up, hi, lo), -c / s)
    A[:, 4:, :4] = torch.where(act[:, :, None], N, 0.0)
    A[:, 4:, 4:] = torch.where(act[:, :, None], 0.0, eye)
    rhs[:, 4:] = torch.where(act, b, 0.0)
    sol, info = torch.linalg.solve_ex(A, rhs)
    bad = (info != 0) | ~torch.isfinite(sol).all(1)
    x, mu = sol[:, :4], sol[:, 4:] * s
    g = (Q @ x[:, :, None])[:, :, 0] + c + (N.transpose(1, 2) @ mu[:, :, None])[:, :, 0]
    tol = 1e-11 * s
    move = lo < hi
    below, above = (lo - x) * ~fx, (x - hi) * ~fx
    drop = torch.where(fx & move, torch.where(up, g, -g), 0.0) / s
    row = torch.where(on & ~act, (N @ x[:, :, None])[:, :, 0] - b, 0.0)
    rdrop = torch.where(act, -mu, 0.0) / s
    size = torch.cat([below, above, drop, row, rdrop], 1)
    return x, mu, size, bad | (size.amax(1) > 1e-11)


def _line_qp(Q, c, lo, hi, N, b, on, sets):
    """Unique KKT point of every branch's strictly convex QP, from the active
    sets of the previous call: corrections of the set, then every set in turn
    for what is left.  Updates ``sets``."""
    fx, up, act = sets
    x = torch.zeros_like(c)
    mu = torch.zeros_like(b)
    todo = torch.arange(c.shape[0], device=c.device)
    for it in range(30):
        a = [v[todo] for v in (Q, c, lo, hi, N, b, on, fx, up, act)]
        xs, ms, size, wrong = _kkt(*a)
        x[todo], mu[todo] = xs, ms
        todo, size = todo[wrong], size[wrong]
        if not todo.numel():
            return x, mu
        ask = size > 1e-11
        if it >= 6:  # one change at a time from here on
            ask &= size >= size.amax(1, keepdim=True)
        below, above, drop, row, rdrop = ask.split(4, 1)
        fixed = lo[todo] >= hi[todo]
        fx[todo] = ((fx[todo] | below | above) & ~drop) | fixed
        up[todo] = (up[todo] | above) & ~below
        act[todo] = (act[todo] | row) & ~rdrop
    best = torch.full((todo.numel(),), math.inf, dtype=torch.float64, device=c.device)
    fixed = lo[todo] >= hi[todo]
    q = [v[todo] for v in (Q, c, lo, hi, N, b, on)]
    for code in range(81 * 12):  # every working set: bounds free, low or high; rows; one angle row at most
        side = torch.tensor([(code // 3 ** i) % 3 for i in range(4)], device=c.device)
        r = code // 81
        rows = torch.tensor([r & 1, (r >> 1) & 1, (r >> 2) == 1, (r >> 2) == 2], device=c.device).bool()
        f_, u_, a_ = fixed | (side > 0), (side == 2) & ~fixed, rows & on[todo]
        xs, ms, size, _ = _kkt(*q, f_, u_, a_)
        off = torch.nan_to_num(size.amax(1), nan=math.inf)
        t = off < best
        best = torch.where(t, off, best)
        k = todo[t]
        x[k], mu[k], fx[k], up[k], act[k] = xs[t], ms[t], f_[t], u_[t], a_[t]
    return x, mu


def _exact_qp(case, grids):
    """The QP at the flat start (w = 1, theta = 0, wR = 1, wI = 0, pi = 0) by the
    component ADMM: there the Hessian of the Lagrangian vanishes, d_wR = (d_wi +
    d_wj) / 2 and d_wI = d_thi - d_thj."""
    m = _Model(grids)
    L = m.L
    A = torch.tensor([[1, 0, 0, 0], [0, 0, 1, 0], [0.5, 0, 0.5, 0], [0, 1, 0, -1]], dtype=torch.float64, device="cuda")
    F = m.J @ A  # flow changes over (d_wi, d_thi, d_wj, d_thj)
    flow = m.J.sum(2) - m.J[:, :, 3]
    Q = RHO * (F.transpose(1, 2) @ F + torch.eye(4, dtype=torch.float64, device="cuda"))
    wl, wh = torch.clamp(m.wmin - 1, min=-1.0), torch.clamp(m.wmax - 1, max=1.0)
    tb = torch.where(m.ref, 0.0, 1.0)
    lo = torch.stack([wl[m.f], -tb[m.f], wl[m.t], -tb[m.t]], 1)
    hi = torch.stack([wh[m.f], tb[m.f], wh[m.t], tb[m.t]], 1)
    N = torch.zeros(L, 4, 4, dtype=torch.float64, device="cuda")
    b = torch.zeros(L, 4, dtype=torch.float64, device="cuda")
    on = torch.zeros(L, 4, dtype=torch.bool, device="cuda")
    norm = torch.ones(L, 2, dtype=torch.float64, device="cuda")
    for e in range(2):
        p, q = flow[:, 2 * e], flow[:, 2 * e + 1]
        row = 2 * p[:, None] * F[:, 2 * e] + 2 * q[:, None] * F[:, 2 * e + 1]
        norm[:, e] = row.norm(dim=1)
        on[:, e] = (m.rate > 0) & (norm[:, e] > 0)
        norm[:, e] = torch.where(on[:, e], norm[:, e], 1.0)
        N[:, e] = row / norm[:, e, None]
        b[:, e] = (m.rate ** 2 - p ** 2 - q ** 2) / norm[:, e]
    N[:, 2, 1], N[:, 2, 3], N[:, 3, 1], N[:, 3, 3] = 1.0, -1.0, -1.0, 1.0
    b[:, 2], b[:, 3] = m.angmax, -m.angmin
    on[:, 2:] = ((m.angmin > -2 * math.pi) & (m.angmax < 2 * math.pi))[:, None]
    pg, qg = 0.5 * (m.pmin + m.pmax), 0.5 * (m.qmin + m.qmax)
    sums = m.at_buses(flow.reshape(L, 2, 2), -torch.stack([pg, qg], 1))
    pk, qk = m.pd + m.gs + sums[:, 0], m.qd - m.bs + sums[:, 1]
    g1, g2 = 2 * m.c2 * pg + m.c1, 2 * m.c2
    lp, up_ = torch.clamp(m.pmin - pg, min=-1.0), torch.clamp(m.pmax - pg, max=1.0)
    lq, uq = torch.clamp(m.qmin - qg, min=-1.0), torch.clamp(m.qmax - qg, max=1.0)
    one_e, one_g = torch.ones(L, 2, 1, dtype=torch.float64, device="cuda"), torch.ones(m.G, 1, dtype=torch.float64,
                                                                                      device="cuda")
    s_inv = m.at_buses(one_e, one_g)[:, 0] / RHO
    qw = m.at_buses(one_e)[:, 0] * RHO
    z, lam = (torch.zeros(L, 2, 4, dtype=torch.float64, device="cuda") for _ in range(2))  # per end: p, q, w, theta
    zg, lg = (torch.zeros(m.G, 2, dtype=torch.float64, device="cuda") for _ in range(2))
    held = lo >= hi
    sets = [held, torch.zeros_like(held), torch.zeros_like(on)]
    for _ in range(case["iters"]):
        t = RHO * zg - lg
        xg = torch.stack([torch.clamp((t[:, 0] - g1) / (g2 + RHO), lp, up_), torch.clamp(t[:, 1] / RHO, lq, uq)], 1)
        r = lam - RHO * z
        c = (F.transpose(1, 2) @ r[:, :, :2].reshape(L, 4, 1))[:, :, 0] + r[:, :, 2:].reshape(L, 4)
        v, mu = _line_qp(Q, c, lo, hi, N, b, on, sets)
        x = torch.cat([(F @ v[:, :, None]).reshape(L, 2, 2), v.reshape(L, 2, 2)], 2)
        a, ag = lam + RHO * x, lg + RHO * xg
        sm = m.at_buses(torch.cat([-a[:, :, :2] / RHO, a[:, :, 2:]], 2))
        sg = m.at_buses(torch.zeros_like(a), torch.cat([ag / RHO, torch.zeros_like(ag)], 1))
        n1, n2, dw = _bus_system(m, s_inv, sm[:, 0] + sg[:, 0] - pk, sm[:, 1] + sg[:, 1] - qk, qw, sm[:, 2])
        dth = torch.where(m.ref, 0.0, sm[:, 3] / qw)
        nu, bus = torch.stack([n1, n2], 1), torch.stack([dw, dth], 1)
        zg = (ag - nu[m.gbus]) / RHO
        lg = ag - RHO * zg
        ends = torch.stack([m.f, m.t], 1)
        z = torch.cat([(a[:, :, :2] + nu[ends]) / RHO, bus[ends]], 2)
        lam = a - RHO * z
    dwr, dwi = 0.5 * (dw[m.f] + dw[m.t]), dth[m.f] - dth[m.t]
    u = mu[:, :2] / norm * on[:, :2]
    force = lam[:, :, :2].reshape(L, 4) + 2 * u.repeat_interleave(2, 1) * flow
    grad = (m.J[:, :, 2:].transpose(1, 2) @ force[:, :, None])[:, :, 0]
    pi = torch.stack([-grad[:, 0] / 2, grad[:, 1], -u[:, 0], -u[:, 1]], 1)
    return dict(d=m.split(grids, (xg[:, 0], xg[:, 1], dw, dth, dwr, dwi)), pi=pi.reshape(-1).cpu().numpy())


def _exact_projection(grids, pred, rho=0.5, eps=1e-4, check=25):
    """The projection's component ADMM to the same tolerance: residuals of every
    instance at most eps, looked at every ``check`` iterations."""
    m = _Model(grids)
    g0 = grids[0]
    ng, nb, nl = g0.ngen, g0.nbus, g0.nbranch
    x0 = _t(pred)
    parts = [p.reshape(-1) for p in x0[:, :2 * (ng + nb + nl)].split([ng, ng, nb, nb, nl, nl], 1)]
    pg0, qg0 = torch.clamp(parts[0], m.pmin, m.pmax), torch.clamp(parts[1], m.qmin, m.qmax)
    w0, th, own = torch.clamp(parts[2], m.wmin, m.wmax), parts[3], torch.stack(parts[4:], 1)
    lo, hi = (torch.stack([v[m.f], v[m.t]], 1) for v in (m.wmin, m.wmax))
    h = rho * (m.J.transpose(1, 2) @ m.J) + torch.diag(torch.tensor([rho, rho, 2.0, 2.0], dtype=torch.float64,
                                                                    device="cuda"))
    solve = {}  # inverse on the free variables, by which of (w_i, w_j) are held
    for held in ((0, 0), (1, 0), (0, 1), (1, 1)):
        keep = [i for i in range(4) if i > 1 or not held[i]]
        inv = torch.zeros_like(h)
        inv[:, torch.tensor(keep)[:, None], torch.tensor(keep)] = torch.linalg.inv(h[:, keep][:, :, keep])
        solve[held] = inv
    v = torch.cat([w0[m.f, None], w0[m.t, None], own], 1)
    x = torch.cat([(m.J @ v[:, :, None]).reshape(m.L, 2, 2), v[:, :2, None]], 2)
    z, lam = x.clone(), torch.zeros_like(x)
    zg = torch.stack([pg0, qg0], 1)
    lg = torch.zeros_like(zg)
    one_e, one_g = torch.ones(m.L, 2, 1, dtype=torch.float64, device="cuda"), torch.ones(m.G, 1, dtype=torch.float64,
                                                                                        device="cuda")
    s_inv = m.at_buses(one_e, one_g)[:, 0] / rho
    qw = 2 + rho * m.at_buses(one_e)[:, 0]
    ends = torch.stack([m.f, m.t], 1)
    for it in range(1, 20001):
        xg = torch.stack([torch.clamp((2 * pg0 - lg[:, 0] + rho * zg[:, 0]) / (2 + rho), m.pmin, m.pmax),
                          torch.clamp((2 * qg0 - lg[:, 1] + rho * zg[:, 1]) / (2 + rho), m.qmin, m.qmax)], 1)
        r = lam - rho * z
        c = (m.J.transpose(1, 2) @ r[:, :, :2].reshape(m.L, 4, 1))[:, :, 0]
        c = c + torch.cat([r[:, :, 2], -2 * own], 1)
        v = torch.zeros_like(c)
        found = torch.zeros(m.L, dtype=torch.bool, device="cuda")
        for held, inv in solve.items():
            for side in range(2 ** sum(held)):
                bound = torch.zeros_like(c)
                at_hi = [side & 1, side >> 1 if held[0] else side & 1]
                for i in range(2):
                    if held[i]:
                        bound[:, i] = hi[:, i] if at_hi[i] else lo[:, i]
                y = bound - (inv @ (c + (h @ bound[:, :, None])[:, :, 0])[:, :, None])[:, :, 0]
                g = (h @ y[:, :, None])[:, :, 0] + c
                ok = ~found
                for i in range(2):
                    if held[i]:
                        ok &= (g[:, i] <= 0) if at_hi[i] else (g[:, i] >= 0)
                    else:
                        ok &= (y[:, i] >= lo[:, i]) & (y[:, i] <= hi[:, i])
                v = torch.where(ok[:, None], y, v)
                found |= ok
        x = torch.cat([(m.J @ v[:, :, None]).reshape(m.L, 2, 2), v[:, :2, None]], 2)
        a, ag = lam + rho * x, lg + rho * xg
        sm = m.at_buses(torch.cat([-a[:, :, :2] / rho, a[:, :, 2:]], 2))
        sg = torch.zeros(m.B, 2, dtype=torch.float64, device="cuda").index_add_(0, m.gbus, ag / rho)
        n1, n2, w = _bus_system(m, s_inv, sm[:, 0] + sg[:, 0] - m.pd, sm[:, 1] + sg[:, 1] - m.qd, qw,
                                2 * w0 + sm[:, 2])
        nu = torch.stack([n1, n2], 1)
        zgn = (ag - nu[m.gbus]) / rho
        zn = torch.cat([(a[:, :, :2] + nu[ends]) / rho, w[ends][:, :, None]], 2)
        if it % check == 0:
            rp = max(float((x - zn).abs().max()), float((xg - zgn).abs().max()))
            rd = rho * max(float((zn - z).abs().max()), float((zgn - zg).abs().max()))
        z, zg, lam, lg = zn, zgn, a - rho * zn, ag - rho * zgn
        if it % check == 0 and rp <= eps and rd <= eps:
            break
    th = torch.where(m.ref, 0.0, torch.clamp(th, -2 * math.pi, 2 * math.pi))
    return m.split(grids, (xg[:, 0], xg[:, 1], torch.clamp(w, m.wmin, m.wmax), th, v[:, 2], v[:, 3]))


def _exact_network(case, seed):
    _, dims, X, T = _network_data(case, seed)

    def standardise(a):
        a = a.double()
        mean, dev = a.mean(0), a.std(0, unbiased=False)
        return mean, torch.where(dev <= 1e-12 * (1 + mean.abs()), 1.0, dev)

    (mx, sx), (my, sy) = standardise(X), standardise(T)
    flat, o, W, b = _t(gridgen.mlp_init(dims, seed)), 0, [], []
    for i, n in zip(dims, dims[1:]):
        W.append(flat[o:o + i * n].reshape(n, i).clone())
        b.append(flat[o + i * n:o + i * n + n].clone())
        o += i * n + n

    def layers(x):
        acts, zs = [x], []
        for k in range(len(W)):
            zs.append(acts[-1] @ W[k].T + b[k])
            acts.append(torch.nn.functional.gelu(zs[-1]) if k + 1 < len(W) else zs[-1])
        return acts, zs

    if case["kind"] == "predict":
        return layers((X[:case["rows"]].double() - mx) / sx)[0][-1] * sy + my
    rng = np.random.default_rng(seed)
    n, steps, batch = case["rows"], case["steps"], case["batch"]
    order = np.concatenate([rng.permutation(n) for _ in range((steps * batch) // n + 1)])
    params = W + b
    mom = [[torch.zeros_like(p) for p in params] for _ in range(2)]
    losses = []
    for k in range(steps):
        idx = torch.from_numpy(order[k * batch:(k + 1) * batch]).cuda()
        acts, zs = layers((X[idx].double() - mx) / sx)
        d = acts[-1] - (T[idx].double() - my) / sy
        losses.append(float((d * d).mean()))
        d = 2 * d / d.numel()
        gW, gb = [None] * len(W), [None] * len(W)
        for l in range(len(W) - 1, -1, -1):
            gW[l], gb[l] = d.T @ acts[l], d.sum(0)
            if l:
                zl = zs[l - 1]
                d = (d @ W[l]) * (0.5 * (1 + torch.erf(zl / math.sqrt(2)))
                                  + zl * torch.exp(-0.5 * zl * zl) / math.sqrt(2 * math.pi))
        lr = max(1e-3 * 0.5 * (1 + math.cos(math.pi * k / steps)), 1e-7)
        for p, g, m1, m2 in zip(params, gW + gb, *mom):
            m1.mul_(0.9).add_(g, alpha=0.1)
            m2.mul_(0.999).addcmul_(g, g, value=0.001)
            p.sub_(lr * (m1 / (1 - 0.9 ** (k + 1))) / ((m2 / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8))
    params = torch.cat([torch.cat([w.reshape(-1), v]) for w, v in zip(W, b)])
    return dict(losses=torch.tensor(losses, dtype=torch.float64), params=params)
