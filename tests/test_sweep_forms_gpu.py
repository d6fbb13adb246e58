"""The sweep's dispatch at the sizes where it changes: four lanes, one lane or
no resident lane per branch (FP64, device-wide and in clusters), and bus tasks
of 31 to 33 entries (a full warp task, a task of its own)."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu
KEYS = ("x", "z", "lam", "xg", "zg", "lg", "zb", "nu", "ul")


def _shunts(g, seed=5):
    r = np.random.default_rng(seed)
    return replace(g, gs=r.uniform(-0.05, 0.05, g.nbus), bs=r.uniform(-0.1, 0.1, g.nbus),
                   tap=r.uniform(0.95, 1.05, g.nbranch), shift=r.uniform(-0.05, 0.05, g.nbranch))


def _state(grids, precision, shape, iters, rho=None):
    s = binding.Solver(grids, precision=precision)
    s.tune(*shape)
    s.build_qp(1.0, 2e4, True)
    o = binding.default_admm()
    # two launches, so that a sweep also starts from a state with active sets
    s.admm_iterate(iters // 2, o)
    s.admm_iterate(iters - iters // 2, o)
    got = [s.get_admm_state(k) for k in range(len(grids))]
    s.close()
    return got


# four lanes per branch: device-wide up to 9,600 branches, in a cluster up to
# 4,096 threads; one lane beyond; streaming where that does not fit either
@pytest.mark.parametrize("buses,shape", [(300, (64, 0, 3)), (300, (256, 0, 4)), (750, (256, 0, 4)), (780, (256, 0, 4)),
                                         (7000, (256, 0, 3)), (7500, (256, 0, 3)), (30000, (256, 0, 3))])
def test_fp64_forms_agree(buses, shape):
    grids = [_shunts(gg.geometric_grid(buses, seed=buses))]
    want = _state(grids, "fp64", (256, 0, 0), 40)
    got = _state(grids, "fp64", shape, 40)
    for a, b in zip(got, want):
        for k in KEYS:
            # both forms return the line subproblems' unique KKT points
            np.testing.assert_allclose(a[k], b[k], rtol=0, atol=1e-9 * max(1.0, np.abs(b[k]).max()), err_msg=k)


@pytest.mark.parametrize("solver", [0, 1])
def test_fp64_forms_agree_on_a_batch(solver):
    """Instances of unequal size in one cluster launch, and the augmented
    Lagrangian (line_solver 1), which keeps no set."""
    grids = [gg.grid_30bus(), _shunts(gg.geometric_grid(118, seed=7)), gg.hub_grid(40)]
    out = []
    for shape in ((256, 0, 0), (64, 0, 3), (64, 0, 4)):
        s = binding.Solver(grids, precision="fp64")
        s.tune(*shape)
        s.build_qp(1.0, 2e4, True)
        s.admm_iterate(30, binding.default_admm(line_solver=solver))
        out.append([s.get_admm_state(k) for k in range(len(grids))])
        s.close()
    for got in out[1:]:
        for a, b in zip(got, out[0]):
            for k in KEYS:
                np.testing.assert_allclose(a[k], b[k], rtol=0, atol=1e-9 * max(1.0, np.abs(b[k]).max()), err_msg=k)


@pytest.mark.parametrize("spokes", [30, 31, 32, 33])
@pytest.mark.parametrize("shape", [(256, 0, 0), (64, 0, 3), (64, 0, 4)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_bus_tasks_of_a_full_warp(spokes, shape, precision):
    """A hub whose entries fill a warp task to 30..33 lanes, with a generator at
    some of its buses, against the oracle."""
    import oracle

    g = _shunts(gg.hub_grid(spokes))
    m = oracle.Model(g)
    x, _ = binding.Solver(g).get_iterate(0)
    qp = m.build(x, None, 1.0, 1)
    st, _ = m.admm(qp, m.new_state(2e4), rho=2e4, eps=0.0, max_iter=6)
    got = _state([g], precision, shape, 6)[0]
    # FP64: 1e-7 of the scale as in the parity tests; FP32: 2^-24 amplified by the penalty (3e-4)
    tol = 1e-7 if precision == "fp64" else 3e-4
    for k, ok in (("x", "xl"), ("z", "zl"), ("lam", "ll"), ("zb", "zb"), ("nu", "nu")):
        np.testing.assert_allclose(got[k], st[ok], rtol=0, atol=tol * max(1.0, np.abs(st[ok]).max()), err_msg=k)


def test_bus_tasks_of_a_batch_that_thins_out():
    """Bus tasks in runs per CTA while most instances take part, round all
    warps after that, or (many warps) round all warps throughout: an instance's
    arithmetic is the same, bit for bit."""
    grids = [gg.grid_30bus()] * 6 + gg.scenarios_cholesky(gg.grid_2000bus(), 6, 1)
    o = binding.default_sqp(tol=1e-2, max_sqp=8, admm=dict(rho=2e4, max_iter=200, eps=1e-3, eps_dual=5e-3))
    out = []
    for shape in ((64, 1, 0), (256, 0, 0)):
        s = binding.Solver(grids, precision="mixed")
        s.tune(*shape)
        s.sqp_solve(o)
        out.append([(s.get_residuals(k), s.get_iterate(k)) for k in range(len(grids))])
        s.close()
    assert len({r["sqp_iter"] for r, _ in out[0]}) > 1  # the batch did thin out
    for (ra, ia), (rb, ib) in zip(*out):
        assert (ra["sqp_iter"], ra["admm_iter"]) == (rb["sqp_iter"], rb["admm_iter"])
        for a, b in zip(ia, ib):
            np.testing.assert_array_equal(a, b)
