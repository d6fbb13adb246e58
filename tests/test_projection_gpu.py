"""The linear projection (eq. linfeas) where its kernels' branches change: box
QPs with both end voltages at their bounds, buses with a fixed voltage, shunts
and a hub of more than 31 entries, and a grid longer than one window of the
degree ordering."""
from dataclasses import replace

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grids(name):
    from paper_2310_13143_gb300 import gridgen as gg

    g = {"30": gg.grid_30bus, "hub": lambda: gg.hub_grid(40), "1100": lambda: gg.geometric_grid(1100, seed=4)}[name]()
    r = np.random.default_rng(2)
    vmin, vmax = np.full(g.nbus, 0.99), np.full(g.nbus, 1.01)
    fixed = r.random(g.nbus) < 0.2
    vmin[fixed] = vmax[fixed] = 1.0
    return replace(g, vmin=vmin, vmax=vmax, gs=r.uniform(-0.1, 0.1, g.nbus), bs=r.uniform(-0.2, 0.2, g.nbus))


@pytest.mark.parametrize("name", ["30", "hub", "1100"])
def test_projection_with_tight_voltage_bounds(name):
    import oracle
    from oracle import linfeas as olf
    from paper_2310_13143_gb300 import binding

    g = _grids(name)
    r = np.random.default_rng(7)
    x0 = np.concatenate([r.uniform(0, 1, 2 * g.ngen), 1 + 0.2 * r.standard_normal(g.nbus),
                         0.1 * r.standard_normal(g.nbus), 1 + 0.2 * r.standard_normal(g.nbranch),
                         0.2 * r.standard_normal(g.nbranch)])
    s = binding.Solver([g, g], precision="fp64")
    for k in range(2):
        s.set_iterate(k, x0)
    it, rp, rd = s.project_linear(rho=0.5, eps=1e-10, max_iter=100000)
    assert rp <= 1e-10 and rd <= 1e-10, (it, rp, rd)
    want, _ = olf.project(oracle.Model(g), x0)
    w = want[2 * g.ngen:2 * g.ngen + g.nbus]
    at = (w <= g.vmin ** 2 + 1e-9) | (w >= g.vmax ** 2 - 1e-9)
    assert np.sum(at[g.f] & at[g.t]) >= 3  # branches whose two ends are at their bounds
    for k in range(2):
        # residuals of 1e-10 leave the point within about 1e-8 of the projection
        np.testing.assert_allclose(s.get_iterate(k)[0], want, atol=2e-7)
    s.close()


def test_nan_start_does_not_pass_the_residual_test():
    from paper_2310_13143_gb300 import binding, gridgen as gg

    g = gg.grid_30bus()
    s = binding.Solver(g, precision="fp64")
    x, _ = s.get_iterate(0)
    x[2 * g.ngen + 3] = np.nan
    s.set_iterate(0, x)
    it, rp, _ = s.project_linear(rho=0.5, eps=1e-4, max_iter=100)
    assert it == 100 and rp > 1e-4
    s.close()
