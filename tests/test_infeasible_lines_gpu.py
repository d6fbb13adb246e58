"""FP64 line subproblems without a feasible point (an angle window that the
trust region cannot reach), next to feasible ones: the forms that keep active
sets leave them to the general solves and agree with the form that keeps none."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu
KEYS = ("x", "z", "lam", "xg", "zg", "lg", "zb", "nu", "ul")


@pytest.mark.parametrize("share", [0.1, 1.0])
def test_forms_agree_on_infeasible_lines(share):
    g = gg.geometric_grid(60, seed=4)
    r = np.random.default_rng(5)
    tight = r.random(g.nbranch) < share
    g = replace(g, angmin=np.where(tight, -0.01, -1.0), angmax=np.where(tight, 0.01, 1.0))
    theta = 0.3 * r.standard_normal(g.nbus)
    # a branch cannot reach its window when its ends' steps of at most delta leave it outside
    delta = 0.05
    far = tight & (np.abs(theta[g.f] - theta[g.t]) > 0.01 + 2 * delta)
    assert far.sum() >= 3
    out = []
    for shape in ((256, 0, 0), (32, 0, 3), (256, 0, 3), (64, 0, 4)):
        s = binding.Solver(g, precision="fp64")
        s.tune(*shape)
        x, _ = s.get_iterate(0)
        x[2 * g.ngen + g.nbus:2 * (g.ngen + g.nbus)] = theta
        s.set_iterate(0, x)
        s.build_qp(delta, 2e4, True)
        for n in (3, 5):
            s.admm_iterate(n, binding.default_admm())
        out.append(s.get_admm_state(0))
        s.close()
    for got in out[1:]:
        for k in KEYS:
            # the bound of the agreement of the forms on feasible subproblems
            np.testing.assert_allclose(got[k], out[0][k], rtol=0, atol=1e-9 * max(1.0, np.abs(out[0][k]).max()), err_msg=k)
