"""The FP64 generator update (eq. gen_kernel) of the forms that keep the
reciprocals of its divisors has the bits of the form that divides."""
import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu


def test_generator_update_is_the_quotient():
    g = gg.geometric_grid(118, seed=7)
    rng = np.random.default_rng(3)
    st = {"zg": rng.uniform(-0.5, 1.5, (g.ngen, 2)), "lg": 1e3 * rng.standard_normal((g.ngen, 2))}
    out = []
    for shape in ((256, 0, 0), (64, 0, 3), (64, 0, 4)):
        s = binding.Solver(g, precision="fp64")
        s.tune(*shape)
        s.build_qp(1.0, 2e4, True)
        inside = 0
        for k in range(20):
            s.set_admm_state(0, {n: v * (1 + 0.01 * k) for n, v in st.items()})
            s.admm_iterate(1, binding.default_admm())
            out.append(s.get_admm_state(0)["xg"])
            inside += np.sum((out[-1] != out[-1].max()) & (out[-1] != 0))
        assert inside > 20
        s.close()
    for k in range(20):
        np.testing.assert_array_equal(out[20 + k], out[k])
        np.testing.assert_array_equal(out[40 + k], out[k])
