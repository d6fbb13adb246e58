"""Handles of different launch shapes used in turn: the sweeps' kernels are
shared by all handles of a device, so nothing that one handle sets for its own
launch may reach another's."""
import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu
KEYS = ("x", "z", "lam", "xg", "zg", "lg", "zb", "nu", "ul")


def _open(buses, threads, stages, precision):
    s = binding.Solver(gg.geometric_grid(buses, seed=buses), precision=precision)
    s.tune(threads, 0, stages)
    s.build_qp(1.0, 2e4, True)
    return s


# FP64 clusters with one lane per branch: kept operators of 59,392 and 29,696
# bytes per CTA, on both sides of what a kernel may take without a raised limit;
# with four lanes 14,848 and 3,712.  FP64 device-wide with one lane, and FP32
# clusters with the exchanged state in shared memory
@pytest.mark.parametrize("precision,stages,large,small", [
    ("fp64", 4, (2000, 256), (1000, 128)), ("fp64", 4, (300, 256), (300, 64)), ("fp64", 3, (9000, 256), (4000, 64)),
    ("mixed", 4, (2000, 256), (300, 64))])
def test_handles_of_two_shapes_in_turn(precision, stages, large, small):
    o = binding.default_admm()
    want = []
    for buses, threads in (large, small):
        s = _open(buses, threads, stages, precision)
        for _ in range(2):
            s.admm_iterate(4, o)
        want.append(s.get_admm_state(0))
        s.close()
    a, b = _open(*large, stages, precision), _open(*small, stages, precision)
    for s in (a, b, a, b):
        s.admm_iterate(4, o)
    for s, w in zip((a, b), want):
        got = s.get_admm_state(0)
        for k in KEYS:
            np.testing.assert_array_equal(got[k], w[k], err_msg=k)
        s.close()
