"""Read-outs of one instance (acopf_get_iterate, _step, _solution): every block
in the caller's order, for generators given out of bus order and instances of
unequal size read in any order, on the default and on another stream."""
import ctypes as C
from dataclasses import replace

import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu


def _shuffled(g, seed):
    p = np.random.default_rng(seed).permutation(g.ngen)
    return replace(g, **{n: getattr(g, n)[p] for n in ("gbus", "pmin", "pmax", "qmin", "qmax", "c2", "c1", "c0")})


@pytest.mark.parametrize("order", [(0, 1, 2, 3), (3, 2, 1, 0)])
@pytest.mark.parametrize("own_stream", [False, True])
def test_values_come_back_where_they_were_put(order, own_stream):
    import torch

    grids = [gg.two_bus(), _shuffled(gg.grid_30bus(), 1), _shuffled(gg.geometric_grid(118, seed=7), 2),
             _shuffled(gg.geometric_grid(257, seed=9), 3)]
    s = binding.Solver(grids, precision="mixed")
    stream = torch.cuda.Stream() if own_stream else None
    if stream:
        s.set_stream(stream.cuda_stream)
    rng = np.random.default_rng(4)
    put = []
    for k, g in enumerate(grids):
        x, pi = 1 + 0.1 * rng.standard_normal(s.nvars(k)), rng.standard_normal(4 * g.nbranch)
        s.set_iterate(k, x, pi)
        put.append((x, pi))
    for k in order:
        x, pi = s.get_iterate(k)
        np.testing.assert_array_equal(x, put[k][0])
        np.testing.assert_array_equal(pi, put[k][1])
        sol, G, B = s.get_solution(k), grids[k].ngen, grids[k].nbus
        np.testing.assert_array_equal(np.concatenate([sol["pg"], sol["qg"]]), x[:2 * G])
        np.testing.assert_array_equal(sol["vm"], np.sqrt(x[2 * G:2 * G + B]))
        np.testing.assert_array_equal(np.concatenate([sol["va"], sol["wr"], sol["wi"]]), x[2 * G + B:])
    # the step: the generators' x and the buses' values of the ADMM state, FP32 values exactly
    s.admm_solve_qp(0.5, binding.default_admm(eps=0.0, max_iter=5, warm=0))
    for k in order:
        g, st = grids[k], s.get_admm_state(k)
        d, pi = s.get_step(k)
        np.testing.assert_array_equal(d[:2 * g.ngen], st["xg"].T.ravel())
        np.testing.assert_array_equal(d[2 * g.ngen:2 * (g.ngen + g.nbus)], st["zb"].T.ravel())
        only = np.zeros(4 * g.nbranch)  # pi without the step
        assert binding.lib().acopf_get_step(s.h, k, None, only.ctypes.data_as(C.POINTER(C.c_double))) == 0
        np.testing.assert_array_equal(only, pi)
    s.close()
