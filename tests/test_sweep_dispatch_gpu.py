"""The sweep's dispatch on both sides of its lines, with the sizes taken from
the device's number of SMs: four FP64 lanes per branch as long as generators
and branches fit the co-resident threads, and bus tasks in contiguous runs per
CTA where warps have four or more and most of the batch takes part."""
import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KEYS = ("x", "z", "lam", "xg", "zg", "lg", "zb", "nu", "ul")


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _tasks(grids):
    """Warp tasks of a batch: consecutive whole buses of one instance with at
    most 32 generators and branch ends; buses with more are not among them."""
    n = 0
    for g in grids:
        entries = np.bincount(g.f, minlength=g.nbus) + np.bincount(g.t, minlength=g.nbus) + np.bincount(g.gbus, minlength=g.nbus)
        held = 0
        for e in entries:
            if e > 32 or held + e > 32:
                n += held > 0
                held = 0
            held += e if e <= 32 else 0
        n += held > 0
    return n


@pytest.mark.parametrize("fits", [True, False])
def test_four_lanes_device_wide_to_the_last_thread(fits):
    room = _sms() * 256  # one CTA of 256 threads per SM
    need = lambda g: g.ngen + 4 * g.nbranch
    buses, beyond = room // 7, room // 5  # 5.6 threads per bus
    while beyond - buses > 1:
        mid = (buses + beyond) // 2
        buses, beyond = (mid, beyond) if need(gg.geometric_grid(mid, seed=1)) <= room else (buses, mid)
    g = gg.geometric_grid(buses if fits else beyond, seed=1)
    assert (need(g) <= room) == fits and abs(need(g) - room) < 64
    out = []
    for shape in ((256, 0, 0), (256, 0, 3)):
        s = binding.Solver(g, precision="fp64")
        s.tune(*shape)
        s.build_qp(1.0, 2e4, True)
        for _ in range(2):
            s.admm_iterate(10, binding.default_admm())
        out.append(s.get_admm_state(0))
        s.close()
    for k in KEYS:
        # both forms return the line subproblems' unique KKT points
        np.testing.assert_allclose(out[1][k], out[0][k], rtol=0, atol=1e-9 * max(1.0, np.abs(out[0][k]).max()), err_msg=k)


def test_runs_of_bus_tasks_in_a_batch_that_thins_out():
    """An instance's arithmetic is the same bit for bit in runs per CTA, round
    all warps once most instances have finished, and round all warps
    throughout."""
    grids = [gg.grid_30bus()] * 6 + gg.scenarios_cholesky(gg.grid_2000bus(), 6, 1)
    tasks, work = _tasks(grids), sum(g.ngen + g.nbranch for g in grids)
    few, many = (32, 1, 0), (256, 0, 0)
    assert -(-work // 32) > _sms() and tasks >= 4 * _sms()  # one warp per SM, at least four tasks each: runs
    assert -(-work // 256) <= _sms() and tasks < 4 * 8 * -(-work // 256)  # eight warps per 256 components: no runs
    o = binding.default_sqp(tol=1e-2, max_sqp=8, admm=dict(rho=2e4, max_iter=200, eps=1e-3, eps_dual=5e-3))
    out = []
    for shape in (few, many):
        s = binding.Solver(grids, precision="mixed")
        s.tune(*shape)
        s.sqp_solve(o)
        out.append([(s.get_residuals(k), s.get_iterate(k)) for k in range(len(grids))])
        s.close()
    iters = [r["admm_iter"] for r, _ in out[0]]
    assert sum(i < max(iters) for i in iters) > len(grids) // 4  # fewer than three in four take part at the end
    for (ra, ia), (rb, ib) in zip(*out):
        assert (ra["sqp_iter"], ra["admm_iter"]) == (rb["sqp_iter"], rb["admm_iter"])
        for a, b in zip(ia, ib):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("case", ["large grid", "many instances"])
def test_many_passes_and_tasks_per_warp(case):
    """More than eight passes over the components and more than 32 tasks per
    warp: tasks round all warps for a large grid, in runs for many instances;
    the same bits as with many threads."""
    sms = _sms()
    if case == "large grid":
        grids = [gg.geometric_grid(60000 * sms // 152, seed=3)]
    else:
        grids = gg.scenarios_cholesky(gg.grid_2000bus(), 32 * sms // 152, 2)
    tasks, work = _tasks(grids), sum(g.ngen + g.nbranch for g in grids)
    assert work > 8 * 32 * sms and tasks > 32 * sms  # one warp per SM
    assert (tasks > 1024 * len(grids)) == (case == "large grid")
    out = []
    for shape in ((32, 1, 0), (256, 0, 0)):
        s = binding.Solver(grids, precision="mixed")
        s.tune(*shape)
        s.build_qp(1.0, 2e4, True)
        s.admm_iterate(6, binding.default_admm())
        out.append([s.get_admm_state(k) for k in range(len(grids))])
        s.close()
    for a, b in zip(*out):
        for k in KEYS:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
