"""Values given to a handle on a stream of its own arrive there, whatever the
default stream is doing: each setter is followed at once by a read-out or a
kernel of the handle's stream while another thread keeps the default stream
busy."""
import threading

import numpy as np
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def busy_default_stream():
    stop = threading.Event()

    def work():
        while not stop.is_set():
            torch.cuda._sleep(1_000_000)  # about half a millisecond
            torch.cuda.default_stream().synchronize()

    t = threading.Thread(target=work)
    t.start()
    yield
    stop.set()
    t.join()


def test_solver_setters(busy_default_stream):
    grids = [gg.grid_30bus(), gg.geometric_grid(118, seed=7)]
    s = binding.Solver(grids, precision="fp64")
    s.set_stream(torch.cuda.Stream().cuda_stream)
    rng = np.random.default_rng(2)
    for i in range(20):
        k = i % 2
        L, G = grids[k].nbranch, grids[k].ngen
        x, pi = rng.standard_normal(s.nvars(k)), rng.standard_normal(4 * L)
        s.set_iterate(k, x, pi)
        got = s.get_iterate(k)
        np.testing.assert_array_equal(got[0], x)
        np.testing.assert_array_equal(got[1], pi)
        x = rng.standard_normal(s.nvars(k))
        s.set_warm_start(k, x0=x, lambda0=rng.standard_normal(8 * L + 2 * G), rho=np.full(L + G, 10.0 + i))
        got = s.get_iterate(k)
        np.testing.assert_array_equal(got[0], x)
        np.testing.assert_array_equal(got[1], 0.0)
        st = {"x": rng.standard_normal((L, 8)), "zg": rng.standard_normal((G, 2)), "nu": rng.standard_normal((grids[k].nbus, 2))}
        s.set_admm_state(k, st)
        got = s.get_admm_state(k)
        for n, v in st.items():
            np.testing.assert_array_equal(got[n], v)
    s.close()


def test_network_parameters(busy_default_stream):
    dims = [64, 512, 512, 136]
    flat = [gg.mlp_init(dims, seed=k) for k in range(2)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        X = torch.randn(128, 64, device="cuda")
        Y = [torch.zeros(128, 136, device="cuda") for _ in range(2)]
    out = []
    for i in range(6):
        net = binding.Mlp(dims, max_batch=128)
        net.set_stream(stream.cuda_stream)
        net.set_params(flat[i % 2])
        net.forward(X.data_ptr(), 128, Y[i % 2].data_ptr())
        with torch.cuda.stream(stream):
            out.append(Y[i % 2].clone().cpu())
        net.close()
    for k in range(2):
        assert torch.equal(out[k], out[k + 2]) and torch.equal(out[k], out[k + 4])
    assert not torch.equal(out[0], out[1])
