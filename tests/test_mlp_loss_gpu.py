"""The training loss over the range of FP32: its squares are summed in FP64, so
errors whose squares lie outside the FP32 range still give the mean's value."""
import numpy as np
import pytest

from paper_2310_13143_gb300 import binding

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _loss(T, rows):
    """Loss of a zero network, whose errors are -T."""
    net = binding.Mlp([8, T.shape[1]], max_batch=rows)
    net.set_params(np.zeros(net.nparams, np.float32))
    X, Td = torch.zeros(rows, 8, device="cuda"), torch.from_numpy(T).cuda()
    out = torch.full((1,), -1.0, device="cuda")
    net.train_step(X.data_ptr(), Td.data_ptr(), None, rows, 1e-3, out.data_ptr())
    net.sync()
    net.close()
    return out.item()


@pytest.mark.parametrize("value", [1e-21, 1e-19, 3e-5, 1.0, 1e18, 2e19, 3e20])
@pytest.mark.parametrize("rows,width", [(128, 8), (130, 200)])
def test_loss_of_one_large_and_many_small_errors(value, rows, width):
    rng = np.random.default_rng(rows)
    T = (1e-3 * value * rng.standard_normal((rows, width))).astype(np.float32)
    T[rows // 2, width // 3] = value
    want = np.mean(T.astype(np.float64) ** 2)
    # the FP64 mean rounded to FP32, of which a subnormal has fewer digits
    assert abs(_loss(T, rows) - want) <= 2.0 ** -24 * want * (1 + 1e-9) + 2.0 ** -149


def test_loss_of_infinite_and_nan_errors():
    T = np.zeros((128, 16), np.float32)
    T[5, 3] = np.inf
    assert _loss(T, 128) == np.inf
    T[5, 3] = np.nan
    assert np.isnan(_loss(T, 128))


# one run of rows and several: a wide layer, one whose last run is shorter, one
# of a single column block with as many runs as row tiles, one row tile
@pytest.mark.parametrize("width,rows", [(40000, 300), (2600, 1000), (8, 2000), (712, 4100), (72, 100)])
def test_loss_and_output_bias_gradient_over_runs_of_rows(width, rows):
    rng = np.random.default_rng(width + rows)
    T = rng.standard_normal((rows, width)).astype(np.float32)
    net = binding.Mlp([8, width], max_batch=rows)
    net.set_params(np.zeros(net.nparams, np.float32))
    X, Td = torch.zeros(rows, 8, device="cuda"), torch.from_numpy(T).cuda()
    out = torch.zeros(1, device="cuda")
    net.train_step(X.data_ptr(), Td.data_ptr(), None, rows, 1e-3, out.data_ptr())
    net.sync()
    want = np.mean(T.astype(np.float64) ** 2)
    assert abs(out.item() - want) <= 2.0 ** -23 * want
    # 2 (Y - T) / (rows N) rounded to bfloat16, summed in FP32 in row order: the same bits
    g = torch.from_numpy(np.float32(2) * -T / (np.float32(rows) * np.float32(width))).bfloat16().float().numpy()
    s = np.zeros(width, np.float32)
    for r in range(rows):
        s = s + g[r]
    np.testing.assert_array_equal(net.get_grads()[8 * width:], s)
    net.close()


@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_loss_at_any_address(offset):
    """The loss may be asked for at any byte address of device memory."""
    rows, T = 128, torch.ones(128, 16, device="cuda")
    net = binding.Mlp([8, 16], max_batch=rows)
    net.set_params(np.zeros(net.nparams, np.float32))
    X, out = torch.zeros(rows, 8, device="cuda"), torch.full((12,), 7, dtype=torch.uint8, device="cuda")
    net.train_step(X.data_ptr(), T.data_ptr(), None, rows, 1e-3, out.data_ptr() + offset)
    net.sync()
    got = out.cpu().numpy()
    assert got[offset:offset + 4].copy().view(np.float32)[0] == 1.0
    assert (got[:offset] == 7).all() and (got[offset + 4:] == 7).all()
    net.close()
