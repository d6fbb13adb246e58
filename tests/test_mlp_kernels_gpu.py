"""The network's kernels at the edges of their tiles: widths that end inside a
64-column tile, batches of one row, of one less and one more than a row tile,
a single layer, and data that is only 4-byte aligned.  Gradients, the bias
gradients and the loss of one training step against the FP64 oracle, then two
further steps against the oracle's Adam on the kernels' own gradients."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2310_13143_gb300 import binding, gridgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _split(flat, dims):
    out, o = [], 0
    for i, n in zip(dims, dims[1:]):
        w = flat[o:o + i * n].reshape(n, i)
        o += i * n
        out.append((w, flat[o:o + n]))
        o += n
    return out


def _on_device(a, offset):
    """A device copy whose address is 4 * offset bytes past an aligned one."""
    t = torch.zeros(a.size + offset, device="cuda")
    t[offset:] = torch.from_numpy(a).reshape(-1).cuda()
    return t, t.data_ptr() + 4 * offset


@pytest.mark.parametrize("dims,rows,offset", [([8, 8], 1, 0), ([24, 72, 72], 127, 0), ([72, 136, 200], 129, 1),
                                              ([40, 64, 64, 8], 130, 3), ([64, 512, 512, 712], 100, 0)])
def test_training_steps_at_tile_edges(dims, rows, offset):
    rng = np.random.default_rng(sum(dims) + rows)
    n = rows + 5
    X = (1.0 + rng.standard_normal((n, dims[0]))).astype(np.float32)
    T = (2.0 * rng.standard_normal((n, dims[-1])) - 1.0).astype(np.float32)
    net = binding.Mlp(dims, max_batch=rows)
    flat = gg.mlp_init(dims, seed=3)
    for (_, b) in _split(flat, dims):
        b[:] = 0.1 * rng.standard_normal(b.size)
    net.set_params(flat)
    (xk, xp), (tk, tp) = _on_device(X, offset), _on_device(T, offset)
    net.fit_standardiser(xp, tp, n)
    mx, sx, my, sy = net.get_standardiser()
    idx = rng.permutation(n)[:rows].astype(np.int32)
    idxd = torch.from_numpy(idx).cuda()
    loss = torch.zeros(1, device="cuda")
    m = v = 0.0
    for step in range(1, 4):
        before = net.get_params().astype(np.float64)
        net.train_step(xp, tp, idxd.data_ptr(), rows, 1e-3, loss.data_ptr())
        net.sync()
        g = net.get_grads().astype(np.float64)
        # oracle of this step from the parameters the kernels started from
        params = [(w.astype(np.float64), b.astype(np.float64)) for w, b in _split(before, dims)]
        Y, cache = omlp.forward(params, (X[idx].astype(np.float64) - mx) / sx, q=omlp.bf16_round)
        ol, dY = omlp.mse(Y, (T[idx].astype(np.float64) - my) / sy)
        assert abs(loss.item() - ol) <= 1e-3 * ol
        for (gw, gb), (ow, ob) in zip(_split(g, dims), omlp.backward(params, cache, dY, q=omlp.bf16_round)):
            # bfloat16 gradients: a rounding that falls differently moves a term by 2^-8
            assert np.max(np.abs(gw - ow)) <= 2 ** -7 * (np.max(np.abs(ow)) + 1e-30)
            assert np.max(np.abs(gb - ob)) <= 2 ** -7 * (np.max(np.abs(ob)) + 1e-30)
        # Adam on the kernels' own gradients: FP32 rounding of a step of at most 1e-3
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        want = before - 1e-3 * (m / (1 - 0.9 ** step)) / (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
        after = net.get_params()
        np.testing.assert_allclose(after, want, rtol=2 ** -22, atol=1e-3 * 2 ** -12)
    net.close()
    del xk, tk


@pytest.mark.parametrize("dims,batch,rows", [([16, 32, 24], 128, 1), ([64, 512, 512, 712], 128, 129),
                                             ([40, 72, 20488], 256, 128), ([40, 72, 20488], 256, 130),
                                             ([4104, 264, 136], 256, 257)])
def test_inference_at_tile_edges(dims, batch, rows):
    """Outputs straight from the product's epilogue: one row, one more than a
    block of rows, an output layer whose tiles are narrower for one block of
    rows than for two, and a first layer summed from splits; nothing is
    written past the rows asked for."""
    rng = np.random.default_rng(dims[-1] + rows)
    X = rng.standard_normal((rows, dims[0])).astype(np.float32)
    T = (3.0 * rng.standard_normal((64, dims[-1])) + 1.0).astype(np.float32)
    fit = rng.standard_normal((64, dims[0])).astype(np.float32)
    net = binding.Mlp(dims, max_batch=batch)
    flat = gg.mlp_init(dims, seed=4)
    for (_, b) in _split(flat, dims):
        b[:] = 0.1 * rng.standard_normal(b.size)
    net.set_params(flat)
    Xd, Td, Fd = (torch.from_numpy(a).cuda() for a in (X, T, fit))
    net.fit_standardiser(Fd.data_ptr(), Td.data_ptr(), 64)
    mx, sx, my, sy = net.get_standardiser()
    Yd = torch.full((rows + 1, dims[-1]), 7.0, device="cuda")
    net.forward(Xd.data_ptr(), rows, Yd.data_ptr())
    params = [(w.astype(np.float64), b.astype(np.float64)) for w, b in _split(flat, dims)]
    Y, _ = omlp.forward(params, (X.astype(np.float64) - mx) / sx, q=omlp.bf16_round)
    got = Yd.cpu().double().numpy()
    want = Y * sy + my
    assert np.max(np.abs(got[:rows] - want)) <= 2 ** -7 * np.max(np.abs(want))
    assert (got[rows] == 7.0).all()
    net.close()
