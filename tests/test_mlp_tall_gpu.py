"""Inference in chunks of more rows than a grid's second dimension has tiles of
32: the same bits as in chunks of 4,096 rows."""
import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tall_chunk():
    rows, dims = 32 * 65536 + 100, [8, 16, 8]
    X = torch.randn(rows, 8, device="cuda")
    out = []
    for batch in (4096, rows):
        net = binding.Mlp(dims, max_batch=batch)
        net.set_params(gg.mlp_init(dims, seed=1))
        Y = torch.full((rows, 8), float("nan"), device="cuda")
        net.forward(X.data_ptr(), rows, Y.data_ptr())
        net.close()
        out.append(Y)
    assert torch.isfinite(out[0]).all() and torch.equal(*out)
