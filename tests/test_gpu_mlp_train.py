"""Training launches of the learned proposal at the edges of their tiles: row counts around the 16-row halves and 32-row
tiles of a block, and beyond the blocks of one wave (each then takes several tiles), against the reference with the
kernels' BF16 rounding points; training reproduces itself bit for bit (no atomics on the gradient), also with a last
batch of a single row.

Tolerance of a gradient block, relative to its norm: FP32 sums of m terms in chains of 16 and 32 and then over blocks
carry below (16 + 2 + m / 32) u of the sum of magnitudes, which for m <= 20001 stays below 1e-4 of it; a block's
gradient is at least a tenth of that sum here; the reference rounds A1 and dH2 to BF16 from FP64 rather than FP32
values, which moves one in 2^16 operands by 2^-8: another 1e-4. Held to 2e-3, ten times their sum, as in test_gpu_mlp.py."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import emppp, inputs  # noqa: E402

_BLOCKS = [(mlp.OFF_W1, mlp.OFF_B1), (mlp.OFF_B1, mlp.OFF_W2), (mlp.OFF_W2, mlp.OFF_B2), (mlp.OFF_B2, mlp.OFF_W3),
           (mlp.OFF_W3, mlp.OFF_B3), (mlp.OFF_B3, mlp.NUM_PARAMS)]


def _data(m, seed):
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(m, 10)).astype(np.float32)
    return X, (1.0 + 0.3 * X[:, 0] + 0.1 * rng.normal(size=m)).astype(np.float32)


@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 31, 32, 33, 48, 1000, 9729, 20001])
def test_gradient_at_tile_edges(m):
    X, T = _data(m, m)
    p = inputs.mlp_init_params(7)
    loss, g = emppp.mlp_gradient(p, X, T)
    loss_r, g_r = mlp.loss_and_grad(p, X, T, rounding=True)
    assert abs(loss - loss_r) <= 1e-3 * loss_r
    for a, b in _BLOCKS:
        assert np.linalg.norm(g[a:b] - g_r[a:b]) <= 2e-3 * np.linalg.norm(g_r[a:b]), (m, a)


@pytest.mark.parametrize("rows,batch", [(257, 256), (700, 64), (33, 33), (12000, 10000)])
def test_training_is_reproducible(rows, batch):
    X, T = _data(rows, 3)
    p0 = inputs.mlp_init_params(8)
    a, la = emppp.mlp_train(p0, X, T, epochs=2, batch=batch, lr=1e-3, lr_final=1e-4)
    b, lb = emppp.mlp_train(p0, X, T, epochs=2, batch=batch, lr=1e-3, lr_final=1e-4)
    assert np.array_equal(a, b)
    assert np.all(np.isfinite(a)) and not np.array_equal(a, p0)
    assert np.allclose(la, lb, rtol=1e-5) and la[1] < la[0]
