"""The training gradient is a sum over blocks of samples: that sum adds one
rounding, whatever the number of blocks, and its order is fixed.

B copies of the same eight samples make B blocks with the same partial sums
(one block per eight samples up to one block per SM).  With B a power of two
the factor 1/n scales every term exactly, so the gradient of the B copies is
that of the eight samples to the last bit; adding the blocks to an FP32 word
one after the other rounds at every block that is no power of two."""
import numpy as np
import pytest

import oracle
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def learned():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import learned as lr
    return lr


def samples(n, seed):
    rng = np.random.default_rng(seed)
    X = mlp.features(rng.uniform(1.5, 4.5, n), 20.0, 1.6, 12.0)
    T = rng.standard_normal((n, 4))
    y = rng.standard_normal(n) * 0.3
    w = rng.uniform(0.5, 2.0, n)
    return np.ascontiguousarray(np.concatenate([X, T, y[:, None], w[:, None]], 1), np.float32)


@pytest.mark.parametrize("copies", [2, 16, 32, 64, 128])
def test_equal_blocks_add_up_exactly(learned, copies):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count < copies:
        pytest.skip("fewer blocks than copies")
    net = learned.Network(mlp.init_params(11, scale_out=0.8).astype(np.float32))
    S = samples(8, 5)
    loss1, g1 = net.loss_grad(S)
    loss, g = net.loss_grad(np.ascontiguousarray(np.tile(S, (copies, 1))))
    net.close()
    assert np.abs(g1).max() > 0
    np.testing.assert_array_equal(g, g1)
    assert abs(loss - loss1) <= 1e-14 * abs(loss1)  # FP64 sums of 64 terms at most per thread


@pytest.mark.parametrize("n", [1050, 65536])
def test_gradient_is_the_same_on_every_call(learned, n):
    net = learned.Network(mlp.init_params(12, scale_out=0.8).astype(np.float32))
    S = samples(n, 6)
    loss, g = net.loss_grad(S)
    for _ in range(3):
        again = net.loss_grad(S)
        assert again[0] == loss
        np.testing.assert_array_equal(again[1], g)
    net.close()


@pytest.mark.parametrize("n", [8, 16, 17, 248, 256, 264, 1216, 1224, 38912, 38913])
def test_numbers_of_blocks_around_a_row_of_the_sum(learned, n):
    """One block, two, counts around the 32 rows that are summed side by side, the
    first that gives a block of 152 SMs a second unit, and the last with one block
    per SM and the first with two."""
    th = mlp.init_params(13, scale_out=0.8).astype(np.float32)
    net = learned.Network(th)
    S = samples(n, n)
    loss, g = net.loss_grad(S)
    rl, rg = mlp.loss_grad(th.astype(np.float64), S.astype(np.float64),
                           oracle.fd_coefficients(4))
    assert abs(loss - rl) <= 1e-5 * abs(rl)
    assert np.linalg.norm(g - rg) <= 1e-4 * np.linalg.norm(rg)
    net.close()
