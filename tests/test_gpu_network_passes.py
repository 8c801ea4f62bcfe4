"""Network kernels over more than one pass of the GPU: inference on rows and on
a grid's cells (chunks of 128, four blocks per SM) where a block takes second
and third chunks and the activation tile is used again, and the gradient where
its staged samples are double-buffered (chunks of 64)."""
import numpy as np
import pytest

import oracle
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def learned(fd):
    from paper_2312_13094_gb300 import learned as lr
    return lr


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("size", ["127", "128", "129", "one pass and a row", "two and a half passes"])
def test_rows(learned, size):
    one = 4 * sms() * 128
    n = {"one pass and a row": one + 1, "two and a half passes": 5 * one // 2}.get(size) or int(size)
    th = mlp.init_params(5, scale_out=0.8).astype(np.float32)
    net = learned.Network(th)
    X = mlp.features(np.random.default_rng(n).uniform(1.5, 4.5, n), 20.0, 1.6, 12.0).astype(np.float32)
    got = net.coefficients(X)
    ref = mlp.coefficients(th.astype(np.float64), X.astype(np.float64), oracle.fd_coefficients(4))
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
    net.close()


@pytest.mark.parametrize("chunks", [1.0, 1.5, 2.5, 3.25])
def test_gradient(learned, chunks):
    """Chunks of 64, one block per SM up to four chunks and two beyond: two chunks of
    one block, three, two and a part of two blocks, and three and a part, so that
    both staging buffers are used again."""
    n = int(2 * sms() * 64 * chunks) + (3 if chunks > 1 else 0)
    rng = np.random.default_rng(n)
    S = np.concatenate([mlp.features(rng.uniform(1.5, 4.5, n), 20.0, 1.6, 12.0),
                        rng.standard_normal((n, 4)), 0.3 * rng.standard_normal((n, 1)),
                        rng.uniform(0.5, 2.0, (n, 1))], 1).astype(np.float32)
    th = mlp.init_params(8, scale_out=0.8).astype(np.float32)
    net = learned.Network(th)
    loss, g = net.loss_grad(np.ascontiguousarray(S))
    rl, rg = mlp.loss_grad(th.astype(np.float64), S.astype(np.float64), oracle.fd_coefficients(4))
    assert abs(loss - rl) <= 1e-5 * abs(rl)
    assert np.linalg.norm(g - rg) <= 1e-4 * np.linalg.norm(rg)
    net.close()


@pytest.mark.parametrize("n", [(67, 59, 61), (64, 32, 38), (65, 3, 5)])
def test_every_cell_of_a_grid_takes_its_own_weights(fd, learned, n):
    """One step from a random state with a velocity of its own in every cell,
    element by element: u+ = 2u - u- + A sum_j c_j d_j.  A <= 0.09 and |d_j| <= 12,
    so four weights within 1e-5 of the largest (below 2.4) leave 1.04e-4, and the
    FP32 sums 5e-6 more; a neighbour's weights differ by far more at most cells."""
    h, v_max = 20.0, 4.5
    dt = 0.3 * h / v_max
    rng = np.random.default_rng(7)
    shape = n[::-1]
    v = rng.uniform(1.5, v_max, shape).astype(np.float32)
    um, u = (rng.uniform(-1, 1, shape).astype(np.float32) for _ in range(2))
    th = mlp.init_params(9, scale_out=1.0).astype(np.float32)
    net = learned.Network(th)
    with fd.Grid(n, h, 8, 0, dt, 4) as g:
        g.set_model(v)
        fd.check(fd.fd_set_learned_coefficients(g.handle, net.handle, 12.0), "learned")
        g.set_wavefield(um, u)
        fd.check(g.propagate(0, 1), "fd_propagate")
        got = np.zeros(shape, np.float32)
        g.get_wavefield(np.zeros(shape, np.float32), got)
    net.close()
    c = mlp.coefficients(th.astype(np.float64),
                         mlp.features(v.astype(np.float64), h, dt, 12.0).reshape(-1, 4),
                         oracle.fd_coefficients(4)).reshape(shape + (4,))
    p = np.pad(u.astype(np.float64), 4)
    lap = np.zeros(shape)
    for j in range(1, 5):
        s = -6.0 * u.astype(np.float64)
        for axis in range(3):
            for o in (-j, j):
                at = [slice(4, 4 + m) for m in shape]
                at[axis] = slice(4 + o, 4 + o + shape[axis])
                s = s + p[tuple(at)]
        lap += c[..., j - 1] * s
    want = 2.0 * u - um + (v.astype(np.float64) * dt / h) ** 2 * lap
    assert np.abs(got - want).max() <= 1.1e-4
