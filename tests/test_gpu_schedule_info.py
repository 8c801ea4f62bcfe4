"""What fd_grid_info says of a run under AUTO: per-cell weights on column waves
above the limit of the bricks (the same bits as equal shares) and on bricks
below it, whatever ran before, and the CTAs of a step on bricks."""
import numpy as np
import pytest

from test_gpu_brick import equal, forward, workload

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


def percell(fd, w):
    import oracle
    rng = np.random.default_rng(4)
    c = (oracle.fd_coefficients(4)[1:] *
         (1 + 0.1 * rng.uniform(-1, 1, w["v"].shape + (4,)))).astype(np.float32)
    return lambda g: fd.check(
        fd.fd_set_coefficients(g.handle, c.ctypes.data, fd.FD_COEF_PER_CELL), "per-cell")


def test_percell_weights_run_column_waves_above_the_bricks(fd):
    w = workload(8, (150, 131, 137), 4, 8)
    a, info = forward(fd, w, False, percell(fd, w))
    assert info["schedule"] == fd.FD_SCHED_WAVES
    assert (info["tile_x"], info["tile_y"]) in [(32, 16), (64, 8)]
    b, shares = forward(fd, w, True, percell(fd, w))
    assert shares["schedule"] == fd.FD_SCHED_SHARES
    equal(a, b)


def test_percell_run_replaces_the_schedule_of_the_run_before(fd):
    w = workload(8, (40, 31, 25), 4, 8)
    with fd.Grid.from_workload(w) as g:
        g.set_model(w["v"])
        rec = np.zeros((w["nt"], len(w["rec"])), np.float32)
        g.set_schedule(fd.FD_SCHED_WAVES)
        fd.check(g.forward(w["src"], w["wavelet"], w["rec"], rec), "fd_forward")
        assert g.info()["schedule"] == fd.FD_SCHED_WAVES
        percell(fd, w)(g)
        g.set_schedule(fd.FD_SCHED_AUTO)
        fd.check(g.forward(w["src"], w["wavelet"], w["rec"], rec), "fd_forward")
        assert g.info()["schedule"] == fd.FD_SCHED_SHARES


@pytest.mark.parametrize("n,nbl,bricks", [((32, 8, 8), 0, 1), ((33, 9, 9), 0, 8),
                                          ((53, 38, 41), 6, 3 * 7 * 7)])
def test_ctas_of_a_step_on_bricks(fd, n, nbl, bricks):
    _, info = forward(fd, workload(8, n, nbl, 8), False)
    assert info["ctas"] == bricks
