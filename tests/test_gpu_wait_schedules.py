"""A bounded device wait that runs out (the load of one plane is never issued)
on each kernel that serves a forward step: bricks, equal shares and column
waves, with one and with split staging of u^n, and per-cell weights under both
schedules.  The run reports the time-out, and the grid keeps working."""
import numpy as np
import pytest

from test_gpu_brick import workload

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


@pytest.mark.parametrize("sched", ["auto", "shares", "waves"])
@pytest.mark.parametrize("so,percell", [(4, False), (8, False), (12, False), (8, True)])
def test_time_out_and_recovery(fd, sched, so, percell):
    n = (45, 38, 41)
    w = workload(so, n, 4, 20)
    with fd.Grid.from_workload(w) as g:
        g.set_schedule({"auto": fd.FD_SCHED_AUTO, "shares": fd.FD_SCHED_SHARES,
                        "waves": fd.FD_SCHED_WAVES}[sched])
        g.set_model(w["v"])
        if percell:
            import oracle
            rng = np.random.default_rng(3)
            c = (oracle.fd_coefficients(4)[1:] *
                 (1 + 0.1 * rng.uniform(-1, 1, w["v"].shape + (4,)))).astype(np.float32)
            fd.check(fd.fd_set_coefficients(g.handle, c.ctypes.data, fd.FD_COEF_PER_CELL))
        ref = np.zeros((w["nt"], len(w["rec"])), np.float32)
        fd.check(g.forward(w["src"], w["wavelet"], w["rec"], ref), "clean run")
        assert np.abs(ref).max() > 0
        g.set_debug(fd.FD_DEBUG_SPIN_LIMIT, 2_000_000)
        g.set_debug(fd.FD_DEBUG_SKIP_PLANE, 5)
        rec = np.zeros_like(ref)
        assert g.forward(w["src"], w["wavelet"], w["rec"], rec) == fd.FD_ERR_TIMEOUT
        assert "wait" in fd.fd_last_error().decode()
        g.set_debug(fd.FD_DEBUG_SKIP_PLANE, -1)
        again = np.zeros_like(ref)
        fd.check(g.forward(w["src"], w["wavelet"], w["rec"], again), "after recovery")
        np.testing.assert_array_equal(again, ref)
