"""Gradients of many short segments, each recomputed in its checkpoint's own
memory with tensor maps of its own at the same descriptor address, against the
gradient of one segment, bit for bit: on bricks, column waves and equal shares,
with one and with split staging of u^n, and with the segment counts of one grid
changing from call to call."""
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


@pytest.mark.parametrize("so", [4, 8, 12])
@pytest.mark.parametrize("sched", ["auto", "waves", "shares"])
def test_segment_count_does_not_change_a_bit(fd, so, sched):
    import torch
    n = (61, 45, 52)
    w = workload(so, n, 6, 60)
    obs = np.zeros((w["nt"], len(w["rec"])), np.float32)
    with fd.Grid.from_workload(w) as g:
        g.set_schedule({"auto": fd.FD_SCHED_AUTO, "waves": fd.FD_SCHED_WAVES,
                        "shares": fd.FD_SCHED_SHARES}[sched])
        g.set_model(w["v"])
        grads = []
        for segments in (1, 30, 1, 20, 7):
            grad = torch.zeros(n[::-1], device="cuda")
            st, _ = g.adjoint_gradient(w["src"], w["wavelet"], w["rec"], obs, segments, grad)
            fd.check(st, "fd_adjoint_gradient")
            grads.append(grad)
    assert float(grads[0].abs().max()) > 0
    for grad in grads[1:]:
        assert torch.equal(grad, grads[0])
