"""Fold of the padded gradient onto the physical cells: a gradient whose layer
cells matter, on extents where an x end shares its warp with others, is alone in
it, or is both ends at once, against the FP64 oracle's adjoint."""
import numpy as np
import pytest

import oracle
from paper_2312_13094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nbl", [((1, 9, 8), 3), ((33, 1, 7), 3), ((130, 6, 1), 5),
                                   ((129, 5, 9), 0), ((20, 18, 16), 12)])
def test_folded_gradient_against_the_oracle(n, nbl):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import binding as fd
    h, dt, nt = 10.0, 1.0, 90
    rng = np.random.default_rng(5)
    v = (1.5 + 0.5 * rng.random(n[::-1])).astype(np.float32)
    src = np.array([[0.5 * (n[0] - 1) * h, 0.4 * (n[1] - 1) * h, 0.6 * (n[2] - 1) * h]])
    rec = np.array([[x, 0.0, (n[2] - 1) * h] for x in np.linspace(0.0, (n[0] - 1) * h, 5)])
    wav = wl.ricker(nt, dt, 40.0).reshape(nt, 1).astype(np.float32)
    d_obs = np.zeros((nt, len(rec)), np.float32)
    og = oracle.Grid(n=n, h=h, dt=dt, R=2, nbl=nbl)
    want = oracle.adjoint_gradient(og, 1.0 / v.astype(np.float64) ** 2, nt, src, wav, rec,
                                   d_obs=d_obs.astype(np.float64))[0]
    desc = dict(n=n, h=h, space_order=4, nbl=nbl, dt=dt, nt=nt)
    with fd.Grid.from_workload(desc) as g:
        g.set_model(v)
        grad = np.zeros(n[::-1], np.float32)
        st, _ = g.adjoint_gradient(src, wav, rec, d_obs, 3, grad)
        fd.check(st, "fd_adjoint_gradient")
    assert np.abs(want).max() > 0
    assert np.linalg.norm(grad - want) <= 1e-4 * np.linalg.norm(want)
