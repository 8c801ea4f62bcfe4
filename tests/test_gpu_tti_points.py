"""Receivers of the anisotropic step in one block and, where there are thousands,
in launches of several: the same receivers in one run and split over two runs
give the same bits, with and without a source."""
import numpy as np
import pytest

from paper_2312_13094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrec", [1, 511, 513, 4096, 4097])
@pytest.mark.parametrize("sources", [0, 2])
def test_receivers_do_not_depend_on_how_many_there_are(nrec, sources):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import binding as fd
    n, h, nt, dt = (24, 20, 18), 10.0, 12, 0.8
    rng = np.random.default_rng(3)
    ext = np.array([(m - 1) * h for m in n])
    src = (rng.random((sources, 3)) * ext).astype(np.float32)
    rec = (rng.random((nrec, 3)) * ext).astype(np.float32)
    wav = np.repeat(wl.ricker(nt, dt, 40.0).reshape(nt, 1), max(sources, 1), 1).astype(np.float32)
    field = lambda c: np.full(n[::-1], c, np.float32)
    p0 = rng.standard_normal((18 + 8, 20 + 8, 24 + 8)).astype(np.float32)

    def run(points):
        with fd.TtiGrid(n, h, 4, 4, dt, nt) as g:
            g.set_model(field(2.0), field(0.1), field(0.05), field(0.3), field(0.2))
            g.set_state(p=p0, q=p0)
            out = np.zeros((nt, len(points)), np.float32)
            fd.check(g.propagate(0, nt, src if sources else None, wav if sources else None, points,
                                 out))
            return out

    whole = run(rec)
    assert np.abs(whole).max() > 0
    k = (nrec + 1) // 2
    np.testing.assert_array_equal(whole[:, :k], run(rec[:k]))
    if k < nrec:
        np.testing.assert_array_equal(whole[:, k:], run(rec[k:]))
