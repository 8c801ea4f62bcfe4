"""Extremes and bad values of a model, wherever they stand: sizes below one load
per thread, with a remainder behind the rounds of four loads, and with several
rounds per thread."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [(3, 2, 1), (16, 16, 1), (32, 16, 2), (33, 31, 29),
                               (128, 97, 103), (220, 210, 233)])
def test_extremes_and_bad_values_are_found_everywhere(fd, n):
    import torch
    size = n[0] * n[1] * n[2]
    rng = np.random.default_rng(size)
    base = torch.from_numpy(rng.uniform(2.0, 2.5, n[::-1]).astype(np.float32)).cuda()
    at = sorted({0, size - 1, size // 2, size * 3 // 4, int(rng.integers(size))})
    with fd.Grid(n, 10.0, 4, 0, 0.5, 4) as g:
        for i in at:
            v = base.clone()
            v.view(-1)[i] = 3.25
            g.set_model(v)
            assert g.info()["v_max"] == 3.25
            m = 1.0 / (base * base)
            m.view(-1)[i] = 0.0625  # v = 4, exactly
            g.set_model(m, fd.FD_MODEL_M)
            assert g.info()["v_max"] == 4.0
            for bad in (float("nan"), 0.0, -1.0, float("inf")):
                v = base.clone()
                v.view(-1)[i] = bad
                with pytest.raises(fd.FDError) as e:
                    g.set_model(v)
                assert e.value.status == fd.FD_ERR_ARG
        g.set_model(base)
        assert g.info()["v_max"] == float(base.max())
