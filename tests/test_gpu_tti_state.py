"""State of the anisotropic grid from and to the caller's arrays in every mix of
host and device arrays, absent ones and one array given twice, on rows shorter and
longer than a block and on more rows than one launch takes."""
import numpy as np
import pytest

from paper_2312_13094_gb300 import workloads as wl

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


def host(a):
    return a if isinstance(a, np.ndarray) else a.cpu().numpy()


@pytest.mark.parametrize("n", [(131, 6, 5), (7, 330, 217)])
@pytest.mark.parametrize("where", ["dddd", "hhhh", "dhdh", "ddhh", "d-d-", "-d-d", "dd--", "--dd",
                                   "-dd-", "dd-d"])
def test_state_in_every_mix_of_arrays(fd, n, where):
    import torch
    nbl = 2
    shp = tuple(m + 2 * nbl for m in n[::-1])
    st = [wl.random_state(shp, 30 + i).astype(np.float32) for i in range(4)]
    other = [wl.random_state(shp, 50 + i).astype(np.float32) for i in range(4)]
    take = {"d": lambda a: torch.from_numpy(a).cuda(), "h": lambda a: a.copy(), "-": lambda a: None}
    with fd.TtiGrid(n, 10.0, 8, nbl, 0.5, 4) as g:
        g.set_state(*other)
        g.set_state(*[take[w](a) for w, a in zip(where, st)])
        out = [np.zeros(shp, np.float32) for _ in range(4)]
        for i, name in enumerate(("p_prev", "p", "q_prev", "q")):
            g.get_state(**{name: out[i]})
        for w, a, b, o in zip(where, st, other, out):
            np.testing.assert_array_equal(o, b if w == "-" else a)
        want = [o.copy() for o in out]
        got = [take[w](np.zeros(shp, np.float32)) for w in where]
        g.get_state(*got)
        for a, b in zip(want, got):
            if b is not None:
                np.testing.assert_array_equal(host(b), a)


def test_one_array_given_twice(fd):
    import torch
    n, nbl = (20, 9, 8), 2
    shp = tuple(m + 2 * nbl for m in n[::-1])
    a, b = (wl.random_state(shp, 70 + i).astype(np.float32) for i in range(2))
    with fd.TtiGrid(n, 10.0, 8, nbl, 0.5, 4) as g:
        da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        g.set_state(p_prev=da, p=db, q_prev=da, q=da)
        out = [np.zeros(shp, np.float32) for _ in range(4)]
        g.get_state(*out)
        for o, want in zip(out, (a, b, a, a)):
            np.testing.assert_array_equal(o, want)
        buf = torch.zeros(shp, device="cuda")
        g.get_state(p=buf, q_prev=buf)  # q_prev is written after p
        np.testing.assert_array_equal(buf.cpu().numpy(), a)
