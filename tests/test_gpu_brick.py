"""Brick kernel of small grids and the wave tile of larger ones (grids left to
AUTO) against the equal-share sweep, bit for bit: sizes around the 32 x 8 x 8
bricks, grids smaller than one, every space order, both learned weight modes,
the adjoint, runs continued in pieces, and grids just above the brick limit."""
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


def workload(so, n, nbl, nt, seed=9):
    h = 10.0
    v = wl.layered_model(n, h, seed, vmin=1.5, vmax=3.0)
    dt = 0.35 * h / float(v.max())
    ext = [(d - 1) * h for d in n]
    src = np.array([[0.37 * ext[0], 0.61 * ext[1], 0.45 * ext[2]],
                    [0.8 * ext[0], 0.2 * ext[1], 0.9 * ext[2]]])
    rec = np.array([[x, 0.33 * ext[1], z] for x in np.linspace(0.0, ext[0], 17)
                    for z in np.linspace(0.0, ext[2], 9)])
    wav = np.stack([wl.ricker(nt, dt, 25.0), 0.5 * wl.ricker(nt, dt, 18.0)], 1)
    return dict(n=n, h=h, space_order=so, nbl=nbl, dt=dt, nt=nt, v=v, src=src, rec=rec,
                wavelet=np.ascontiguousarray(wav, np.float32))


def forward(fd, w, shares, prepare=None, pieces=None):
    with fd.Grid.from_workload(w) as g:
        if shares:
            g.set_schedule(fd.FD_SCHED_SHARES)
        g.set_model(w["v"])
        if prepare:
            prepare(g)
        rec = np.zeros((w["nt"], len(w["rec"])), np.float32)
        if pieces:
            n0 = 0
            for k in pieces:
                fd.check(g.propagate(n0, k, w["src"], w["wavelet"], w["rec"], rec[n0:n0 + k]))
                n0 += k
        else:
            fd.check(g.forward(w["src"], w["wavelet"], w["rec"], rec), "fd_forward")
        prev = np.zeros(g.padded_shape, np.float32)
        cur = np.zeros(g.padded_shape, np.float32)
        g.get_wavefield(prev, cur)
        return (rec, prev, cur), g.info()


def equal(a, b):
    assert np.abs(a[2]).max() > 0
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("so", range(2, 18, 2))
@pytest.mark.parametrize("n,nbl", [((32, 8, 8), 0), ((33, 9, 9), 0), ((31, 7, 15), 0),
                                   ((5, 4, 3), 2), ((53, 38, 41), 6)])
def test_bricks_equal_the_sweep(fd, so, n, nbl):
    w = workload(so, n, nbl, 24)
    a, info = forward(fd, w, False)
    assert (info["tile_x"], info["tile_y"]) == (32, 8)
    equal(a, forward(fd, w, True)[0])


def test_brick_pieces_equal_one_run(fd):
    w = workload(8, (53, 38, 41), 6, 24)
    equal(forward(fd, w, False, pieces=(1, 7, 16))[0], forward(fd, w, True)[0])


@pytest.mark.parametrize("table", [0, 2, 64])
@pytest.mark.parametrize("n", [(33, 9, 17), (60, 44, 39)])
def test_bricks_equal_the_sweep_with_learned_weights(fd, table, n):
    from oracle import mlp
    from paper_2312_13094_gb300 import learned
    w = workload(8, n, 5, 30)
    net = learned.Network(mlp.init_params(9, scale_out=1.0).astype(np.float32))

    def weights(g):
        if table:
            fd.check(fd.fd_set_learned_table(g.handle, net.handle, 12.0, table))
        else:
            fd.check(fd.fd_set_learned_coefficients(g.handle, net.handle, 12.0))

    equal(forward(fd, w, False, weights)[0], forward(fd, w, True, weights)[0])
    net.close()


@pytest.mark.parametrize("so,n,nbl", [(2, (33, 9, 17), 0), (4, (53, 38, 41), 6),
                                      (8, (40, 31, 25), 4), (16, (35, 30, 28), 8)])
def test_brick_gradient_equals_the_sweeps(fd, so, n, nbl):
    import torch
    w = workload(so, n, nbl, 40)
    obs = 0.5 * forward(fd, w, True)[0][0]
    out = []
    for shares in (False, True):
        with fd.Grid.from_workload(w) as g:
            if shares:
                g.set_schedule(fd.FD_SCHED_SHARES)
            g.set_model(w["v"])
            grad = torch.zeros(n[::-1], device="cuda")
            st, loss = g.adjoint_gradient(w["src"], w["wavelet"], w["rec"], obs, 5, grad)
            fd.check(st, "fd_adjoint_gradient")
            out.append((grad, loss))
    assert float(out[0][0].abs().max()) > 0
    assert torch.equal(out[0][0], out[1][0])
    assert abs(out[0][1] - out[1][1]) <= 1e-12 * abs(out[1][1])  # (a sum by atomics)


@pytest.mark.parametrize("so,n", [(4, (200, 180, 178)), (8, (171, 158, 160)), (12, (250, 126, 140)),
                                  (8, (64, 700, 101))])
def test_wave_tile_equals_the_sweep_above_the_brick_limit(fd, so, n):
    w = workload(so, n, 4, 12)
    a, info = forward(fd, w, False)
    assert info["schedule"] == fd.FD_SCHED_WAVES
    assert (info["tile_x"], info["tile_y"]) in [(32, 16), (64, 8)]
    equal(a, forward(fd, w, True)[0])
