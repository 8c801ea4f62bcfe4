"""The calls that a user of this library makes, at the sizes they are made at.

Five families, each through its public entry point:

* ``forward``   one shot of isotropic acoustic modelling (binding.Grid.forward)
* ``tti``       one shot of anisotropic modelling (binding.TtiGrid.forward)
* ``gradient``  the adjoint gradient of one shot (binding.Grid.adjoint_gradient),
                or one shot of an inversion loop with its model update
                (fwi.AdjointShots, fwi.device_update)
* ``batch``     many shots per launch (binding.batch_forward)
* ``learned``   coarse modelling with network weights (weight table, or per-cell
                weights that a new model needs first), and ``mlp``, the loss
                gradient of one mini-batch that trains that network

Sizes are those of the workloads module, the benchmark and the tests, or lie
between them.  Inputs are made on the GPU from the seed; sources and receivers
lie off the grid nodes near the surface, so that arrivals reach the receivers.
``exact`` is the same recurrence in plain FP64 torch.
"""
import math
import os

import numpy as np
import torch

from paper_2312_13094_gb300 import binding as fd
from paper_2312_13094_gb300 import checkpoint, fwi, learned

DEV = "cuda"
PKG = os.path.dirname(os.path.abspath(fd.__file__))
PARAMS = os.path.join(PKG, "data", "learned_coarse_h20_so8_12hz.fdck")


def listed():
    return [
        # the smallest shot: the 64^3 correctness workload (SO 4, 100 steps), as
        # in a smoke check or a small survey; its time is launches and latency
        {"name": "forward_64_so4", "kind": "forward", "nx": 64, "ny": 64, "nz": 64, "so": 4,
         "nbl": 10, "nt": 100, "h": 10.0, "nrec": 64},
        # an ordinary shot window of odd sizes, too short for the tuner
        {"name": "forward_ragged_so8", "kind": "forward", "nx": 211, "ny": 157, "nz": 123,
         "so": 8, "nbl": 20, "nt": 300, "h": 10.0, "nrec": 101},
        # the benchmark grid, 512^3 with a 40-cell layer at SO 8: the paper's
        # single-GPU acoustic run (400 of its 1000 steps)
        {"name": "forward_512_so8", "kind": "forward", "nx": 512, "ny": 512, "nz": 512, "so": 8,
         "nbl": 40, "nt": 400, "h": 10.0, "nrec": 512},
        # the widest stencil, the order the paper's accuracy runs end at
        {"name": "forward_300_so16", "kind": "forward", "nx": 300, "ny": 300, "nz": 300,
         "so": 16, "nbl": 40, "nt": 400, "h": 10.0, "nrec": 150},
        # anisotropic modelling at the order the paper quotes
        {"name": "tti_256_so8", "kind": "tti", "nx": 256, "ny": 256, "nz": 256, "so": 8,
         "nbl": 40, "nt": 100, "h": 10.0, "nrec": 128},
        # anisotropic modelling with the 769-point stencil on odd sizes
        {"name": "tti_ragged_so16", "kind": "tti", "nx": 203, "ny": 141, "nz": 167, "so": 16,
         "nbl": 20, "nt": 60, "h": 10.0, "nrec": 77},
        # the gradient workload: 256^3, 500 steps, 25 checkpoints, 32 x 32 receivers
        {"name": "gradient_256_so8", "kind": "gradient", "nx": 256, "ny": 256, "nz": 256,
         "so": 8, "nbl": 20, "nt": 500, "h": 10.0, "nrec": 1024, "nc": 25, "update": False},
        # one shot of an inversion loop on a small window: new model, gradient,
        # descent step
        {"name": "inversion_ragged_so4", "kind": "gradient", "nx": 117, "ny": 96, "nz": 71,
         "so": 4, "nbl": 16, "nt": 150, "h": 10.0, "nrec": 144, "nc": 10, "update": True},
        # uneven shots in one launch (the batch workload's window range)
        {"name": "batch_12_so8", "kind": "batch", "shots": 12, "lo": 128, "hi": 320, "so": 8,
         "nbl": 20, "nt": 200, "h": 10.0, "nrec": 128},
        # the coarse solve with tabulated network weights, 256^3 at h = 20 m
        {"name": "learned_table_256", "kind": "learned", "nx": 256, "ny": 256, "nz": 256,
         "nbl": 20, "nt": 625, "h": 20.0, "nrec": 128, "table": 256},
        # a new model under per-cell network weights: model, inference, shot
        {"name": "learned_cells_ragged", "kind": "learned", "nx": 190, "ny": 173, "nz": 141,
         "nbl": 20, "nt": 200, "h": 20.0, "nrec": 90, "table": 0},
        # one mini-batch of the network's training, from its initial parameters
        {"name": "mlp_65536", "kind": "mlp", "n": 65536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "tti", "tti", "gradient", "batch",
                       "learned", "mlp"])
    if kind == "mlp":
        return {"kind": kind, "n": _log(rng, 500, 1 << 20)}
    if kind == "batch":
        lo = rng.randint(64, 160)
        return {"kind": kind, "shots": rng.randint(3, 12), "lo": lo,
                "hi": rng.randint(lo + 20, 320), "so": rng.choice([4, 8, 8, 12]),
                "nbl": rng.choice([10, 20]), "nt": rng.randint(60, 200), "h": 10.0,
                "nrec": rng.randint(20, 128)}
    top = {"forward": 512, "tti": 256, "gradient": 256, "learned": 256}[kind]
    n = [_log(rng, 48, top) for _ in range(3)]
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "nrec": rng.randint(20, 300)}
    if kind == "forward":
        c.update(so=2 * rng.randint(1, 8), nbl=rng.choice([0, 10, 20, 40]), nt=_log(rng, 60, 500),
                 h=10.0)
    elif kind == "tti":
        c.update(so=rng.choice([4, 8, 8, 12, 16]), nbl=rng.choice([10, 20, 40]),
                 nt=rng.randint(20, 100), h=10.0)
    elif kind == "gradient":
        c.update(so=rng.choice([4, 8, 8, 12]), nbl=rng.choice([10, 20]), nt=_log(rng, 80, 500),
                 h=10.0, nrec=rng.randint(5, 32) ** 2, nc=rng.randint(4, 25),
                 update=rng.random() < 0.5)
    else:
        c.update(nbl=rng.choice([10, 20]), nt=rng.randint(100, 500), h=20.0,
                 table=rng.choice([0, 256]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ricker(nt, dt, f_hz):
    t = np.arange(nt) * dt - 1000.0 / f_hz
    a = (np.pi * f_hz / 1000.0 * t) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32).reshape(nt, 1)


def _smooth(x, reps):
    """Repeated three-point means along every axis (edges reflected)."""
    for _ in range(reps):
        for a in range(3):
            p = torch.cat([x.narrow(a, 0, 1), x, x.narrow(a, x.shape[a] - 1, 1)], a)
            n = x.shape[a]
            x = (p.narrow(a, 0, n) + p.narrow(a, 1, n) + p.narrow(a, 2, n)) * (1.0 / 3.0)
    return x


def _velocity(n, h, seed, vmin, vmax):
    """Layered medium with smooth lateral noise of 5 % (km/s), [nz][ny][nx]."""
    rng = np.random.default_rng(seed)
    nl = rng.integers(3, 7)
    depth = np.sort(rng.uniform(0.1, 0.95, nl - 1)) * n[2] * h
    vel = np.sort(rng.uniform(vmin, vmax / 1.05, nl))
    z = np.arange(n[2]) * h
    col = np.full(n[2], vel[0])
    for d, a, b in zip(depth, vel[:-1], vel[1:]):
        col += (b - a) * 0.5 * (1.0 + np.tanh((z - d) / 20.0))
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    small = torch.randn([(m + 3) // 4 + 1 for m in n[::-1]], device=DEV, generator=gen)
    small = _smooth(small, 2)
    p = small
    for a in range(3):
        p = p.repeat_interleave(4, a).narrow(a, 0, n[2 - a])
    p = _smooth(p, 3)
    p = p * (0.05 / p.abs().max())
    v = torch.from_numpy(col.astype(np.float32)).to(DEV)[:, None, None] * (1.0 + p)
    return v.clamp(vmin * 0.95, vmax).contiguous()


def _points(case, n, h, seed):
    """One source in the upper third, off the nodes, and receivers near the
    surface: a line, or for gradients a square of them."""
    rng = np.random.default_rng(seed + 1000)
    ext = [(m - 1) * h for m in n]
    src = np.array([[ext[0] * rng.uniform(0.4, 0.6), ext[1] * rng.uniform(0.4, 0.6),
                     min(ext[2] * 0.3, h * rng.uniform(8.0, 16.0))]])
    if case["kind"] == "gradient":
        k = math.isqrt(case["nrec"])
        x, y = np.meshgrid(np.linspace(0.0, ext[0], k), np.linspace(0.0, ext[1], k))
        x, y = x.ravel(), y.ravel()
    else:
        x = np.linspace(0.0, ext[0], case["nrec"])
        y = np.full(case["nrec"], src[0, 1] + 0.3 * h)
    rec = np.stack([x, y, np.full(len(x), 2.5 * h)], 1)
    return src.astype(np.float32), rec.astype(np.float32)


def _shot(case, seed, n=None, vmin=1.5, vmax=3.2, courant=0.4, f_hz=15.0):
    n = n or (case["nx"], case["ny"], case["nz"])
    h = case["h"]
    dt = courant * h / vmax
    src, rec = _points(case, n, h, seed)
    amp = np.float32(1.0 + 0.1 * (seed % 7))
    return {"n": n, "h": h, "dt": dt, "nt": case["nt"], "nbl": case["nbl"],
            "so": case.get("so", 8), "v": _velocity(n, h, seed, vmin, vmax), "src": src,
            "rec": rec, "wavelet": _ricker(case["nt"], dt, f_hz) * amp, "f_hz": f_hz}


def _tti_shot(case, seed):
    s = _shot(case, seed, vmax=3.5, courant=0.3)
    shape = s["v"].shape
    rng = np.random.default_rng(seed + 2000)

    def field():
        ax = [torch.sin(torch.linspace(0.0, float(rng.uniform(3, 9)), m, device=DEV)
                        + float(rng.uniform(0, 6))) for m in shape]
        return 0.5 + 0.5 * ax[0][:, None, None] * ax[1][None, :, None] * ax[2][None, None, :]

    s["eps"] = (0.05 + 0.15 * field()).contiguous()
    s["delta"] = (0.5 * s["eps"]).contiguous()
    s["theta"] = (0.6 * field()).contiguous()
    s["phi"] = (1.2 * field()).contiguous()
    return s


def _obs(s, seed):
    """Receiver data of another medium: noise-like arrivals of the right size."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
    nt, nrec = s["nt"], len(s["rec"])
    d = torch.randn((nt, nrec), device=DEV, generator=gen)
    d = _smooth(d[None], 4)[0]
    return (d * (2e-4 / d.abs().max())).contiguous()


def _grid(cls, s):
    return cls(s["n"], s["h"], s["so"], s["nbl"], s["dt"], s["nt"])


def _wav(s):
    return torch.from_numpy(s["wavelet"]).to(DEV)


def _samples(n, seed):
    """Training samples [n, 10] as fd_mlp_make_samples lays them out: features,
    stencil sums, target near the plain prediction, weight."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    S = torch.empty((n, fd.FD_MLP_SAMPLE), device=DEV)
    S[:, 0] = (1.5 + 3.0 * torch.rand(n, device=DEV, generator=gen)) * 1.6 / 20.0
    S[:, 1], S[:, 2], S[:, 3] = 2.0, 1.6, 1.2
    u = torch.randn(n, device=DEV, generator=gen)
    for j in range(1, 5):
        S[:, 3 + j] = u * j * j * (1.0 - 0.02 * j * j) + 0.05 * torch.randn(
            n, device=DEV, generator=gen)
    c = torch.tensor([8 / 5, -1 / 5, 8 / 315, -1 / 560], device=DEV)
    S[:, 8] = (S[:, 4:8] * c).sum(1) + 0.02 * torch.randn(n, device=DEV, generator=gen)
    S[:, 9] = 1.0 / (0.5 + u * u)
    return S.contiguous()


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return {"kind": kind, "net": learned.Network(learned.init_params(seed)),
                "samples": _samples(case["n"], seed)}
    if kind == "batch":
        rng = np.random.default_rng(case["shots"])
        shots, keep = [], []
        for i in range(case["shots"]):
            n = tuple(int(m) // 4 * 4 for m in rng.integers(case["lo"], case["hi"] + 1, 3))
            s = _shot(case, 100 * seed + i, n=n, vmax=4.5)
            g = _grid(fd.Grid, s)
            g.set_model(s["v"])
            rec = torch.zeros((s["nt"], len(s["rec"])), device=DEV)
            shots.append((g, s["src"], _wav(s), s["rec"], rec))
            keep.append(rec)
        return {"kind": kind, "shots": shots, "rec": keep}
    if kind == "tti":
        s = _tti_shot(case, seed)
        g = _grid(fd.TtiGrid, s)
        g.set_model(s["v"], s["eps"], s["delta"], s["theta"], s["phi"])
        st = {k: torch.zeros(g.padded_shape, device=DEV) for k in ("p", "q")}
        return {"kind": kind, "grid": g, "src": s["src"], "wav": _wav(s), "points": s["rec"],
                "rec": torch.zeros((s["nt"], len(s["rec"])), device=DEV), **st}
    if kind == "learned":
        s = _shot(case, seed, vmax=4.5, courant=0.36, f_hz=12.0)
        params, _ = checkpoint.load(PARAMS)
        g, net = _grid(fd.Grid, s), learned.Network(params)
        if case["table"]:
            g.set_model(s["v"])
            fd.check(fd.fd_set_learned_table(g.handle, net.handle, s["f_hz"], case["table"]))
        return {"kind": kind, "table": case["table"], "grid": g, "net": net, "v": s["v"],
                "f_hz": s["f_hz"], "src": s["src"], "wav": _wav(s), "points": s["rec"],
                "rec": torch.zeros((s["nt"], len(s["rec"])), device=DEV),
                "u": torch.zeros(g.phys_shape, device=DEV)}
    s = _shot(case, seed)
    g = _grid(fd.Grid, s)
    if kind == "gradient":
        m = (1.0 / s["v"].double() ** 2).float().contiguous()
        g.set_model(m, fd.FD_MODEL_M)
        st = {"kind": kind, "grid": g, "m": m, "src": s["src"], "wav": _wav(s),
              "points": s["rec"], "obs": _obs(s, seed), "nc": case["nc"],
              "update": case["update"]}
        if case["update"]:
            st["shots"] = fwi.AdjointShots(g, [s["src"]], st["wav"], s["rec"], [st["obs"]],
                                           case["nc"])
            st["step"] = fwi.device_update(1.0 / 3.4 ** 2, 1.0 / 1.3 ** 2)
        else:
            st["grad"] = torch.zeros_like(m)
        return st
    g.set_model(s["v"])
    return {"kind": kind, "grid": g, "src": s["src"], "wav": _wav(s), "points": s["rec"],
            "rec": torch.zeros((s["nt"], len(s["rec"])), device=DEV),
            "u": torch.zeros(g.phys_shape, device=DEV)}


def run(state):
    kind = state["kind"]
    if kind == "mlp":
        loss, grad = state["net"].loss_grad(state["samples"])
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        fd.check(fd.batch_forward(state["shots"], fd.FD_BATCH_GRAPH | fd.FD_BATCH_AUTOTUNE))
        return state["rec"]
    g = state["grid"]
    if kind == "gradient":
        if state["update"]:
            grad, loss = state["shots"](0, state["m"])
            return {"m": state["step"](state["m"], grad, 0.02), "grad": grad, "loss": loss}
        status, loss = g.adjoint_gradient(state["src"], state["wav"], state["points"],
                                          state["obs"], state["nc"], state["grad"])
        fd.check(status)
        return {"grad": state["grad"], "loss": loss}
    if kind == "tti":
        fd.check(g.forward(state["src"], state["wav"], state["points"], state["rec"]))
        g.get_state(p=state["p"], q=state["q"])
        return {"rec": state["rec"], "p": state["p"], "q": state["q"]}
    if kind == "learned" and not state["table"]:
        g.set_model(state["v"])
        fd.check(fd.fd_set_learned_coefficients(g.handle, state["net"].handle, state["f_hz"]))
    fd.check(g.forward(state["src"], state["wav"], state["points"], state["rec"], state["u"]))
    return {"rec": state["rec"], "u": state["u"]}


def _padded(case):
    return [case[k] + 2 * case["nbl"] for k in ("nx", "ny", "nz")]


def work(case):
    """Bytes: every step reads u^n, u^{n-1} and the model and writes u^{n+1};
    flops: one multiply-add per symmetric neighbour pair and the update."""
    kind = case["kind"]
    if kind == "mlp":
        # three dense layers forward, twice that backward
        mac = 4 * 64 + 64 * 64 + 64 * 8
        return {"bytes": 40 * case["n"] + 2 * 20000, "flops": case["n"] * 2 * 3 * mac}
    if kind == "batch":
        rng = np.random.default_rng(case["shots"])
        pts = 0
        for _ in range(case["shots"]):
            n = [int(m) // 4 * 4 + 2 * case["nbl"]
                 for m in rng.integers(case["lo"], case["hi"] + 1, 3)]
            pts += n[0] * n[1] * n[2]
        R = case["so"] // 2
        return {"bytes": 16 * pts * case["nt"], "flops": (9 * R + 8) * pts * case["nt"]}
    N = _padded(case)
    pts, nt = N[0] * N[1] * N[2], case["nt"]
    R = case.get("so", 8) // 2
    if kind == "tti":
        # per field: three second derivatives, dx, dy and three sums of those
        return {"bytes": 48 * pts * nt, "flops": (2 * (3 * 3 * R + 5 * 3 * R) + 60) * pts * nt}
    step = (9 * R + 8) * pts * nt
    if kind == "gradient":
        # forward, recomputation storing e, adjoint with the imaging sum
        return {"bytes": 64 * pts * nt, "flops": 3 * step}
    if kind == "learned":
        each = 16 if case["table"] else 32
        net = 0 if case["table"] else 2 * (4 * 64 + 64 * 64 + 64 * 8) * pts
        return {"bytes": each * pts * nt, "flops": step + 12 * pts * nt + net}
    return {"bytes": 16 * pts * nt, "flops": step}


# ---------------------------------------------------------------------------
# the same in plain FP64 torch
# ---------------------------------------------------------------------------

def _weights2(R):
    c = [0.0] * (R + 1)
    for j in range(1, R + 1):
        r = 1.0
        for k in range(1, j + 1):
            r *= (R - k + 1) / (R + k)
        c[j] = (2.0 if j & 1 else -2.0) * r / (j * j)
    c[0] = -2.0 * sum(c[1:])
    return c


def _weights1(R):
    return [0.0] + [(0.5 * j) * c for j, c in enumerate(_weights2(R)) if j]


def _add(out, u, axis, j, w):
    """out += w u(i + j) along the axis, zero beyond the grid (w a number or a
    field)."""
    n = u.shape[axis] - abs(j)
    if n <= 0:
        return
    o, s = out.narrow(axis, max(0, -j), n), u.narrow(axis, max(0, j), n)
    if isinstance(w, float):
        o.add_(s, alpha=w)
    else:
        o.addcmul_(s, w.narrow(axis, max(0, -j), n))


def _laplacian(u, c):
    """sum_j c_j (S_j - 6 u): c_j numbers (c[0] = -2 sum) or fields c[1..R]."""
    R = len(c) - 1
    if isinstance(c[1], float):
        out = u * (3.0 * c[0])
    else:
        out = u * (-6.0 * sum(c[1:]))
    for a in range(3):
        for j in range(1, R + 1):
            _add(out, u, a, j, c[j])
            _add(out, u, a, -j, c[j])
    return out


def _first(u, axis, d):
    out = torch.zeros_like(u)
    for j in range(1, len(d)):
        _add(out, u, axis, j, d[j])
        _add(out, u, axis, -j, -d[j])
    return out


def _second(u, axis, c):
    out = u * c[0]
    for j in range(1, len(c)):
        _add(out, u, axis, j, c[j])
        _add(out, u, axis, -j, c[j])
    return out


class _Exact:
    """Padded FP64 model, damping and point weights of one shot."""

    def __init__(self, s, vmax=None, v=None):
        v = (s["v"] if v is None else v).double()
        self.n, self.nbl, self.h, self.dt, self.nt = s["n"], s["nbl"], s["h"], s["dt"], s["nt"]
        self.idx = [torch.arange(m + 2 * self.nbl, device=DEV).sub(self.nbl).clamp(0, m - 1)
                    for m in self.n[::-1]]
        vmax = float(v.max()) if vmax is None else vmax
        self.A = self.dt ** 2 / self.h ** 2 * self.pad(v) ** 2
        dep = []
        for m in self.n[::-1]:
            i = torch.arange(m + 2 * self.nbl, device=DEV)
            dep.append(torch.maximum(self.nbl - i, i - (m + self.nbl - 1)).clamp(min=0).double() ** 2)
        d2 = dep[0][:, None, None] + dep[1][None, :, None] + dep[2][None, None, :]
        b = 0.0
        if self.nbl:
            b = 3.0 * vmax * math.log(1000.0) / (2.0 * self.nbl * self.h) * self.dt / 2.0 / self.nbl ** 2
        self.den, self.num = 1.0 + b * d2, 1.0 - b * d2
        self.si, self.sw = self.weights(s["src"])
        self.ri, self.rw = self.weights(s["rec"])
        self.q = torch.from_numpy(s["wavelet"]).to(DEV).double()

    def pad(self, x):
        return x[self.idx[0]][:, self.idx[1]][:, :, self.idx[2]].contiguous()

    def weights(self, pts):
        """Flat padded indices and trilinear weights, [points, 8]."""
        N = [m + 2 * self.nbl for m in self.n]
        s = np.asarray(pts, np.float32).astype(np.float64) / self.h
        i0 = np.floor(s).astype(np.int64)
        f = s - i0
        idx, w = [], []
        for c in range(8):
            hi = np.array([(c >> a) & 1 for a in range(3)])
            node = np.minimum(i0 + hi, np.array(self.n) - 1) + self.nbl
            wt = np.prod(np.where(hi == 1, f, 1.0 - f), axis=1)
            idx.append((node[:, 2] * N[1] + node[:, 1]) * N[0] + node[:, 0])
            w.append(wt)
        return (torch.from_numpy(np.stack(idx, 1)).to(DEV), torch.from_numpy(np.stack(w, 1)).to(DEV))

    def zeros(self):
        return torch.zeros_like(self.A)

    def phys(self, u):
        for a in range(3):
            u = u.narrow(a, self.nbl, self.n[2 - a])
        return u

    def record(self, u):
        return (u.reshape(-1)[self.ri] * self.rw).sum(1)

    def rhs(self, u, c, idx, val):
        """A (lap u + h^2 s) with point terms val at idx (already h^2 s)."""
        lap = _laplacian(u, c)
        lap.view(-1).index_add_(0, idx.reshape(-1), val.reshape(-1))
        return lap.mul_(self.A)

    def source(self, n):
        return self.sw * self.q[n][:, None] / self.h

    def step(self, prev, u, e):
        """(1 + b) u+ = 2 u - (1 - b) u- + e, into prev."""
        return prev.mul_(self.num).neg_().add_(u, alpha=2.0).add_(e).div_(self.den)


def _exact_forward(s, c, x=None):
    x = x or _Exact(s)
    prev, u = x.zeros(), x.zeros()
    rec = torch.zeros((x.nt, len(s["rec"])), device=DEV, dtype=torch.float64)
    for n in range(x.nt):
        rec[n] = x.record(u)
        prev, u = u, x.step(prev, u, x.rhs(u, c, x.si, x.source(n)))
    return rec, x.phys(u).contiguous()


def _exact_gradient(case, seed):
    s = _shot(case, seed)
    m = (1.0 / s["v"].double() ** 2).float().double()
    x = _Exact(s, v=1.0 / m.sqrt())
    c = _weights2(case["so"] // 2)
    obs = _obs(s, seed).double()
    L = max(1, int(math.sqrt(x.nt)))
    prev, u = x.zeros(), x.zeros()
    rec = torch.zeros((x.nt, len(s["rec"])), device=DEV, dtype=torch.float64)
    keep = {}
    for n in range(x.nt):
        if n % L == 0:
            keep[n] = (prev.clone(), u.clone())
        rec[n] = x.record(u)
        prev, u = u, x.step(prev, u, x.rhs(u, c, x.si, x.source(n)))
    r = rec - obs
    z2, z1, g = x.zeros(), x.zeros(), x.zeros()
    for n0 in sorted(keep, reverse=True):
        prev, u = keep.pop(n0)
        es = []
        for n in range(n0, min(n0 + L, x.nt)):
            es.append(x.rhs(u, c, x.si, x.source(n)))
            prev, u = u, x.step(prev, u, es[-1])
        for n in range(min(n0 + L, x.nt) - 1, n0 - 1, -1):
            g.addcmul_(z1, es.pop(), value=-1.0 / x.dt ** 2)
            z2, z1 = z1, x.step(z2, z1, x.rhs(z1, c, x.ri, x.rw * r[n][:, None] * x.h ** 2))
    # fold the layer's replicated cells onto the physical ones
    for a in range(3):
        out = torch.zeros([x.n[2 - k] if k == a else g.shape[k] for k in range(3)], device=DEV,
                          dtype=torch.float64)
        g = out.index_add_(a, x.idx[a], g)
    res = {"grad": g, "loss": float(0.5 * (r ** 2).sum())}
    if case["update"]:
        alpha = 0.02 * float(m.abs().max()) / float(g.abs().max())
        res["m"] = (m - alpha * g).clamp(1.0 / 3.4 ** 2, 1.0 / 1.3 ** 2)
    return res


def _exact_tti(case, seed):
    s = _tti_shot(case, seed)
    vp, eps, delta = s["v"].double(), s["eps"].double(), s["delta"].double()
    x = _Exact(s, vmax=float((vp * torch.sqrt(1.0 + 2.0 * eps)).max()))
    e2, dl = x.pad(1.0 + 2.0 * eps), x.pad(torch.sqrt(1.0 + 2.0 * delta))
    th, ph = x.pad(s["theta"].double()), x.pad(s["phi"].double())
    nv = (torch.cos(th), torch.sin(th) * torch.sin(ph), torch.sin(th) * torch.cos(ph))  # z, y, x
    c, d = _weights2(case["so"] // 2), _weights1(case["so"] // 2)

    def parts(u):
        """(Laplacian, H_z) of one field."""
        lap, hz = torch.zeros_like(u), torch.zeros_like(u)
        for a in range(3):
            t = _second(u, a, c)
            lap += t
            hz.addcmul_(nv[a] * nv[a], t)
        for b in (2, 1):
            f = _first(u, b, d)
            for a in range(b):
                hz.addcmul_(nv[a] * nv[b], _first(f, a, d), value=2.0)
        return lap, hz

    pm, p, qm, q = (x.zeros() for _ in range(4))
    rec = torch.zeros((x.nt, len(s["rec"])), device=DEV, dtype=torch.float64)
    for n in range(x.nt):
        rec[n] = x.record(p)
        lap, hzp = parts(p)
        hzq = parts(q)[1]
        h0 = lap - hzp
        rp, rq = e2 * h0 + dl * hzq, dl * h0 + hzq
        val = x.source(n).reshape(-1)
        for f in (rp, rq):
            f.view(-1).index_add_(0, x.si.reshape(-1), val)
            f.mul_(x.A)
        pm, p = p, x.step(pm, p, rp)
        qm, q = q, x.step(qm, q, rq)
    return {"rec": rec, "p": p, "q": q}


def _network(params, X):
    """Outputs of the 4-64-64-8 network: (s_1..s_4, layers)."""
    t = torch.from_numpy(np.asarray(params, np.float64)).to(DEV)
    W1, b1, W2, b2, W3, b3 = torch.split(t, [256, 64, 4096, 64, 512, 8])
    W1, W2, W3 = W1.view(64, 4), W2.view(64, 64), W3.view(8, 64)
    h1 = (X @ W1.T + b1).clamp(min=0.0)
    h2 = (h1 @ W2.T + b2).clamp(min=0.0)
    o = h2 @ W3.T + b3
    return 0.5 * (o[:, :4] + o[:, 4:]), h1, h2, W2, W3


def _network_weights(params, X):
    cT = torch.tensor(_weights2(4)[1:], device=DEV, dtype=torch.float64)
    return cT * (1.0 + 0.5 * torch.tanh(_network(params, X)[0]))


def _exact_learned(case, seed):
    s = _shot(case, seed, vmax=4.5, courant=0.36, f_hz=12.0)
    x = _Exact(s)
    params, _ = checkpoint.load(PARAMS)

    def weights(A):
        X = torch.empty((A.numel(), 4), device=DEV, dtype=torch.float64)
        X[:, 0] = A.reshape(-1).sqrt()
        X[:, 1], X[:, 2], X[:, 3] = s["h"] / 10.0, s["dt"], s["f_hz"] / 10.0
        return torch.cat([_network_weights(params, b) for b in X.split(1 << 20)])

    if case["table"]:
        k = case["table"]
        lo, hi = float(x.phys(x.A).min()), float(x.phys(x.A).max())
        T = weights(torch.linspace(lo, hi, k, device=DEV, dtype=torch.float64))
        at = ((x.A.reshape(-1) - lo) * ((k - 1) / (hi - lo))).clamp(0.0, k - 1.0)
        i = at.floor().long().clamp(max=k - 2)
        w = T[i] + (at - i)[:, None] * (T[i + 1] - T[i])
    else:
        w = weights(x.A)
    c = [None] + [w[:, j].reshape(x.A.shape).contiguous() for j in range(4)]
    rec, u = _exact_forward(s, c, x)
    return {"rec": rec, "u": u}


def _exact_mlp(case, seed):
    params = learned.init_params(seed)
    S = _samples(case["n"], seed).double()
    cT = torch.tensor(_weights2(4)[1:], device=DEV, dtype=torch.float64)
    total, loss = torch.zeros(5000, device=DEV, dtype=torch.float64), 0.0
    for b in S.split(1 << 18):
        X, T, y, w = b[:, :4], b[:, 4:8], b[:, 8], b[:, 9]
        s, h1, h2, W2, W3 = _network(params, X)
        th = torch.tanh(s)
        r = (cT * (1.0 + 0.5 * th) * T).sum(1) - y
        loss += float((w * r * r).sum()) / case["n"]
        ds = (2.0 * w * r / case["n"])[:, None] * T * cT * 0.5 * (1.0 - th * th)
        do = 0.5 * torch.cat([ds, ds], 1)
        d2 = (do @ W3) * (h2 > 0)
        d1 = (d2 @ W2) * (h1 > 0)
        total += torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0),
                            (do.T @ h2).reshape(-1), do.sum(0)])
    return {"loss": loss, "grad": total.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "tti":
        return _exact_tti(case, seed)
    if kind == "learned":
        return _exact_learned(case, seed)
    c = _weights2(case["so"] // 2)
    if kind == "batch":
        rng = np.random.default_rng(case["shots"])
        out = []
        for i in range(case["shots"]):
            n = tuple(int(m) // 4 * 4 for m in rng.integers(case["lo"], case["hi"] + 1, 3))
            out.append(_exact_forward(_shot(case, 100 * seed + i, n=n, vmax=4.5), c)[0])
        return out
    rec, u = _exact_forward(_shot(case, seed), c)
    return {"rec": rec, "u": u}
