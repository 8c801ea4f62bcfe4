"""A batch whose grids run on streams of their own with work pending on them: the
sweep on the first grid's stream has to wait for the point tables and wavelets
that the other grids' streams still hold, and for a wavelet that the caller
writes there.  A bounded delay kernel on the later streams makes the order show;
receivers equal the single-shot runs bit for bit."""
import numpy as np
import pytest

from paper_2312_13094_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

DELAY = 20_000_000  # clock cycles, about 10 ms


def moved(w, k):
    """The shot with as many points elsewhere and another wavelet."""
    ext = np.array([(m - 1) * w["h"] for m in w["n"]], np.float32)
    turn = lambda p: (ext - np.asarray(p, np.float32)) if k % 2 else np.asarray(p, np.float32)
    return dict(w, src=turn(w["src"]), rec=turn(w["rec"]),
                wavelet=np.ascontiguousarray(np.asarray(w["wavelet"]) * np.float32(1 + k)))


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("host_wavelet", [True, False])
def test_batch_waits_for_the_other_grids_streams(tuned, host_wavelet):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import binding as fd
    shots = wl.batched_shots(nshots=4, nt=30, lo=24, hi=60, nbl=6)
    streams = [torch.cuda.Stream() for _ in shots]
    grids = [fd.Grid.from_workload(w, stream=s.cuda_stream) for w, s in zip(shots, streams)]
    for g, w in zip(grids, shots):
        g.set_model(w["v"])
    flags = fd.FD_BATCH_GRAPH | (fd.FD_BATCH_AUTOTUNE if tuned else 0)
    for k in range(3):
        now = [moved(w, k) for w in shots]
        outs = [np.zeros((w["nt"], len(w["rec"])), np.float32) for w in now]
        spec = []
        for i, (g, w, s, out) in enumerate(zip(grids, now, streams, outs)):
            wav = w["wavelet"]
            with torch.cuda.stream(s):
                if not host_wavelet:
                    ready = torch.from_numpy(wav).cuda()
                    wav = torch.zeros_like(ready)
                if i:
                    torch.cuda._sleep(DELAY)
                if not host_wavelet:
                    wav.copy_(ready)
            spec.append((g, w["src"], wav, w["rec"], out))
        fd.check(fd.batch_forward(spec, flags), "fd_batch_forward")
        for g, w, out in zip(grids, now, outs):
            single = np.zeros_like(out)
            fd.check(g.forward(w["src"], w["wavelet"], w["rec"], single), "fd_forward")
            assert np.abs(single).max() > 0
            np.testing.assert_array_equal(out, single)
    for g in grids:
        g.close()


@pytest.mark.parametrize("nrec", [3, 20000])
def test_point_tables_outlive_a_call_that_only_queues_them(nrec):
    """One grid whose stream is busy while the tables of a run go up (small ones,
    and ones of hundreds of kilobytes), run after run with other points."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_13094_gb300 import build
    build.build()
    from paper_2312_13094_gb300 import binding as fd
    w = wl.small_acoustic(24)
    w["nt"] = 20
    w["wavelet"] = w["wavelet"][:20]
    ext = np.array([(d - 1) * w["h"] for d in w["n"]])
    stream = torch.cuda.Stream()
    with fd.Grid.from_workload(w, stream=stream.cuda_stream) as busy, \
            fd.Grid.from_workload(w) as idle:
        for g in (busy, idle):
            g.set_model(w["v"])
        for k in range(3):
            rec = (np.random.default_rng(k).random((nrec, 3)) * ext).astype(np.float32)
            got, want = (np.zeros((w["nt"], nrec), np.float32) for _ in range(2))
            with torch.cuda.stream(stream):
                torch.cuda._sleep(DELAY)
            fd.check(busy.forward(w["src"], w["wavelet"], rec, got), "fd_forward")
            fd.check(idle.forward(w["src"], w["wavelet"], rec, want), "fd_forward")
            assert np.abs(want).max() > 0
            np.testing.assert_array_equal(got, want)
