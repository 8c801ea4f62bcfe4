"""Which arrays the anisotropic state's kernels address themselves, on CPU: those
of the grid's own device and managed ones.  Host arrays, and arrays of another
device, which a kernel could not reach without peer access, go through copies."""
import os
import shutil
import subprocess

import pytest

from test_sched_host import CSRC, ROOT, _cuda_include

UNREGISTERED, HOST, DEVICE, MANAGED = range(4)  # cudaMemoryType


def test_only_local_memory_is_addressed(tmp_path):
    gxx, inc = shutil.which("g++"), _cuda_include()
    if not gxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "pointer_check")
    subprocess.check_call([gxx, "-std=c++17", "-I", inc, "-I", CSRC,
                           os.path.join(ROOT, "tests", "native", "pointer_check.cpp"),
                           "-o", exe])
    rows = [tuple(map(int, r.split())) for r in
            subprocess.check_output([exe], text=True).strip().split("\n")]
    assert len(rows) == 24
    for kind, owner, device, answer in rows:
        want = kind == MANAGED or (kind == DEVICE and owner == device)
        assert bool(answer) == want, (kind, owner, device)


def test_state_copies_ask_for_the_grids_device():
    """The state copy decides by the grid's device, and its staged copies leave
    the direction to the driver (the array may be another device's)."""
    src = open(os.path.join(CSRC, "fd_tti.cu")).read()
    body = src[src.index("fd_status copy_state("):]
    body = body[:body.index("\n}\n")]
    assert "is_local_ptr(user, t->d.device)" in body
    assert "is_device_ptr" not in body
    assert body.count("cudaMemcpyDefault") == 2
