"""The load model that picks a wave tile, on CPU: wave_load (closed form over
runs of items) equals the busiest CTA of the schedule that wave_schedule lays
out, for tile counts around multiples of the CTA count."""
import os
import shutil
import subprocess

import pytest

from test_sched_host import CSRC, ROOT, _cuda_include


def test_predicted_load_is_that_of_the_schedule(tmp_path):
    gxx, inc = shutil.which("g++"), _cuda_include()
    if not gxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "wave_load_check")
    subprocess.check_call([gxx, "-std=c++17", "-O2", "-I", inc, "-I", CSRC, "-x", "c++",
                           os.path.join(CSRC, "fd_sched.cu"),
                           os.path.join(ROOT, "tests", "native", "wave_load_check.cpp"),
                           "-o", exe])
    rows = [tuple(map(int, r.split())) for r in
            subprocess.check_output([exe], text=True).strip().split("\n")]
    assert len(rows) == 3 * 4 * 8 * 4 + 2
    for G, R, predicted, found in rows:
        assert predicted == found, (G, R, predicted, found)
