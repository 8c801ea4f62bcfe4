"""Scratch slots of the descent step, on CPU: a call that leaves with work still
queued waits for it before its slot can be taken again."""
import os
import shutil
import subprocess

import pytest

from test_sched_host import CSRC, ROOT


def test_slot_is_held_until_its_work_is_done(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    exe = str(tmp_path / "slots_check")
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC,
                           os.path.join(ROOT, "tests", "native", "slots_check.cpp"), "-o", exe])
    out = subprocess.check_output([exe], text=True).split("\n")
    assert out[0] == "idle 0 1 0"
    assert out[1] == "busy 1 1 0"
    assert out[2] == "slots 0 1 2 3"
    assert out[3] == "again 0"
    assert out[4] == "clashes 0"
