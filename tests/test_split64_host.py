"""Host parts of the FP64 digit split."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def _native(tmp_path, name):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / name)
    subprocess.run([cxx, "-O2", "-std=c++17", os.path.join(HERE, "native", name + ".cpp"), "-o", exe],
                   check=True)
    return subprocess.run([exe], capture_output=True, text=True)


def test_operand_slots_are_not_overwritten_before_they_are_read(tmp_path):
    r = _native(tmp_path, "slot_ring_check")
    assert r.returncode == 0 and "ring ok" in r.stdout, r.stdout


def test_batches_fit_the_scratch_they_are_placed_in(tmp_path):
    r = _native(tmp_path, "scratch_check")
    assert r.returncode == 0 and "scratch ok" in r.stdout, r.stdout
