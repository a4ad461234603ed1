"""The choice of the on-chip tridiagonalisation's class (csrc/tri_pick.h), also
where larger clusters cannot be resident; the C++ check in tests/cpp is compiled
with the host compiler and run."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_block_that_fits_has_a_class_that_holds_it(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "tri_pick_test")
    src = os.path.join(HERE, "cpp", "tri_pick_test.cpp")
    subprocess.run([cxx, "-O2", "-std=c++17", src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
