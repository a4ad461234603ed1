"""The Householder reflector of the on-chip tridiagonalisation (csrc/reflector.h):
FP32 scalars as rounded FP64 ones, small tails beside a large first entry kept.
The C++ check in tests/cpp is compiled with the host compiler and run."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_reflector_scalars(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "reflector_test")
    src = os.path.join(HERE, "cpp", "reflector_test.cpp")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
