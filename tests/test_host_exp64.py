"""The FP64 segment weight (vet_exp64.h) on the host: against long double over
depths of every size, at its seams, and what it refuses.  No GPU."""
import os
import shutil
import subprocess

import pytest

from test_host_geometry import CSRC, ROOT, _cuda_include


def test_weight_matches_long_double(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    exe = str(tmp_path / "exp64_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", inc, "-I", CSRC, os.path.join(ROOT, "tests", "host", "exp64_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
