"""The FP64 segment weight (vet_exp64.h) on the host at the edges of its premise, under the
undefined-behaviour sanitizer where the compiler has it.  No GPU."""
import os
import shutil
import subprocess

import pytest

from test_host_geometry import CSRC, ROOT, _cuda_include


def test_edges_of_the_premise(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    exe = str(tmp_path / "exp64_edges")
    cmd = [cxx, "-O1", "-std=c++17", "-I", inc, "-I", CSRC, os.path.join(ROOT, "tests", "host", "exp64_edges.cpp"), "-o", exe]
    sanitize = ["-fsanitize=undefined", "-fno-sanitize-recover=all"]
    if subprocess.run(cmd + sanitize, capture_output=True).returncode:
        subprocess.run(cmd, check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
