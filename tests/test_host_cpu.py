"""Host code of the library on a fake CUDA runtime: tests/host_check.cpp is
linked with the library's own objects and tests/fake_cudart.h in place of the
CUDA runtime (no GPU) and run."""
import os
import shutil
import subprocess

import pytest

from test_planner_cpu import cuda_include

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_host_code(tmp_path):
    gxx = shutil.which("g++")
    inc = cuda_include()
    if not gxx or not inc:
        pytest.skip("g++ or the CUDA headers are missing")
    from paper_1612_08091_gb300 import build

    build.build()
    objs = [os.path.join(build.BUILD, src + ".o") for src in build.SOURCES]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    exe = str(tmp_path / "host_check")
    cmd = [gxx, "-O1", "-std=c++17", "-I", inc, os.path.join(ROOT, "tests", "host_check.cpp")]
    cmd += objs + ["-ldl", "-lpthread", "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
