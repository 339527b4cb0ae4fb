"""The planning of the one-warp windows and strips (no GPU): they cover each member once and,
replayed with node numbers in place of values, pull the right nodes at every step: the windows in
every form (positions a lane, lane groups, steps between trades, clusters or not), periodic and
bounded (tests/wave_check.cu), the strips with several members' segments in a warp
(tests/strip_check.cu), through the library's exported host functions."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("check", ["wave_check", "strip_check"])
def test_one_warp_plans(tmp_path, check):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    from paper_0907_1720_gb300 import build as B
    libdir = os.path.dirname(B.build())
    exe = str(tmp_path / check)
    cmd = [nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_0907_1720_gb300", "csrc"),
           os.path.join(ROOT, "tests", check + ".cu"), "-o", exe, "-L", libdir, "-llbhpde", "-lcudart",
           "-Xlinker", "-rpath=" + libdir]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout[-2000:]
