"""Accesses of a warp's lanes to shared data are ordered by what CUDA defines
(warp and block barriers, fences with atomics), not by how a warp happens to
run: device code on the CPU, one coroutine per thread, every access checked
(lanes/lanes.h)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


@pytest.mark.parametrize("program", ["solve_share", "hand_over", "trackers"])
def test_accesses_are_ordered(program, tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / program)
    src = os.path.join(HERE, "lanes", program + ".cpp")
    # compiled with the sanitizer's calls, linked without its library: lanes.h has them
    subprocess.check_call([gxx, "-std=c++17", "-O2", "-w", "-fsanitize=thread",
                           "-ffp-contract=off", "-I" + CUDA, "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(ROOT, "paper_2112_03444_gb300", "csrc"),
                           "-c", src, "-o", exe + ".o"])
    subprocess.check_call([gxx, exe + ".o", "-o", exe])
    run = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
