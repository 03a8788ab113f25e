"""Pinned memory and events that threads hand on when they end, on a made-up CUDA runtime: no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_03420_gb300", "csrc")


def test_threads_that_end_hand_on_what_they_kept(tmp_path):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "thread_kit_host")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", CSRC, "-I", cuda, "-x", "c++", os.path.join(CSRC, "thread_kit.cu"),
                    os.path.join(ROOT, "tests", "thread_kit_host.cpp"), "-o", exe, "-lpthread"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
