"""The kept arena blocks (csrc/blocks.cu): host code, here on a made-up CUDA runtime that ends the program where work on a
block is not ordered behind the block's last use.  No GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_03420_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = next((d for d in ("/usr/local/cuda/include",) if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)
    if not shutil.which("g++") or not cuda:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("blocks") / "blocks_host")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", CSRC, "-I", cuda, "-x", "c++", os.path.join(CSRC, "blocks.cu"),
                    os.path.join(ROOT, "tests", "blocks_host.cpp"), "-o", exe, "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("case", ["abandoned set", "failed wait", "work after the wait", "second attempt", "another stream's work",
                                  "the library's stream", "given back to the pool", "waited for",
                                  "taken block", "near size", "smallest that fits", "idle first", "changing budgets",
                                  "passed over", "a quarter of the memory", "number of blocks", "small ones", "out of memory",
                                  "trim", "events", "last graph"])
def test_blocks(program, case):
    r = subprocess.run([program, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
