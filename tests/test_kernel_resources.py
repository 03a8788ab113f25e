"""The join kernels keep their state in registers and shared memory: what the compiler says of their spills.  A few words
that are set once a unit may be spilled; the row pass and the slot tiles, which need all 64 registers, must not pay for what
the kernel around them keeps.  No GPU."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_03420_gb300", "csrc")


@pytest.mark.parametrize("source,kernel,variants", [("batch.cu", "k_batch", 4), ("join.cu", "k_query", 2)])
def test_spills(tmp_path, source, kernel, variants):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-lineinfo", "-std=c++17", "-Xptxas", "-v",
                        "-cubin", "-o", str(tmp_path / "out.cubin"), os.path.join(CSRC, source)], capture_output=True, text=True,
                       check=True)
    found = re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr, re.S)
    spills = [(int(s), int(l)) for name, s, l in found if kernel + "I" in name]
    assert len(spills) == variants
    assert max(s for s, _ in spills) <= 64 and max(l for _, l in spills) <= 64, spills
