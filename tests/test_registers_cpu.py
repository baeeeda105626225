"""Kernels that run at their register limit without a spill keep to it: a kernel of few instructions per byte that saves
registers to local memory pays for it in every thread.  Read off the compiler's own report."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not shutil.which(NVCC), reason="needs nvcc")
def test_topk_kernels_do_not_spill(tmp_path):
    csrc = os.path.join(ROOT, "paper_2507_12000_b200", "csrc")
    r = subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
                        "-I", os.path.join(ROOT, "include"), "-I", csrc, "-c", "-o", str(tmp_path / "topk.o"), os.path.join(csrc, "topk_verify.cu")],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    kernels = re.findall(r"Function properties for (\S+)\n\s*(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr)
    assert sum("topk_fold_kernel" in k[0] for k in kernels) == 3 and len(kernels) >= 9
    assert not [k for k in kernels if k[2] != "0" or k[3] != "0"]
