"""Spills of the shared-link kernel's FP32 builds (compiled here; no GPU needed): its 80-register build
leaves little room, and 200 bytes of spills per thread cost a quarter of the kernel's speed."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1901_07294_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SRC = """
#include "dslash_mrhs.cuh"
namespace wd {
%s
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_shared_link_fp32_builds_do_not_spill(tmp_path):
    inst = [f"template __global__ void hop_mrhs_kernel<PREC_F32, {r}, {d}, {x}, 3, {d}>(HopArgs, int, int);"
            for r in (18, 12) for d in ("false", "true") for x in ("false", "true")]
    (tmp_path / "k.cu").write_text(SRC % "\n".join(inst))
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-lineinfo",
                        "--expt-relaxed-constexpr", "-Xptxas", "-v", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        "-c", str(tmp_path / "k.cu"), "-o", str(tmp_path / "k.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    kernels = re.findall(r"entry function '(\S*hop_mrhs\S*)'.*?(\d+) bytes spill stores", r.stderr, re.S)
    assert len(kernels) == 8
    for name, spill in kernels:
        assert int(spill) <= 48, (name, spill)
