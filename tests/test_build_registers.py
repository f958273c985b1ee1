"""Registers that a kernel's speed rests on, as the compiler reports them (no GPU needed)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_the_epilogue_of_wide_passes_fits_eight_times_on_an_sm(tmp_path):
    """tc_epilogue_kernel waits for memory most of its time and needs all 2048 threads of an SM: 8 CTAs of 256 threads share its
    65,536 registers at 32 per thread.  In passes of up to 64 rows and in those of more (grouped), for every epilogue."""
    src = tmp_path / "epi.cu"
    src.write_text('#include "gemm.cuh"\nnamespace ls {\n' + "".join(
        f"template __global__ void tc_epilogue_kernel<{e}, {g}>(const __grid_constant__ TcEpiParams);\n"
        for e in ("EPI_QKV", "EPI_RESID", "EPI_SWIGLU") for g in ("false", "true")) + "}\n")
    r = subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-Xptxas=-v",
                        "-I", os.path.join(ROOT, "paper_2609_17184_b200", "csrc"), "-c", str(src), "-o", str(tmp_path / "epi.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\S*tc_epilogue_kernel\S*)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", r.stderr, re.S)
    assert len(found) == 6, r.stderr
    assert all(int(regs) <= 32 and int(spill) == 0 for _, spill, regs in found), found
