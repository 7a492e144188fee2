"""The CUDA-core kernels for a few columns keep two CTAs of 256 threads on an SM: at most
128 registers a thread of the SM's 65536.  Their folds hold up to three numbers per sum,
which must not decide the registers of the loops before them.  ptxas reports what it
allotted; no GPU is needed."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

SOURCE = """
#include "scaled_kernels.cuh"
#include "wz2_kernels.cuh"
namespace whff {
namespace dev {
#define WZ2(RATE, LIFT, GL) \\
  template __global__ void wz2_gemv_kernel<RATE, LIFT, 4, 2, GL>( \\
      const uint8_t*, int64_t, int64_t, int64_t, int64_t, const float*, int64_t, bool, int64_t, int, double*, double*, \\
      int64_t, double*, double, bool, unsigned*);
#define SCALED(FMT, R, GL) \\
  template __global__ void scaled_range_kernel<FMT, R, GL>( \\
      const uint8_t*, const float*, int64_t, int64_t, int64_t, int64_t, const float*, int64_t, bool, int64_t, int, \\
      double*, double*, int64_t, double*, double, bool, unsigned*);
WZ2(16, true, 32) WZ2(16, true, 8) WZ2(24, false, 32)
SCALED(2, 2, 32) SCALED(2, 2, 8) SCALED(7, 2, 32) SCALED(7, 4, 8)
}  // namespace dev
}  // namespace whff
"""


def test_few_columns_fit_two_ctas(tmp_path):
    if not shutil.which(NVCC):
        pytest.skip("no nvcc")
    src = tmp_path / "few.cu"
    src.write_text(SOURCE)
    cmd = [NVCC, "-std=c++17", "-O3", "-I", os.path.join(ROOT, "include"), "-I",
           os.path.join(ROOT, "paper_1902_08018_gb300", "csrc"), "-gencode", "arch=compute_103a,code=sm_103a", "-Xptxas",
           "-v", "-cubin", str(src), "-o", str(tmp_path / "few.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", r.stderr,
                       re.S)
    found = {name: (int(regs), int(spill)) for name, spill, regs in found if "wz2_gemv" in name or "scaled_range" in name}
    assert len(found) == 7
    for name, (regs, spill) in found.items():
        assert regs <= 128 and spill <= 32, (name, regs, spill)
