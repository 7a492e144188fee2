"""The dynamic shared-memory limit of a kernel belongs to one device.  A host program
stands in for the CUDA runtime with two devices that each keep their own limits and
refuse a launch above them, and takes tensor-core passes of every format through both:
no GPU is needed, as no kernel runs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <map>
#include <utility>

#include <cuda_runtime.h>

#include "wz2_dispatch.h"

static int g_device = 0, g_refused = 0, g_launches = 0, g_large = 0;
static std::map<std::pair<int, const void*>, size_t> g_limit;

extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[{g_device, f}] = (size_t)v;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { return *k = (cudaKernel_t)f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  ++g_launches;
  if (smem <= 48 * 1024) return cudaSuccess;
  ++g_large;
  const auto it = g_limit.find({g_device, (const void*)k});
  if (it != g_limit.end() && smem <= it->second) return cudaSuccess;
  ++g_refused;
  return cudaErrorInvalidValue;
}
}

int main() {
  alignas(64) static unsigned char map[256] = {};
  for (int device = 0; device < 2; ++device) {
    g_device = device;
    for (int fmt = 2; fmt <= 4; ++fmt)
      for (int R : {8, 32})
        for (const void* tmap : {(const void*)map, (const void*)nullptr}) {
          whff::ScaledMmaStep a{};
          a.fmt = fmt, a.M = 256, a.N = 256, a.ld = 256, a.TN = 2, a.ldx = 256, a.R = R, a.L = 1, a.ctas = 8, a.maxseg = 4;
          a.ldy = 256, a.spin = 1, a.tmap = tmap, a.device = device;
          if (whff::scaled_mma_launch(a, nullptr)) return 2;
        }
    for (int rate = 8; rate <= 24; rate += 4)
      for (int R : {8, 32}) {
        whff::MmaStep a{};
        a.rate = rate, a.lift = true, a.M = 256, a.N = 256, a.BM = 64, a.BN = 64, a.ldx = 256, a.R = R, a.L = 1, a.ctas = 8;
        a.maxseg = 4, a.ldy = 256, a.spin = 1, a.map = map, a.device = device;
        if (whff::mma_launch(a, nullptr)) return 3;
      }
    whff::Wz2Step b{};  // the bulk-staged pass
    b.M = 256, b.N = 256, b.BM = 64, b.BN = 64, b.ldx = 256, b.L = 4096, b.maxseg = 1, b.ldy = 256, b.ctas = 1, b.unroll = 2;
    b.lift = true, b.R = 1, b.staged = true, b.device = device;
    if (whff::wz2_launch<8>(b, nullptr) || whff::wz2_launch<16>(b, nullptr) || whff::wz2_launch<24>(b, nullptr)) return 6;
  }
  std::printf("%d launches, %d large, %d refused\n", g_launches, g_large, g_refused);
  return g_large < 20 ? 4 : g_refused ? 5 : 0;
}
"""


def test_every_device_gets_its_limits(tmp_path):
    import paper_1902_08018_gb300 as W

    W.library()  # built and up to date
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "limits.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "limits"
    lib = os.path.join(ROOT, "paper_1902_08018_gb300")
    cmd = [gxx, "-std=c++17", "-rdynamic", "-I", os.path.join(lib, "csrc"), "-I", os.path.join(ROOT, "include"),
           "-I", "/usr/local/cuda/include", str(src), "-L", lib, "-lwhff", f"-Wl,-rpath,{lib}", "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
