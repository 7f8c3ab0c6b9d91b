"""The kernels' quotients and roots that spare the FP64 pipe
(csrc/exact_arith.cuh) against the IEEE operations, bit for bit: on the host
with the FP32 seeds moved within their error bound, and on the device with its
own seeds.  Operands: any bit pattern, significands next to a power of two,
quotients and roots next to representable numbers and to midpoints."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2503_10263_gb300", "csrc")

HOST = r"""
#include <cstdint>
#include <cstring>
static uint64_t g_move;
static float moved(float y) {            // the seeds' bound: two units of FP32
  int b; std::memcpy(&b, &y, 4);
  g_move = g_move * 6364136223846793005ULL + 1442695040888963407ULL;
  b += (int)((g_move >> 33) % 5) - 2;
  std::memcpy(&y, &b, 4);
  return y;
}
#define XA_SEED(y) moved(y)
#include "exact_arith.cuh"
#include "exact_arith_check.h"
extern "C" long long run(long long first, long long n) {
  long long bad = 0;
  for (long long i = first; i < first + n; ++i) bad += chk_one((uint64_t)i);
  return bad;
}
"""

DEVICE = r"""
#include "exact_arith.cuh"
#include "exact_arith_check.h"
__global__ void k(long long first, long long n, unsigned long long* bad) {
  unsigned long long c = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    c += chk_one((uint64_t)(first + i));
  if (c) atomicAdd(bad, c);
}
extern "C" long long run(long long first, long long n) {
  unsigned long long *d, h = 1;
  if (cudaMalloc(&d, 8) || cudaMemset(d, 0, 8)) return -1;
  k<<<1024, 256>>>(first, n, d);
  if (cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost)) return -2;
  cudaFree(d);
  return (long long)h;
}
"""


def _load(tmp_path, text, ext, cmd):
    src, lib = tmp_path / f"check{ext}", tmp_path / "check.so"
    src.write_text(text)
    subprocess.run(cmd + ["-I", CSRC, "-I", HERE, "-o", str(lib), str(src)], check=True)
    f = ctypes.CDLL(str(lib)).run
    f.argtypes, f.restype = [ctypes.c_longlong] * 2, ctypes.c_longlong
    return f


def test_host_bits(tmp_path):
    f = _load(tmp_path, HOST, ".cpp", ["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared",
                                      "-fPIC"])
    assert f(0, 4_000_000) == 0


@pytest.mark.gpu
def test_device_bits(tmp_path):
    from paper_2503_10263_gb300 import build
    f = _load(tmp_path, DEVICE, ".cu", [build._nvcc(), *build.ARCH, "-O3", "-std=c++17",
                                        "-fmad=false", "-shared", "-Xcompiler", "-fPIC"])
    assert f(10_000_000, 400_000_000) == 0
