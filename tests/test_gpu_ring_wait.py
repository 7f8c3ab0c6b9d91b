"""A claim on the shared ring whose cells do not come in time: the wait ends by
its deadline, the run's error is set, and the warp's queue holds no place that
was not read (csrc/event.cuh, ring_to_queue)."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2503_10263_gb300", "csrc")

CODE = r"""
#include "event.cuh"
using namespace karl;
__global__ void k(Ring R, Control* ctl, int more, int qleft, unsigned long long deadline, int* out) {
  __shared__ WarpQueue Q;
  const int lane = threadIdx.x;
  Q.s[lane].ev = 1000u + lane;
  if (lane == 0) Q.top = qleft;
  __syncwarp();
  const int n = ring_to_queue(R, ctl, 0, more, Q, qleft, deadline);
  if (lane == 0) { out[0] = n; out[1] = Q.top; }
  out[2 + lane] = (int)Q.s[lane].ev;
}
// a ring of 64 cells whose first `ready` are written (particle i has event index i)
extern "C" int run(int ready, int more, int qleft, int* out, int* error, int* abort) {
  const int cap = 64;
  Ring R;
  Control* ctl;
  int* d;
  unsigned long long seq[cap];
  unsigned ev[cap];
  for (int i = 0; i < cap; ++i) { seq[i] = i < ready ? i + 1 : i; ev[i] = (unsigned)i; }
  char* m;
  if (cudaMalloc(&m, 9 * cap * 8) || cudaMemset(m, 0, 9 * cap * 8) ||
      cudaMalloc(&ctl, sizeof(Control)) || cudaMemset(ctl, 0, sizeof(Control)) ||
      cudaMalloc(&d, 34 * 4)) return -1;
  R.z = (double*)m; R.eq = (long long*)(m + cap * 8); R.mu = (double*)(m + 2 * cap * 8);
  R.node = (unsigned long long*)(m + 3 * cap * 8); R.tal = (double*)(m + 4 * cap * 8);
  R.pid = (unsigned long long*)(m + 5 * cap * 8); R.seq = (unsigned long long*)(m + 6 * cap * 8);
  R.ev = (unsigned*)(m + 7 * cap * 8); R.sj = (unsigned*)(m + 8 * cap * 8);
  R.cap = cap; R.mask = cap - 1;
  if (cudaMemcpy(R.seq, seq, sizeof seq, cudaMemcpyHostToDevice) ||
      cudaMemcpy(R.ev, ev, sizeof ev, cudaMemcpyHostToDevice)) return -2;
  k<<<1, 32>>>(R, ctl, more, qleft, ready >= more ? ~0ULL : 1ULL, d);
  Control c;
  if (cudaMemcpy(out, d, 34 * 4, cudaMemcpyDeviceToHost) ||
      cudaMemcpy(&c, ctl, sizeof c, cudaMemcpyDeviceToHost)) return -3;
  *error = c.error;
  *abort = c.abort;
  cudaFree(m); cudaFree(ctl); cudaFree(d);
  return 0;
}
"""
ERR_TIMEOUT = 4


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2503_10263_gb300 import build
    d = tmp_path_factory.mktemp("ring")
    src, lib = d / "ring.cu", d / "ring.so"
    src.write_text(CODE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    f = ctypes.CDLL(str(lib)).run

    def call(ready, more, qleft):
        out, err, ab = (ctypes.c_int * 34)(), ctypes.c_int(), ctypes.c_int()
        assert f(ready, more, qleft, out, ctypes.byref(err), ctypes.byref(ab)) == 0
        return out[0], out[1], list(out)[2:], err.value, ab.value
    return call


@pytest.mark.parametrize("more,qleft", [(1, 0), (9, 7), (16, 0), (16, 15)])
def test_whole_claim_joins_the_queue(run, more, qleft):
    n, top, ev, err, ab = run(more, more, qleft)
    assert (n, top, err, ab) == (qleft + more, qleft + more, 0, 0)
    assert ev[qleft:qleft + more] == list(range(more))
    assert ev[:qleft] == [1000 + i for i in range(qleft)]


@pytest.mark.parametrize("ready,more,qleft", [(0, 1, 0), (0, 16, 15), (8, 9, 7), (3, 16, 0)])
def test_a_cell_that_does_not_come_leaves_the_queue_as_it_was(run, ready, more, qleft):
    n, top, ev, err, ab = run(ready, more, qleft)
    assert (n, top) == (qleft, qleft)
    assert ev[:qleft] == [1000 + i for i in range(qleft)]
    assert (err, ab) == (ERR_TIMEOUT, 1)
