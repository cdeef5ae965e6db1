"""The bounded waits of the tensor-core kernels give one answer per warp.

A one-CTA kernel over the waits of csrc/tc_gemm.cuh: half of a warp's lanes
wait with one limit, the other half with another, and a second warp arrives on
the barrier after a while or never.  What follows such a wait in the GEMM
kernels needs the whole warp, so all lanes have to go the same way, also when
some of them ran out of polls before the arrival and the others did not."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "tc_gemm.cuh"
using namespace cbddc::tc;
// warp 0 waits, lanes below 16 with lim0, the others with lim1; warp 1
// arrives after delay clocks (delay < 0: never); out[0:32] the answers,
// out[32:64] those of the abort flag that only lane 3 of warp 0 sets
__global__ void wait_kernel(unsigned lim0, unsigned lim1, long long delay, int* out) {
  __shared__ uint64_t bar;
  __shared__ int flag[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) {
    out[lane] = warp_wait(&bar, 0, lane < 16 ? lim0 : lim1) ? 1 : 0;
    flag[lane] = lane == 3 ? 1 : 0;
    __syncwarp();
    out[32 + lane] = warp_aborted(&flag[lane]) ? 1 : 0;
  } else if (lane == 0 && delay >= 0) {
    const long long t0 = clock64();
    for (int i = 0; i < (1 << 22) && clock64() - t0 < delay; ++i) {}
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
  }
}
extern "C" int run(unsigned lim0, unsigned lim1, long long delay, int* host) {
  int* d = nullptr;
  if (cudaMalloc(&d, 64 * sizeof(int)) != cudaSuccess) return 1;
  wait_kernel<<<1, 64>>>(lim0, lim1, delay, d);
  const cudaError_t e = cudaMemcpy(host, d, 64 * sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("wait")
    src = d / "wait.cu"
    src.write_text(SOURCE)
    so = d / "libwait.so"
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode=arch=compute_103a,code=sm_103a", "-shared", "-Xcompiler",
                    "-fPIC", "-I", os.path.join(ROOT, "paper_2208_06191_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    L = ctypes.CDLL(str(so))
    L.run.argtypes = [ctypes.c_uint, ctypes.c_uint, ctypes.c_longlong, ctypes.c_void_p]
    return L


MANY = 1 << 20


# no polls at all gives up at once; MANY polls outlast the delay by far
@pytest.mark.parametrize("lim0,lim1,delay,answer", [
    (MANY, MANY, 100000, 1),   # every lane sees the arrival
    (0, MANY, 100000, 0),      # half of the lanes give up before it
    (MANY, 0, 100000, 0),
    (0, 0, 0, 0),
    (3, 3, -1, 0),             # nothing ever arrives
])
def test_one_answer_per_warp(lib, lim0, lim1, delay, answer):
    torch.cuda.synchronize()
    out = np.full(64, -1, np.int32)
    assert lib.run(lim0, lim1, delay, out.ctypes.data) == 0
    assert (out[:32] == answer).all()
    assert (out[32:] == 1).all()
