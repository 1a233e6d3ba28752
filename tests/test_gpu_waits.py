"""The bounded wait of the operator kernels gives every lane of a warp the same answer, also when only some of
its lanes have run out of tries: the warp then takes one path, and the kernel returns its error."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# Warp 0 waits, the odd lanes with one try of at most 1 ms, the even ones with 1,000; warp 1 completes the phase
# after 8 ms or more (late = 1) or at once (late = 0).
SOURCE = r"""
#include "lp_ptx.cuh"
__global__ void k_wait(int late, int* out) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    stdg::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    out[threadIdx.x] = stdg::warp_wait_gave_up(&bar, 0, (threadIdx.x & 1) ? 0 : 1000) ? 1 : 0;
  } else if (threadIdx.x == 32) {
    unsigned long long t0, t1;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int k = 0; late && k < 100000; ++k) {
      __nanosleep(100000);
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
      if (t1 - t0 > 8000000) break;
    }
    stdg::mbar_arrive(&bar);
  }
  __syncthreads();
}
extern "C" int run(int late, int* out) {
  k_wait<<<1, 64>>>(late, out);
  const cudaError_t e = cudaGetLastError();
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1601_07384_gb300 import build as b
    d = tmp_path_factory.mktemp("wait")
    (d / "wait.cu").write_text(SOURCE)
    so = str(d / "wait.so")
    subprocess.run([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-I", b.CSRC, "-Xcompiler", "-fPIC", "-shared", "-o", so,
                    str(d / "wait.cu")], check=True, capture_output=True)
    assert os.path.exists(so)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("late", [0, 1])
def test_all_lanes_of_a_warp_agree(lib, late):
    out = torch.full((32,), -1, dtype=torch.int32, device="cuda")
    assert lib.run(late, ctypes.c_void_p(out.data_ptr())) == 0
    assert out.cpu().tolist() == [late] * 32
