"""The bounded barrier wait of the kernels: it returns when the phase completes, when another thread has flagged a failure, and by
itself within its limit where nothing ever arrives.  A kernel of one warp, compiled here against the library's own header."""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "razer_ptx.cuh"
using namespace razer;
// mode 0: nothing arrives; 1: nothing arrives and the failure flag is up; 2: the phase completes
__global__ void wait_kernel(unsigned long long* out, int mode) {
  __shared__ __align__(8) unsigned long long barrier;
  __shared__ uint32_t flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&barrier), 1);
    flag = mode == 1;
    if (mode == 2) mbar_arrive(smem_u32(&barrier));
  }
  __syncthreads();
  const unsigned long long t0 = global_ns();
  const bool got = mbar_wait(smem_u32(&barrier), 0, &flag);
  if (threadIdx.x == 0) { out[0] = got; out[1] = global_ns() - t0; out[2] = WAIT_LIMIT_NS; }
}
extern "C" int run_wait(unsigned long long* out, int mode) {
  wait_kernel<<<1, 32>>>(out, mode);
  return (int)cudaDeviceSynchronize();
}
"""


def test_barrier_wait_ends_within_its_limit(tmp_path):
    (tmp_path / "wait.cu").write_text(SOURCE)
    lib = tmp_path / "wait.so"
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_2501_04052_b200", "csrc"), "-o", str(lib), str(tmp_path / "wait.cu")],
                   check=True)
    run = ctypes.CDLL(str(lib)).run_wait
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    results = []
    for mode in (0, 1, 2):
        torch.cuda.synchronize()
        assert run(ctypes.c_void_p(out.data_ptr()), mode) == 0
        results.append(out.tolist())
    (gave_up, long_ns, limit), (flagged, flag_ns, _), (done, done_ns, _) = results
    assert gave_up == 0 and 0.5 * limit <= long_ns <= 1.02 * limit       # 2 % for the poll at hand
    assert flagged == 0 and flag_ns <= 0.01 * limit
    assert done == 1 and done_ns <= 1e-4 * limit
