"""The bounded waits of csrc/ptx.cuh with a short limit: a wait that nothing ends
returns false and sets the abort flag and the status word; after that the wait
for a copy in flight still goes on until the data are there."""
import ctypes
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1009_3308_gb300", "csrc")

SRC = r"""
#define SPH_WAIT_LIMIT (1u << 12)
#include <cuda_runtime.h>
#include "ptx.cuh"
using namespace sph;
constexpr int N = 2048;   // 16 KB of doubles

__global__ void k(const double* src, int* out, unsigned* status) {
    __shared__ __align__(128) double buf[N];
    __shared__ uint64_t copy, never;
    __shared__ int flag;
    if (threadIdx.x == 0) {
        flag = 0;
        mbar_init(&copy, 1);
        mbar_init(&never, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int* abort = &flag;
        out[0] = mbar_wait(&never, 0, abort, status);
        out[1] = *abort;
        out[2] = *status;
        mbar_arrive_expect_tx(&copy, N * sizeof(double));
        bulk_g2s(buf, src, N * sizeof(double), &copy, policy_evict_first());
        out[3] = mbar_drain(&copy, 0, status);
        int same = 0;
        for (int i = 0; i < N; ++i) same += buf[i] == src[i];
        out[4] = same;
        out[5] = mbar_wait2(&copy, 0, &never, 0, abort, status);
    }
}

extern "C" int run(const double* src, int* out, unsigned* status) {
    k<<<1, 32>>>(src, out, status);
    return cudaDeviceSynchronize();
}
"""


def test_waits_end_and_copies_are_awaited(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    src, lib = tmp_path / "w.cu", tmp_path / "libw.so"
    src.write_text(SRC)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    x = torch.arange(2048, dtype=torch.float64, device="cuda") + 1
    out = torch.full((6,), -1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert ctypes.CDLL(str(lib)).run(p(x), p(out), p(status)) == 0
    assert out.tolist() == [0, 1, 1, 1, 2048, 0] and status.item() == 1
