"""A step of one call goes on beside another kernel that holds some of the SMs
(for a fixed time, waiting for nothing)."""
import ctypes as C
import subprocess
import time

import numpy as np
import pytest

from paper_2106_08950_gb300 import build as B
from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
// one block to an SM, for ns nanoseconds
__global__ void hold(unsigned long long ns) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    } while (t - t0 < ns);
}
extern "C" int hold_sms(int blocks, unsigned long long ns, void *stream) {
    const int smem = 200 * 1024;
    cudaError_t e = cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) hold<<<blocks, 32, smem, (cudaStream_t)stream>>>(ns);
    return e == cudaSuccess ? (int)cudaGetLastError() : (int)e;
}
"""


@pytest.fixture(scope="module")
def holder(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("hold")
    (d / "hold.cu").write_text(SRC)
    lib = str(d / "libhold.so")
    subprocess.check_call([B.nvcc(), *B.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", lib, str(d / "hold.cu")])
    L = C.CDLL(lib)
    L.hold_sms.argtypes = [C.c_int, C.c_ulonglong, C.c_void_p]
    return L


@pytest.mark.parametrize("batched", [False, True])
def test_one_step_beside_a_resident_kernel(holder, batched):
    import torch
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    prob = W.periodic_suspension(n=1024, count=100, seed=2)
    a, b = (D.Simulation(prob, stream=int(side.cuda_stream)) for _ in range(2))
    run = D.Batch([a]) if batched else a
    run.step(1)                                 # (loads the kernels)
    run.sync()
    b.step(3)
    assert holder.hold_sms(76, 400_000_000, int(other.cuda_stream)) == 0
    time.sleep(0.02)
    t = time.monotonic()
    run.step(1)
    run.step(1)
    run.sync()
    took = time.monotonic() - t
    assert not other.query(), "the other kernel ended first"
    assert took < 0.2
    other.synchronize()
    assert np.array_equal(a.populations(), b.populations())
    for x, y in zip(a.forces(), b.forces()):
        assert np.array_equal(x, y)
    if batched:
        run.close()
    a.close()
    b.close()
