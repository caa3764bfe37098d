"""The sweep's reciprocal and square root give the correctly rounded result:
compared with CUDA's __frcp_rn and __fsqrt_rn over every FP32 value of their
domains (densities: normal values with a normal reciprocal, of either sign;
squared distances: 0 and from 1e-30 to 2^63)."""
import ctypes as C
import subprocess

import pytest

from paper_2106_08950_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "dilbm_kernels.cuh"
using namespace dilbm;
// out[0]: reciprocals compared, out[1]: differing; out[2], out[3]: square roots
__global__ void compare(unsigned long long *out) {
    unsigned long long n[4] = {0, 0, 0, 0};
    const unsigned step = gridDim.x * blockDim.x;
    for (unsigned long long q = blockIdx.x * blockDim.x + threadIdx.x; q < 1ull << 31; q += step) {
        // a pair: the value and its neighbour above
        const unsigned a = (unsigned)q, b = a + 1 < 0x80000000u ? a + 1 : a;
        const float2 v = make_float2(__uint_as_float(a), __uint_as_float(b));
        const bool in = v.x >= 1.17549435e-38f && v.x <= 8.507059e37f && v.y <= 8.507059e37f;
        if (in) {
            for (int s = 0; s < 2; ++s) {
                const float2 w = s ? make_float2(-v.x, -v.y) : v;
                const float2 r = recip2(w);
                n[0] += 2;
                n[1] += (__float_as_uint(r.x) != __float_as_uint(__frcp_rn(w.x))) + (__float_as_uint(r.y) != __float_as_uint(__frcp_rn(w.y)));
            }
        }
        if (a == 0 || (v.x >= 1e-30f && v.y <= 9.2233720e18f)) {
            const float2 w = a == 0 ? make_float2(0.f, 1.f) : v;
            const float2 r = sqrt2(w);
            n[2] += 2;
            n[3] += (__float_as_uint(r.x) != __float_as_uint(__fsqrt_rn(w.x))) + (__float_as_uint(r.y) != __float_as_uint(__fsqrt_rn(w.y)));
        }
    }
    for (int k = 0; k < 4; ++k) atomicAdd(out + k, n[k]);
}
extern "C" int run_compare(unsigned long long *host) {
    unsigned long long *d = nullptr;
    cudaError_t e = cudaMalloc((void **)&d, 32);
    if (e == cudaSuccess) e = cudaMemset(d, 0, 32);
    if (e == cudaSuccess) {
        compare<<<1216, 256>>>(d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(host, d, 32, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


def test_reciprocal_and_square_root_are_correctly_rounded(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (tmp_path / "round.cu").write_text(SRC)
    lib = str(tmp_path / "libround.so")
    subprocess.check_call([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-fmad=false", "-shared", "-Xcompiler", "-fPIC",
                           "-I", B.CSRC, "--expt-relaxed-constexpr", "-o", lib, str(tmp_path / "round.cu")])
    out = (C.c_ulonglong * 4)()
    assert C.CDLL(lib).run_compare(out) == 0
    assert out[0] > 4_000_000_000 and out[2] > 2_000_000_000
    assert out[1] == 0, f"{out[1]} of {out[0]} reciprocals differ"
    assert out[3] == 0, f"{out[3]} of {out[2]} square roots differ"
