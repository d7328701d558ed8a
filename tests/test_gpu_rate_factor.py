"""The device fact behind the rate factors that are taken as 1: networks without the rate
cache skip a rate pass while |c u| <= 2^-26 for every reaction, because ex2.approx of any
such number is 1.  PTX gives the instruction a relative error of 2^-22, so this is a
property of the device and is tried here on every one of those numbers."""
import ctypes as C
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
// the numbers of bits [0, last] and both signs whose ex2.approx is not 1
__global__ void count_kernel(unsigned last, unsigned long long* bad) {
    unsigned long long n = 0;
    for (unsigned b = blockIdx.x * blockDim.x + threadIdx.x; b <= last; b += gridDim.x * blockDim.x)
        for (unsigned s = 0; s < 2; ++s) {
            float y;
            asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(b | s << 31)));
            n += y != 1.0f;
        }
    atomicAdd(bad, n);
}
extern "C" long long count_not_one(unsigned last) {
    unsigned long long *d, h = ~0ull;
    if (cudaMalloc(&d, 8) != cudaSuccess) return -1;
    cudaMemset(d, 0, 8);
    count_kernel<<<1216, 512>>>(last, d);
    const cudaError_t e = cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? (long long)h : -1;
}
"""


def test_ex2_of_small_numbers_is_one(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_5826_gb300 import build
    (tmp_path / "ex2.cu").write_text(SRC)
    so = str(tmp_path / "ex2.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", so, str(tmp_path / "ex2.cu")],
                   check=True)
    f = C.CDLL(so).count_not_one
    f.restype, f.argtypes = C.c_longlong, [C.c_uint]
    last = (127 - 26) << 23  # the bits of 2^-26
    assert f(last) == 0
    # and it is not so for all numbers: 2^-23 to 2^-22 gives others than 1
    assert f((127 - 22) << 23) > 0
