"""The check that a launch fits before it is captured: a launch refused in there would be missing
from the graph. Nothing is launched here that does not fit."""
import ctypes
import importlib
import subprocess

import pytest

build = importlib.import_module("paper_1001_3301_gb300.build")  # (the package has a function of that name)

pytestmark = pytest.mark.gpu

SRC = """
#include "rt_internal.cuh"
__global__ void __launch_bounds__(512) k_static(float *out)
{
    __shared__ float s[1668];  // 6672 bytes
    extern __shared__ float d[];
    s[threadIdx.x] = d[threadIdx.x] = threadIdx.x;
    __syncthreads();
    out[threadIdx.x] = s[blockDim.x - 1 - threadIdx.x] + d[threadIdx.x];
}
extern "C" int fits(int threads, int smem) { return rt::launch_fits((const void *)k_static, threads, (size_t)smem); }
extern "C" int raise_limit(int smem)
{
    return (int)cudaFuncSetAttribute(k_static, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}
extern "C" int run(int threads, int smem)
{
    float *p = nullptr;
    cudaMalloc(&p, 4096);
    k_static<<<1, threads, smem>>>(p);
    const int e = (int)cudaGetLastError(), f = (int)cudaDeviceSynchronize();
    cudaFree(p);
    return e ? e : f;
}
"""


def test_launch_fits(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (tmp_path / "t.cu").write_text(SRC)
    so = tmp_path / "libfits.so"
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-cudart", "static", str(tmp_path / "t.cu"),
                                                                     "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    edge = 48 * 1024 - 6672  # with the static part 48 KB
    assert lib.fits(512, 4096) and lib.fits(512, edge) and lib.run(512, edge) == 0
    assert not lib.fits(512, edge + 16) and not lib.fits(512, 48 * 1024) and not lib.fits(512, 64 * 1024)
    assert not lib.fits(1024, 4096)
    assert lib.raise_limit(64 * 1024) == 0
    assert lib.fits(512, edge + 16) and lib.fits(512, 64 * 1024) and lib.run(512, 64 * 1024) == 0
    assert not lib.fits(512, 64 * 1024 + 16)
