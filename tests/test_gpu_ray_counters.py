"""The ray counters of a persistent CTA: per-thread counts whose sum over the CTA exceeds 32 bits reach
the 64-bit totals whole."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1703_09707_gb300 import build as B  # noqa: E402

CODE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
#include "mlens_dev.cuh"
__global__ void k(const unsigned *v, unsigned long long *stats)
{
    __shared__ unsigned long long sred[3];
    if (threadIdx.x < 3) sred[threadIdx.x] = 0ull;
    __syncthreads();
    const unsigned *t = v + 3 * (blockIdx.x * blockDim.x + threadIdx.x);
    mlens::stats_add_cta(t[0], t[1], t[2], sred, stats);
}
extern "C" int run(const unsigned *v, int ctas, int threads, unsigned long long *out)
{
    unsigned *d = nullptr;
    unsigned long long *s = nullptr;
    const size_t n = sizeof(unsigned) * 3 * ctas * threads;
    if (cudaMalloc(&d, n) != cudaSuccess || cudaMalloc(&s, 24) != cudaSuccess) return 1;
    cudaMemcpy(d, v, n, cudaMemcpyHostToDevice);
    cudaMemset(s, 0, 24);
    k<<<ctas, threads>>>(d, s);
    const cudaError_t e = cudaMemcpy(out, s, 24, cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(s);
    return e != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("counters")
    src, so = os.path.join(d, "counters.cu"), os.path.join(d, "counters.so")
    with open(src, "w") as f:
        f.write(CODE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-o", so, src], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("ctas,threads", [(1, 32), (1, 256), (3, 256)])
@pytest.mark.parametrize("top", [9, 1 << 16, 1 << 25, 1 << 32])
def test_sums_beyond_32_bits(lib, ctas, threads, top):
    v = np.random.default_rng(top).integers(0, top, (ctas * threads, 3), dtype=np.uint64).astype(np.uint32)
    v[: threads // 2, 1] = top - 1
    out = np.zeros(3, np.uint64)
    assert lib.run(v.ctypes.data_as(C.c_void_p), ctas, threads, out.ctypes.data_as(C.c_void_p)) == 0
    assert np.array_equal(out, v.astype(np.uint64).sum(0))
