"""The float32 dot-product accumulation of the Arnoldi passes (common.cuh: dotacc).

A thread's running sum takes the four products of a vector at once.  2^24 + 4 x 0.5 is exact that way
and loses every product when they are added one by one; a sum of 64 vectors errs by at most one
rounding of the running sum and three of the (smaller) vector sums each.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "common.cuh"
__global__ void dots(const float4* a, const float4* b, const float* c, float* out, int threads, int vectors) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= threads) return;
    float s = c[i];
    for (int k = 0; k < vectors; ++k) s = jfnk::dotacc(a[i * vectors + k], b[i * vectors + k], s);
    out[i] = s;
}
extern "C" int run(const void* a, const void* b, const void* c, void* out, int threads, int vectors) {
    dots<<<(threads + 255) / 256, 256>>>((const float4*)a, (const float4*)b, (const float*)c, (float*)out, threads, vectors);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def dots(tmp_path_factory):
    from paper_2007_10411_gb300 import build as b
    d = tmp_path_factory.mktemp("dot")
    (d / "dot.cu").write_text(SOURCE)
    nv = b.nvcc()
    subprocess.run([nv, *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared", "-I", b.CSRC,
                    "-I", os.path.join(b.HERE, "..", "include"), str(d / "dot.cu"), "-o", str(d / "dot.so"),
                    "-Xlinker", "-rpath", "-Xlinker", b.cuda_lib_dir(nv)], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "dot.so"))

    def run(a, b, c):
        ta, tb, tc = (torch.from_numpy(x).cuda() for x in (a, b, c))
        out = torch.empty_like(tc)
        torch.cuda.synchronize()
        assert lib.run(*(ctypes.c_void_p(t.data_ptr()) for t in (ta, tb, tc, out)), len(c), a.shape[1]) == 0
        return out.cpu().numpy()

    return run


def test_products_meet_before_the_running_sum(dots):
    a = np.full((1, 64, 4), 0.5, np.float32)
    got = dots(a, np.ones_like(a), np.array([2.0**24], np.float32))
    assert got[0] == 2.0**24 + 128


def test_running_sum_error(dots):
    rng = np.random.default_rng(4)
    a, b = (rng.standard_normal((4096, 64, 4)).astype(np.float32) for _ in range(2))
    got = dots(a, b, np.zeros(4096, np.float32))
    p = (a.astype(np.float64) * b).sum(2)
    s = np.cumsum(p, axis=1)
    size = np.abs(s).sum(1) + 3 * (np.abs(a.astype(np.float64) * b)).sum((1, 2))
    assert np.all(np.abs(got - s[:, -1]) <= 1.01 * 2.0**-24 * size)
