"""The float64 square roots of the kernels (common.cuh: root, root_pair) over the whole range.

Random mantissas at every normal exponent, perfect squares and their neighbours, the smallest and
largest normals, subnormals, zeros, negatives, infinities and NaN, against the correctly rounded
square root.  Bounds, from the roundings of the iteration: the last step adds a residual that is
exact up to 2^-54 of the root to a root good to about 39 bits, so the result is within one unit in
the last place; the reciprocal carries half of three roundings and one whole one, 2.5 x 2^-53.
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
__global__ void roots(const double* x, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = jfnk::root(x[i]);
    jfnk::root_pair(x[i], out[n + i], out[2 * n + i]);
}
extern "C" int run(const double* x, double* out, int n) {
    roots<<<(n + 255) / 256, 256>>>(x, out, n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    from paper_2007_10411_gb300 import build as b
    d = tmp_path_factory.mktemp("root")
    (d / "roots.cu").write_text(SOURCE)
    nv = b.nvcc()
    subprocess.run([nv, *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared", "-I", b.CSRC,
                    "-I", os.path.join(b.HERE, "..", "include"), str(d / "roots.cu"), "-o", str(d / "roots.so"),
                    "-Xlinker", "-rpath", "-Xlinker", b.cuda_lib_dir(nv)], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "roots.so"))

    def run(x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        out = torch.empty(3, t.numel(), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(out.data_ptr()), t.numel()) == 0
        return out.cpu().numpy()

    return run


def test_roots_of_normal_numbers(roots):
    rng = np.random.default_rng(1)
    e = np.arange(-1022, 1024)
    x = np.ldexp(1.0 + rng.random((e.size, 512)), e[:, None]).ravel()
    k = rng.integers(1, 2**26, 20000).astype(np.float64) ** 2
    lim = np.array([np.finfo(np.float64).tiny, np.finfo(np.float64).max, 1.0, 2.0, 4.0])
    x = np.concatenate([x, k, np.nextafter(k, 0.0), np.nextafter(k, np.inf), lim, np.nextafter(lim[2:], 0.0)])
    x = x[np.isfinite(x)]
    root, g, ig = roots(x)
    ref = np.sqrt(x)
    for got in (root, g):
        assert np.max(np.abs(got - ref) / np.spacing(ref)) <= 1.0
    rel = np.abs(ig.astype(np.longdouble) * np.sqrt(x.astype(np.longdouble)) - 1)
    assert rel.max() <= 2.5 * 2.0**-53 + 2.0**-60


def test_roots_of_special_operands(roots):
    sub = np.concatenate([np.ldexp(1.0, np.arange(-1074, -1022)), np.random.default_rng(2).random(1000) * 2.0**-1022])
    with np.errstate(all="ignore"):
        root, g, ig = roots(sub)
        ref = np.sqrt(sub)
        assert np.array_equal(root, ref) and np.array_equal(g, ref) and np.array_equal(ig, 1.0 / ref)
    x = np.array([0.0, -0.0, -1.0, -np.inf, -2.0**-1060, np.inf, np.nan, -np.nan])
    root, g, ig = roots(x)
    with np.errstate(all="ignore"):
        assert np.array_equal(root, np.sqrt(x), equal_nan=True)
    assert np.array_equal(g, [0, 0, 0, 0, 0, np.inf, np.nan, np.nan], equal_nan=True)
    assert np.array_equal(ig, [0, 0, 0, 0, 0, 0, np.nan, np.nan], equal_nan=True)
