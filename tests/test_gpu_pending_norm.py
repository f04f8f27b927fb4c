"""The finite-difference step from pending partial sums of ||z||^2 (common.cuh: pending_eps).

A preconditioner apply leaves one partial per block, a float-float pair (field blocks) or a float64
(Schur complement); every block of the Jacobian product adds them.  Whatever its size, a block has to
obtain the same step, from sums as exact as its parts: float-float additions within a warp err by
2^-44 each (ff_add), all others by 2^-53, halved by the root; the root errs by 2 x 2^-53, its
reciprocal by 2.5 x 2^-53, the product with the numerator by 2^-53.
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
__global__ void setup(jfnk::Ctl* ctl, int np) {
    ctl->eps_num = 1.0;
    ctl->inv_eps_num = 1.0;
    ctl->eps_part = np;
}
__global__ void step(const jfnk::Ctl* ctl, const double* part, double* out) {
    const double2 e = jfnk::pending_eps(ctl, part);
    if (threadIdx.x == blockDim.x - 1) {
        out[0] = e.x;
        out[1] = e.y;
    }
}
extern "C" size_t ctl_bytes() { return sizeof(jfnk::Ctl); }
extern "C" int run(void* ctl, int np, const double* part, double* out, int threads) {
    setup<<<1, 1>>>((jfnk::Ctl*)ctl, np);
    step<<<1, threads>>>((const jfnk::Ctl*)ctl, part, out);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def pending(tmp_path_factory):
    from paper_2007_10411_gb300 import build as b
    d = tmp_path_factory.mktemp("pending")
    (d / "pending.cu").write_text(SOURCE)
    nv = b.nvcc()
    subprocess.run([nv, *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared", "-I", b.CSRC,
                    "-I", os.path.join(b.HERE, "..", "include"), str(d / "pending.cu"), "-o", str(d / "pending.so"),
                    "-Xlinker", "-rpath", "-Xlinker", b.cuda_lib_dir(nv)], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "pending.so"))
    lib.ctl_bytes.restype = ctypes.c_size_t

    def run(part, np_, threads):
        t = torch.from_numpy(part.view(np.float64)).cuda()
        ctl = torch.zeros(lib.ctl_bytes(), dtype=torch.uint8, device="cuda")
        out = torch.empty(2, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(ctypes.c_void_p(ctl.data_ptr()), np_, ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                       threads) == 0
        return out.cpu().numpy()

    return run


def float_float(v):
    hi = v.astype(np.float32)
    return np.stack([hi, (v - hi.astype(np.float64)).astype(np.float32)], axis=1)


def check(pending, part, np_, total, tol):
    got = [pending(part, np_, threads) for threads in (128, 256)]
    assert np.array_equal(got[0], got[1])
    norm = np.sqrt(np.longdouble(total))
    assert abs(got[0][0] * norm - 1) < tol and abs(got[0][1] / norm - 1) < tol


@pytest.mark.parametrize("n", [1, 31, 128, 129, 512, 700])
def test_float_float_partials(pending, n):
    p = float_float(np.random.default_rng(n).random(n) + 1e-3)
    check(pending, p, n, p.astype(np.longdouble).sum(), ((n + 127) // 128 + 5) * 2.0**-44 + 8 * 2.0**-53)


def test_sums_across_warps_are_float64(pending):
    v = np.zeros(128)
    v[::32] = np.random.default_rng(8).random(4)      # one part a warp: float-float additions err by 1e-15 here
    p = float_float(v)
    check(pending, p, 128, p.astype(np.longdouble).sum(), 5 * 2.0**-53)


@pytest.mark.parametrize("n", [1, 33, 128, 304, 608])
def test_float64_partials(pending, n):
    p = np.random.default_rng(n).random(n) + 1e-3
    check(pending, p, -n, p.astype(np.longdouble).sum(), ((n + 127) // 128 + 5 + 8) * 2.0**-53)
