"""Rounding of F(u) in float32 (a mixed handle's jfnk_rhs) against a plain float32 evaluation.

F_j = -1/2 D(u_j u) - 1/2 u_j D u + D(K D u) for theta = p = 0 and constant K.  The plain evaluation
rounds every product and every difference once; so does a flux K D u - 1/2 u_j u whose velocity
product enters a fused multiply-add.  A flux that rounds the product and the sum errs sqrt(2) times
as much: the bound lies half way, 1.2.
"""
import numpy as np
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def evaluate(u, K, h, T):
    """-1/2 D_j(u_j u) - 1/2 u_j D_j u + D_j(K D_j u) of every velocity component in type T."""
    h = [T(v) for v in h]
    axes = (2, 1, 0) if len(u) == 3 else (2, 0)
    u = [a.astype(T) for a in u]
    iw = len(u) - 1

    def d(f, axis, hj, parity):
        if axis == 0:
            n = f.shape[0]
            e = np.concatenate([T(parity) * f[:2][::-1], f, T(parity) * f[-2:][::-1]])
            t = {k: e[2 + k:2 + k + n] for k in (-2, -1, 1, 2)}
        else:
            t = {k: np.roll(f, -k, axis) for k in (-2, -1, 1, 2)}
        return (T(2.0 / 3.0) * (t[1] - t[-1]) - T(1.0 / 12.0) * (t[2] - t[-2])) * (T(1.0) / hj)

    out = []
    for f in range(len(u)):
        par = -1.0 if f == iw else 1.0            # free slip: u, v even, w odd at the walls
        r = T(0)
        for j, a in enumerate(axes):
            g = d(u[f], a, h[j], par)
            r = r - T(0.5) * d(u[j] * u[f], a, h[j], -par) - T(0.5) * u[j] * g + d(T(K) * g, a, h[j], -par)
        out.append(r)
    return out


@pytest.mark.parametrize("grid", [(256, 128), (250, 119), (96, 80, 48)])
def test_float32_flux_is_rounded_once(grid):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    three = len(grid) == 3
    c = synth.case(("thermal3d_%dx%dx%d" if three else "thermal_stable_%dx%d") % grid)
    c["sgs"].update(mode=synth.SGS_CONST, K_M=10.0, K_H=14.1)
    c["opts"]["precision"] = synth.PREC_MIXED
    g = c["grid"]
    nx, nz, ny = g["nx"], g["nz"], g["ny"] if three else 1
    h = [g["lx"] / nx, g["ly"] / ny, g["lz"] / nz] if three else [g["lx"] / nx, g["lz"] / nz]
    x, z = 2 * np.pi * np.arange(nx) / nx, np.pi * (np.arange(nz) + 0.5) / nz
    y = 2 * np.pi * np.arange(ny) / ny
    nf = 5 if three else 4
    nv = nf - 2
    u = np.zeros((nf, nz, ny, nx))
    for f in range(nv):
        prof = np.sin(z) if f == nv - 1 else np.cos(z)
        u[f] = (4.0 + f) * prof[:, None, None] * (1.2 + np.cos(x + f) + 0.4 * np.cos(3 * x + 2 * f))[None, None, :]
        if three:
            u[f] *= (1.0 + 0.5 * np.cos(y + 0.7 * f))[None, :, None]
    u = u.astype(np.float32).astype(np.float64)
    ref, plain = evaluate(u[:nv], 10.0, h, np.float64), evaluate(u[:nv], 10.0, h, np.float32)
    shape = synth.shape(c)
    F = torch.empty(shape, dtype=torch.float64, device="cuda")
    jfnk.Solver(c).rhs(torch.from_numpy(u.reshape(shape)).cuda(), F)
    got = F.cpu().numpy().reshape(u.shape)
    ratio = [np.linalg.norm(got[f] - ref[f]) / np.linalg.norm(plain[f] - ref[f]) for f in range(nv)]
    assert max(ratio) < 1.2, ratio
