"""The divergence of F's pressure equation: no axis is weighted against the others (float64).

F_p = -gamma_p pbar div(u) for p = 0.  For a nearly solenoidal flow the parts of the axes cancel, so
that a rounded derivative weight of one axis would show as an error proportional to that axis's part.
The reference is evaluated in extended precision with the weights 2/3 and 1/12 times 1/h; the error's
projections on the parts have to be a small fraction of a unit in the last place of a weight (0.1 x
2^-53; the unsystematic roundings of the N points leave 2^-53 / sqrt(N)).
"""
import numpy as np
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.mark.parametrize("grid", [(250, 119), (120, 50), (70, 33), (48, 40, 33), (130, 77, 45)])
def test_divergence_weights(grid):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    three = len(grid) == 3
    c = synth.case(("thermal3d_%dx%dx%d" if three else "thermal_stable_%dx%d") % grid)
    c["opts"]["precision"] = synth.PREC_FP64
    g, s = c["grid"], c["strat"]
    nx, nz, ny = g["nx"], g["nz"], g["ny"] if three else 1
    h = [g["lx"] / nx, g["ly"] / ny, g["lz"] / nz] if three else [g["lx"] / nx, g["lz"] / nz]
    x, z = 2 * np.pi * np.arange(nx) / nx, np.pi * (np.arange(nz) + 0.5) / nz
    y = 2 * np.pi * np.arange(ny) / ny
    u = np.zeros((5 if three else 4, nz, ny, nx))
    iw = len(u) - 3
    for k, a, ph in ((1, 3.0, 0.3), (3, 1.1, 1.9), (7, 0.7, 4.0)):          # rolls of all horizontal scales
        for axis, pos in ((0, x[None, None, :]), (1, y[None, :, None]))[: 2 if three else 1]:
            length = g["lx"] if axis == 0 else g["ly"]
            u[axis] += a * np.cos(z)[:, None, None] * np.cos(k * pos + ph + axis)
            u[iw] += a * g["lz"] / np.pi * np.sin(z)[:, None, None] * (2 * np.pi * k / length) * np.sin(k * pos + ph + axis)
    shape = synth.shape(c)
    F = torch.empty(shape, dtype=torch.float64, device="cuda")
    jfnk.Solver(c).rhs(torch.from_numpy(u.reshape(shape)).cuda(), F)
    got = F.cpu().numpy().reshape(u.shape)[-1].astype(L)

    def deriv(f, axis, h_):
        f = f.astype(L)
        if axis == 0:                                                       # z: w is odd at both walls
            e = np.concatenate([-f[:2][::-1], f, -f[-2:][::-1]])
            t = {k: e[2 + k:2 + k + nz] for k in (-2, -1, 1, 2)}
        else:
            t = {k: np.roll(f, -k, axis) for k in (-2, -1, 1, 2)}
        return (L(2.0 / 3.0) * (t[1] - t[-1]) - L(1.0 / 12.0) * (t[2] - t[-2])) * L(1.0 / h_)

    axes = (2, 1, 0) if three else (2, 0)
    parts = [-L(s["gamma_p"]) * L(s["pbar"]) * deriv(u[i], a, h[i]) for i, a in enumerate(axes)]
    err = (got - sum(parts)).astype(np.float64).ravel()
    A = np.stack([p.astype(np.float64).ravel() for p in parts[:-1]], axis=1)
    coef = np.linalg.lstsq(A, err, rcond=None)[0]
    assert np.all(np.abs(coef) <= 0.1 * 2.0**-53), coef * 2.0**53
