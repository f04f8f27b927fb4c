"""Rounding of the Schur complement's Helmholtz sweeps on smooth right-hand sides, against the oracle.

H = (2/dt) I - a sum_j D_j D_j with large a / h^2: applied through coefficients of x that add up to
zero, it rounds at a / h^2 times x instead of at the size of its result.  Through differences of x a
sweep adds about three roundings of the pressure (residual, direction, iterate) and the sweeps'
roundings are independent: 3 sqrt(32) x 2^-24 after 32 sweeps in float32 (relative L2 of p).  The
reference is evaluated in extended precision.
"""
import numpy as np
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SWEEPS = 32
L = np.longdouble


def pressure(c, r):
    """p of the Schur complement's solution for r [field][z][y][x], extended precision."""
    g, st, o = c["grid"], c["strat"], c["opts"]
    three = g["dim"] == 3
    h = {2: L(g["lx"]) / L(g["nx"]), 0: L(g["lz"]) / L(g["nz"])}
    if three:
        h[1] = L(g["ly"]) / L(g["ny"])
    axes = (2, 1, 0) if three else (2, 0)
    A, B = L(2) / L(3), L(1) / L(12)

    def d(f, axis, parity=1.0):
        if axis == 0:
            n = f.shape[0]
            e = np.concatenate([L(parity) * f[:2][::-1], f, L(parity) * f[-2:][::-1]])
            t = {k: e[2 + k:2 + k + n] for k in (-2, -1, 1, 2)}
        else:
            t = {k: np.roll(f, -k, axis) for k in (-2, -1, 1, 2)}
        return (A * (t[1] - t[-1]) - B * (t[2] - t[-2])) / h[axis]

    half, su, sp = L(o["dt"]) / 2, L(o["scale_u"]), L(o["scale_p"])
    cg = L(st["gamma_p"]) * L(st["pbar"])
    a = cg * L(st["theta0"]) * half
    rhs = r[-1] * sp - cg * half * sum(d(su * r[i], ax, -1.0 if ax == 0 else 1.0) for i, ax in enumerate(axes))
    lo = 1 / half
    hi = lo + L(2.25) * a * sum(1 / v**2 for v in h.values())
    theta, delta = (hi + lo) / 2, (hi - lo) / 2
    rho = delta / theta
    x = dk = rhs / theta
    for _ in range(1, SWEEPS):
        new = 1 / (2 * theta / delta - rho)
        hx = lo * x - a * sum(d(d(x, ax), ax, -1.0 if ax == 0 else 1.0) for ax in axes)
        dk = new * rho * dk + 2 * new / delta * (rhs - hx)
        x, rho = x + dk, new
    return x / sp


@pytest.mark.parametrize("grid", [(1024, 512), (512, 129), (1023, 300), (64, 64, 32), (63, 50, 40)])
def test_smooth_right_hand_side(grid):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    three = len(grid) == 3
    c = synth.case(("thermal3d_%dx%dx%d" if three else "thermal_stable_%dx%d") % grid)
    c["opts"].update(precision=synth.PREC_MIXED, precond=synth.PC_SCHUR, pc_sweeps=SWEEPS, krylov_m=2)
    g = c["grid"]
    nx, nz, ny = g["nx"], g["nz"], g["ny"] if three else 1
    x = 2 * np.pi * np.arange(nx) / nx
    z = np.pi * (np.arange(nz) + 0.5) / nz
    y = 2 * np.pi * np.arange(ny) / ny
    r = np.zeros((5 if three else 4, nz, ny, nx))
    for f in range(len(r)):
        prof = np.sin(z) if f == len(r) - 3 else 1.0 + 0.5 * np.cos(2 * z)
        r[f] = prof[:, None, None] * (1.0 + 0.3 * np.cos(y + f))[None, :, None] * np.cos(x + 0.8 * f)[None, None, :]
    shape = synth.shape(c)
    r = r.astype(np.float32).astype(np.float64)
    ref = pressure(c, r.astype(L)).reshape(shape[1:])
    r = r.reshape(shape)
    u = synth.random_state(c, 1, amp=(0.2, 0.1, 0.001))
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    jfnk.Solver(c).precond_apply(torch.from_numpy(u).cuda(), torch.from_numpy(r).cuda(), out)
    got = out.cpu().numpy()
    err = np.sqrt(float(((got[-1] - ref) ** 2).sum() / (ref ** 2).sum()))
    assert err < 3 * np.sqrt(SWEEPS) * 2.0**-24, err
