"""Tile and march edges of the 3-D passes (strain, plane, column) and field-block sweeps.

Grids one column, row or plane past and short of the 32 x 16 (float32) and 32 x 8 (float64)
plane tiles, the 32-column CTAs and the marches of the column pass and the sweeps; rows of
16-byte (nx = 36, 64), 8-byte (34) and single-element (33, 5) vectors; the smallest nz.
Tolerances (relative L2 per field), those of the other 3-D checks: float64 1e-12, mixed
Jacobian product 1e-4, mixed preconditioner 1e-5.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(5, 3, 4), (33, 17, 9), (34, 16, 17), (36, 9, 5), (64, 33, 8)]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("closure", [synth.SGS_CONST, synth.SGS_SMAGORINSKY, synth.SGS_DEARDORFF])
@pytest.mark.parametrize("prec", [synth.PREC_FP64, synth.PREC_MIXED])
def test_passes3d_tile_edges(grid, closure, prec):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    nx, ny, nz = grid
    c = synth.case("uhi3d_%dx%dx%d" % grid)
    c["grid"].update(lx=150.0 * nx, ly=130.0 * ny, lz=90.0 * nz)
    c["sgs"]["mode"] = closure
    c["sgs"]["K_M"], c["sgs"]["K_H"] = 1.0e3, 1.4e3
    c["opts"]["precision"] = prec
    c["init"] = {"kind": "rest", "H0": 200.0, "patch_halfwidth": 150.0 * nx / 5, "xi": 0.1, "l": 1.5}
    un, u = (synth.random_state(c, k, amp=(0.5, 0.3, 0.002)) for k in (5, 6))
    r = synth.random_vector(c, 7)
    H = synth.heat_flux(c)
    m = Model(c)
    m.set_heat_flux(H)

    def cu(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def check(got, ref, tol):
        got = got.cpu().numpy()
        for f in range(5):
            err = np.linalg.norm(got[f] - ref[f]) / max(np.linalg.norm(ref[f]), 1e-300)
            assert err < tol, (f, err)

    for sweeps in (2, 3, 4):
        c["opts"]["pc_sweeps"] = sweeps
        s = jfnk.Solver(c)
        s.set_surface_flux(cu(H))
        out = torch.empty_like(cu(u))
        s.precond_apply(cu(u), cu(r), out)
        check(out, m.precond(u, r, sweeps), 1e-12 if prec == synth.PREC_FP64 else 1e-5)
    if prec == synth.PREC_FP64:
        s.rhs(cu(u), out)
        check(out, m.F(u), 1e-12)
    s.residual(cu(un), cu(u), out)
    check(out, m.residual(u, m.rhs_f(un)), 1e-12)
    if prec == synth.PREC_MIXED:
        v = m.unscale(m.scale(r) / np.linalg.norm(m.scale(r)))
        s.jv(cu(u), cu(v), out, eps=1e-4)
        check(out, m.jv(u, m.F(u), v, 1e-4), 1e-4)
