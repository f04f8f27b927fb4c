"""Tile edges of the 2-D preconditioner sweeps: field blocks and the Schur complement's Helmholtz sweeps.

Row vectors of 16 bytes (nx a multiple of 4), 8 bytes (even) and one element (odd), grids smaller
than a tile and its halo, one point past a tile in x and z (64 x 32 Helmholtz, 64 x 16 and smaller
field blocks), and nz down to the smallest a launch of one, two, three or four sweeps takes.
Every CTA size of the field-block sweep gives bitwise the same result.
Tolerances (relative L2 per field), those of the other checks: float64 1e-12, mixed 1e-5.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(1, 4), (5, 7), (8, 12), (63, 15), (66, 17), (68, 33), (130, 40), (260, 96)]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("prec", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("kind", ["const", "smag", "dear", "schur"])
def test_sweeps2d_tile_edges(grid, prec, kind):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    nx, nz = grid
    c = synth.case("uhi_%dx%d" % grid)
    c["grid"].update(lx=150.0 * nx, lz=90.0 * nz)
    c["sgs"]["mode"] = {"const": synth.SGS_CONST, "dear": synth.SGS_DEARDORFF}.get(kind, synth.SGS_SMAGORINSKY)
    c["sgs"]["K_M"], c["sgs"]["K_H"] = 1.0e3, 1.4e3
    c["opts"].update(precision=prec, precond=synth.PC_SCHUR if kind == "schur" else synth.PC_BLOCK)
    u, r = synth.random_state(c, 21, amp=(0.5, 0.3, 0.002)), synth.random_vector(c, 22)
    m = Model(c)
    d_u, d_r = torch.from_numpy(u).cuda(), torch.from_numpy(r).cuda()
    for sweeps in (2, 3, 4, 5, 9):
        c["opts"]["pc_sweeps"] = sweeps
        ref = m.schur_precond(u, r, sweeps) if kind == "schur" else m.precond(u, r, sweeps)
        s = jfnk.Solver(c)
        z = torch.empty_like(d_r)
        s.precond_apply(d_u, d_r, z)
        got = z.cpu().numpy()
        for f in range(4):
            err = np.linalg.norm(got[f] - ref[f]) / np.linalg.norm(ref[f])
            assert err < (1e-12 if prec == synth.PREC_FP64 else 1e-5), (sweeps, f, err)
        if prec == synth.PREC_MIXED and kind != "schur":
            for tile in (1, 2, 3):
                s.set_tiles(0, tile)
                y = torch.empty_like(d_r)
                s.precond_apply(d_u, d_r, y)
                assert torch.equal(y, z), (sweeps, tile)
