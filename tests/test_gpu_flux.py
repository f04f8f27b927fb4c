"""Tile edges of the 2-D flux stencil: F(u) and R(u^n, u) in float64 against the oracle.

The sizes take every tile shape of the launcher's rule (8x8, 16x8, 16x16, 32x16), exact
multiples and remainders of one row or column, and grids smaller than a tile and its halo.
Tolerance: relative L2 per field 1e-12, the bound of the float64 operators (about 130
operations a point of 2^-53 each, the largest terms exceeding F by no more than 1e2).
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(1, 4), (5, 5), (8, 8), (9, 9), (17, 10), (96, 96), (129, 67), (250, 119), (256, 144), (510, 257), (1027, 130)]


@pytest.mark.parametrize("nx,nz", SIZES)
@pytest.mark.parametrize("closure", [synth.SGS_CONST, synth.SGS_SMAGORINSKY, synth.SGS_DEARDORFF])
def test_flux_stencil_tile_edges(nx, nz, closure):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    c = synth.case("uhi_%dx%d" % (nx, nz))          # no-slip ground: K must take its image row there
    c["grid"].update(lx=150.0 * nx, lz=90.0 * nz)
    c["sgs"]["mode"] = closure
    c["opts"]["precision"] = synth.PREC_FP64
    c["init"] = {"kind": "rest", "H0": 200.0, "patch_halfwidth": 150.0 * nx / 5, "xi": 0.1, "l": 1.5}
    un, u = (synth.random_state(c, k, amp=(1.0, 0.5, 0.005)) for k in (5, 6))
    H = synth.heat_flux(c)
    model = Model(c)
    model.set_heat_flux(H)
    s = jfnk.Solver(c)
    s.set_surface_flux(torch.from_numpy(H).cuda())
    d_un, d_u = torch.from_numpy(un).cuda(), torch.from_numpy(u).cuda()
    F, R = torch.empty_like(d_u), torch.empty_like(d_u)
    s.rhs(d_u, F)
    s.residual(d_un, d_u, R)
    torch.cuda.synchronize()
    for got, ref in ((F, model.F(u)), (R, model.residual(u, model.rhs_f(un)))):
        got = got.cpu().numpy()
        for f in range(4):
            err = np.linalg.norm(got[f] - ref[f]) / max(np.linalg.norm(ref[f]), 1e-300)
            assert err < 1e-12, (f, err)
