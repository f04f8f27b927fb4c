"""The mixed 2-D Jacobian product on rows that are no multiple of a vector load, against the oracle.

Rows of single elements (odd nx), pairs (even nx) and one 16-byte case; grids smaller than a tile and its
halo, one column or row past a tile (32, 64 x 4, 8, 16), both CTA sizes.  No-slip ground, so that
the eddy coefficients of ghost rows are those of their images.  Tolerance (relative L2 per field)
that of the other mixed products, 1e-4.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(1, 4), (5, 7), (33, 9), (67, 40), (131, 17), (2, 5), (6, 9), (66, 17), (130, 41), (68, 33)])
@pytest.mark.parametrize("closure", [synth.SGS_CONST, synth.SGS_SMAGORINSKY, synth.SGS_DEARDORFF])
def test_jv2d_rows(grid, closure):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    nx, nz = grid
    c = synth.case("uhi_%dx%d" % grid)
    c["grid"].update(lx=150.0 * nx, lz=90.0 * nz)
    c["sgs"]["mode"] = closure
    c["sgs"]["K_M"], c["sgs"]["K_H"] = 1.0e3, 1.4e3
    c["opts"]["precision"] = synth.PREC_MIXED
    u, r = synth.random_state(c, 21, amp=(0.5, 0.3, 0.002)), synth.random_vector(c, 22)
    m = Model(c)
    v = m.unscale(m.scale(r) / np.linalg.norm(m.scale(r)))
    ref = m.jv(u, m.F(u), v, 1e-4)
    s = jfnk.Solver(c)
    d_u, d_v = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    for tile in (0, 2):
        s.set_tiles(tile, 0)
        out = torch.empty_like(d_u)
        s.jv(d_u, d_v, out, eps=1e-4)
        got = out.cpu().numpy()
        for f in range(4):
            err = np.linalg.norm(got[f] - ref[f]) / np.linalg.norm(ref[f])
            assert err < 1e-4, (tile, f, err)
