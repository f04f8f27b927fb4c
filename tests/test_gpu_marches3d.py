"""Long marches of the 3-D sweeps (16, 32 and 64 planes a CTA, with a remainder), against the oracle.

The march lengths follow the number of CTAs, so they need wide grids.  The input repeats a small block
periodically in x and y, which the result then does as well: the oracle evaluates the block, and no
block length divides a tile.  Planes per CTA of each case, for the Helmholtz sweeps (float32,
float64) and the float32 field-block sweeps:
    260 x 250 x 70   32, 64; 64      260 x 250 x 35   16, 32; 64
    132 x 100 x 50    8,  8; 16      132 x 200 x 40    8,  8; 32
    261 x 208 x 66   64, 64; 64 (single elements)
    262 x 250 x 70   64, 64; 64 (pairs of float32)
    516 x 403 x 66   64 (16-byte rows of float32)
Three sweeps and four: the Helmholtz marches run both ways.  Tolerances (relative L2 per field), those
of the other preconditioner checks: float64 1e-12, mixed 1e-5.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOTH = (synth.PREC_FP64, synth.PREC_MIXED)
CASES = [((260, 250, 70), (52, 50), BOTH), ((260, 250, 35), (52, 50), BOTH), ((132, 100, 50), (44, 25), BOTH),
         ((132, 200, 40), (44, 40), BOTH), ((261, 208, 66), (29, 26), BOTH), ((262, 250, 70), (131, 50), BOTH),
         ((516, 403, 66), (43, 31), (synth.PREC_MIXED,))]


@pytest.mark.parametrize("grid,block,prec", [(g, b, p) for g, b, ps in CASES for p in ps])
@pytest.mark.parametrize("kind", ["schur", "smag", "dear"])
def test_long_marches(grid, block, prec, kind):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    (nx, ny, nz), (bx, by) = grid, block
    rx, ry = nx // bx, ny // by
    assert rx * bx == nx and ry * by == ny

    def params(nx_, ny_):
        c = synth.case("uhi3d_%dx%dx%d" % (nx_, ny_, nz))
        c["grid"].update(lx=150.0 * nx_, ly=130.0 * ny_, lz=90.0 * nz)
        c["sgs"]["mode"] = synth.SGS_DEARDORFF if kind == "dear" else synth.SGS_SMAGORINSKY
        c["opts"].update(precision=prec, precond=synth.PC_SCHUR if kind == "schur" else synth.PC_BLOCK, krylov_m=1)
        return c

    c = params(bx, by)
    u, r = synth.random_state(c, 11, amp=(0.5, 0.3, 0.002)), synth.random_vector(c, 12)
    m = Model(c)
    big = params(nx, ny)

    def tiled(a):
        return torch.from_numpy(a).cuda().repeat(1, 1, ry, rx).contiguous()

    d_u, d_r = tiled(u), tiled(r)
    for sweeps in (3, 4):
        ref = m.schur_precond(u, r, sweeps) if kind == "schur" else m.precond(u, r, sweeps)
        big["opts"]["pc_sweeps"] = sweeps
        s = jfnk.Solver(big)
        z = torch.empty_like(d_r)
        s.precond_apply(d_u, d_r, z)
        want = tiled(ref)
        for f in range(5):
            err = float((z[f] - want[f]).norm() / want[f].norm())
            assert err < (1e-12 if prec == synth.PREC_FP64 else 1e-5), (sweeps, f, err)
        s.close()
