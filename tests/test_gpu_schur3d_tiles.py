"""Tile and march edges of the 3-D Helmholtz sweeps, against the oracle's Schur preconditioner.

Rows of 16-byte vectors and single elements (nx odd), one column or row past a 64 x 16 (float32),
64 x 8 (float64) or 32 x 8 (unaligned) tile, the smallest nz, and nz past a march of 8 and 64 planes.
Tolerances (relative L2 per field): float64 1e-12, mixed 1e-5, those of the other Schur checks.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(4, 1, 4), (5, 3, 4), (21, 13, 9), (33, 9, 17), (64, 16, 8), (68, 17, 5), (12, 8, 70)])
@pytest.mark.parametrize("prec", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("sweeps", [2, 3, 6])
def test_schur3d_tile_edges(grid, prec, sweeps):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    c = synth.case("tiny3d_%dx%dx%d" % grid)
    c["opts"].update(precision=prec, precond=synth.PC_SCHUR, pc_sweeps=sweeps)
    u, r = synth.random_state(c, 11), synth.random_vector(c, 12)
    ref = Model(c).schur_precond(u, r, sweeps)
    s = jfnk.Solver(c)
    d_u, d_r = torch.from_numpy(u).cuda(), torch.from_numpy(r).cuda()
    z = torch.empty_like(d_r)
    s.precond_apply(d_u, d_r, z)
    got = z.cpu().numpy()
    for f in range(5):
        err = np.linalg.norm(got[f] - ref[f]) / np.linalg.norm(ref[f])
        assert err < (1e-12 if prec == synth.PREC_FP64 else 1e-5), (f, err)
