"""Float64 Arnoldi passes B and CA over every basis size of a cycle, against the oracle's GMRES.

One Newton correction by one whole cycle of 8 to 32 Krylov steps (the forcing term is out of
reach): each instantiation (8, 12, 16, 24 and 32 vectors, the empty ones skipped four at a time,
one CTA per SM above 16) at its ends.  Tolerance (scaled L2 of the correction): 5e-3.  The
finite-difference product divides rounding by its step, so a relative error of 4e-16 in the
oracle's F moves this correction by up to 5e-4; a basis vector left out of the projections moves
it by 8e-2 at least.
"""
import numpy as np
import pytest

from oracle.newton import implicit_step
from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [8, 9, 12, 13, 16, 17, 21, 24, 25, 29, 32])
@pytest.mark.parametrize("grid", [(33, 17), (64, 32)])
def test_fp64_passes_every_basis_size(m, grid):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    nx, nz = grid
    c = synth.case("uhi_%dx%d" % grid)
    c["grid"].update(lx=150.0 * nx, lz=90.0 * nz)
    c["opts"].update(precision=synth.PREC_FP64, precond=synth.PC_BLOCK, krylov_m=m, dt=5.0,
                     max_newton=1, max_restarts=0, eta=1e-13)
    U = synth.random_state(c, 41, amp=(0.3, 0.1, 0.001))
    model, ref_st = Model(c), {}
    ref = implicit_step(model, U, c["opts"], ref_st)
    u = torch.from_numpy(U).cuda()
    st = jfnk.Solver(c).step(u)
    assert st["gmres_iters"] == m and ref_st["gmres_iters"] == [m]
    err = np.linalg.norm(model.scale(u.cpu().numpy() - ref)) / np.linalg.norm(model.scale(ref - U))
    assert err < 5e-3, err
