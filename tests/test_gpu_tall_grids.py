"""2-D grids of more tile rows than one grid dimension of a launch holds (65 535).

Narrow grids whose height is past 65 535 rows of the smallest tiles (8 rows); rows of 16-byte,
8-byte and single-element vectors.  Against the oracle, tolerances (relative L2 per field) those
of the other checks: float64 1e-12, mixed preconditioner 1e-5, mixed Jacobian product 1e-4.
"""
import numpy as np
import pytest

from oracle.operators import Model
from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 2, 4])
def test_tall_grid(nx):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    nz = 8 * 65535 + 21
    c = synth.case("uhi_%dx%d" % (nx, nz))
    c["grid"].update(lx=150.0 * nx, lz=90.0 * nz)
    c["sgs"]["mode"] = synth.SGS_SMAGORINSKY
    c["opts"].update(krylov_m=2, precond=synth.PC_BLOCK, pc_sweeps=2)
    u, r = synth.random_state(c, 21, amp=(0.5, 0.3, 0.002)), synth.random_vector(c, 22)
    m = Model(c)
    v = m.unscale(m.scale(r) / np.linalg.norm(m.scale(r)))
    F, z, w = m.F(u), m.precond(u, r, 2), m.jv(u, m.F(u), v, 1e-4)
    d_u, d_r, d_v = (torch.from_numpy(a).cuda() for a in (u, r, v))
    out = torch.empty_like(d_u)

    def check(ref, tol):
        got = out.cpu().numpy()
        for f in range(4):
            err = np.linalg.norm(got[f] - ref[f]) / max(np.linalg.norm(ref[f]), 1e-300)
            assert err < tol, (f, err)

    for prec in (synth.PREC_FP64, synth.PREC_MIXED):
        c["opts"]["precision"] = prec
        s = jfnk.Solver(c)
        if prec == synth.PREC_FP64:
            s.rhs(d_u, out)
            check(F, 1e-12)
        s.precond_apply(d_u, d_r, out)
        check(z, 1e-12 if prec == synth.PREC_FP64 else 1e-5)
        if prec == synth.PREC_MIXED:
            s.jv(d_u, d_v, out, eps=1e-4)
            check(w, 1e-4)
        s.close()
