"""State and residual arrays of 8-byte alignment (the ABI's requirement) against 16-byte aligned ones.

The grids have rows that are whole 16-byte vectors of float64 and tiles inside the periodic box, so
that an aligned array takes the vector loads.  The float64 passes read the caller's arrays; the same
values at an odd multiple of 8 bytes have to give the same result bitwise, and with the Schur
complement, whose kernels are other instantiations for such rows, to 1e-12 (relative L2 per field,
the tolerance of the other float64 preconditioner checks).
"""
import numpy as np
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def offset(a):
    """A copy of a whose data start 8 bytes past a 16-byte boundary."""
    base = torch.empty(a.numel() + 2, dtype=a.dtype, device="cuda")
    first = 1 if base.data_ptr() % 16 == 0 else 2
    v = base[first:first + a.numel()].view(a.shape)
    assert v.data_ptr() % 16 == 8
    return v.copy_(a)


@pytest.mark.parametrize("grid", [(96, 40), (256, 128), (512, 260), (64, 36, 12)])
@pytest.mark.parametrize("prec", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("precond", [synth.PC_BLOCK, synth.PC_SCHUR])
def test_element_aligned_arrays(grid, prec, precond):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    c = synth.case(("tiny_%dx%d" if len(grid) == 2 else "tiny3d_%dx%dx%d") % grid)
    c["sgs"]["mode"] = synth.SGS_SMAGORINSKY
    c["opts"].update(precision=prec, precond=precond, pc_sweeps=4, krylov_m=10)
    s = jfnk.Solver(c)
    un, u = (torch.from_numpy(synth.random_state(c, k, amp=(0.2, 0.1, 0.001))).cuda() for k in (3, 4))
    r = torch.from_numpy(synth.random_vector(c, 5)).cuda()

    def calls(at):
        out = {}
        for name, call in (("rhs", lambda o: s.rhs(at(u), o)), ("residual", lambda o: s.residual(at(un), at(u), o)),
                           ("jv", lambda o: s.jv(at(u), at(r), o, eps=1e-4)),
                           ("precond", lambda o: s.precond_apply(at(u), at(r), o))):
            o = at(torch.zeros_like(u))
            call(o)
            out[name] = o
        w = at(u)
        s.step(w)
        out["step"] = w
        return out

    a, b = calls(lambda t: t.clone()), calls(offset)
    for name in a:
        if precond == synth.PC_SCHUR and prec == synth.PREC_FP64 and name == "precond":
            for f in range(len(u)):
                assert float((a[name][f] - b[name][f]).norm() / a[name][f].norm()) < 1e-12, (name, f)
        else:
            assert torch.equal(a[name], b[name]), name
