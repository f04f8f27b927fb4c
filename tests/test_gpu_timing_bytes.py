"""Bytes that the kernel timing reports for a Schur-complement preconditioner apply, against the
launches it makes: planes read and written once per launch, listed here launch by launch."""
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def planes(groups, nf):
    """rhs kernel and back-substitution, then one entry of `groups` (its sweeps) per Helmholtz launch."""
    b = nf + 2 * nf - 1
    for i in range(len(groups)):
        b += (1 if i == 0 else 3) + (1 if i == len(groups) - 1 else 2)
    return b


@pytest.mark.parametrize("grid,prec,groups", [
    ((64, 48), synth.PREC_MIXED, [4] * 7 + [3]),            # 31 sweeps: float32 row vectors, four a launch
    ((62, 48), synth.PREC_MIXED, [2] * 15 + [1]),           # rows that are no 16-byte vectors: pairs
    ((64, 48), synth.PREC_FP64, [2] * 15 + [1]),
    ((64, 13), synth.PREC_MIXED, [3] * 10 + [1]),           # one reflection of 13 rows: three a launch
    ((64, 6), synth.PREC_MIXED, [1] * 31),
    ((32, 16, 8), synth.PREC_MIXED, [1] * 31),
])
def test_schur_apply_bytes(grid, prec, groups):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    assert sum(groups) == 31
    three = len(grid) == 3
    c = synth.case(("tiny3d_%dx%dx%d" if three else "tiny_%dx%d") % grid)
    c["opts"].update(precision=prec, precond=synth.PC_SCHUR, pc_sweeps=32, krylov_m=10)
    s = jfnk.Solver(c)
    u = torch.from_numpy(synth.random_state(c, 3, amp=(0.2, 0.1, 0.001))).cuda()
    s.kernel_timing(families=("precond",))
    s.step(u)
    kt = s.kernel_timing_read()["precond"]
    npt = u[0].numel()
    assert kt["launches"] > 0
    assert kt["bytes"] == kt["launches"] * planes(groups, 5 if three else 4) * npt * (8 if prec == synth.PREC_FP64 else 4)


@pytest.mark.parametrize("grid", [(64, 48), (32, 16, 8)])
@pytest.mark.parametrize("prec", [synth.PREC_FP64, synth.PREC_MIXED])
@pytest.mark.parametrize("closure", [synth.SGS_CONST, synth.SGS_SMAGORINSKY])
@pytest.mark.parametrize("sweeps", [1, 2, 4])
def test_field_block_apply_bytes(grid, prec, closure, sweeps):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    three = len(grid) == 3
    nf = 5 if three else 4
    c = synth.case(("tiny3d_%dx%dx%d" if three else "tiny_%dx%d") % grid)
    c["sgs"]["mode"] = closure
    c["opts"].update(precision=prec, precond=synth.PC_BLOCK, pc_sweeps=sweeps, krylov_m=10)
    s = jfnk.Solver(c)
    u = torch.from_numpy(synth.random_state(c, 3, amp=(0.2, 0.1, 0.001))).cuda()
    s.kernel_timing(families=("precond",))
    s.step(u)
    kt = s.kernel_timing_read()["precond"]
    eddy = 0 if closure == synth.SGS_CONST else 1
    # planes of one launch: each diffused field's r and x, d in after the first sweep and out before
    # the last, the eddy field; p read and written by the last sweep
    b = {1: 2 * nf, 2: 2 * (nf - 1) + eddy + 2, 4: (nf - 1) * (3 + 5 + 4) + 3 * eddy + 2}[sweeps]
    assert kt["launches"] > 0
    assert kt["bytes"] == kt["launches"] * b * u[0].numel() * (8 if prec == synth.PREC_FP64 else 4)
