"""The autotuner's choice is between kernels that differ.

Tile indices that launch the same kernel (0, 1 and 3 of the Jacobian product; all of them in 3-D and,
for the preconditioner, with the Schur complement) are one candidate: the smallest index.
"""
import pytest

from paper_2007_10411_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,precond,jv,pc", [
    ((250, 119), synth.PC_BLOCK, {0, 2}, {0, 1, 3}),          # index 0 is 128 threads there, as index 2
    ((1024, 512), synth.PC_BLOCK, {0, 2}, {0, 2, 3}),         # and 256 here, as index 1
    ((256, 128), synth.PC_SCHUR, {0, 2}, {0}),
    ((64, 64, 32), synth.PC_BLOCK, {0}, {0}),
])
def test_autotune_candidates(grid, precond, jv, pc):
    import __graft_entry__
    from paper_2007_10411_gb300 import jfnk
    __graft_entry__.build()
    c = synth.case(("thermal3d_%dx%dx%d" if len(grid) == 3 else "thermal_stable_%dx%d") % grid)
    c["opts"].update(precision=synth.PREC_MIXED, precond=precond, pc_sweeps=4, krylov_m=4)
    s = jfnk.Solver(c)
    u = torch.from_numpy(synth.random_state(c, 3, amp=(0.2, 0.1, 0.001))).cuda()
    picks = [s.autotune(u) for _ in range(8)]
    assert {p[0] for p in picks} <= jv and {p[1] for p in picks} <= pc, picks
