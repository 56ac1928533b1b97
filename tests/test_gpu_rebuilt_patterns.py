"""Problem.build_patterns called again: S and H follow to the new patterns, so that their
products keep using the lists of the new plans (few launches), with the same results."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")
from paper_1704_00512_gb300 import solve  # noqa: E402

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("order", [None, "hilbert"])
def test_matrices_follow_the_patterns(order):
    pb = solve.problem_from_system(synth.make_system(100, 8.0, 3), 3.0, DEV, cg.F64, order=order)
    runs = []
    for again in (False, True):
        if again:
            pb.build_patterns()
        for M in (pb.S, pb.H):
            assert M.row_ptr is pb.P_H.row_ptr and M.col_idx is pb.P_H.col_idx
        l0 = cg.launch_count()
        r = solve.powers(pb, bounds_S=(0.05, 5.0), n_terms=40)
        runs.append((cg.launch_count() - l0, r["acc"], r["moments"]))
    assert runs[0][0] == runs[1][0] < 20
    assert torch.equal(runs[0][2], runs[1][2])
    assert all(torch.equal(a, b) for a, b in zip(runs[0][1], runs[1][1]))
