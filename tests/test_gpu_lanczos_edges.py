"""Lanczos bounds (csrc/lanczos.cu) at the ends of the number range, and of a tridiagonal
whose highest Ritz value is an eigenvalue to the last bit: then the last pivot of the
inverse iteration is exactly zero, and the residual still counts.

Bars: the recursion's rounding, 1e-12 of the interval; at subnormal scale one unit there."""
import numpy as np
import pytest
import torch

from oracle import ref

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def diagonal(blocks):
    b = torch.as_tensor(np.asarray(blocks), dtype=torch.float64, device=DEV)
    n = b.shape[0]
    return cg.Bsr(torch.arange(n + 1, device=DEV), torch.arange(n, dtype=torch.int32, device=DEV), b)


@pytest.mark.parametrize("c", [2.5, 3e-310, -3e-310, 1e-320, 1e-290])
def test_a_multiple_of_the_identity_at_every_scale(c):
    e0, e1, th = cg.bounds(diagonal(np.tile(c * np.eye(4), (9, 1, 1))), 20)
    unit = max(36 * 2.0 ** -52 * abs(c), 36 * 2.0 ** -1074)
    assert abs(th[0] - c) <= unit and abs(th[1] - c) <= unit
    assert e0 <= th[0] and e1 >= th[1] and np.isfinite([e0, e1]).all()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -400, 2.0 ** 400])
def test_a_highest_ritz_value_that_is_exact(scale):
    # v0 = e_1 gives T = [[0, 2], [2, 3]] after two steps: eigenvalues -1 and 4, the next
    # beta 1, so the residuals are the last components 1/sqrt(5) and 2/sqrt(5)
    M = np.array([[0.0, 2.0, 0.0, 0.0], [2.0, 3.0, 1.0, 0.0], [0.0, 1.0, 1.0, 1.0], [0.0, 0.0, 1.0, 2.0]]) * scale
    v0 = torch.tensor([1.0, 0.0, 0.0, 0.0], dtype=torch.float64, device=DEV)
    e0, e1, th = cg.bounds(diagonal(M[None]), 2, v0=v0)
    want = np.array([-1.0 - 2.0 / 5 ** 0.5, 4.0 + 4.0 / 5 ** 0.5, -1.0, 4.0]) * scale
    assert np.abs(np.array([e0, e1, *th]) - want).max() <= 1e-12 * 5 * scale
    o0, o1, _, _ = ref.ritz_bounds(np.array([0.0, 3.0]), np.array([2.0, 1.0]))
    assert abs(e0 / scale - o0) <= 1e-9 and abs(e1 / scale - o1) <= 1e-9


def test_one_step_of_values_beyond_1e300():
    e0, e1, th = cg.bounds(diagonal(np.diag([3e302, 3e302, 3e302, 3e302])[None]), 1)
    assert abs(th[0] / 3e302 - 1.0) <= 1e-14 and th[0] == th[1]
