"""Lanczos bounds (csrc/lanczos.cu) against the oracle at the sizes where the kernels
can go wrong: one block row, rows of one block beside rows of many (around the four
and eight blocks a warp reads at once), one step, as many steps as the interface
takes, and a breakdown at the first step.

Bars: the first few steps are the recursion's rounding, (k + row sum) u with a margin
of 1e3 of them; later ones lose orthogonality alike on both sides and agree at the
extremes to 1e-9 of the width."""
import numpy as np
import pytest
import torch

from oracle import ref

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def matrix(nbr, seed):
    """Symmetric, row 0 with as many blocks as there are, others with 1 to about 12."""
    rng = np.random.default_rng(seed)
    on = np.eye(nbr, dtype=bool)
    on[0, : nbr // 2 + 1] = True
    for i in range(1, nbr):
        on[i, rng.integers(0, nbr, size=i % 6)] = True
    on |= on.T
    D = np.where(on.repeat(4, 0).repeat(4, 1), rng.normal(size=(4 * nbr, 4 * nbr)), 0.0)
    D = 0.5 * (D + D.T)
    I, J = np.nonzero(on)
    vals = D.reshape(nbr, 4, nbr, 4).transpose(0, 2, 1, 3)[I, J]
    rp = np.concatenate([[0], np.cumsum(on.sum(1))])
    return ref.Bsr(rp.astype(np.int64), J.astype(np.int32), np.ascontiguousarray(vals)), D


def dev(M, shift=0):
    buf = torch.zeros(M.vals.size + shift, dtype=torch.float64, device=DEV)
    buf[shift:] = torch.as_tensor(M.vals.reshape(-1), device=DEV)
    return cg.Bsr(torch.as_tensor(M.row_ptr, device=DEV), torch.as_tensor(M.col_idx, device=DEV),
                  buf[shift:].view(-1, 4, 4))


@pytest.mark.parametrize("nbr,k", [(1, 1), (1, 3), (3, 1), (3, 2), (50, 5), (50, 40), (100, 512), (700, 6), (2500, 30)])
def test_bounds_sizes(nbr, k):
    M, D = matrix(nbr, nbr + k)
    v0 = 1.0 + np.random.default_rng(k).uniform(size=4 * nbr)
    a, b = ref.lanczos(M, v0, k)
    o0, o1, t0, t1 = ref.ritz_bounds(a, b)
    e0, e1, th = cg.bounds(dev(M), k, v0=torch.as_tensor(v0, device=DEV))
    width = max(o1 - o0, abs(o0), abs(o1))
    tol = 1e-9 if k > 6 else 1e3 * 2.0 ** -53 * (k + 4 * (nbr // 2 + 12))
    assert abs(th[0] - t0) < tol * width and abs(th[1] - t1) < tol * width
    assert abs(e0 - o0) < 1e-6 * width and abs(e1 - o1) < 1e-6 * width
    # values on an 8-byte boundary only: the same sums
    assert cg.bounds(dev(M, 1), k, v0=torch.as_tensor(v0, device=DEV)) == (e0, e1, th)


def test_breakdown_at_the_first_step():
    nbr = 9
    M = ref.Bsr(np.arange(nbr + 1, dtype=np.int64), np.arange(nbr, dtype=np.int32),
                np.tile(2.5 * np.eye(4), (nbr, 1, 1)))
    a, b = ref.lanczos(M, np.ones(4 * nbr), 20)
    o0, o1, t0, t1 = ref.ritz_bounds(a, b)
    e0, e1, th = cg.bounds(dev(M), 20)
    assert abs(th[0] - 2.5) < 1e-14 * 100 and abs(th[1] - 2.5) < 1e-14 * 100
    assert abs(e0 - o0) < 1e-12 and abs(e1 - o1) < 1e-12
