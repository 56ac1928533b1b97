"""Digit products (csrc/colstep.cu, csrc/product.cu) of operands whose rows and columns
have different scales: an operator element is held to 2^-60 (FP64) or 2^-30 (FP32) of its
scalar row's largest, a column's of its own, and a product column that the digits cannot
resolve is multiplied in FP64.

Bars, element by element: K products, each with both operands known to the working
precision u of their row's or column's largest element -- 4 K u max|row| max|column|; where
the scales of rows and columns cancel within a product, K u of the sum of |products|."""
import numpy as np
import pytest
import torch

import synth
from oracle import pipelines, ref

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)

SCALES = 2.0 ** -torch.tensor([0.0, 13.0, 27.0, 45.0], dtype=torch.float64)


def band(n, width):
    i = np.arange(n)
    on = np.abs(i[:, None] - i[None, :]) <= width
    rp = np.concatenate([[0], np.cumsum(on.sum(1))])
    return (torch.as_tensor(rp, dtype=torch.int64, device=DEV),
            torch.as_tensor(np.nonzero(on)[1], dtype=torch.int32, device=DEV))


def rows_of(P):
    return torch.repeat_interleave(torch.arange(len(P[0]) - 1, device=DEV), P[0][1:] - P[0][:-1])


def dense(P, vals):
    n = len(P[0]) - 1
    out = torch.zeros((n, n, 4, 4), dtype=torch.float64, device=DEV)
    out[rows_of(P), P[1].long()] = vals
    return out.permute(0, 2, 1, 3).reshape(4 * n, 4 * n)


def blocks(P, D):
    n = len(P[0]) - 1
    return D.reshape(n, 4, n, 4).permute(0, 2, 1, 3)[rows_of(P), P[1].long()]


def rand(P, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn((len(P[1]), 4, 4), generator=g, dtype=torch.float64, device=DEV)


def row_column_bar(A, B):
    return A.abs().amax(1)[:, None] * B.abs().amax(0)[None, :]


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_products_of_graded_rows_and_columns(shift):
    L, P = band(203, 30), band(203, 47)
    plan = cg.Plan(cg.Bsr(*P), cg.F64).attach_operator(cg.Bsr(*L))
    assert cg.plan_col_info(plan)[0] >= 1
    d = SCALES.roll(shift).to(DEV)
    for Q, A in ((L, rand(L, 1) * d[:, None]), (P, rand(P, 2) * d[:, None])):
        B = rand(P, 3) * d.flip(0)[None, :]
        C = torch.empty_like(B)
        cg.masked_product(plan, cg.Bsr(Q[0], Q[1], A), B, C)
        DA, DB = dense(Q, A), dense(P, B)
        bar = 4 * (4 * 95) * 2.0 ** -53 * row_column_bar(DA, DB)
        assert ((C - blocks(P, DA @ DB)).abs() <= blocks(P, bar)).all()


@pytest.mark.parametrize("width", [24, 60])
def test_products_whose_inner_scales_cancel(width):
    # the large elements of every row meet the small ones of every column
    L, P = band(181, 29), band(181, width)
    plan = cg.Plan(cg.Bsr(*P), cg.F64).attach_operator(cg.Bsr(*L))
    assert cg.plan_col_info(plan)[0] >= 1
    d = SCALES.to(DEV)
    for Q, A in ((L, rand(L, 1) / d[None, :]), (P, rand(P, 2) / d[None, :])):
        B = rand(P, 3) * d[:, None]
        B[:, :, 2] = 0.0  # (a zero column is exact by digits)
        C = torch.full_like(B, 9.0)
        cg.masked_product(plan, cg.Bsr(Q[0], Q[1], A), B, C)
        DA, DB = dense(Q, A), dense(P, B)
        bar = 2 * (4 * (2 * width + 1)) * 2.0 ** -53 * (DA.abs() @ DB.abs())
        assert ((C - blocks(P, DA @ DB)).abs() <= blocks(P, bar)).all()


@pytest.mark.parametrize("prec,u", [(cg.F64, 2.0 ** -53), (cg.F64X, 2.0 ** -48), (cg.F32, 2.0 ** -24)])
@pytest.mark.parametrize("stepwise", [True, False])
def test_expansions_of_an_operator_with_graded_rows(prec, u, stepwise):
    # T_2 = 2 M M - I alone, scalar rows of one block row 2^-45 apart
    s = synth.make_system(90, 8.0, 11)
    S, H, P_out = pipelines.system_mats(s, 3.0)
    Ht = ref.scale(H, -12.0, 12.0)
    vals = torch.as_tensor(Ht.vals, device=DEV) * SCALES.to(DEV)[:, None]
    Q = (torch.as_tensor(Ht.row_ptr, device=DEV), torch.as_tensor(Ht.col_idx, dtype=torch.int32, device=DEV))
    P = (torch.as_tensor(P_out.row_ptr, device=DEV), torch.as_tensor(P_out.col_idx, dtype=torch.int32, device=DEV))
    plan = cg.Plan(cg.Bsr(*P), prec).attach_operator(cg.Bsr(*Q))
    assert cg.plan_col_info(plan)[0] >= 1
    acc = torch.zeros((P_out.nnzb, 4, 4), dtype=torch.float64, device=DEV)
    c = torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device=DEV)
    cg.expand(plan, cg.Bsr(Q[0], Q[1], vals), 3, c, [acc], precision=prec, stepwise=stepwise)
    M = dense(Q, vals)
    want = blocks(P, 2.0 * M @ M) - blocks(P, torch.eye(M.shape[0], dtype=torch.float64, device=DEV))
    bar = blocks(P, 2 * 4 * (4 * 90) * u * row_column_bar(M, M)) + 2 * u * want.abs()
    assert ((acc - want).abs() <= bar).all()
