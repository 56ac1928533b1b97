"""The longest columns that the column kernel's panels hold: 667 rows in FP32, 577 in FP64
(the next row longer gets no lists and runs on the ranking kernel), against dense products.
Bar: T_2 = 2 M M - I of K = 4 * rows products, 4 K u max|row| max|column|."""
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("prec,u,n,listed", [
    (cg.F32, 2.0 ** -24, 667, True), (cg.F32, 2.0 ** -24, 668, False),
    (cg.F64, 2.0 ** -53, 577, True), (cg.F64, 2.0 ** -53, 578, False),
])
def test_full_columns_at_the_capacity(prec, u, n, listed):
    # an output pattern of full columns, an operator of 61 blocks a row
    i = torch.arange(n, device=DEV)
    on = (i[:, None] - i[None, :]).abs() <= 30
    L = cg.Bsr(torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), on.sum(1).cumsum(0)]),
               on.nonzero()[:, 1].to(torch.int32))
    P = cg.Bsr(torch.arange(n + 1, device=DEV) * n, i.to(torch.int32).repeat(n))
    g = torch.Generator(device=DEV).manual_seed(n)
    vals = torch.randn((L.nnzb, 4, 4), generator=g, dtype=torch.float64, device=DEV) / 16.0
    plan = cg.Plan(P, prec).attach_operator(L)
    assert (cg.plan_col_info(plan)[0] >= 1) == listed
    acc = torch.zeros((P.nnzb, 4, 4), dtype=torch.float64, device=DEV)
    c = torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device=DEV)
    cg.expand(plan, L.with_vals(vals), 3, c, [acc], precision=prec, stepwise=True)
    M = torch.zeros((n, n, 4, 4), dtype=torch.float64, device=DEV)
    M[on] = vals
    M = M.permute(0, 2, 1, 3).reshape(4 * n, 4 * n)
    want = 2.0 * M @ M - torch.eye(4 * n, dtype=torch.float64, device=DEV)
    got = acc.view(n, n, 4, 4).permute(0, 2, 1, 3).reshape(4 * n, 4 * n)
    bar = 2 * 4 * (4 * 61) * u * M.abs().amax(1)[:, None] * M.abs().amax(0)[None, :] + 2 * u * want.abs()
    assert ((got - want).abs() <= bar).all()
