"""FP64 masked products by digits (csrc/product.cu) against dense products: both left
patterns (the operator's and the output's), panels whose union fits and panels that
run column by column, groups of more quads than the exact sums hold, values beyond the
grids, several streams, and a captured call (which takes the FP64 pipe).

Bar: both sides sum K = 4 * (longest row) products, K u each of the largest product,
u = 2^-53, and the grids add less."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)

U = 2.0 ** -53


def band(n, width, order=None):
    """|i - j| <= width, rows and columns in the given order, as (row_ptr, col_idx, mask)."""
    i = np.arange(n) if order is None else np.asarray(order)
    on = np.abs(i[:, None] - i[None, :]) <= width
    rp = np.concatenate([[0], np.cumsum(on.sum(1))])
    return (torch.as_tensor(rp, dtype=torch.int64, device=DEV),
            torch.as_tensor(np.nonzero(on)[1], dtype=torch.int32, device=DEV), torch.as_tensor(on, device=DEV))


def pairs_apart(n, d):
    """An order in which columns 2k and 2k + 1 are d apart."""
    return [b + k + h * d for b in range(0, n, 2 * d) for k in range(d) for h in (0, 1) if b + k + h * d < n]


def dense(P, vals):
    rp, ci, on = P
    n = len(rp) - 1
    out = torch.zeros((n, n, 4, 4), dtype=torch.float64, device=DEV)
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    out[row, ci.long()] = vals
    return out.permute(0, 2, 1, 3).reshape(4 * n, 4 * n)


def blocks(P, D):
    rp, ci, on = P
    n = len(rp) - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    return D.reshape(n, 4, n, 4).permute(0, 2, 1, 3)[row, ci.long()]


def rand(P, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn((len(P[1]), 4, 4), generator=g, dtype=torch.float64, device=DEV)


def setup(n, w_op, w_out, order=None):
    L, P = band(n, w_op, order), band(n, w_out, order)
    plan = cg.Plan(cg.Bsr(P[0], P[1]), cg.F64).attach_operator(cg.Bsr(L[0], L[1]))
    assert cg.plan_col_info(plan)[0] >= 1
    return L, P, plan


def check(got, P, A, B, alpha, beta, D, K):
    want = alpha * blocks(P, A @ B) + (beta * D if D is not None else 0.0)
    bar = 2 * K * U * abs(alpha) * A.abs().max() * B.abs().max() + (2 * U * abs(beta) * D.abs().max() if D is not None else 0.0)
    assert (got - want).abs().max() <= bar


@pytest.mark.parametrize("n,w_op,w_out,order", [
    (50, 49, 49, None),                          # full rows, an odd half group
    (51, 50, 50, None),                          # an odd last column
    (203, 30, 47, None),
    (700, 30, 260, None),                        # rows near the longest that fit, more than 126 quads a group
    (900, 30, 255, pairs_apart(900, 90)),        # unions of two columns that do not fit
    (1300, 30, 285, None),                       # rows that do not fit: the FP64 pipe
])
def test_products_on_both_patterns(n, w_op, w_out, order):
    L, P, plan = setup(n, w_op, w_out, order)
    H, A, B, D = rand(L, 1), rand(P, 2), rand(P, 3), rand(P, 4)
    K = 4 * int((P[0][1:] - P[0][:-1]).max())
    C = torch.full_like(A, 9.0)
    cg.masked_product(plan, cg.Bsr(L[0], L[1], H), B, C)
    check(C, P, dense(L, H), dense(P, B), 1.0, 0.0, None, K)
    cg.masked_product(plan, cg.Bsr(P[0], P[1], A), B, C, alpha=-0.5, D=D, beta=1.5)
    check(C, P, dense(P, A), dense(P, B), -0.5, 1.5, D, K)
    C2 = torch.empty_like(C)
    cg.masked_product(plan, cg.Bsr(P[0], P[1], A), B, C2, alpha=-0.5, D=D, beta=1.5)
    assert torch.equal(C, C2)


@pytest.mark.parametrize("pa,pb", [(450, 0), (-430, 20), (0, 420), (3, -450)])
def test_values_beyond_the_grids(pa, pb):
    L, P, plan = setup(203, 30, 47)
    A, B = rand(P, 5), rand(P, 6)
    C = torch.empty_like(A)
    cg.masked_product(plan, cg.Bsr(P[0], P[1], A * 2.0 ** pa), B * 2.0 ** pb, C)
    check(C * 2.0 ** -(pa + pb), P, dense(P, A), dense(P, B), 1.0, 0.0, None, 4 * 95)


def test_what_is_not_finite_stays_where_it_belongs():
    L, P, plan = setup(203, 30, 47)
    A, B = rand(P, 5), rand(P, 6)
    B[int(P[0][100]) + 3, 2, 1] = float("inf")
    C = torch.empty_like(A)
    cg.masked_product(plan, cg.Bsr(P[0], P[1], A), B, C)
    bad = ~torch.isfinite(C).all(-1).all(-1)
    col = int(P[1][int(P[0][100]) + 3])
    assert bad.any() and (P[1][bad].long() == col).all()


def test_streams_share_the_digits_in_turn():
    L, P, plan = setup(203, 30, 47)
    A = [rand(P, 10 + i) for i in range(4)]
    want = []
    for i in range(4):
        C = torch.empty_like(A[0])
        cg.masked_product(plan, cg.Bsr(P[0], P[1], A[i]), A[(i + 1) % 4], C)
        want.append(C)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(4)]
    got = [[torch.empty_like(A[0]) for _ in range(5)] for _ in range(4)]
    torch.cuda.synchronize()
    for r in range(5):
        for i, st in enumerate(streams):
            cg.masked_product(plan, cg.Bsr(P[0], P[1], A[i]), A[(i + 1) % 4], got[i][r], stream=st)
    torch.cuda.synchronize()
    for i in range(4):
        for r in range(5):
            assert torch.equal(got[i][r], want[i])


def test_a_captured_product():
    L, P, plan = setup(203, 30, 47)
    A, B = rand(P, 5), rand(P, 6)
    C = torch.zeros_like(A)
    st = torch.cuda.Stream()
    Ab = cg.Bsr(P[0], P[1], A)
    with torch.cuda.stream(st):
        cg.masked_product(plan, Ab, B, C, stream=st)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            cg.masked_product(plan, Ab, B, C, stream=st)
    C.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    check(C, P, dense(P, A), dense(P, B), 1.0, 0.0, None, 4 * 95)
