"""The column-order kernel's digit products (csrc/colstep.cu) where they can go
wrong: FP64 and FP64-accurate plans with long operator rows against the oracle and
against the per-step kernels, term counts around the accumulation groups and the
launch boundary, batches, and the plain path taken by values beyond the grid.

Bars: the perturbation bound of the recursion, 8 u sum_k |c_k| (k+1)^2 sqrt(elements),
u = 2^-53 or 2^-24; whole equality where the arithmetic is exact."""
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


def dbsr(M, vals=True):
    return cg.Bsr(torch.as_tensor(M.row_ptr, dtype=torch.int64, device=DEV),
                  torch.as_tensor(M.col_idx, dtype=torch.int32, device=DEV),
                  torch.as_tensor(np.ascontiguousarray(M.vals), dtype=torch.float64, device=DEV) if vals else None)


def system(n_atoms, r_c, r_buf, seed):
    s = synth.make_system(n_atoms, r_c, seed)
    S, H, P_out = pipelines.system_mats(s, r_buf)
    return ref.scale(H, -12.0, 12.0), P_out


def run(plan, dM, n, c, G, nnzb, prec, stepwise=True):
    acc = [torch.zeros((nnzb, 4, 4), dtype=torch.float64, device=DEV) for _ in range(len(c))]
    t, g = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
    cg.expand(plan, dM, n, torch.as_tensor(c, device=DEV) if len(c) else None, acc, moments=t,
              G=torch.as_tensor(G, device=DEV), gmoments=g, precision=prec, stepwise=stepwise)
    return [a.cpu().numpy() for a in acc], t.cpu().numpy(), g.cpu().numpy()


@pytest.mark.parametrize("prec", [cg.F64, cg.F64X, cg.F32])
@pytest.mark.parametrize("n_atoms,n,nf,stepwise", [
    (61, 3, 1, True),      # every row full, one step beyond the start
    (61, 4, 8, False),     # one whole accumulation group
    (150, 6, 2, True),     # a group and a rest
    (231, 99, 1, False),   # one term beyond the first launch's steps
    (230, 101, 3, True),   # ... and the next group's rest
    (640, 5, 1, True),     # more panels (FP64) than the launch order sorts
])
def test_digit_products_against_the_oracle(prec, n_atoms, n, nf, stepwise):
    Ht, P_out = system(n_atoms, 8.0, 3.0, 600 + n_atoms)
    rng = np.random.default_rng(n_atoms + n)
    c = rng.normal(size=(nf, n)) / (1.0 + np.arange(n)) ** 1.5
    G = rng.normal(size=(P_out.nnzb, 4, 4))
    ex = ref.chebyshev_expand(Ht, P_out, c, G=P_out.with_vals(G))
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(Ht))
    dM = cg.Bsr(*plan._op_pattern, torch.as_tensor(Ht.vals, device=DEV))
    assert cg.plan_col_info(plan)[0] >= 1
    acc, t, g = run(plan, dM, n, c, G, P_out.nnzb, prec, stepwise)
    u = 2.0 ** -24 if prec == cg.F32 else 2.0 ** -53
    k = np.arange(n)
    for j in range(nf):
        bound = 8 * u * np.sum(np.abs(c[j]) * (1 + k) ** 2) * np.sqrt(P_out.nnzb * 16)
        assert np.linalg.norm(acc[j] - ex.acc[j].vals) < bound
    grow = 8 * u * (1 + k) ** 2
    assert np.all(np.abs(t - ex.t) <= grow * 4 * P_out.nbr)
    assert np.all(np.abs(g - ex.g) <= grow * np.linalg.norm(G) * np.sqrt(4 * P_out.nbr))
    acc2, t2, g2 = run(plan, dM, n, c, G, P_out.nnzb, prec, not stepwise)
    for x, y in zip(acc + [t, g], acc2 + [t2, g2]):
        assert np.array_equal(x, y)  # both forms are the same kernel


@pytest.mark.parametrize("prec,power,n", [
    (cg.F32, 25, 6),    # T_4 leaves the grid's exponents
    (cg.F32, 40, 4), (cg.F32, -40, 4),    # the operator does
    (cg.F64, 300, 4), (cg.F64, 450, 3), (cg.F64, -420, 4),
])
def test_values_beyond_the_grid_take_the_plain_products(prec, power, n):
    # an operator scaled by 2^power; the result must stay a rounding of the oracle's
    Ht, P_out = system(80, 8.0, 2.0, 9)
    M = ref.Bsr(Ht.row_ptr, Ht.col_idx, np.ldexp(Ht.vals, power))
    c = np.ldexp(np.ones((1, n)), -np.arange(n) * max(power, 0))
    ex = ref.chebyshev_expand(M, P_out, c)
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(M))
    dM = cg.Bsr(*plan._op_pattern, torch.as_tensor(M.vals, device=DEV))
    assert cg.plan_col_info(plan)[0] >= 1
    acc, t, g = run(plan, dM, n, c, np.zeros((P_out.nnzb, 4, 4)), P_out.nnzb, prec)
    u = 2.0 ** -24 if prec == cg.F32 else 2.0 ** -53
    err = np.linalg.norm(acc[0] - ex.acc[0].vals) / np.linalg.norm(ex.acc[0].vals)
    assert err < 8 * u * n * n * 64  # (rows of up to 80 blocks summed in any order)


@pytest.mark.parametrize("prec", [cg.F64, cg.F32])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_elements_that_are_not_finite_stay_where_the_products_put_them(prec, value):
    Ht, P_out = system(90, 8.0, 2.0, 10)
    vals = Ht.vals.copy()
    vals[7, 1, 2] = value
    M = ref.Bsr(Ht.row_ptr, Ht.col_idx, vals)
    c = np.ones((1, 5))
    G = np.ones((P_out.nnzb, 4, 4))
    with np.errstate(invalid="ignore"):
        ex = ref.chebyshev_expand(M, P_out, c, G=P_out.with_vals(G))
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(M))
    dM = cg.Bsr(*plan._op_pattern, torch.as_tensor(vals, device=DEV))
    acc, t, g = run(plan, dM, 5, c, G, P_out.nnzb, prec)
    assert np.array_equal(np.isfinite(acc[0]), np.isfinite(ex.acc[0].vals))
    assert np.array_equal(np.isfinite(t), np.isfinite(ex.t))
    assert np.array_equal(np.isfinite(g), np.isfinite(ex.g))


@pytest.mark.parametrize("prec", [cg.F64, cg.F32, cg.BF16])
def test_zero_operator(prec):
    # T_k = I, 0, -I, 0, I: all digits zero in every other step
    Ht, P_out = system(70, 8.0, 2.0, 11)
    M = ref.Bsr(Ht.row_ptr, Ht.col_idx, np.zeros_like(Ht.vals))
    c = np.array([[0.5, 3.0, 1.0, 7.0, 2.0]])
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(M))
    dM = cg.Bsr(*plan._op_pattern, torch.as_tensor(M.vals, device=DEV))
    acc, t, g = run(plan, dM, 5, c, np.zeros((P_out.nnzb, 4, 4)), P_out.nnzb, prec)
    I = np.repeat(np.arange(P_out.nbr), np.diff(P_out.row_ptr))
    want = np.where((I == P_out.col_idx)[:, None, None], np.eye(4) * (0.25 - 1.0 + 2.0), 0.0)
    assert np.array_equal(acc[0], want)
    assert np.array_equal(t, 4.0 * P_out.nbr * np.array([1.0, 0.0, -1.0, 0.0, 1.0]))


@pytest.mark.parametrize("prec", [cg.F64, cg.F32])
def test_batch_through_the_lists_equals_the_systems_alone(prec):
    # the panels of a batch do not straddle systems and are those of the systems alone
    sizes, terms = (60, 101, 75), (99, 40, 5)
    parts = [system(n, 8.0, 2.0, 20 + n) for n in sizes]
    rng = np.random.default_rng(3)
    cs = [rng.normal(size=n) / (1.0 + np.arange(n)) for n in terms]
    Gs = [rng.normal(size=(P.nnzb, 4, 4)) for _, P in parts]
    bd = cg.block_diag([dbsr(M) for M, _ in parts])
    bo = cg.block_diag([dbsr(ref.Bsr(P.row_ptr, P.col_idx, np.zeros((P.nnzb, 4, 4)))) for _, P in parts], with_vals=False)
    starts = np.concatenate([[0], np.cumsum(sizes)]).tolist()
    plan = cg.BatchedPlan(bo, starts, prec).attach_operator(bd)
    assert cg.plan_col_info(plan)[0] >= 3
    k = max(terms)
    acc = torch.zeros((bo.nnzb, 4, 4), dtype=torch.float64, device=DEV)
    t, g = (torch.zeros((3, k), dtype=torch.float64, device=DEV) for _ in range(2))
    off = np.concatenate([[0], np.cumsum(terms)])[:-1]
    cg.expand_batched(plan, bd, k, torch.tensor(terms, dtype=torch.int32, device=DEV),
                      torch.as_tensor(np.concatenate(cs), device=DEV), torch.as_tensor(off, dtype=torch.int64, device=DEV),
                      0, [acc], moments=t, G=torch.as_tensor(np.concatenate(Gs), device=DEV), gmoments=g, moment_stride=k,
                      precision=prec)
    b0 = 0
    for i, ((M, P), n) in enumerate(zip(parts, terms)):
        one = cg.Plan(dbsr(P, False), prec).attach_operator(dbsr(M))
        dM = cg.Bsr(*one._op_pattern, torch.as_tensor(M.vals, device=DEV))
        a1, t1, g1 = run(one, dM, n, cs[i][None], Gs[i], P.nnzb, prec)
        assert np.array_equal(acc[b0:b0 + P.nnzb].cpu().numpy(), a1[0])
        assert np.array_equal(t[i, :n].cpu().numpy(), t1) and not t[i, n:].any()
        assert np.array_equal(g[i, :n].cpu().numpy(), g1) and not g[i, n:].any()
        b0 += P.nnzb


@pytest.mark.parametrize("n_atoms,sparse", [(61, False), (230, False), (230, True)])
def test_wide_lists_from_both_builders(n_atoms, sparse):
    Ht, P_out = system(n_atoms, 9.0, 2.0, 30)
    if sparse:  # rows of uneven length, some without a neighbour
        keep = np.flatnonzero((np.repeat(np.arange(Ht.nbr), np.diff(Ht.row_ptr)) * 7 + Ht.col_idx) % 5 < 3)
        rows = np.repeat(np.arange(Ht.nbr), np.diff(Ht.row_ptr))[keep]
        Ht = ref.Bsr(np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=Ht.nbr))]).astype(np.int64),
                     Ht.col_idx[keep], Ht.vals[keep])
    dP, dM = dbsr(P_out, False), dbsr(Ht)
    a = cg.Plan(dP, cg.F64).attach_operator(dM)
    b = cg.Plan(dP, cg.F64).attach_operator(dM, gather="host")
    assert cg.plan_col_info(a) == cg.plan_col_info(b) and cg.plan_col_info(a)[0] >= 1
    for x, y in zip(cg.plan_col_lists(a), cg.plan_col_lists(b)):
        assert torch.equal(x, y)
