"""Expansions whose spectrum leaves the interval: T_k grows until it is no longer finite.
The steps at and beyond that point cost about what the others do, the traces leave the
finite numbers where the ranking kernel's do, and up to there they agree with it."""
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


def system(n_atoms, reach):
    """H scaled so that its largest |eigenvalue| is reach."""
    s = synth.make_system(n_atoms, 8.0, 5)
    S, H, P_out = pipelines.system_mats(s, 3.0)
    half = np.abs(np.linalg.eigvalsh(synth.to_dense(H.row_ptr, H.col_idx, H.vals))).max() / reach
    return ref.scale(H, -half, half), P_out


def run(plan, M, n, G, prec):
    t, g = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
    acc = torch.zeros_like(G)
    c = torch.full((1, n), 2.0 ** -140, dtype=torch.float64, device=DEV)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    torch.cuda.synchronize()
    e[0].record()
    cg.expand(plan, M, n, c, [acc], moments=t, G=G, gmoments=g, precision=prec, stepwise=True)
    e[1].record()
    torch.cuda.synchronize()
    return t, g, acc, e[0].elapsed_time(e[1])


@pytest.mark.parametrize("prec,n", [(cg.F32, 400), (cg.BF16, 400), (cg.F64, 3000)])
def test_steps_beyond_the_finite_numbers_are_not_slower(prec, n):
    # (T_k grows by 1.56 a term: FP32 is left near term 200, FP64 near term 1,600)
    times = []
    for reach in (0.9, 1.1):
        Ht, P_out = system(250, reach)
        plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(Ht))
        assert cg.plan_col_info(plan)[0] >= 1
        M = cg.Bsr(*plan._op_pattern, torch.as_tensor(Ht.vals, device=DEV))
        G = torch.ones((P_out.nnzb, 4, 4), dtype=torch.float64, device=DEV)
        runs = [run(plan, M, n, G, prec) for _ in range(4)]
        times.append(min(r[3] for r in runs))
        finite = torch.isfinite(runs[0][0])
        assert bool(finite.all()) == (reach < 1.0) and torch.isfinite(runs[0][0][:60]).all()
    assert times[1] < 1.6 * times[0], times


@pytest.mark.parametrize("prec,reach", [(cg.F32, 1.1), (cg.F32, 8.0), (cg.BF16, 1.1), (cg.F64, 60.0)])
def test_overflow_agrees_with_the_ranking_kernel(prec, reach):
    Ht, P_out = system(100, reach)
    n = 260
    G = torch.rand((P_out.nnzb, 4, 4), dtype=torch.float64, device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(Ht))
    assert cg.plan_col_info(plan)[0] >= 1
    M = cg.Bsr(*plan._op_pattern, torch.as_tensor(Ht.vals, device=DEV))
    t, g, acc, _ = run(plan, M, n, G, prec)
    t2, g2, acc2, _ = run(cg.Plan(dbsr(P_out, False), prec), dbsr(Ht), n, G, prec)
    first = [int((~torch.isfinite(x)).nonzero()[0]) for x in (t, t2)]
    assert abs(first[0] - first[1]) <= 1
    m = min(first) - 1
    # every step's rounding grows like T_k itself: n u of the largest term so far, u of the stored T_k
    u = {cg.F32: 2.0 ** -24, cg.BF16: 2.0 ** -9, cg.F64: 2.0 ** -53}[prec]
    scale = torch.cummax(t2[:m].abs(), 0).values + 4 * P_out.nbr
    assert ((t[:m] - t2[:m]).abs() <= 64 * n * u * scale).all()
    assert not torch.isfinite(t[max(first) + 3:]).any() and not torch.isfinite(g[max(first) + 3:]).any()
    assert torch.equal(torch.isfinite(acc), torch.isfinite(acc2))
