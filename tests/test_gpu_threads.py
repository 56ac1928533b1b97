"""Two threads with plans of different shared-memory sizes on streams of their own: every
call succeeds and gives what it gives alone."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def full(n, seed):
    rp = torch.arange(n + 1, device=DEV) * n
    ci = torch.arange(n, dtype=torch.int32, device=DEV).repeat(n)
    g = torch.Generator(device=DEV).manual_seed(seed)
    return cg.Bsr(rp, ci, torch.randn((n * n, 4, 4), generator=g, dtype=torch.float64, device=DEV) / (8.0 * n ** 0.5))


def product(n):
    A = full(n, n)
    plan = cg.Plan(cg.Bsr(A.row_ptr, A.col_idx), cg.F64).attach_operator(A)
    outs = [torch.empty_like(A.vals) for _ in range(2)]

    def call(i, stream):
        cg.masked_product(plan, A, A.vals, outs[i], stream=stream)
        return outs[i]
    return call


def expansion(n, prec, listed, stepwise):
    A = full(n, n)
    plan = cg.Plan(cg.Bsr(A.row_ptr, A.col_idx), prec)
    if listed:
        plan.attach_operator(A)
    acc = [torch.empty_like(A.vals) for _ in range(2)]
    c = torch.ones((1, 3), dtype=torch.float64, device=DEV)
    ws = cg.expand(plan, A, 3, c, [acc[0]], precision=prec, stepwise=stepwise)

    def call(i, stream):
        cg.expand(plan, A, 3, c, [acc[i]], precision=prec, stepwise=stepwise, ws=ws, stream=stream)
        return acc[i]
    return call


@pytest.mark.parametrize("make", [
    product,
    lambda n: expansion(n, cg.F64, True, True),
    lambda n: expansion(n, cg.F32, True, True),
    lambda n: expansion(n, cg.F64, False, True),
    lambda n: expansion(n, cg.F32, False, False),
])
def test_two_plans_in_two_threads(make):
    calls = [make(64), make(71), make(80), make(72)]
    want = [call(0, None).clone() for call in calls]
    torch.cuda.synchronize()
    bad, start = [], threading.Barrier(len(calls))

    def work(call, ref):
        torch.cuda.set_device(DEV)
        st = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(1500):
                call(1, st)
            got = call(1, st)
            st.synchronize()
            if not torch.equal(got, ref):
                bad.append("result")
        except cg.ChebError as e:
            bad.append(str(e))

    th = [threading.Thread(target=work, args=a) for a in zip(calls, want)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert not bad, bad


def test_attaching_in_two_threads():
    ops = [full(n, n) for n in (64, 150, 96, 130)]
    bad, start = [], threading.Barrier(len(ops))

    def work(A, prec):
        torch.cuda.set_device(DEV)
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            try:
                for _ in range(40):
                    plan = cg.Plan(cg.Bsr(A.row_ptr, A.col_idx), prec).attach_operator(A)
                    assert cg.plan_col_info(plan)[0] >= 1
            except cg.ChebError as e:
                bad.append(str(e))

    th = [threading.Thread(target=work, args=(A, p)) for A, p in zip(ops, (cg.F32, cg.F64, cg.F64, cg.F32))]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert not bad, bad
