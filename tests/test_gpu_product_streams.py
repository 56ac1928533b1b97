"""Masked products of one plan on several streams: small ones run side by side, as many as
the plan keeps digits for, and any number of streams, plans attached again in between and
calls that change streams give what a product gives alone."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def setup(n, op_width):
    i = torch.arange(n, device=DEV)
    P = cg.Bsr(torch.arange(n + 1, device=DEV) * n, i.to(torch.int32).repeat(n))
    plan = cg.Plan(P, cg.F64)
    attach(plan, n, op_width)
    g = torch.Generator(device=DEV).manual_seed(n)
    vals = [torch.randn((P.nnzb, 4, 4), generator=g, dtype=torch.float64, device=DEV) for _ in range(4)]
    return P, plan, vals


def attach(plan, n, op_width):
    i = torch.arange(n, device=DEV)
    on = (i[:, None] - i[None, :]).abs() <= op_width
    rp = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), on.sum(1).cumsum(0)])
    plan.attach_operator(cg.Bsr(rp, on.nonzero()[:, 1].to(torch.int32)))
    assert cg.plan_col_info(plan)[0] >= 1


def test_small_products_run_side_by_side():
    P, plan, vals = setup(100, 99)
    A = P.with_vals(vals[0])
    outs = [torch.empty_like(vals[1]) for _ in range(8)]
    streams = [torch.cuda.Stream() for _ in range(8)]

    def ms(many):
        best = float("inf")
        for _ in range(12):
            torch.cuda.synchronize()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record(streams[0])
            for s in streams[1:]:
                s.wait_event(e[0])
            for s, C in zip(streams, outs):
                cg.masked_product(plan, A, vals[1], C, stream=s if many else streams[0])
            for s in streams[1:]:
                streams[0].wait_stream(s)
            e[1].record(streams[0])
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    one, many = ms(False), ms(True)
    assert many <= 0.7 * one, (one, many)
    assert all(torch.equal(outs[0], C) for C in outs[1:])


@pytest.mark.parametrize("n,op_widths", [(64, (63, 45)), (150, (40, 149, 30))])
def test_any_number_of_streams(n, op_widths):
    P, plan, vals = setup(n, op_widths[0])
    want = []
    for k in range(4):
        C = torch.empty_like(vals[0])
        cg.masked_product(plan, P.with_vals(vals[k]), vals[(k + 1) % 4], C)
        want.append(C)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(19)]
    for width in op_widths:  # (another operator: another size and number of digits)
        attach(plan, n, width)
        torch.cuda.synchronize()
        got = [(k % 4, torch.empty_like(vals[0])) for k in range(57)]
        torch.cuda.synchronize()
        for i, (k, C) in enumerate(got):
            cg.masked_product(plan, P.with_vals(vals[k]), vals[(k + 1) % 4], C, stream=streams[(5 * i) % 19])
        torch.cuda.synchronize()
        assert all(torch.equal(C, want[k]) for k, C in got)
