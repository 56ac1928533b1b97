"""<T_k, G> of FP32 expansions is summed in pairs of floats (csrc/colstep.cu), each update
exact to 1.5 * 2^-47 of the running sum: the second part is at most half a unit of the
first's last place before and after.

With M = J / 64 on 512 atoms (all 2,048 x 2,048 elements), T_2 = 2 M M - I = J - I exactly,
and with a constant G every lane adds the same 64 products, so the lanes' errors add up:
at most 1.5 * 2^-47 * (64 + 1) / 2 of the sum, plus 2^-44 for the sums of the lanes.  The
constant is one whose roundings go one way (found on the CPU: pairs that are not normalised
after each update lose 2^-40.6 of the sum)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("g", ["0x1.1d7d5f1ffde5bp+0", "0x1.1df7a07b72134p+0"])
def test_lanes_that_add_the_same_products(g):
    g, n = float.fromhex(g), 512
    rp = torch.arange(n + 1, device=DEV) * n
    ci = torch.arange(n, dtype=torch.int32, device=DEV).repeat(n)
    M = cg.Bsr(rp, ci, torch.full((n * n, 4, 4), 1.0 / 64.0, dtype=torch.float64, device=DEV))
    plan = cg.Plan(cg.Bsr(rp, ci), cg.F32).attach_operator(M)
    assert cg.plan_col_info(plan)[0] >= 1
    t, gm = (torch.zeros(3, dtype=torch.float64, device=DEV) for _ in range(2))
    G = torch.full((n * n, 4, 4), g, dtype=torch.float64, device=DEV)
    cg.expand(plan, M, 3, None, [], moments=t, G=G, gmoments=gm, precision=cg.F32, stepwise=True)
    assert t.tolist() == [4.0 * n, 4.0 * n / 64.0, 0.0]
    want = g * (4.0 * n) * (4.0 * n - 1)
    assert abs(gm[2].item() - want) <= (1.5 * 2.0 ** -47 * 32.5 + 2.0 ** -44) * want
