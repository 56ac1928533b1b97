"""The device list builder on the longest patterns: hundreds of thousands of block rows
still get the column kernel's lists, and the expansion on them agrees with the ranking
kernel's.  Bar: FP32 rounding of six terms of rows of three blocks."""
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [300_000, 660_000])
def test_lists_of_long_patterns(n):
    i = torch.arange(n, device=DEV)
    j = (i[:, None] + torch.tensor([-1, 0, 1], device=DEV)).reshape(-1)
    on = (j >= 0) & (j < n)
    ci = j[on].to(torch.int32)
    rp = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), on.reshape(n, 3).sum(1).cumsum(0)])
    g = torch.Generator(device=DEV).manual_seed(n)
    M = cg.Bsr(rp, ci, (torch.rand((ci.numel(), 4, 4), generator=g, dtype=torch.float64, device=DEV) - 0.5) / 6.0)
    plan = cg.Plan(cg.Bsr(rp, ci), cg.F32).attach_operator(M)
    assert cg.plan_col_info(plan)[0] == (n + 3) // 4
    c = torch.full((1, 6), 1.0, dtype=torch.float64, device=DEV)
    acc = [torch.zeros_like(M.vals) for _ in range(2)]
    cg.expand(plan, M, 6, c, acc[:1], precision=cg.F32, stepwise=True)
    cg.expand(cg.Plan(cg.Bsr(rp, ci), cg.F32), M, 6, c, acc[1:], precision=cg.F32, stepwise=True)
    assert (acc[0] - acc[1]).abs().max() <= 2 * 8 * 2.0 ** -24 * 6 ** 2
