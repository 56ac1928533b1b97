"""Operators whose rows name a block column twice, or out of order: masked products add
every block, with and without attached lists.  Bar: as tests/test_gpu_product.py."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("builder", ["device", "host"])
@pytest.mark.parametrize("what", ["repeated", "descending"])
def test_products_add_every_block(what, builder):
    n = 60
    rng = np.random.default_rng(4)
    rows = [list(range(n)) for _ in range(n)]
    for i in range(n):
        if what == "repeated":
            rows[i] = sorted(rows[i] + [(7 * i) % n, (7 * i) % n, (11 * i + 3) % n])
        else:
            rows[i] = rows[i][::-1]
    rp = torch.as_tensor(np.concatenate([[0], np.cumsum([len(r) for r in rows])]), device=DEV)
    ci = torch.as_tensor(np.concatenate(rows).astype(np.int32), device=DEV)
    L = cg.Bsr(rp, ci, torch.as_tensor(rng.normal(size=(ci.numel(), 4, 4)), device=DEV))
    P = cg.Bsr(torch.arange(n + 1, device=DEV) * n, torch.arange(n, dtype=torch.int32, device=DEV).repeat(n))
    B = torch.as_tensor(rng.normal(size=(n * n, 4, 4)), device=DEV)
    A = torch.zeros((n, n, 4, 4), dtype=torch.float64, device=DEV)
    I = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    A.index_put_((I, ci.long()), L.vals, accumulate=True)
    want = torch.einsum("ikab,kjbc->ijac", A, B.view(n, n, 4, 4)).reshape(-1, 4, 4)
    bar = 2 * (4 * 63) * 2.0 ** -53 * L.vals.abs().max() * B.abs().max()
    for attach in (False, True):
        plan = cg.Plan(P, cg.F64)
        if attach:
            plan.attach_operator(L, gather=builder)
        C = torch.empty_like(B)
        cg.masked_product(plan, L, B, C)
        assert (C - want).abs().max() <= bar
