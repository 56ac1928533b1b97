"""The panels of the device builder (csrc/gather.cu: a span per column, then the chain of
starts) against the host builder's: more columns than one window of the chain, rows that
close panels early, the smallest patterns."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def pattern(n, far, seed):
    """Symmetric, the diagonal and far random partners a row."""
    rng = np.random.default_rng(seed)
    i = np.repeat(np.arange(n), far)
    j = rng.integers(0, n, size=n * far)
    key = np.unique(np.concatenate([np.arange(n) * (n + 1), i * n + j, j * n + i]))
    rp = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))])
    return cg.Bsr(torch.as_tensor(rp, dtype=torch.int64, device=DEV),
                  torch.as_tensor(key % n, dtype=torch.int32, device=DEV))


@pytest.mark.parametrize("prec", [cg.F32, cg.F64])
@pytest.mark.parametrize("n,far", [(1, 0), (2, 1), (5, 2), (700, 80), (1500, 150), (32768, 1), (33001, 2)])
def test_device_panels_equal_the_host_builders(prec, n, far):
    P = pattern(n, far, n + far)
    lists = []
    for builder in ("device", "host"):
        cg.set_plan_builder(builder)
        try:
            plan = cg.Plan(P, prec)
            lists.append([t.cpu() for t in cg.plan_lists(plan, (6, 7, 8, 9, 10))])
        finally:
            cg.set_plan_builder("device")
    assert all(torch.equal(a, b) for a, b in zip(*lists))
