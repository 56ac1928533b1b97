"""Scalar steps at the sizes that their fast forms do not suit: a prime number of terms
takes no longer than twice a prime (about the same number of products), and a midpoint
of few nodes is summed without the barriers that one of many needs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


def device_ms(fn, reps=8):
    fn()
    best = float("inf")
    for _ in range(reps):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        fn()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("nf", [1, 4])
def test_prime_transforms(nf):
    # n (n1 + n2) products: n1 + n2 = 9974 / 2 + 2 against 9973 + 1 with half of them by symmetry
    fs = [{"kind": 0, "mu": 0.1 * f, "kT": 0.05} for f in range(nf)]
    t = {n: device_ms(lambda: cg.coeffs(fs, -2.0, 2.0, 0.0, n, device=DEV)) for n in (9973, 9974)}
    assert t[9973] <= 1.4 * t[9974], t


def test_mu_search_over_few_nodes():
    # (no count is within a negative tolerance: 128 midpoints each)
    t = {}
    for n in (16, 300):
        g = torch.as_tensor(2.0 * np.cos(np.arange(n)[:, None] * np.arccos(np.linspace(-0.9, 0.9, 50))[None]).sum(1), device=DEV)
        t[n] = device_ms(lambda: cg.mu_search(g, n, -1.0, 1.0, 0, 0.02, 41.3, -1.0, max_iter=128))
    assert t[16] <= 0.6 * t[300], t
