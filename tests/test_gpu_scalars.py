"""The scalar steps (csrc/coeffs.cu) at the sizes where their kernels can go wrong:
prime and odd transform lengths, odd node counts, fewer nodes than a thread block and
more than the registers keep, the edge of the penalty's cosine table, tolerances beside
a candidate's error.

u = 2^-53.  A transform or a weight sums n products, each known to a few u."""
import numpy as np
import pytest
import torch

from oracle import ref

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)

U = 2.0 ** -53


def moments_of_levels(x, n):
    """sum_j T_k(x_j), k < n."""
    return np.cos(np.arange(n)[:, None] * np.arccos(x)[None, :]).sum(1)


@pytest.mark.parametrize("n", [16, 17, 35, 64, 997, 2048, 2 * 1021, 4095])
def test_transform_lengths(n):
    e0, e1, kT = -1.7, 2.9, 0.11
    fs = [{"kind": 0, "mu": 0.3, "kT": kT}, {"kind": 1, "mu": -0.2, "kT": kT},
          {"kind": 3, "lo": -0.4, "hi": 0.5, "kT": kT}]
    _, c = cg.coeffs(fs, e0, e1, 0.0, n, device=DEV)
    for f, got in zip(fs, c.cpu().numpy()):
        want = ref.cheb_coeffs(ref.Func(f["kind"], mu=f.get("mu", 0.0), kT=kT, lo=f.get("lo", 0.0),
                                        hi=f.get("hi", 0.0)), n, e0, e1)
        # |f| <= 1, a node is known to 4 u max|x| and f' <= 1/kT
        bound = 2 * U * (n + 16) + 2 * 8 * U * max(abs(e0), abs(e1)) / kT
        assert np.max(np.abs(got - want)) < bound


@pytest.mark.parametrize("func,tol,rel,n_max", [
    ({"kind": 0, "mu": 0.2, "kT": 0.011}, 1e-9, False, 8192),   # beyond the first batch of candidates
    ({"kind": 2, "a": -0.5}, 1e-4, True, 100),                   # a small one, the largest not on the ladder
    ({"kind": 0, "mu": 0.2, "kT": 5.0}, 1e-3, False, 16),        # the smallest ladder
])
def test_degree_search_takes_the_ladder_entry_of_the_rule(func, tol, rel, n_max):
    e0, e1 = (0.1, 2.0) if func["kind"] == 2 else (-2.0, 2.5)
    n, _ = cg.coeffs([func], e0, e1, tol, n_max, rel=rel, device=DEV)
    f = ref.Func(func["kind"], mu=func.get("mu", 0.0), kT=func.get("kT", 0.0), a=func.get("a", 0.0))
    assert n == ref.choose_degree(f, e0, e1, tol, n_max, rel=rel)


@pytest.mark.parametrize("factor", [0.96, 1.04, 1.5])
@pytest.mark.parametrize("rel", [False, True])
def test_degree_search_near_the_tolerance(factor, rel):
    f = ref.Func(2, a=0.5) if rel else ref.Func(0, mu=0.2, kT=0.05)
    e0, e1 = (0.05, 3.0) if rel else (-2.0, 2.5)
    tol = factor * ref.max_fit_error(f, 56 if rel else 320, e0, e1, rel)
    n, _ = cg.coeffs([{"kind": f.kind, "mu": 0.2, "kT": 0.05, "a": 0.5}], e0, e1, tol, 1024, rel=rel, device=DEV)
    assert n == ref.choose_degree(f, e0, e1, tol, 1024, rel=rel)
    assert (n <= (56 if rel else 320)) == (factor > 1.0)


@pytest.mark.parametrize("n", [1, 2, 7, 31, 33, 300, 1024, 1025, 2100])
def test_penalty_sizes(n):
    rng = np.random.default_rng(n)
    t = rng.normal(size=n) / (1.0 + np.arange(n))
    alpha = -0.3 * n
    got = cg.penalty_trace(torch.as_tensor(t, device=DEV), n, alpha).item()
    # the penalty is at most 1; its argument alpha (x +- 1) is known to 4 u |alpha|
    want, scale = ref.penalty_trace(t, alpha, -1.0, 1.0), np.abs(t).sum()
    assert abs(got - want) <= 2 * U * (2 * n + 16 + 8 * abs(alpha)) * scale


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("n,max_iter", [(2, 100), (3, 100), (63, 100), (64, 4), (1025, 100), (4095, 100)])
def test_mu_search_sizes(kind, n, max_iter):
    rng = np.random.default_rng(7 * n + kind)
    e0, e1, kT = -3.0, 2.0, 0.06
    N_e = 41.3 if n > 3 else 50.0
    g = 2.0 * moments_of_levels(rng.uniform(-0.95, 0.95, 50), n) if n > 3 else np.array([100.0, 3.0, -7.0])[:n]
    want = ref.mu_bisect(g, kind, kT, e0, e1, N_e, 1e-7, max_iter=max_iter)
    res = cg.decode_mu_result(cg.mu_search(torch.as_tensor(g, device=DEV), n, e0, e1, kind, kT, N_e, 1e-7,
                                           max_iter=max_iter))
    assert res["converged"] == want.converged and res["iters"] == want.iters
    assert res["bits"] == want.bits and abs(res["mu"] - want.mu) <= 1e-15 * max(1.0, abs(want.mu))
    # N sums n occupations times weights, each weight (2/n) times a sum over g
    assert abs(res["N"] - want.counts[-1]) <= 2 * U * (2 * n + 16 + 8 * 3.0 / kT) * 2 * np.abs(g).sum()


def test_mu_search_with_more_nodes_than_the_registers_keep():
    n, e0, e1, kT = 16395, -1.0, 1.0, 0.02
    x = np.random.default_rng(3).uniform(-0.9, 0.9, 40)
    g = moments_of_levels(x, n)
    res = cg.decode_mu_result(cg.mu_search(torch.as_tensor(g, device=DEV), n, e0, e1, 0, kT, 17.2, 1e-7))
    # n is far beyond the degree that resolves kT: N(mu) is the levels' occupation itself
    N = np.sum(1.0 / (1.0 + np.exp((x - res["mu"]) / kT)))
    assert res["converged"] == 1 and abs(res["N"] - 17.2) <= 1e-7
    # the moments' angles k arccos(x) are known to n u / sqrt(1 - x^2), over sum_k |c_k| ~ 2 ln(1/kT)
    assert abs(res["N"] - N) <= 40 * U * (4 * n / np.sqrt(1 - 0.81)) * 2 * np.log(1 / kT) + 1e-12
