"""The mu-proposal network's kernels (csrc/mlp.cu) at batch sizes around the four
samples of a block and the eight parts of the batch sums, against the oracle in FP64.

Bars: sums of at most 128 products in FP32 through three layers, 3 * 128 * 2^-24 =
2.3e-5 of the largest; batch sums add (batch / 8 + 8) 2^-24."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

cg = pytest.importorskip("paper_1704_00512_gb300")

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
if DEV is None:
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 7, 8, 9, 31, 65, 611])
def test_forward_and_backward_at_batch(B):
    rng = np.random.default_rng(B)
    th = (omlp.xavier_init(B).astype(np.float64) + rng.normal(size=omlp.N_PARAMS) * 0.01).astype(np.float32)
    X = (rng.normal(size=(B, omlp.N_IN)) * 0.5).astype(np.float32)
    out_o, cache = omlp.forward(th.astype(np.float64), X.astype(np.float64))
    dout = rng.normal(size=(B, 2)).astype(np.float32) / B
    g_o = omlp.backward(th.astype(np.float64), cache, dout.astype(np.float64))
    pad = 64  # untouched values beyond the buffers
    dth, dX = torch.as_tensor(th, device=DEV), torch.as_tensor(X, device=DEV)
    act, ws = (torch.full((B * 256 + pad,), 7.0, device=DEV) for _ in range(2))
    out, grad = torch.full((B * 2 + pad,), 7.0, device=DEV), torch.full((omlp.N_PARAMS + pad,), 7.0, device=DEV)
    cg.mlp_forward(dth, dX, act, out)
    got = out[: 2 * B].view(B, 2).cpu().numpy()
    bar = 3 * 128 * 2.0 ** -24
    assert np.max(np.abs(got - out_o)) < bar * max(1.0, np.max(np.abs(out_o)))
    cg.mlp_backward(dth, dX, act, torch.as_tensor(dout, device=DEV), grad, ws)
    gg = grad[: omlp.N_PARAMS].cpu().numpy()
    assert np.linalg.norm(gg - g_o) < (bar + (B / 8 + 8) * 2.0 ** -24) * np.linalg.norm(g_o)
    for t, n in ((act, 256 * B), (ws, 256 * B), (out, 2 * B), (grad, omlp.N_PARAMS)):
        assert torch.all(t[n:] == 7.0)
    grad2 = torch.empty_like(grad)
    cg.mlp_backward(dth, dX, act, torch.as_tensor(dout, device=DEV), grad2, ws)
    assert torch.equal(grad[: omlp.N_PARAMS], grad2[: omlp.N_PARAMS])
