"""Workspaces at any address: the header asks for no alignment of a call's workspace, so
bounds, coefficients and expansions on the column kernel give the same bits with one that
starts on an 8-byte boundary only, at exactly the size that the call asks for."""
import ctypes

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


def system():
    s = synth.make_system(80, 8.0, 3)
    S, H, P_out = pipelines.system_mats(s, 2.0)
    return ref.scale(H, -12.0, 12.0), P_out


def at(buf, shift):
    assert buf.data_ptr() % 256 == 0
    return ctypes.c_void_p(buf.data_ptr() + shift)


def p(t):
    return ctypes.c_void_p(t.data_ptr())


SHIFTS = (0, 8, 248)


def all_equal(results):
    return all(torch.equal(a, b) for r in results[1:] for a, b in zip(results[0], r))


def test_bounds():
    lib = cg._lib.load()
    M = dbsr(system()[0])
    nb, cb, res = ctypes.c_size_t(), M.c(), []
    cg._lib._check(lib.cheb_bounds_workspace_size(M.nbr, 12, ctypes.byref(nb)))
    for shift in SHIFTS:
        ws = torch.empty(nb.value + shift, dtype=torch.uint8, device=DEV)
        lo, hi, th = ctypes.c_double(), ctypes.c_double(), (ctypes.c_double * 2)()
        cg._lib._check(lib.cheb_bounds(ctypes.byref(cb), 12, None, 0.01, ctypes.byref(lo), ctypes.byref(hi), th,
                                       at(ws, shift), nb.value, cg._lib._stream()))
        res.append([torch.tensor([lo.value, hi.value, th[0], th[1]])])
    assert all_equal(res)


@pytest.mark.parametrize("tol", [0.0, 1e-7])
def test_coeffs(tol):
    lib = cg._lib.load()
    nb, res = ctypes.c_size_t(), []
    cg._lib._check(lib.cheb_coeffs_workspace_size(2, 600, ctypes.byref(nb)))
    f = cg._lib.make_funcs([{"kind": 0, "mu": 0.3, "kT": 0.1}, {"kind": 1, "mu": 0.1, "kT": 0.2}])
    for shift in SHIFTS:
        ws = torch.empty(nb.value + shift, dtype=torch.uint8, device=DEV)
        out, n = torch.zeros((2, 600), dtype=torch.float64, device=DEV), ctypes.c_int32()
        cg._lib._check(lib.cheb_coeffs(f, 2, -2.0, 2.5, tol, 0, 600, ctypes.byref(n), p(out), at(ws, shift), nb.value,
                                       cg._lib._stream()))
        res.append([out, torch.tensor([n.value])])
    assert all_equal(res)


@pytest.mark.parametrize("prec", [cg.F64, cg.F32])
@pytest.mark.parametrize("stepwise", [True, False])
def test_expansions_on_the_column_kernel(prec, stepwise):
    lib = cg._lib.load()
    Ht, P_out = system()
    plan = cg.Plan(dbsr(P_out, False), prec).attach_operator(dbsr(Ht))
    M = cg.Bsr(*plan._op_pattern, torch.as_tensor(Ht.vals, device=DEV))
    assert cg.plan_col_info(plan)[0] >= 1
    nb, cb, n, res = ctypes.c_size_t(), M.c(), 9, []
    if stepwise:
        cg._lib._check(lib.cheb_expand_stepwise_workspace_size(plan.handle, ctypes.byref(cb), prec, ctypes.byref(nb)))
    else:
        cg._lib._check(lib.cheb_expand_workspace_size(plan.handle, ctypes.byref(cb), prec, n, ctypes.byref(nb)))
    c = torch.linspace(1.0, 0.2, n, dtype=torch.float64, device=DEV)
    G = torch.ones((P_out.nnzb, 4, 4), dtype=torch.float64, device=DEV)
    for shift in SHIFTS:
        ws = torch.empty(nb.value + shift, dtype=torch.uint8, device=DEV)
        acc = torch.zeros((P_out.nnzb, 4, 4), dtype=torch.float64, device=DEV)
        t, g = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
        fn = lib.cheb_expand_stepwise if stepwise else lib.cheb_expand
        cg._lib._check(fn(plan.handle, ctypes.byref(cb), n, p(c), n, 1, (ctypes.c_void_p * 1)(acc.data_ptr()), p(t), p(G),
                          p(g), prec, at(ws, shift), nb.value, cg._lib._stream()))
        res.append([acc, t, g])
    assert all_equal(res)
