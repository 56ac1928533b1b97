"""What users of this framework have it do, as cases that can be timed and checked.

Every case goes through the public entry points (paper_1704_00512_gb300 and its
solve module).  Systems are atom-centred: four s-type Gaussians per atom at the
density of 200 atoms per (18 bohr)^3, the overlap S, the Hamiltonian H and the
block patterns of a cutoff r_c (operator) and r_c + r_buf (output), the sizes
and cutoffs of the benchmark's and the tests' configurations.

Kinds:
  expand    the recursion of a density-matrix pass: the scaled operator, an
            expansion with nf accumulators, Tr T_k and <T_k, G>.  A program that
            asks for FP32 (BF16) products keeps their results as float32
            (bfloat16): the containers the library writes are FP64, the values
            have the precision of the products.
  powers    S^-1, S^1/2, S^-1/2 from one recursion (solve.powers).
  foe       one whole density-matrix solve (solve.foe, two-pass form).
  batched   many uneven systems in one batched expansion.
  products  the masked products of a solve: H' = P_H(A P_out(H A)) and
            F = P_out(A P_out(p A)).
  scalars   what a solve does between its passes: the penalty check, the mu
            bisection, the degree search and the coefficients at several mu.
  bounds    Lanczos bounds of a Hamiltonian.
  mlp       one training step of the mu-proposal network.
"""
import math

import numpy as np
import torch

import paper_1704_00512_gb300 as cg
from paper_1704_00512_gb300 import solve

DEV = "cuda"
EXPS = (0.6, 2.4, 9.6, 38.4)
PREC = {"f64": cg.F64, "f32": cg.F32, "bf16": cg.BF16, "f64x": cg.F64X}
KEEP = {"f64": torch.float64, "f64x": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the accumulation pass of the 40,000-row mixed-precision density matrix (a stretch of its steps)
        dict(name="expand_f32_40k", kind="expand", prec="f32", n_atoms=10000, r_c=10.0, r_buf=4.0, n_terms=48, nf=1,
             order="hilbert"),
        # the accumulation pass with four chemical potentials at once, 12,000 rows
        dict(name="expand_f32_12k_mu4", kind="expand", prec="f32", n_atoms=3000, r_c=10.0, r_buf=4.0, n_terms=96, nf=4,
             order="hilbert"),
        # a system that fills the GPU about once, in the caller's atom order
        dict(name="expand_f32_4k", kind="expand", prec="f32", n_atoms=1000, r_c=8.0, r_buf=4.0, n_terms=64, nf=1,
             order="none"),
        # the BF16 product mode on a small, odd-sized system, two accumulators
        dict(name="expand_bf16_2k", kind="expand", prec="bf16", n_atoms=501, r_c=8.0, r_buf=4.0, n_terms=48, nf=2,
             order="none"),
        # the matrix powers of the 12,000-row benchmark at half its size, FP64
        dict(name="powers_f64_6k", kind="powers", prec="f64", n_atoms=1500, r_c=10.0, r_buf=4.0, n_terms=72),
        # the same with FP64-accurate products on the FP32 pipe; the size where one launch runs all steps
        dict(name="powers_f64x_4k", kind="powers", prec="f64x", n_atoms=1000, r_c=8.0, r_buf=4.0, n_terms=64),
        # one whole FP64 solve of the 800-row configuration, at a smearing for geometry optimisation
        dict(name="foe_f64_800", kind="foe", prec="f64", n_atoms=200, r_c=8.0, r_buf=4.0, kT=0.05),
        # a batch of uneven independent systems, FP32 products
        dict(name="batched_f32", kind="batched", prec="f32", n_sys=16, atoms_lo=125, atoms_hi=500, r_c=8.0, r_buf=4.0,
             n_terms=64),
        # orthogonalisation and post-processing around the passes, FP64
        dict(name="products_f64_6k", kind="products", n_atoms=1500, r_c=10.0, r_buf=4.0),
        # the scalar steps between the passes at the 40,000-row solve's degree
        dict(name="scalars_9216", kind="scalars", n_terms=9216, n_mu=4, kT=0.005, n_max=16384),
        # Lanczos bounds of a 20,000-row Hamiltonian, 40 steps
        dict(name="bounds_20k", kind="bounds", n_atoms=5000, r_c=10.0, steps=40),
        # the smallest calls: one training step of the mu proposal on its own training-set size
        dict(name="mlp_step", kind="mlp", batch=346),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("expand", "expand", "expand", "powers", "foe", "batched", "products", "scalars", "bounds", "mlp"))
    if kind == "expand":
        prec = rng.choice(("f32", "f32", "f32", "bf16", "f64", "f64x"))
        hi = {"f32": 8000, "bf16": 800, "f64": 1500, "f64x": 1500}[prec]
        return dict(kind=kind, prec=prec, n_atoms=_log_int(rng, 150, hi), r_c=rng.choice((8.0, 10.0)), r_buf=4.0,
                    n_terms=rng.randint(20, 44), nf=rng.randint(0, 4) if prec != "bf16" else rng.randint(1, 4),
                    order=rng.choice(("hilbert", "none")))
    if kind == "powers":
        return dict(kind=kind, prec=rng.choice(("f64", "f64x")), n_atoms=_log_int(rng, 150, 1400),
                    r_c=rng.choice((8.0, 10.0)), r_buf=4.0, n_terms=rng.randint(32, 64))
    if kind == "foe":
        return dict(kind=kind, prec="f64", n_atoms=rng.randint(60, 180), r_c=round(rng.uniform(4.0, 5.5), 2),
                    r_buf=round(rng.uniform(1.5, 3.0), 2), kT=round(rng.uniform(0.05, 0.1), 3))
    if kind == "batched":
        return dict(kind=kind, prec=rng.choice(("f32", "f32", "f64")), n_sys=rng.randint(3, 14), atoms_lo=125,
                    atoms_hi=rng.randint(160, 500), r_c=8.0, r_buf=4.0, n_terms=rng.randint(24, 64))
    if kind == "products":
        return dict(kind=kind, n_atoms=_log_int(rng, 150, 1500), r_c=rng.choice((8.0, 10.0)), r_buf=4.0)
    if kind == "scalars":
        n = _log_int(rng, 300, 9216)  # (the degree follows the smearing)
        return dict(kind=kind, n_terms=n, n_mu=rng.randint(1, 8), kT=round(46.0 / n * rng.uniform(1.0, 1.5), 5), n_max=16384)
    if kind == "bounds":
        return dict(kind=kind, n_atoms=_log_int(rng, 200, 5000), r_c=rng.choice((8.0, 10.0)), steps=rng.randint(8, 60))
    return dict(kind=kind, batch=_log_int(rng, 1, 2000))


# ---------------------------------------------------------------------------
# synthetic systems (torch only)

def _box(n):
    return 18.0 * (n / 200.0) ** (1.0 / 3.0)


def _atoms(n, dev, which=0):
    """n atoms on randomly chosen cells of a grid, displaced within them, in Morton order.

    One geometry for every seed (a self-consistent loop, or one geometry with
    several bases): the seed gives the values on its patterns."""
    g = torch.Generator().manual_seed(which * 7919 + n)
    L, m = _box(n), math.ceil(round(n ** (1.0 / 3.0), 9))
    cell = torch.randperm(m ** 3, generator=g)[:n]
    ijk = torch.stack((cell // (m * m), cell // m % m, cell % m), 1)
    xyz = (ijk.double() + 0.5 + 0.4 * (torch.rand((n, 3), generator=g, dtype=torch.float64) - 0.5)) * (L / m)
    q = (xyz / L * 1024).long().clamp_(0, 1023)
    key = torch.zeros(n, dtype=torch.int64)
    for b in range(10):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return xyz[torch.argsort(key)].contiguous().to(dev), L


def _delta(xyz, L, I, J):
    d = xyz[J] - xyz[I]
    return d - L * torch.round(d / L)


def _mix(x):
    x = (x ^ ((x >> 31) & 0x1FFFFFFFF)) * 0x7FB5D329728EA185
    x = (x ^ ((x >> 27) & 0x1FFFFFFFFF)) * -0x7E25210B43D22BB3
    return x ^ ((x >> 33) & 0x7FFFFFFF)


def _overlap(xyz, L, I, J, seed):
    u = np.random.default_rng([int(seed), 3]).random(4)
    a = torch.tensor([e * (1.0 + 0.1 * x) for e, x in zip(EXPS, u)], dtype=torch.float64, device=xyz.device)
    pref = (2.0 * torch.sqrt(a[:, None] * a[None, :]) / (a[:, None] + a[None, :])) ** 1.5
    red = a[:, None] * a[None, :] / (a[:, None] + a[None, :])
    r2 = _delta(xyz, L, I, J).square().sum(1)
    return pref * torch.exp(-red * r2[:, None, None])


def _hamiltonian(S, I, J, seed):
    """H = -S/2 (1 + 0.1 z) with z(i, j) = z(j, i) normal; diagonal elements uniform in [-1.2, 0.3]."""
    r = torch.arange(4, device=S.device)
    i = (4 * I)[:, None, None] + r[:, None]
    j = (4 * J)[:, None, None] + r[None, :]
    h = _mix((torch.minimum(i, j) << 32) ^ torch.maximum(i, j) ^ (int(seed) * 1000003))
    h2 = _mix(h)
    u1 = ((h & 0x7FFFFFFF).double() + 0.5) / 2147483648.0
    u2 = (h2 & 0x7FFFFFFF).double() / 2147483648.0
    H = -0.5 * S * (1.0 + 0.1 * torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2))
    on_site = (I == J)[:, None, None]
    H = torch.where(on_site & (i != j), torch.zeros_like(H), H)
    return torch.where(on_site & (i == j), -1.2 + 1.5 * u2, H)


def _gershgorin(v, I, J, n):
    """An interval that holds the spectrum: centres and radii of the scalar rows."""
    on = (I == J)[:, None, None] & torch.eye(4, dtype=torch.bool, device=v.device)
    rad = torch.zeros((n, 4), dtype=torch.float64, device=v.device)
    rad.index_add_(0, I, torch.where(on, torch.zeros_like(v), v).abs().sum(2))
    dia = torch.zeros((n, 4), dtype=torch.float64, device=v.device)
    dia.index_add_(0, I, torch.where(on, v, torch.zeros_like(v)).sum(2))
    # (outward to a grid, so that the order of the sums above does not show)
    return math.floor((dia - rad).min().item() * 4096) / 4096, math.ceil((dia + rad).max().item() * 4096) / 4096


def _pattern(xyz, L, r):
    rp, ci = cg.pattern_build(xyz, L, r)
    I = torch.repeat_interleave(torch.arange(xyz.shape[0], device=xyz.device), rp[1:] - rp[:-1])
    return cg.Bsr(rp, ci), I, ci.long()


def _near(xyz, L, r):
    """The block pattern by plain distances: (I, J) in row order, and a dense mask of elements."""
    d = xyz[None, :, :] - xyz[:, None, :]
    d = d - L * torch.round(d / L)
    m = d.square().sum(2) <= r * r
    I, J = torch.nonzero(m, as_tuple=True)
    return I, J, m


def _dense(I, J, v, n):
    A = torch.zeros((n, n, 4, 4), dtype=torch.float64, device=v.device)
    A[I, J] = v
    return A.permute(0, 2, 1, 3).reshape(4 * n, 4 * n)


def _blocks(A, I, J):
    n = A.shape[0] // 4
    return A.view(n, 4, n, 4).permute(0, 2, 1, 3)[I, J]


def _ordered(xyz, L, order):
    if order != "hilbert":
        return xyz
    perm = cg._lib.locality_order(xyz, L)
    return cg._lib.gather_rows(xyz.reshape(-1), perm, 3).view(-1, 3)


def _fermi_funcs(c, e0, e1):
    """Fermi functions around the middle of the interval, one per accumulator."""
    kT = 0.02 * (e1 - e0)
    return [{"kind": cg.FERMI, "mu": e0 + (0.40 + 0.05 * f) * (e1 - e0), "kT": kT} for f in range(c["nf"])]


# ---------------------------------------------------------------------------

def _prep_expand(c, seed):
    prec = PREC[c["prec"]]
    xyz, L = _atoms(c["n_atoms"], DEV)
    xyz = _ordered(xyz, L, c["order"])
    PH, I, J = _pattern(xyz, L, c["r_c"])
    PO, IO, JO = _pattern(xyz, L, c["r_c"] + c["r_buf"])
    H = _hamiltonian(_overlap(xyz, L, I, J, seed), I, J, seed)
    e0, e1 = _gershgorin(H, I, J, c["n_atoms"])
    Ht = PH.with_vals(cg.scale(PH.with_vals(H), e0, e1))
    plan = cg.Plan(PO, prec).attach_operator(PH)
    n = c["n_terms"]
    coef = cg.coeffs(_fermi_funcs(c, e0, e1), e0, e1, 0.0, n, device=DEV)[1] if c["nf"] else None
    acc = [torch.zeros((PO.nnzb, 4, 4), dtype=torch.float64, device=DEV) for _ in range(c["nf"])]
    t, g = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
    return dict(c=c, plan=plan, Ht=Ht, n=n, coef=coef, acc=acc, t=t, g=g, G=_overlap(xyz, L, IO, JO, seed), prec=prec, ws=None)


def _run_expand(s):
    s["ws"] = cg.expand(s["plan"], s["Ht"], s["n"], s["coef"], s["acc"], moments=s["t"], G=s["G"], gmoments=s["g"],
                        precision=s["prec"], ws=s["ws"], stepwise=True)
    keep = KEEP[s["c"]["prec"]]
    return {"acc": [a.to(keep) for a in s["acc"]], "t": s["t"].to(keep), "g": s["g"].to(keep)}


def _dct(f, n):
    """Chebyshev coefficients of f on [-1, 1] at n nodes."""
    k = torch.arange(n, dtype=torch.float64)
    x = torch.cos(math.pi * (k + 0.5) / n)
    v = f(x)
    out = torch.empty(n, dtype=torch.float64)
    for j0 in range(0, n, 512):
        j = torch.arange(j0, min(n, j0 + 512))
        ang = (j[:, None] * (2 * torch.arange(n) + 1)[None, :]) % (4 * n)
        out[j0:j0 + 512] = (2.0 / n) * (torch.cos(math.pi * ang.double() / (2.0 * n)) @ v)
    return out


def _recursion(M, mask, n, coefs, G=None):
    """The truncated recursion on dense matrices."""
    dev, N = M.device, M.shape[0]
    Tm, T = torch.eye(N, dtype=torch.float64, device=dev), M.clone()
    acc = [0.5 * c[0] * Tm + c[1] * T for c in coefs]
    t, g = [Tm.trace(), T.trace()], [] if G is None else [(Tm * G).sum(), (T * G).sum()]
    for k in range(2, n):
        Tn = torch.matmul(M, T).mul_(2.0).mul_(mask).sub_(Tm)
        Tm, T = T, Tn
        for a, c in zip(acc, coefs):
            a.add_(T, alpha=float(c[k]))
        t.append(T.trace())
        if G is not None:
            g.append((T * G).sum())
    return acc, torch.stack(t), torch.stack(g) if g else None


def _exact_device():
    return DEV if torch.cuda.is_available() else "cpu"


def _fermi(x, mu, kT):
    return 1.0 / (1.0 + torch.exp((x - mu) / kT))


def _exact_expand(c, seed):
    if c["n_atoms"] > 1100 or c["order"] == "hilbert":
        return None
    n = c["n_atoms"]
    xyz, L = _atoms(n, _exact_device())
    I, J, _ = _near(xyz, L, c["r_c"])
    IO, JO, mO = _near(xyz, L, c["r_c"] + c["r_buf"])
    H = _hamiltonian(_overlap(xyz, L, I, J, seed), I, J, seed)
    e0, e1 = _gershgorin(H, I, J, n)
    sig, tau = 2.0 / (e1 - e0), 0.5 * (e0 + e1)
    M = sig * (_dense(I, J, H, n) - tau * torch.eye(4 * n, dtype=torch.float64, device=H.device))
    mask = mO.double().repeat_interleave(4, 0).repeat_interleave(4, 1)
    coefs = [_dct(lambda x: _fermi(x / sig + tau, f["mu"], f["kT"]), c["n_terms"]) for f in _fermi_funcs(c, e0, e1)]
    G = _dense(IO, JO, _overlap(xyz, L, IO, JO, seed), n)
    acc, t, g = _recursion(M, mask, c["n_terms"], coefs, G)
    return {"acc": [_blocks(a, IO, JO) for a in acc], "t": t, "g": g}


# ---------------------------------------------------------------------------

EXPONENTS = (-1.0, 0.5, -0.5)


def _problem(c, seed, prec):
    xyz, L = _atoms(c["n_atoms"], DEV)
    _, I, J = _pattern(xyz, L, c["r_c"])
    S = _overlap(xyz, L, I, J, seed)
    H = _hamiltonian(S, I, J, seed)
    pb = solve.Problem(xyz.cpu().numpy(), L, c["r_c"], c["r_buf"], S.cpu().numpy(), H.cpu().numpy(), DEV, prec)
    return pb, xyz, L


def _powers_bounds(S, I, J, n):
    return 0.05, _gershgorin(S, I, J, n)[1]  # (a lower bound kept from an earlier geometry)


def _prep_powers(c, seed):
    pb, xyz, L = _problem(c, seed, PREC[c["prec"]])
    I = torch.repeat_interleave(torch.arange(c["n_atoms"], device=DEV), pb.S.row_ptr[1:] - pb.S.row_ptr[:-1])
    return dict(c=c, pb=pb, b=_powers_bounds(pb.S.vals, I, pb.S.col_idx.long(), c["n_atoms"]), prec=PREC[c["prec"]])


def _run_powers(s):
    r = solve.powers(s["pb"], EXPONENTS, bounds_S=s["b"], n_terms=s["c"]["n_terms"], precision=s["prec"])
    return {"acc": r["acc"], "moments": r["moments"]}


def _exact_powers(c, seed):
    n = c["n_atoms"]
    if n > 1100:
        return None
    xyz, L = _atoms(n, _exact_device())
    I, J, _ = _near(xyz, L, c["r_c"])
    IO, JO, mO = _near(xyz, L, c["r_c"] + c["r_buf"])
    S = _overlap(xyz, L, I, J, seed)
    e0, e1 = _powers_bounds(S, I, J, n)
    sig, tau = 2.0 / (e1 - e0), 0.5 * (e0 + e1)
    M = sig * (_dense(I, J, S, n) - tau * torch.eye(4 * n, dtype=torch.float64, device=S.device))
    mask = mO.double().repeat_interleave(4, 0).repeat_interleave(4, 1)
    coefs = [_dct(lambda x: (x / sig + tau) ** a, c["n_terms"]) for a in EXPONENTS]
    acc, t, _ = _recursion(M, mask, c["n_terms"], coefs)
    return {"acc": [_blocks(a, IO, JO) for a in acc], "moments": t}


# ---------------------------------------------------------------------------

def _prep_foe(c, seed):
    pb, _, _ = _problem(c, seed, PREC[c["prec"]])
    return dict(c=c, pb=pb)


def _run_foe(s):
    r = solve.foe(s["pb"], s["c"]["kT"], 2.0 * s["c"]["n_atoms"], tol=1e-9)
    return {"F": r["F"], "p": r["p"], "mu": r["mu"], "trace_FS": r["trace_FS"], "n_terms": r["n_terms"]}


# ---------------------------------------------------------------------------

def _batch_sizes(c):
    g = np.random.default_rng([c["n_sys"], c["atoms_hi"]])
    atoms = g.integers(c["atoms_lo"], c["atoms_hi"] + 1, c["n_sys"])
    terms = g.integers(max(2, c["n_terms"] // 2), c["n_terms"] + 1, c["n_sys"])
    terms[0] = c["n_terms"]
    return atoms.tolist(), terms.tolist()


def _batch_func(e0, e1):
    return {"kind": cg.FERMI, "mu": e0 + 0.45 * (e1 - e0), "kT": 0.02 * (e1 - e0)}


def _prep_batched(c, seed):
    prec = PREC[c["prec"]]
    atoms, terms = _batch_sizes(c)
    Hs, POs, Gs, cs, offs = [], [], [], [], [0]
    for i, (n, m) in enumerate(zip(atoms, terms)):
        xyz, L = _atoms(n, DEV, i)
        PH, I, J = _pattern(xyz, L, c["r_c"])
        PO, IO, JO = _pattern(xyz, L, c["r_c"] + c["r_buf"])
        H = _hamiltonian(_overlap(xyz, L, I, J, seed), I, J, int(seed) + i)
        e0, e1 = _gershgorin(H, I, J, n)
        Hs.append(PH.with_vals(cg.scale(PH.with_vals(H), e0, e1)))
        POs.append(PO)
        Gs.append(_overlap(xyz, L, IO, JO, seed))
        cs.append(cg.coeffs([_batch_func(e0, e1)], e0, e1, 0.0, max(16, m), device=DEV)[1].reshape(-1))
        offs.append(offs[-1] + max(16, m))
    Ht = cg.block_diag(Hs)
    PO = cg.block_diag(POs, with_vals=False)
    starts = np.concatenate([[0], np.cumsum(atoms)]).tolist()
    plan = cg.BatchedPlan(PO, starts, prec).attach_operator(cg.Bsr(Ht.row_ptr, Ht.col_idx))
    k = max(terms)
    return dict(c=c, plan=plan, Ht=Ht, k=k, nt=torch.tensor(terms, dtype=torch.int32, device=DEV), coef=torch.cat(cs),
                off=torch.tensor(offs[:-1], dtype=torch.int64, device=DEV), G=torch.cat(Gs), prec=prec, ws=None,
                acc=torch.zeros((PO.nnzb, 4, 4), dtype=torch.float64, device=DEV),
                t=torch.zeros((c["n_sys"], k), dtype=torch.float64, device=DEV),
                g=torch.zeros((c["n_sys"], k), dtype=torch.float64, device=DEV))


def _run_batched(s):
    s["ws"] = cg.expand_batched(s["plan"], s["Ht"], s["k"], s["nt"], s["coef"], s["off"], 0, [s["acc"]], moments=s["t"],
                                G=s["G"], gmoments=s["g"], moment_stride=s["k"], precision=s["prec"], ws=s["ws"])
    keep = KEEP[s["c"]["prec"]]
    return {"acc": s["acc"].to(keep), "t": s["t"].to(keep), "g": s["g"].to(keep)}


def _exact_batched(c, seed):
    atoms, terms = _batch_sizes(c)
    accs, ts, gs, k = [], [], [], max(terms)
    dev = _exact_device()
    for i, (n, m) in enumerate(zip(atoms, terms)):
        xyz, L = _atoms(n, dev, i)
        I, J, _ = _near(xyz, L, c["r_c"])
        IO, JO, mO = _near(xyz, L, c["r_c"] + c["r_buf"])
        H = _hamiltonian(_overlap(xyz, L, I, J, seed), I, J, int(seed) + i)
        e0, e1 = _gershgorin(H, I, J, n)
        sig, tau = 2.0 / (e1 - e0), 0.5 * (e0 + e1)
        M = sig * (_dense(I, J, H, n) - tau * torch.eye(4 * n, dtype=torch.float64, device=dev))
        mask = mO.double().repeat_interleave(4, 0).repeat_interleave(4, 1)
        f = _batch_func(e0, e1)
        coef = _dct(lambda x: _fermi(x / sig + tau, f["mu"], f["kT"]), max(16, m))
        acc, t, g = _recursion(M, mask, m, [coef], _dense(IO, JO, _overlap(xyz, L, IO, JO, seed), n))
        accs.append(_blocks(acc[0], IO, JO))
        ts.append(torch.nn.functional.pad(t, (0, k - m)))
        gs.append(torch.nn.functional.pad(g, (0, k - m)))
    return {"acc": torch.cat(accs), "t": torch.stack(ts), "g": torch.stack(gs)}


# ---------------------------------------------------------------------------

def _near_identity(S, I, J, a):
    on = ((I == J)[:, None, None] & torch.eye(4, dtype=torch.bool, device=S.device)).double()
    return on + a * (S - on)


def _prep_products(c, seed):
    pb, xyz, L = _problem(c, seed, cg.F64)
    IO = torch.repeat_interleave(torch.arange(c["n_atoms"], device=DEV), pb.P_out.row_ptr[1:] - pb.P_out.row_ptr[:-1])
    S = _overlap(xyz, L, IO, pb.P_out.col_idx.long(), seed)
    JO = pb.P_out.col_idx.long()
    return dict(pb=pb, A=_near_identity(S, IO, JO, -0.4), p=_near_identity(S, IO, JO, 0.3))


def _run_products(s):
    Hp = solve.orthogonalise(s["pb"], s["A"])
    return {"Hp": Hp.vals, "F": solve.postprocess(s["pb"], s["A"], s["p"])}


def _exact_products(c, seed):
    n = c["n_atoms"]
    xyz, L = _atoms(n, _exact_device())
    I, J, mH = _near(xyz, L, c["r_c"])
    IO, JO, mO = _near(xyz, L, c["r_c"] + c["r_buf"])
    Sc = _overlap(xyz, L, I, J, seed)
    H = _dense(I, J, _hamiltonian(Sc, I, J, seed), n)
    S = _overlap(xyz, L, IO, JO, seed)
    A, p = (_dense(IO, JO, _near_identity(S, IO, JO, a), n) for a in (-0.4, 0.3))
    mask = mO.double().repeat_interleave(4, 0).repeat_interleave(4, 1)
    out = {"Hp": _blocks(torch.matmul(A, torch.matmul(H, A) * mask), I, J)}
    out["F"] = _blocks(torch.matmul(A, torch.matmul(p, A) * mask), IO, JO)
    return out


# ---------------------------------------------------------------------------

E0, E1 = -12.5, 4.5  # the scaled interval of the benchmark's Hamiltonians, about 17 Ha wide


def _levels(seed):
    g = np.random.default_rng([int(seed), 77])
    return np.concatenate([g.normal(-0.55, 0.35, 1200), g.normal(0.9, 0.6, 700), g.uniform(-9.0, 3.5, 100)]).clip(-11.9, 3.9)


def _prep_scalars(c, seed):
    e = torch.tensor(_levels(seed), device=DEV)
    th = torch.acos((2.0 * e - (E0 + E1)) / (E1 - E0))
    k = torch.arange(c["n_terms"], device=DEV, dtype=torch.float64)
    g = torch.cos(k[:, None] * th[None, :]).sum(1)
    return dict(c=c, g=g, N_e=1000.25 + (int(seed) % 97))


def _run_scalars(s):
    c, g = s["c"], s["g"]
    n = c["n_terms"]
    verdict, value = cg.penalty_check(g, min(n, 512), -200.0, 1.0)
    r = cg.decode_mu_result(cg.mu_search(g, n, E0, E1, cg.FERMI, c["kT"], s["N_e"], 1e-6 * s["N_e"]))
    nd, cd = cg.coeffs([{"kind": cg.FERMI, "mu": 0.5 * (E0 + E1), "kT": c["kT"]}], E0, E1, 1e-7, c["n_max"], device=DEV)
    mus = cg.mu_nodes(r["mu"], 0.02 * c["kT"], c["n_mu"])
    _, cm = cg.coeffs([{"kind": cg.FERMI, "mu": m, "kT": c["kT"]} for m in mus], E0, E1, 0.0, n, device=DEV)
    return {"verdict": verdict, "value": value, "mu": r["mu"], "N": r["N"], "iters": r["iters"],
            "bits": np.array((r["bits"] + [2] * 128)[:128], dtype=np.int64), "degree": nd, "c_degree": cd, "c_mu": cm}


def _exact_scalars(c, seed):
    n, kT, N_e = c["n_terms"], c["kT"], 1000.25 + (int(seed) % 97)
    sig, tau = 2.0 / (E1 - E0), 0.5 * (E0 + E1)
    th = torch.acos((2.0 * torch.tensor(_levels(seed)) - (E0 + E1)) / (E1 - E0))
    g = torch.cat([torch.cos(k[:, None] * th[None, :]).sum(1) for k in torch.arange(n, dtype=torch.float64).split(512)])
    # N(mu) of the n-term series = sum over the nodes of f times the moments' transform
    w = torch.empty(n, dtype=torch.float64)
    gh = g.clone()
    gh[0] *= 0.5
    for i in torch.arange(n).split(512):
        ang = (torch.arange(n)[None, :] * (2 * i + 1)[:, None]) % (4 * n)
        w[i] = (2.0 / n) * (torch.cos(math.pi * ang.double() / (2.0 * n)) @ gh)
    x = torch.cos(math.pi * (torch.arange(n, dtype=torch.float64) + 0.5) / n) / sig + tau
    lo, hi, N = E0, E1, 0.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        N = float((_fermi(x, mid, kT) * w).sum())
        if abs(N - N_e) <= 1e-6 * N_e:
            break
        lo, hi = (lo, mid) if N > N_e else (mid, hi)
    half = 0.02 * kT
    mus = [mid + half * math.cos(math.pi * (i + 0.5) / c["n_mu"]) for i in range(c["n_mu"])]
    cm = torch.stack([_dct(lambda v: _fermi(v / sig + tau, m, kT), n) for m in mus])
    return {"verdict": None, "value": None, "mu": mid, "N": N, "iters": None, "bits": None, "degree": None, "c_degree": None,
            "c_mu": cm}


# ---------------------------------------------------------------------------

def _prep_bounds(c, seed):
    xyz, L = _atoms(c["n_atoms"], DEV)
    PH, I, J = _pattern(xyz, L, c["r_c"])
    return dict(c=c, H=PH.with_vals(_hamiltonian(_overlap(xyz, L, I, J, seed), I, J, seed)))


def _run_bounds(s):
    e0, e1, th = cg.bounds(s["H"], s["c"]["steps"])
    return {"bounds": np.array([e0, e1]), "theta": np.array(th)}


# ---------------------------------------------------------------------------

N_IN, N_HID = 35, 128
SIZES = (N_HID * N_IN, N_HID, N_HID * N_HID, N_HID, 2 * N_HID, 2)


def _mlp_data(c, seed):
    g = torch.Generator().manual_seed(int(seed) * 31 + 5)
    B = c["batch"]
    theta = torch.cat([torch.randn(s, generator=g) * a for s, a in zip(SIZES, (0.12, 0.05, 0.09, 0.05, 0.1, 0.5))])
    X = torch.randn((B, N_IN), generator=g) * 0.3
    m = torch.randn(theta.numel(), generator=g) * 1e-3
    v = (torch.randn(theta.numel(), generator=g) * 1e-2).square() + 1e-6
    xs = torch.randn(B, generator=g) * 0.1
    sc = torch.rand(B, generator=g) * 0.5 + 0.2
    return theta, X, m, v, xs, sc


def _prep_mlp(c, seed):
    theta, X, m, v, xs, sc = (a.to(DEV).contiguous() for a in _mlp_data(c, seed))
    B = c["batch"]
    e = lambda *n: torch.empty(n, dtype=torch.float32, device=DEV)  # noqa: E731
    return dict(theta=theta, X=X, m=m, v=v, xs=xs, sc=sc, act=e(B * 256), out=e(B, 2), dout=e(B, 2), ws=e(B * 256),
                grad=torch.empty_like(theta), loss=torch.zeros(1, dtype=torch.float64, device=DEV), t=9)


def _run_mlp(s):
    cg.mlp_forward(s["theta"], s["X"], s["act"], s["out"])
    cg.mlp_loss(s["out"], s["xs"], s["sc"], s["dout"], s["loss"])
    cg.mlp_backward(s["theta"], s["X"], s["act"], s["dout"], s["grad"], s["ws"])
    s["t"] += 1
    cg.mlp_adam(s["theta"], s["grad"], s["m"], s["v"], s["t"], 1e-3)
    return {"out": s["out"], "grad": s["grad"], "theta": s["theta"], "m": s["m"], "v": s["v"], "loss": s["loss"].float()}


def _exact_mlp(c, seed):
    theta, X, m, v, xs, sc = (a.double() for a in _mlp_data(c, seed))
    theta = theta.requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(theta, SIZES)
    h = torch.relu(X @ W1.view(N_HID, N_IN).T + b1)
    h = torch.relu(h @ W2.view(N_HID, N_HID).T + b2)
    out = h @ W3.view(2, N_HID).T + b3
    d, w = (out[:, 0] - xs) / sc, torch.exp(out[:, 1]) / sc
    ad = d.abs()
    loss = (torch.where(ad <= 1.0, 0.5 * d * d, ad - 0.5) + torch.relu(ad - w) + 0.01 * w).mean()
    loss.backward()
    gr = theta.grad
    m2, v2 = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
    th2 = theta.detach() - 1e-3 * (m2 / (1 - 0.9 ** 10)) / (torch.sqrt(v2 / (1 - 0.999 ** 10)) + 1e-8)
    return {"out": out.detach(), "grad": gr, "theta": th2, "m": m2, "v": v2, "loss": loss.detach().view(1)}


# ---------------------------------------------------------------------------

PREPARE = dict(expand=_prep_expand, powers=_prep_powers, foe=_prep_foe, batched=_prep_batched, products=_prep_products,
               scalars=_prep_scalars, bounds=_prep_bounds, mlp=_prep_mlp)
RUN = dict(expand=_run_expand, powers=_run_powers, foe=_run_foe, batched=_run_batched, products=_run_products,
           scalars=_run_scalars, bounds=_run_bounds, mlp=_run_mlp)
EXACT = dict(expand=_exact_expand, powers=_exact_powers, batched=_exact_batched, products=_exact_products,
             scalars=_exact_scalars, mlp=_exact_mlp)


def prepare(case, seed):
    return dict(kind=case["kind"], s=PREPARE[case["kind"]](case, seed))


def run(state):
    return RUN[state["kind"]](state["s"])


def exact(case, seed):
    f = EXACT.get(case["kind"])
    return f(case, seed) if f else None


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _count(n, r):
    return min(float(n), 1.0 + (n / _box(n) ** 3) * 4.0 / 3.0 * math.pi * r ** 3)


def _triples(n, r1, r2, r3):
    """Triples (I, K, J) with |I-K| <= r1, |K-J| <= r2, |I-J| <= r3, r1 <= r2 = r3 (lens volumes)."""
    m, s, wsum = 400, 0.0, 0.0
    for i in range(m):
        d = r1 * (i + 0.5) / m
        lens = math.pi / 12.0 * (4.0 * r3 + d) * max(0.0, 2.0 * r3 - d) ** 2
        s += d * d * lens
        wsum += d * d
    frac = s / wsum / (4.0 / 3.0 * math.pi * r3 ** 3)
    cO = _count(n, r3)
    return n * _count(n, r1) * cO * min(1.0, max(frac, cO / n))


def _expand_work(n, r_c, r_o, steps, nf, with_g, size):
    """Operator and G read once, accumulators written once; the products of every step."""
    nh, no = n * _count(n, r_c), n * _count(n, r_o)
    return (nh * 16 * size + no * 16 * 8 * (nf + (1 if with_g else 0)), 128.0 * steps * _triples(n, r_c, r_o, r_o))


def work(case):
    c, kind = case, case["kind"]
    if kind == "expand":
        b, f = _expand_work(c["n_atoms"], c["r_c"], c["r_c"] + c["r_buf"], c["n_terms"] - 2, c["nf"], True, 8)
    elif kind == "powers":
        b, f = _expand_work(c["n_atoms"], c["r_c"], c["r_c"] + c["r_buf"], c["n_terms"] - 2, 3, False, 8)
    elif kind == "foe":
        # S^-1/2 and two passes of the degree that kT needs, and the products around them
        terms = 2 * min(16384, int(16 * 17.0 / c["kT"] / 8)) + 100
        b, f = _expand_work(c["n_atoms"], c["r_c"], c["r_c"] + c["r_buf"], terms, 1, True, 8)
    elif kind == "batched":
        n, s = 0.5 * (c["atoms_lo"] + c["atoms_hi"]), c["n_sys"]
        b, f = _expand_work(n, c["r_c"], c["r_c"] + c["r_buf"], 0.75 * c["n_terms"], 1, True, 8)
        b, f = b * s, f * s
    elif kind == "products":
        n, ro = c["n_atoms"], c["r_c"] + c["r_buf"]
        nh, no = n * _count(n, c["r_c"]), n * _count(n, ro)
        b = 128.0 * (2 * nh + 3 * no)
        f = 128.0 * (_triples(n, c["r_c"], ro, ro) + 3 * _triples(n, ro, ro, ro))
    elif kind == "scalars":
        n = c["n_terms"]
        b = 8.0 * (n * (1 + c["n_mu"]) + c["n_max"])
        # transforms by their fast form, the bisection's node sums, the degree check of the chosen candidate
        f = 5.0 * n * math.log2(n) * (1 + c["n_mu"]) + 25 * 20.0 * n + 3.0 * n * (8193 + 2 * n)
    elif kind == "bounds":
        nh = c["n_atoms"] * _count(c["n_atoms"], c["r_c"])
        b, f = nh * 132.0, 32.0 * nh * c["steps"]
    else:
        p = sum(SIZES)
        b, f = 4.0 * (7 * p + c["batch"] * 40), 6.0 * p * c["batch"]
    return {"bytes": float(b), "flops": float(f)}
