"""Workloads of the finite-PEPS library, each one call of the Python binding as an optimisation
loop or an estimator makes it: evaluations (psi, E_loc, O), Metropolis and direct sampling, and
MinSR steps.

A case is a dict of plain values.  `kind` names the call:

  evaluate    ln psi, E_loc and O of a batch of stored configurations
  amplitudes  ln psi alone
  sample      Metropolis sweeps of a batch of chains
  direct      the double-layer environments of the parameters, then independent configurations
  minsr       one MinSR step from O and E_loc

Tensors are drawn as the workloads of paper_2503_12557_gb300.inputs draw them (a biased Gaussian
with algebraically decaying virtual legs; complex: mean-zero Gaussian entries), configurations
from the S^z = 0 sector (spin models) or uniformly (Rydberg arrays).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_12557_gb300 import inputs as I
from paper_2503_12557_gb300 import peps as P

PREC = {"fp64": P.PREC_FP64, "fp32": P.PREC_FP32, "mixed": P.PREC_MIXED}


# ------------------------------------------------------------------------------------- cases

def _peps_case(kind, model, Lx, Ly, D, chi, prec, ns, **more):
    return dict(kind=kind, model=model, Lx=Lx, Ly=Ly, D=D, chi=chi, prec=prec, ns=ns, **more)


def listed():
    cases = [
        # the 4x4 exact-chi problem a user starts with: a small call, bound by launches and latency
        ("evaluate 4x4 fp64", _peps_case("evaluate", "heisenberg", 4, 4, 2, 4, "fp64", 256)),
        # a handful of amplitudes (a proposal's acceptance, a spot check): few CTAs, the upper side only
        ("amplitudes 8x8 fp32 few", _peps_case("amplitudes", "heisenberg", 8, 8, 4, 16, "fp32", 37)),
        # the estimators of one optimisation step on the 8x8 workload's full batch of chains
        ("evaluate 8x8 fp32", _peps_case("evaluate", "heisenberg", 8, 8, 4, 16, "fp32", 4096)),
        # the Rydberg array's estimators (flip terms inside a row, long diagonal pairs, chi = 24)
        ("evaluate 12x12 rydberg fp32", _peps_case("evaluate", "rydberg", 12, 12, 4, 24, "fp32", 304)),
        # an odd lattice at a bond without a compiled shape (D = 5, chi = D^2), one ragged batch
        ("evaluate 7x9 D5 fp32", _peps_case("evaluate", "heisenberg", 7, 9, 5, 25, "fp32", 100)),
        # complex PEPS with three-site chiral terms over two rows
        ("evaluate 5x5 chiral c64", _peps_case("evaluate", "j1j2_chiral", 5, 5, 3, 9, "fp32", 152)),
        # the sweeps of one optimisation step on the 8x8 workload's chains
        ("sample 8x8 fp32", _peps_case("sample", "heisenberg", 8, 8, 4, 16, "fp32", 4096, move="exchange", sweeps=2)),
        # double-precision flip chains of a small array, fewer chains than SMs
        ("sample 6x6 flips fp64", _peps_case("sample", "rydberg", 6, 6, 3, 9, "fp64", 100, move="flip", sweeps=1)),
        # direct sampling in an optimisation step: the parameters are new, so the double layer is too
        ("direct 8x8 fp32", _peps_case("direct", "heisenberg", 8, 8, 4, 16, "fp32", 304, chi_double=4)),
        # MinSR of the 8x8 workload with the mixed-precision preset (the benchmark's route)
        ("minsr 8x8 mixed", _peps_case("minsr", "heisenberg", 8, 8, 4, 16, "mixed", 4096, lam=1e-4, rcond=0.0)),
        # MinSR in double precision, the paper's thousand samples
        ("minsr 6x6 fp64", _peps_case("minsr", "heisenberg", 6, 6, 3, 9, "fp64", 1000, lam=1e-4, rcond=0.0)),
        # MinSR with the pseudo-inverse cutoff (eigendecomposition), an odd sample count
        ("minsr 6x6 fp64 cutoff", _peps_case("minsr", "heisenberg", 6, 6, 3, 9, "fp64", 333, lam=1e-4, rcond=1e-8)),
    ]
    return [dict(name=n, **c) for n, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: lattices 4..12 in both directions, D 2..5, 4 to 4096 samples."""
    cap = 0.5 * max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["evaluate", "evaluate", "evaluate", "amplitudes", "sample", "sample", "direct", "minsr", "minsr"])
        Lx, Ly = rng.randint(4, 12), rng.randint(4, 12)
        D = rng.choice([2, 3, 4, 4, 4, 5])
        chi = rng.choice([16, 24]) if D == 4 and rng.random() < 0.7 else rng.randint(D, D * D)
        prec = rng.choice(["fp32", "fp32", "fp64"])
        ns = _log_int(rng, 4, 4096)
        if kind == "minsr":
            D = min(D, 4)
            chi = max(D, min(chi, D * D))
            rcond = rng.choice([0.0, 0.0, 1e-8])
            prec = rng.choice(["mixed", "fp64"])
            ns = max(16, min(ns, 600)) if rcond > 0.0 else max(16, ns)
            c = _peps_case(kind, "heisenberg", Lx, Ly, D, chi, prec, ns, lam=1e-4, rcond=rcond)
            # fewer samples than parameters, as MinSR is made for: T has no further null space
            if ns > I.num_params(_lattice(c)) // 4:
                continue
        elif kind == "sample":
            move = rng.choice(["exchange", "flip"])
            model = "heisenberg" if move == "exchange" else "rydberg"
            c = _peps_case(kind, model, Lx, Ly, D, chi, prec, ns, move=move, sweeps=rng.randint(1, 2))
        elif kind == "direct":
            D = min(D, 4)
            c = _peps_case(kind, "heisenberg", Lx, Ly, D, max(D, min(chi, D * D)), prec, min(ns, 512), chi_double=D)
        elif kind == "amplitudes":
            c = _peps_case(kind, rng.choice(["heisenberg", "rydberg"]), Lx, Ly, D, chi, prec, ns)
        else:
            model = rng.choice(["heisenberg", "heisenberg", "rydberg", "j1j2_chiral"])
            if model == "j1j2_chiral":
                D = min(D, 3)
                chi = rng.randint(D, D * D)
            c = _peps_case(kind, model, Lx, Ly, D, chi, prec, ns)
        if _cost(c) <= cap:
            return c


# ------------------------------------------------------------------------------------ inputs

def _lattice(c):
    return I.Lattice(c["Lx"], c["Ly"], 2, c["D"])


def _complex(c):
    return c["model"] == "j1j2_chiral"


def _theta(c, seed):
    lat = _lattice(c)
    if _complex(c):
        return I.peps_random(lat, seed, scale=0.3, bias=1.0, complex_=True)
    return I.peps_random(lat, seed, scale=0.5, bias=1.0, alpha=1.5)


def _configs(c, seed):
    n, ns = c["Lx"] * c["Ly"], c["ns"]
    rng = np.random.default_rng(seed)
    if c["model"] == "rydberg":
        return rng.integers(0, 2, size=(ns, n), dtype=np.uint8)
    return (np.argsort(rng.random((ns, n)), axis=1) >= n // 2).astype(np.uint8)  # S^z = 0


def _hamiltonian(c):
    return getattr(I, c["model"])(_lattice(c))


def _minsr_inputs(c, seed, device):
    """O (N(0,1) entries with a column offset, each site's block zero for the states its
    configuration does not take, as log-derivatives are), E_loc and weights that leave out one
    sample in 64."""
    lat, ns = _lattice(c), c["ns"]
    g = torch.Generator(device=device).manual_seed(seed)
    npar = I.num_params(lat)
    dtype = torch.float64 if c["prec"] == "fp64" else torch.float32
    O = torch.randn(ns, npar, generator=g, device=device, dtype=dtype)
    O += 0.1 * torch.randn(npar, generator=g, device=device, dtype=dtype)
    S = torch.as_tensor(_configs(c, seed + 1)).to(device)
    offs = I.site_offsets(lat)
    for i in range(lat.nsites):
        blk = (offs[i + 1] - offs[i]) // 2
        O[:, offs[i]:offs[i] + blk] *= (S[:, i:i + 1] == 0)
        O[:, offs[i] + blk:offs[i + 1]] *= (S[:, i:i + 1] == 1)
    e = torch.zeros(ns, 2, device=device, dtype=torch.float64)
    e[:, 0] = 0.23 * lat.nsites + torch.randn(ns, generator=g, device=device, dtype=torch.float64)
    w = (torch.rand(ns, generator=g, device=device, dtype=torch.float64) > 1.0 / 64).double()
    return O, e, w


def prepare(case, seed):
    c = dict(case, seed=int(seed))
    # one MinSR handle solves for its own sample count; its environment store is not used here
    h = P.PEPS(c["Lx"], c["Ly"], 2, c["D"], c["chi"], prec=PREC[c["prec"]], cplx=_complex(c),
               max_samples=1 if c["kind"] == "minsr" else c["ns"])
    if c["kind"] == "minsr":
        return dict(c, h=h, inputs=_minsr_inputs(c, c["seed"], "cuda"))
    h.set_params(torch.as_tensor(_theta(c, c["seed"])).cuda())
    st = dict(c, h=h, S=torch.as_tensor(_configs(c, c["seed"] + 1)).cuda())
    if c["kind"] == "evaluate":
        st["H"] = _hamiltonian(c)
        h.hamiltonian(st["H"])
    return st


def run(st):
    h = st["h"]
    if st["kind"] == "evaluate":
        return h.evaluate(st["H"], st["S"])
    if st["kind"] == "amplitudes":
        return h.amplitudes(st["S"])
    if st["kind"] == "sample":
        move = P.MOVE_EXCHANGE if st["move"] == "exchange" else P.MOVE_FLIP
        # a copy of the chains' start, so that the call can be repeated
        return h.sample(st["S"].clone(), move, st["sweeps"], seed=st["seed"], sweep0=0)
    if st["kind"] == "direct":
        h.direct_prepare(st["chi_double"])
        return h.direct_sample(st["ns"], seed=st["seed"])
    O, e, w = st["inputs"]
    # the update itself; info holds diagnostics (a residual at rounding level) and is not returned
    return h.minsr_step(O, e, w=w, lam=st["lam"], rcond=st["rcond"])[0]


# -------------------------------------------------------------------------------------- work

def _bonds(c, row):
    """Bonds 0..Ly of the boundary MPS that holds `row` + 1 rows (open ends: 1)."""
    Ly, D, chi = c["Ly"], c["D"], c["chi"]
    return [min(chi, D ** min(row + 1, 12), D ** min(k, 12), D ** min(Ly - k, 12)) for k in range(Ly + 1)]


def _row_step_flops(c, row):
    """Multiply-adds x 2 of the row applied to a boundary MPS of `row` rows: exact product,
    left QR sweep, truncation of every cut, at the bonds that occur."""
    D, Ly = c["D"], c["Ly"]
    b, o = _bonds(c, row - 1), _bonds(c, row)
    m = [b[k] * (1 if k in (0, Ly) else D) for k in range(Ly + 1)]
    leg = lambda k: 1 if k in (0, Ly) else D  # noqa: E731
    rho, f = 1, 0.0
    rhos = [1]
    for k in range(Ly - 1):
        f += 2.0 * rho * leg(k) * b[k] * D * b[k + 1] + 2.0 * rho * D * D * leg(k) * b[k + 1] * leg(k + 1)
        r, q = max(rho * D, m[k + 1]), min(rho * D, m[k + 1])
        f += 2.0 * r * q * q - 2.0 * q ** 3 / 3.0
        rho = q
        rhos.append(rho)
    for k in range(Ly - 1, 0, -1):
        lr = D * o[k + 1]
        f += 2.0 * b[k] * D * b[k + 1] * leg(k + 1) * o[k + 1] + 2.0 * m[k] * D * D * leg(k + 1) * o[k + 1]
        f += 1.0 * rhos[k] * m[k] * lr + 4.0 * rhos[k] * lr * o[k] + 2.0 * m[k] * lr * o[k]
    return f


def _absorb_flops(c, x, rows):
    """All columns of one left (or right) partial pass of a sandwich over `rows` rows from row x."""
    D, Ly, Lx = c["D"], c["Ly"], c["Lx"]
    up = _bonds(c, x - 1) if x > 0 else [1] * (Ly + 1)
    lo = _bonds(c, Lx - x - rows - 1) if x + rows < Lx else [1] * (Ly + 1)
    f = 0.0
    for k in range(Ly):
        l = 1 if k == 0 else D
        r = 1 if k == Ly - 1 else D
        du, dd = (D if x > 0 else 1), (D if x + rows < Lx else 1)
        L, R = l ** rows, r ** rows
        f += 2.0 * up[k] * L * lo[k] * du * up[k + 1] + 2.0 * up[k + 1] * R * dd * lo[k] * lo[k + 1]
        if rows == 1:
            f += 2.0 * up[k + 1] * lo[k] * l * du * r * dd
        else:
            f += 2.0 * up[k + 1] * lo[k] * (l * l * du * r * D + l * D * r * r * dd)
    return f


def _work(c):
    lat, ns = _lattice(c), c["ns"]
    npar = I.num_params(lat)
    Lx, Ly = c["Lx"], c["Ly"]
    cx = 4.0 if _complex(c) else 1.0
    osz = (8 if c["prec"] == "fp64" else 4) * (2 if _complex(c) else 1)
    side = sum(_row_step_flops(c, x) for x in range(1, Lx - 1))
    io = ns * Lx * Ly + 8.0 * npar * (2 if _complex(c) else 1)
    if c["kind"] == "minsr":
        return io + ns * npar * osz + 16.0 * ns + 8.0 * npar, 1.0 * ns * ns * npar + 4.0 * ns * npar + ns ** 3 / 3.0
    if c["kind"] == "amplitudes":
        return io + 20.0 * ns, ns * (side + _absorb_flops(c, Lx - 1, 1))
    one = [_absorb_flops(c, x, 1) for x in range(Lx)]
    two = [_absorb_flops(c, x, 2) for x in range(Lx - 1)]
    if c["kind"] == "evaluate":
        f = 2.0 * side + 3.0 * sum(one)  # both sides; left and right partials and the site environments
        row_terms, pair_terms = {"rydberg": (1, 0), "heisenberg": (1, 1), "j1j2_chiral": (1, 8)}[c["model"]]
        f += sum(one) * row_terms  # off-diagonal terms: about one column pass per row and term kind
        if pair_terms:
            f += (2.0 + 0.5 * pair_terms) * sum(two)
        return io + ns * npar * osz + 36.0 * ns, cx * ns * f
    if c["kind"] == "sample":
        f = side * (2 if c["sweeps"] < 2 else 3)
        f += c["sweeps"] * 3.0 * sum(one) + (c["sweeps"] * 2.5 * sum(two) if c["move"] == "exchange" else 0.0)
        return io + ns * (Lx * Ly + 12.0), ns * f
    # direct: the upper rows, and per row the right partials and the d candidates of every site
    cd, D = c["chi_double"], c["D"]
    f = side
    for x in range(Lx):
        n = [v * (1 if k in (0, Ly) else D) for k, v in enumerate(_bonds(c, x - 1) if x else [1] * (Ly + 1))]
        dd = D if x < Lx - 1 else 1
        f += sum(2 * 2.0 * 2 * cd * n[k] * n[k + 1] * dd * (n[k] + cd * dd) for k in range(Ly))
    return io + ns * (Lx * Ly + 12.0), ns * f


def work(case):
    b, f = _work(case)
    return {"bytes": b, "flops": f}


def _cost(c):
    """Work in FP32 units for draw(): FP64 contractions cost about 60 FP32 ones, complex ones and
    shapes without a compiled kernel a few, eigendecompositions and the direct sampler more than
    their operations say."""
    f = _work(c)[1]
    if c["kind"] == "minsr":
        return 0.05 * f + (4e3 * c["ns"] ** 3 if c["rcond"] > 0.0 else 0.0)
    if c["kind"] == "direct":
        return 20.0 * f + 1e11
    return f * (60.0 if c["prec"] == "fp64" else 1.0) * (1.0 if c["D"] == 4 else 3.0) * (2.0 if _complex(c) else 1.0)


# ------------------------------------------------------------------- the same in plain 64 bits

def _project(theta, lat, S):
    """Site tensors (batch, l, u, r, d) of the PEPS projected on every configuration."""
    T = I.theta_to_tensors(lat, theta)
    return [[torch.as_tensor(np.ascontiguousarray(T[x][y][S[:, x * lat.Ly + y]])) for y in range(lat.Ly)]
            for x in range(lat.Lx)]


def _normalised(t):
    m = t.abs().flatten(1).max(1).values
    return t / m.view(-1, *[1] * (t.dim() - 1)), m.log()


def _apply_row(E, A, chi):
    """Boundary MPS E (batch, a, p, b per site) times the row A, truncated to chi from the right
    after the exact left-canonical form; (sites, log factor)."""
    M, n = [], E[0].shape[0]
    for e, t in zip(E, A):
        m = torch.einsum("naub,nlurd->naldbr", e, t)
        M.append(m.reshape(n, m.shape[1] * m.shape[2], m.shape[3], -1))
    for k in range(len(M) - 1):
        q, r = torch.linalg.qr(M[k].flatten(1, 2))
        M[k] = q.reshape(n, M[k].shape[1], M[k].shape[2], -1)
        M[k + 1] = torch.einsum("nij,njdk->nidk", r, M[k + 1])
    for k in range(len(M) - 1, 0, -1):
        u, s, vh = torch.linalg.svd(M[k].flatten(2), full_matrices=False)
        keep = min(chi, s.shape[1])
        shape = M[k].shape
        M[k] = vh[:, :keep].reshape(n, keep, shape[2], shape[3])
        M[k - 1] = torch.einsum("nidj,njk->nidk", M[k - 1], u[:, :, :keep] * s[:, None, :keep])
    out, lg = [], 0.0
    for m in M:
        m, l = _normalised(m)
        out.append(m)
        lg = lg + l
    return out, lg


def _environments(A, chi):
    """Upper environments of rows -1..Lx-2 and lower ones of rows 1..Lx, keyed by row, with logs."""
    Lx, Ly, n = len(A), len(A[0]), A[0][0].shape[0]
    one = [torch.ones(n, 1, 1, 1, dtype=A[0][0].dtype) for _ in range(Ly)]
    up, lo = {-1: (one, torch.zeros(n, dtype=torch.float64))}, {Lx: (one, torch.zeros(n, dtype=torch.float64))}
    for x in range(Lx - 1):
        E, lg = _apply_row(up[x - 1][0], A[x], chi)
        up[x] = (E, up[x - 1][1] + lg)
    for x in range(Lx - 1, 0, -1):
        E, lg = _apply_row(lo[x + 1][0], [t.transpose(2, 4) for t in A[x]], chi)
        lo[x] = (E, lo[x + 1][1] + lg)
    return up, lo


LEFT = {1: "nalb,naux,nlurd,nbdz->nxrz", 2: "naijb,naux,niurv,njvsd,nbdz->nxrsz"}
RIGHT = {1: "nxrz,naux,nlurd,nbdz->nalb", 2: "nxrsz,naux,niurv,njvsd,nbdz->naijb"}


def _partials(rows, eu, el):
    """Left and right partials of the sandwich of one or two rows between two boundary MPS."""
    k, Ly, n = len(rows), len(eu), eu[0].shape[0]
    one = torch.ones(n, *[1] * (k + 2), dtype=eu[0].dtype)
    L, R = [one], [one]
    for y in range(Ly):
        L.append(torch.einsum(LEFT[k], L[-1], eu[y], *[r[y] for r in rows], el[y]))
    for y in range(Ly - 1, -1, -1):
        R.insert(0, torch.einsum(RIGHT[k], R[0], eu[y], *[r[y] for r in rows], el[y]))
    return L, R


def _exact_evaluate(c, seed):
    lat = _lattice(c)
    Lx, Ly, npar = c["Lx"], c["Ly"], I.num_params(lat)
    theta, S = _theta(c, seed), _configs(c, seed + 1).astype(np.int64)
    n = len(S)
    A = _project(theta, lat, S)
    dtype = A[0][0].dtype
    up, lo = _environments(A, c["chi"])
    L, R = _partials([A[Lx - 1]], up[Lx - 2][0], lo[Lx][0])
    top = L[-1].reshape(n)
    logabs, phase = top.abs().log() + up[Lx - 2][1], torch.angle(top)
    if c["kind"] == "amplitudes":
        return [logabs, phase, None]
    H = _hamiltonian(c)
    T = I.theta_to_tensors(lat, theta)
    offs = I.site_offsets(lat)
    O = torch.zeros(n, npar, dtype=dtype)
    e = torch.zeros(n, dtype=torch.complex128)
    for i, j, v in H["pairs"]:
        e += v * torch.as_tensor(S[:, i] * S[:, j]).double()
    e += torch.as_tensor(np.take_along_axis(H["onsite"].T, S, axis=0).sum(1))
    for k in (1, 2):
        for x in range(Lx - k + 1):
            terms = [(s, h) for s, h in H["terms"] if {i // Ly for i in s} == set(range(x, x + k))]
            if k == 2 and not terms:
                continue
            eu, el, rows = up[x - 1][0], lo[x + k][0], A[x:x + k]
            L, R = _partials(rows, eu, el)
            psi = L[-1].reshape(n)
            if k == 1:
                for y in range(Ly):
                    env = torch.einsum("nalb,naux,nxrz,nbdz->nlurd", L[y], eu[y], R[y + 1], el[y]) / psi.view(-1, 1, 1, 1, 1)
                    blk, s = env[0].numel(), torch.as_tensor(S[:, x * Ly + y])
                    O[:, offs[x * Ly + y]:offs[x * Ly + y + 1]].view(n, 2, blk)[torch.arange(n), s] = env.reshape(n, blk)
            for sites, h in terms:
                m = len(sites)
                a = sum(S[:, s] << (m - 1 - t) for t, s in enumerate(sites))
                y0, y1 = min(s % Ly for s in sites), max(s % Ly for s in sites)
                for ia, ib in zip(*np.nonzero(h)):
                    pick = np.nonzero(a == ia)[0]
                    if ia == ib:
                        e[pick] += complex(h[ia, ib])
                        continue
                    if not len(pick):
                        continue
                    t = torch.as_tensor(pick)
                    S2 = S[pick].copy()
                    for q, s in enumerate(sites):
                        S2[:, s] = (ib >> (m - 1 - q)) & 1
                    v = L[y0][t]
                    for y in range(y0, y1 + 1):
                        cols = [torch.as_tensor(np.ascontiguousarray(T[x + r][y][S2[:, (x + r) * Ly + y]])) for r in range(k)]
                        v = torch.einsum(LEFT[k], v, eu[y][t], *cols, el[y][t])
                    e[t] += complex(h[ia, ib]) * (v * R[y1 + 1][t]).flatten(1).sum(1) / psi[t]
    return dict(logabs=logabs, phase=phase, eloc=torch.view_as_real(e), O=O, status=None)


def _exact_minsr(c, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    O, e, w = _minsr_inputs(c, seed, dev)
    w = w / w.sum()
    Ob = O.double()
    Ob = w.sqrt()[:, None] * (Ob - w @ Ob)
    eb = w.sqrt() * (e[:, 0] - w @ e[:, 0])
    T = Ob @ Ob.T
    if c["rcond"] > 0.0:
        lam, V = torch.linalg.eigh(T)
        x = V @ (torch.where(lam > c["rcond"] * lam[-1], 1.0 / (lam + c["lam"]), torch.zeros_like(lam)) * (V.T @ eb))
    else:
        x = torch.linalg.solve(T + c["lam"] * torch.eye(len(T), dtype=T.dtype, device=T.device), eb)
    return (-0.05 * (Ob.T @ x)).cpu()


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "minsr":
        return _exact_minsr(c, int(seed))
    if c["kind"] in ("sample", "direct"):
        return None  # the chains' and draws' decisions are whole numbers; log p has no closed form
    # batched QR and SVD on the host: leave out what takes longer than about 20 seconds
    svds = c["ns"] * (2 if c["kind"] == "evaluate" else 1) * (c["Lx"] - 2) * (c["Ly"] - 1)
    if svds * (4e-5 + 4e-9 * (c["chi"] * c["D"]) ** 3 * (3 if _complex(c) else 1)) > 12.0:
        return None
    return _exact_evaluate(c, int(seed))
