"""The work that programs have this library do, as timed cases.

Every case is a whole call of a public entry point on a seeded synthetic
system (``tbinputs``): silicon supercells and liquid-water boxes from 64 to
4096 atoms, from one right-hand side to several hundred, in plain FP64 and in
mixed precision, for each direction of the path -- Green's-function elements
and full solutions, Mulliken populations, the charge-self-consistency loop,
ragged batches, band-energy gradients with forces, the Mulliken
vector-Jacobian product, and the generalized Lanczos process with its local
densities of states.  The handle is the device copy of a system's matrices,
which a program keeps between calls; everything else is inside ``run``.

Shifts are Gauss-Legendre nodes on the window of the occupied spectrum with a
broadening of 1 to 4 eV, so that every call runs to the stated residual.
"""
import math

import numpy as np
import torch

import paper_1002_1202_gb300 as tb
import tbinputs

G_S = 2.0
INNER_STEPS = 50          # products with S per application of S^-1 (condition number ~10, relative 1e-12 .. 1e-13)
SI_WINDOW = (-20.0, 5.0)
WATER_WINDOW = (-60.0, -8.0)


def listed():
    return [
        # one Green's function element set of one orbital in a small cell, plain FP64: the smallest call, all latency
        {"name": "green_si64_one_column", "kind": "green", "cells": "2x2x2", "cols": 1, "rows": 5, "shifts": 16,
         "eta": 2.0, "precision": "fp64", "tol": 1e-11, "inner_tol": 1e-13},
        # full solutions of a few columns of a small cell in FP64: the parity configuration (64 atoms, 32 shifts, 8 columns)
        {"name": "full_si64_fp64", "kind": "full", "cells": "2x2x2", "cols": 8, "shifts": 32, "eta": 2.0,
         "precision": "fp64", "tol": 1e-11, "inner_tol": 1e-13},
        # the same kind of call in mixed precision on a non-cubic cell with odd counts (a cluster in an MD step)
        {"name": "full_si144_mixed", "kind": "full", "cells": "2x3x3", "cols": 13, "shifts": 24, "eta": 1.0,
         "precision": "mixed", "tol": 1e-11, "inner_tol": 1e-13},
        # populations of selected orbitals in plain FP64, an ordinary size
        {"name": "mulliken_si216_fp64", "kind": "mulliken", "cells": "3x3x3", "cols": 48, "shifts": 64, "eta": 2.0,
         "precision": "fp64", "tol": 1e-10, "inner_tol": 1e-13},
        # populations in mixed precision, an ordinary size: four default panels in flight
        {"name": "mulliken_si512_mixed", "kind": "mulliken", "cells": "4x4x4", "cols": 256, "shifts": 64, "eta": 1.0,
         "precision": "mixed", "tol": 1e-8, "inner_tol": 1e-12},
        # one panel of the full width on a larger crystal
        {"name": "mulliken_si1728_panel256", "kind": "mulliken", "cells": "6x6x6", "cols": 256, "shifts": 128,
         "eta": 2.0, "precision": "mixed", "tol": 1e-8, "inner_tol": 1e-12, "panel": 256},
        # the benchmark crystal with 256 shifts: the largest call
        {"name": "mulliken_si4096_mixed", "kind": "mulliken", "cells": "8x8x8", "cols": 256, "shifts": 256, "eta": 4.0,
         "precision": "mixed", "tol": 1e-8, "inner_tol": 1e-12},
        # ragged batch of independent water boxes (s-only hydrogens, one H3O+ each)
        {"name": "batch_water", "kind": "batch", "boxes": 5, "molecules": 64, "cols": 64, "shifts": 64, "eta": 2.0,
         "precision": "mixed", "tol": 1e-8, "inner_tol": 1e-13},
        # charge self-consistency on a water box: every column, two SCF iterations
        {"name": "csc_water48", "kind": "csc", "molecules": 48, "shifts": 64, "eta": 2.0, "scf": 2,
         "precision": "mixed", "tol": 1e-10, "inner_tol": 1e-13},
        # an MD step: band energy, its gradients at every stored entry of H and S, and the forces
        {"name": "forces_si64_mixed", "kind": "forces", "cells": "2x2x2", "shifts": 64, "eta": 1.0,
         "precision": "mixed", "tol": 1e-11, "inner_tol": 1e-13},
        # backward pass of the charges of a few atoms
        {"name": "vjp_si64_mixed", "kind": "vjp", "cells": "2x2x2", "atoms": 4, "shifts": 32, "eta": 2.0,
         "precision": "mixed", "tol": 1e-11, "inner_tol": 1e-13},
        # local densities of states of many orbitals: Lanczos coefficients and continued fractions
        {"name": "lanczos_si1728_mixed", "kind": "lanczos", "cells": "6x6x6", "cols": 128, "steps": 24, "points": 501,
         "eta": 0.5, "precision": "mixed", "inner_tol": 1e-12},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, lo, hi):
    """Cells along the axes of a silicon supercell with lo .. hi atoms, spread over the logarithm of the count."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        c = [rng.randint(2, 8) for _ in range(3)]
        n = 8 * c[0] * c[1] * c[2]
        if lo <= n <= hi and abs(math.log(n / want)) < 0.35:
            return "%dx%dx%d" % tuple(c)


def draw(rng):
    """Another case of the same ranges; its estimated floating-point work is at most that of the largest listed case of
    its precision, and its steps on small systems (bound by latency) no more than theirs."""
    cap = {"fp64": _flops(listed()[3]), "mixed": _flops(listed()[6])}
    while True:
        kind = rng.choice(["green", "full", "mulliken", "mulliken", "mulliken", "batch", "csc", "forces", "vjp", "lanczos"])
        c = {"kind": kind, "eta": round(math.exp(rng.uniform(math.log(1.0), math.log(4.0))), 3),
             "precision": rng.choice(["mixed", "mixed", "fp64"]), "tol": rng.choice([1e-8, 1e-10]),
             "inner_tol": rng.choice([1e-12, 1e-13])}
        if c["precision"] == "fp64":
            c["eta"] = max(c["eta"], 2.0)
        if kind not in ("mulliken", "batch"):
            c["tol"] = 1e-10 if kind == "csc" else 1e-11
        if kind in ("green", "full"):
            c["cells"] = _cells(rng, 64, 216)
            c["cols"] = _log_int(rng, 1, 24)
            c["shifts"] = _log_int(rng, 4, 64)
            if kind == "green":
                c["rows"] = rng.randint(1, 12)
        elif kind == "mulliken":
            c["cells"] = _cells(rng, 64, 4096 if c["precision"] == "mixed" else 512)
            c["cols"] = min(_log_int(rng, 8, 512), 4 * _atoms(c))
            c["shifts"] = _log_int(rng, 16, 256)
            c["panel"] = rng.choice([0, 0, 64, 128, 256])
        elif kind == "batch":
            c.update(precision="mixed", boxes=rng.randint(2, 6), molecules=_log_int(rng, 36, 64),
                     cols=_log_int(rng, 16, 64), shifts=_log_int(rng, 16, 64))
            c["eta"] = max(c["eta"], 2.0)
        elif kind == "csc":
            c.update(precision="mixed", molecules=_log_int(rng, 27, 56), shifts=_log_int(rng, 16, 64),
                     scf=rng.randint(1, 2))
            c["eta"] = max(c["eta"], 2.0)
        elif kind == "forces":
            c.update(precision="mixed", cells=rng.choice(["2x2x2", "2x2x3", "2x3x2"]), shifts=_log_int(rng, 16, 64))
        elif kind == "vjp":
            c.update(precision="mixed", cells=_cells(rng, 64, 144), atoms=rng.randint(1, 6), shifts=_log_int(rng, 8, 32))
        else:
            c.update(precision="mixed", cells=_cells(rng, 216, 1728), cols=_log_int(rng, 16, 192),
                     steps=rng.randint(12, 24), points=_log_int(rng, 101, 1001), eta=0.5)
            del c["tol"]
        if _flops(c) <= cap[c["precision"]] and c not in listed():
            return c


# ---- sizes and work ---------------------------------------------------------
def _atoms(c):
    if "cells" in c:
        a, b, d = (int(v) for v in c["cells"].split("x"))
        return 8 * a * b * d
    return (3 * c["molecules"] + 1) * c.get("boxes", 1)


def _size(c):
    """Orbitals and stored real entries of S: 17 neighbours of four orbitals in silicon, in water ~39 atoms within the cutoff."""
    n = _atoms(c)
    if "cells" in c:
        return 4 * n, 17.0 * 16 * n
    return 2 * n, 39.0 * 4 * n


def _outer(c):
    """Outer iterations to the residual: ~42 per decade at a broadening of 1 eV, never much more than the orbitals."""
    if c["kind"] == "lanczos":
        return c["steps"]
    n = _size(c)[0] // c.get("boxes", 1)
    return min(n, 42.0 * math.log10(1.0 / c["tol"]) / c["eta"])


def _columns(c):
    n = _size(c)[0]
    return {"forces": n, "csc": n * c.get("scf", 1), "vjp": 8 * c.get("atoms", 1),
            "batch": c.get("cols", 0) * c.get("boxes", 1)}.get(c["kind"], c.get("cols", 0))


def _flops(c):
    """H and S are real, and so is every right-hand side: products of real matrices with real Krylov vectors, INNER_STEPS
    products with S and one with H per column and outer iteration (a batch column meets its own box only), and the
    complex updates of the shifted quantities that are kept."""
    n, nnz = _size(c)
    b = c.get("boxes", 1)
    cols, it = _columns(c), _outer(c)
    kept = {"full": n, "vjp": n, "green": c.get("rows", 1), "forces": 68, "lanczos": 0}.get(c["kind"], 1)
    return cols * it * ((INNER_STEPS + 1) * 2.0 * nnz / b + 16.0 * kept * c.get("shifts", 0))


def work(case):
    n, nnz = _size(case)
    cols, k = _columns(case), case.get("shifts", case.get("points", 0))
    out = {"full": 16.0 * cols * k * n, "green": 16.0 * cols * k * case.get("rows", 1), "mulliken": 8.0 * cols,
           "batch": 8.0 * cols, "csc": 16.0 * _atoms(case) + 8.0 * _atoms(case) ** 2,
           "forces": 16.0 * nnz + 32.0 * nnz, "vjp": 16.0 * nnz,
           "lanczos": 16.0 * cols * k + 16.0 * cols * case.get("steps", 0)}[case["kind"]]
    return {"bytes": 16.0 * nnz + out, "flops": _flops(case)}


# ---- inputs -----------------------------------------------------------------
def _system(case, seed):
    if "cells" in case:
        cells = tuple(int(v) for v in case["cells"].split("x"))
        if case["kind"] in ("forces", "vjp"):
            # thermal motion that keeps the cutoff between the second and the third shell: every seed stores the same
            # number of entries, and so has gradients of the same length
            return tbinputs.si_system(cells, sigma=0.03, seed=seed, cutoff=4.17)
        return tbinputs.si_system(cells, sigma=0.05, seed=seed)
    return tbinputs.water_system(case["molecules"], seed=seed, excess_proton=case["kind"] == "batch")


def _boxes(case, seed):
    """Boxes of a ragged batch: from three quarters of the stated number of molecules up to it, each its own seed."""
    rng = np.random.default_rng(seed)
    return [tbinputs.water_system(int(rng.integers(3 * case["molecules"] // 4, case["molecules"] + 1)),
                                  seed=1000 * (seed % 100000) + i) for i in range(case["boxes"])]


def _grid(case):
    lo, hi = SI_WINDOW if "cells" in case else WATER_WINDOW
    x, w = np.polynomial.legendre.leggauss(case["shifts"])
    return lo + 0.5 * (hi - lo) * (x + 1.0) + 1j * case["eta"], 0.5 * (hi - lo) * w.astype(np.complex128)


def _pick(n, count, rng):
    return np.sort(rng.choice(n, min(n, count), replace=False)).astype(np.int32)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    st = {"kind": case["kind"]}
    opts = {"precision": 1 if case["precision"] == "mixed" else 0, "inner_tol": case["inner_tol"],
            "panel": case.get("panel", 0)}
    if "tol" in case:
        opts["tol"] = case["tol"]
    st["opts"] = tb.tb_default_opts(**opts)
    if case["kind"] == "batch":
        boxes = _boxes(case, seed)
        st["handle"] = tb.tb_create_batch(boxes)
        st["cols"] = np.concatenate([_pick(b.n_orb, case["cols"], rng) + int(o)
                                     for b, o in zip(boxes, st["handle"].orb_off)]).astype(np.int32)
        st["z"], st["w"] = _grid(case)
        return st
    s = _system(case, seed)
    st["handle"] = tb.tb_create_system(s)
    if case["kind"] == "lanczos":
        st["cols"] = _pick(s.n_orb, case["cols"], rng)
        st["steps"] = case["steps"]
        st["z"] = np.linspace(-25.0, 10.0, case["points"]) + 1j * case["eta"]
        return st
    st["z"], st["w"] = _grid(case)
    if case["kind"] in ("full", "green", "mulliken"):
        st["cols"] = _pick(s.n_orb, case["cols"], rng)
    if case["kind"] == "green":
        st["rows"] = np.concatenate([_pick(s.n_orb, case["rows"], rng) for _ in st["cols"]]).astype(np.int32)
        st["row_ptr"] = np.arange(len(st["cols"]) + 1, dtype=np.int64) * (len(st["rows"]) // len(st["cols"]))
    elif case["kind"] == "csc":
        st["gamma"] = torch.tensor(tbinputs.klopman_ohno_gamma(s), device="cuda")
        st["q_ref"] = torch.tensor(tbinputs.valence_populations(s), device="cuda")
        st["copts"] = tb.tb_default_csc_opts(max_scf=case["scf"], mix=0.3, scf_tol=1e-12)
    elif case["kind"] == "forces":
        st["n_values"] = len(s.S_vals)
        st["dS_dd"] = tbinputs.overlap_bond_derivatives(s)
    elif case["kind"] == "vjp":
        st["n_values"] = len(s.S_vals)
        st["v"] = _vjp_weights(case, s, rng)
    return st


def _vjp_weights(case, s, rng):
    v = np.zeros(s.n_orb)
    for a in rng.choice(s.n_atoms, case["atoms"], replace=False):
        v[4 * a:4 * a + 4] = rng.normal()
    return v


def run(state):
    k, h, opts = state["kind"], state["handle"], state["opts"]
    if k == "full":
        return tb.tb_shifted_cocg(h, state["z"], state["cols"], opts=opts)[0]
    if k == "green":
        return tb.tb_green_elements(h, state["z"], state["cols"], state["row_ptr"], state["rows"], opts=opts)[0]
    if k in ("mulliken", "batch"):
        return tb.tb_mulliken_orbital(h, state["z"], state["w"], state["cols"], G_S, opts=opts)[0]
    if k == "csc":
        q, dq, _ = tb.tb_csc_loop(h, state["z"], state["w"], state["gamma"], state["q_ref"], G_S, copts=state["copts"],
                                  opts=opts, allow_unconverged=True)
        return q, dq
    if k == "forces":
        e, gh, gs, _ = tb.tb_band_energy(h, state["z"], state["w"], G_S, opts=opts, n_values=state["n_values"])
        return e, gh, gs, tb.tb_forces(h, gh, gs, state["dS_dd"])
    if k == "vjp":
        gh, gs, _ = tb.tb_mulliken_vjp(h, state["z"], state["w"], state["v"], state["n_values"], G_S, opts=opts)
        return gh, gs
    a, b, norm = tb.tb_generalized_lanczos_batch(h, state["cols"], state["steps"], opts=opts)
    return a, b, norm, tb.tb_lanczos_green_batch(a, b, norm, state["z"])


# ---- the same in 64 bits, by dense linear algebra ---------------------------
def _entries(s):
    """Row and column orbital of every stored entry."""
    rows = np.repeat(np.arange(s.n_atoms), np.diff(s.brow_ptr))
    ni, nj = s.orb_per_atom[rows], s.orb_per_atom[s.bcol]
    off = np.concatenate([[0], np.cumsum(s.orb_per_atom)])
    size = ni.astype(np.int64) * nj
    blk = np.repeat(np.arange(len(size)), size)
    inside = np.arange(size.sum()) - np.repeat(np.cumsum(size) - size, size)
    return off[rows[blk]] + inside // nj[blk], off[s.bcol[blk]] + inside % nj[blk], rows[blk], s.bcol[blk]


def _dense(s):
    a, b, ia, ib = (torch.tensor(v, device="cuda") for v in _entries(s))
    sv = torch.tensor(s.S_vals, device="cuda")
    e = torch.tensor(s.eps, device="cuda")
    hv = torch.where(ia == ib, torch.where(a == b, e[a], torch.zeros_like(sv)), 0.5 * s.K * (e[a] + e[b]) * sv)
    S = torch.zeros(s.n_orb, s.n_orb, dtype=torch.float64, device="cuda")
    H = torch.zeros_like(S)
    S[a, b] = sv
    H[a, b] = hv
    return H, S, a, b


def _modes(H, S):
    """Levels and S-orthonormal modes: G(z) = U diag(1 / (z - level)) U^T."""
    L = torch.linalg.cholesky(S)
    A = torch.linalg.solve_triangular(L, H, upper=False)
    A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
    lev, V = torch.linalg.eigh(0.5 * (A + A.T))
    return lev, torch.linalg.solve_triangular(L.T.contiguous(), V, upper=True)


def _filled(lev, z, w, power=1, with_z=0):
    """-(g_s / pi) Im sum_k w_k z_k^with_z / (z_k - level)^power for every level."""
    zt, wt = torch.tensor(z, device="cuda"), torch.tensor(w, device="cuda")
    return -(G_S / math.pi) * ((wt * zt ** with_z)[:, None] / (zt[:, None] - lev[None, :]) ** power).sum(0).imag


def _populations(H, S, z, w):
    lev, U = _modes(H, S)
    return ((U * (S @ U)) * _filled(lev, z, w)[None, :]).sum(1)


def exact(case, seed):
    k = case["kind"]
    if k == "mulliken" and _size(case)[0] > 2600:
        return None          # the dense eigenproblem of a larger crystal takes minutes
    rng = np.random.default_rng(seed)
    if k == "batch":
        z, w = _grid(case)
        out = []
        for s in _boxes(case, seed):
            H, S, _, _ = _dense(s)
            out.append(_populations(H, S, z, w)[torch.tensor(_pick(s.n_orb, case["cols"], rng).astype(np.int64), device="cuda")])
        return torch.cat(out)
    s = _system(case, seed)
    H, S, a, b = _dense(s)
    if k == "lanczos":
        return _exact_lanczos(case, s, H, S, rng)
    z, w = _grid(case)
    if k in ("full", "green", "mulliken"):
        cols = torch.tensor(_pick(s.n_orb, case["cols"], rng).astype(np.int64), device="cuda")
        if k == "mulliken":
            return _populations(H, S, z, w)[cols]
        lev, U = _modes(H, S)
        zt = torch.tensor(z, device="cuda")
        Uc = U.to(torch.complex128)
        x = torch.stack([Uc @ (Uc[cols] / (zk - lev)[None, :]).T for zk in zt])      # [K][N][R]
        if k == "full":
            return x.transpose(1, 2).contiguous()
        rows = [torch.tensor(_pick(s.n_orb, case["rows"], rng).astype(np.int64), device="cuda") for _ in cols]
        return torch.cat([x[:, r, c].T for c, r in enumerate(rows)]).contiguous()
    if k == "csc":
        gamma = torch.tensor(tbinputs.klopman_ohno_gamma(s), device="cuda")
        q_ref = torch.tensor(tbinputs.valence_populations(s), device="cuda")
        atom = torch.tensor(np.repeat(np.arange(s.n_atoms), s.orb_per_atom), device="cuda")
        dq = torch.zeros(s.n_atoms, dtype=torch.float64, device="cuda")
        for i in range(case["scf"]):
            V = (gamma @ dq)[atom]
            q = torch.zeros_like(dq).index_add_(0, atom, _populations(H + 0.5 * S * (V[:, None] + V[None, :]), S, z, w))
            if i + 1 < case["scf"]:
                dq = dq + 0.3 * ((q - q_ref) - dq)
        return q, dq
    lev, U = _modes(H, S)
    if k == "vjp":
        v = torch.tensor(_vjp_weights(case, s, rng), device="cuda")
        zt, wt = torch.tensor(z, device="cuda"), torch.tensor(w, device="cuda")
        inv = 1.0 / (zt[:, None] - lev[None, :])
        c = (U.T @ S * v[None, :]) @ U
        f = -G_S / math.pi
        m0 = f * (inv.T @ (wt[:, None] * inv)).imag
        m1 = f * (inv.T @ ((wt * zt)[:, None] * inv)).imag
        rho = (U * _filled(lev, z, w)[None, :]) @ U.T
        return (U @ (c * m0) @ U.T)[b, a], v[b] * rho[b, a] - (U @ (c * m1) @ U.T)[b, a]
    rows = lambda f: ((U * f[None, :]) @ U.T)[a, b]  # noqa: E731
    e = float(_filled(lev, z, w, 1, 1).sum())
    gh = rows(_filled(lev, z, w, 2, 1))
    gs = rows(_filled(lev, z, w, 1, 1) - _filled(lev, z, w, 2, 2))
    ds = torch.tensor(tbinputs.overlap_bond_derivatives(s), device="cuda").reshape(3, -1)
    eps = torch.tensor(s.eps, device="cuda")
    _, _, ia, ib = (torch.tensor(x, device="cuda") for x in _entries(s))
    val = torch.where(ia == ib, torch.zeros_like(gs), gs + 0.5 * s.K * (eps[a] + eps[b]) * gh) * ds
    F = torch.zeros(s.n_atoms, 3, dtype=torch.float64, device="cuda")
    F.index_add_(0, ia.long(), val.T.contiguous())
    F.index_add_(0, ib.long(), -val.T.contiguous())
    return e, gh, gs, F


def _exact_lanczos(case, s, H, S, rng):
    cols = torch.tensor(_pick(s.n_orb, case["cols"], rng).astype(np.int64), device="cuda")
    L = torch.linalg.cholesky(S)
    rhs = torch.zeros(s.n_orb, len(cols), dtype=torch.float64, device="cuda")
    rhs[cols, torch.arange(len(cols), device="cuda")] = 1.0
    u = torch.cholesky_solve(rhs, L)
    norm = (u * rhs).sum(0)
    u = u / norm.sqrt()
    n = case["steps"]
    av, bv = torch.zeros(len(cols), n, dtype=torch.float64, device="cuda"), torch.zeros(len(cols), n + 1, dtype=torch.float64, device="cuda")
    up = torch.zeros_like(u)
    for i in range(n):
        y = H @ u
        av[:, i] = (u * y).sum(0)
        wv = torch.cholesky_solve(y, L) - av[:, i] * u - bv[:, i] * up
        bv[:, i + 1] = (wv * (S @ wv)).sum(0).sqrt()
        up, u = u, wv / bv[:, i + 1]
    z = torch.tensor(np.linspace(-25.0, 10.0, case["points"]) + 1j * case["eta"], device="cuda")
    g = torch.zeros(len(cols), len(z), dtype=torch.complex128, device="cuda")
    for i in range(n - 1, -1, -1):
        tail = bv[:, i + 1, None] ** 2 * g if i + 1 < n else 0.0
        g = 1.0 / (z[None, :] - av[:, i, None] - tail)
    return av, bv, norm, norm[:, None] * g
