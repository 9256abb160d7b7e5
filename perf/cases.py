"""The work that users of this library have it do, as measurable cases.

Every case goes through the package's public calls.  The systems are the two
families the library is made for, drawn here from a seed: 4-orbital chains and
PPV-like polymer chains and bundles (14 atoms, 38 orbitals per monomer) with
distance-decay tight-binding elements.  Solves run to a tolerance of 1e-10 or
below, so that their outputs are the solution and not the point at which an
iteration happened to stop.  The geometry (and so the sparsity pattern and the
columns asked for) belongs to the case; the seed draws the matrix elements.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1603_09616_gb300 as gbg
from paper_1603_09616_gb300 import surrogate as sg

R0 = 0.14  # nm, the reference bond length of the decay rules
REPEAT = 0.66  # nm, monomer repeat


# ------------------------------------------------------------------ systems
def _pattern_of(norb, a, b, d, pos=None):
    """Shared CSR pattern of H and S from atoms and interacting pairs at reduced distance d,
    with the places that the drawn elements go to."""
    norb = np.asarray(norb, np.int64)
    first = np.concatenate([[0], np.cumsum(norb)])
    n = int(first[-1])
    cnt = norb[a] * norb[b]
    pid = np.repeat(np.arange(len(a)), cnt)
    loc = np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    r = first[a[pid]] + loc // norb[b[pid]]
    c = first[b[pid]] + loc % norb[b[pid]]
    con = norb * norb
    aid = np.repeat(np.arange(len(norb)), con)
    lo = np.arange(int(con.sum())) - np.repeat(np.cumsum(con) - con, con)
    ro, co = first[aid] + lo // norb[aid], first[aid] + lo % norb[aid]
    rows = np.concatenate([ro, r, c])
    cols = np.concatenate([co, c, r])
    order = np.argsort(rows * n + cols)
    rows, cols = rows[order], cols[order]
    rp = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=rp[1:])
    return SimpleNamespace(n=n, row_ptr=rp, col_idx=cols.astype(np.int32), rows=rows, order=order, on=rows == cols,
                           onsite=np.where(ro == co, ro, -1), decay=np.exp(-d[pid]),
                           orb_atom=np.repeat(np.arange(len(norb)), norb).astype(np.int32), positions=pos,
                           atom_norb=norb.astype(np.int32))


def _fill(p, rng):
    """A system on the pattern p: random onsite energies, couplings that decay with distance."""
    h = -2.7 * math.e * p.decay * rng.uniform(0.5, 1.0, len(p.decay))
    s = 0.1 * p.decay * rng.uniform(0.0, 1.0, len(p.decay))
    e = rng.standard_normal(p.n)
    hv = np.concatenate([np.where(p.onsite >= 0, e[p.onsite], 0.0), h, h])[p.order]
    sv = np.concatenate([(p.onsite >= 0).astype(float), s, s])[p.order]
    off = np.bincount(p.rows, np.where(p.on, 0.0, np.abs(sv)), p.n)
    sv[p.on] = np.maximum(1.0, 1.01 * off)
    return SimpleNamespace(n=p.n, row_ptr=p.row_ptr, col_idx=p.col_idx, h_val=hv, s_val=sv, orb_atom=p.orb_atom,
                           positions=p.positions, atom_norb=p.atom_norb)


@functools.lru_cache(maxsize=4)
def _chain4(sites):
    """Chain of 4-orbital sites, sites up to three apart couple."""
    a = np.concatenate([np.arange(sites - k) for k in (1, 2, 3) if sites > k])
    d = np.concatenate([np.full(sites - k, float(k)) for k in (1, 2, 3) if sites > k])
    return _pattern_of(np.full(sites, 4), a, a + d.astype(np.int64), d)


def _monomers(mono):
    """Positions and orbital counts of a planar PPV-like chain along x.  Odd
    monomers start with two hydrogens, so every carbon's four orbitals fill one
    aligned 4x4 block."""
    t = np.deg2rad(np.arange(0, 360, 60))
    ring = np.stack([0.14 * np.cos(t), 0.14 * np.sin(t), 0 * t], 1)
    hyd = np.stack([0.248 * np.cos(t), 0.248 * np.sin(t), 0 * t], 1)[[2, 4, 1, 5]]
    car = np.vstack([ring, [[0.265, 0.035, 0], [0.395, -0.035, 0]]])
    hyd = np.vstack([hyd, [[0.250, 0.140, 0], [0.410, -0.140, 0]]])
    pos, norb = [], []
    for m in range(mono):
        k = 2 * (m & 1)
        pos.append(np.vstack([hyd[:k], car, hyd[k:]]) + [m * REPEAT, 0.0, 0.0])
        norb += [1] * k + [4] * 8 + [1] * (6 - k)
    return np.vstack(pos), np.array(norb)


def _pairs(pos, cutoff):
    """Atom pairs a < b within the cutoff (a window along the sorted x axis)."""
    o = np.argsort(pos[:, 0], kind="stable")
    x = pos[o]
    hi = np.searchsorted(x[:, 0], x[:, 0] + cutoff, "right")
    w = hi - np.arange(len(x)) - 1
    i = np.repeat(np.arange(len(x)), w)
    j = i + 1 + np.arange(int(w.sum())) - np.repeat(np.cumsum(w) - w, w)
    r = np.sqrt(((x[i] - x[j]) ** 2).sum(1))
    k = r < cutoff
    p, q = o[i[k]], o[j[k]]
    a, b, r = np.minimum(p, q), np.maximum(p, q), r[k]
    s = np.lexsort((b, a))
    return a[s], b[s], r[s]


def _ppv(mono, place=0):
    """One chain, 2 % positional disorder, 0.4 nm cutoff (a banded S)."""
    rng = np.random.default_rng([mono, place, 1])
    pos, norb = _monomers(mono)
    pos = pos + rng.normal(0.0, 0.02 * R0, pos.shape)
    a, b, r = _pairs(pos, 0.4)
    return _pattern_of(norb, a, b, r / R0, pos)


@functools.lru_cache(maxsize=4)
def _bundle(side, mono, place=0):
    """side x side chains 0.45 nm apart, randomly turned and shifted, 0.5 nm cutoff (S is not banded)."""
    rng = np.random.default_rng([side, mono, place, 2])
    chain, norb = _monomers(mono)
    pos = []
    for y in range(side):
        for z in range(side):
            t, dx = rng.uniform(0, 2 * np.pi), rng.uniform(0, REPEAT)
            rot = np.array([[1, 0, 0], [0, np.cos(t), -np.sin(t)], [0, np.sin(t), np.cos(t)]])
            pos.append(chain @ rot.T + [dx, 0.45 * y, 0.45 * z])
    pos = np.vstack(pos)
    pos = pos + rng.normal(0.0, 0.05, pos.shape)
    a, b, r = _pairs(pos, 0.5)
    return _pattern_of(np.tile(norb, side * side), a, b, r / R0, pos)


def _grid(k, eta, lo=-15.0, hi=10.0):
    return np.linspace(lo, hi, k) + 1j * eta if k > 1 else np.array([0.5 * (lo + hi) + 1j * eta])


def _fermi(z, kT=0.1):
    """Real-axis density and energy-density weights at mu = 0."""
    e = z.real
    c = -(2.0 / np.pi) * 0.5 * (1.0 - np.tanh(e / (2 * kT))) * ((e[-1] - e[0]) / max(len(e) - 1, 1))
    return c.astype(complex), (e * c).astype(complex)


def _poles(p, kT):
    """Poles and weights of the Fermi function's continued fraction (spin 2, mu = 0)."""
    m = np.arange(1, 2 * p)
    t = 1.0 / (2.0 * np.sqrt((2 * m - 1.0) * (2 * m + 1.0)))
    b, v = np.linalg.eigh(np.diag(t, 1) + np.diag(t, -1))
    k = b > 0
    a, r = 1.0 / b[k], -v[0, k] ** 2 / (4.0 * b[k] ** 2)
    o = np.argsort(a)
    z = 1j * kT * a[o]
    c = -4.0 * kT * r[o] * 1j
    return z, c, c * z, 1.0, 4.0 * kT * float(r.sum()), 1.0


def _gradients(s):
    """Per-element gradients of H and S with respect to the row atom's position."""
    ai = s.orb_atom[np.repeat(np.arange(s.n), np.diff(s.row_ptr))]
    aj = s.orb_atom[s.col_idx]
    d = s.positions[ai] - s.positions[aj]
    r = np.sqrt((d * d).sum(1))
    u = np.where((ai != aj)[:, None], d / np.where(r > 0, r, 1.0)[:, None], 0.0) / -R0
    return np.ascontiguousarray((s.h_val[:, None] * u).T), np.ascontiguousarray((s.s_val[:, None] * u).T)


def _cols(n, count):
    rng = np.random.default_rng([n, count])
    return np.arange(n, dtype=np.int32) if count >= n else np.sort(rng.choice(n, count, replace=False)).astype(np.int32)


# ------------------------------------------------------------------ cases
def listed():
    return [
        # a quick look at a short chain (48 orbitals, FP64): launches and latency count
        dict(name="solve fp64 48", kind="solve", sites=12, shifts=16, eta=0.2, cols=16, tol=1e-12, prec="fp64"),
        # the plain FP64 solve of a whole 4-orbital chain
        dict(name="solve fp64 480", kind="solve", sites=120, shifts=64, eta=0.1, cols=480, tol=1e-10, prec="fp64"),
        # all columns of a PPV chain on a real-axis grid, then mu from the electron count (mixed precision)
        dict(name="fermi 608", kind="fermi", mono=16, shifts=96, eta=0.25, kT=0.1, tol=1e-10),
        # an MD step: pole expansion on a chain, all columns, the S^-1 terms, the forces
        dict(name="md step 912", kind="md", mono=24, poles=40, kT=0.1, tol=1e-10),
        # local DOS of some orbitals of the 1900-orbital chain: few columns
        dict(name="sampled 1900", kind="solve", mono=50, shifts=128, eta=0.4, cols=24, tol=1e-10, prec="mixed"),
        # uneven chains, each with its own shifts and a few columns, in one launch
        dict(name="batch 96", kind="batch", systems=96, max_mono=32, cols=8, eta=0.3, tol=1e-10, prec="mixed"),
        # labels for the surrogate: all columns of small bundles (S not banded: the iterative inner solve)
        dict(name="labels 2x456", kind="labels", systems=2, side=2, mono=3, shifts=48, eta=0.4, tol=1e-10),
        # the sparse product alone, as a user's own iteration calls it: one column, and a block of eight
        dict(name="spmm fp32 w1", kind="spmm", side=5, mono=25, which=0, w=1, prec="fp32"),
        dict(name="spmm fp64 w8", kind="spmm", side=6, mono=30, which=0, w=8, prec="fp64"),
        # hole wavepackets on the 1900-orbital chain, 0.1 fs steps
        dict(name="wavepacket 1900", kind="wave", mono=50, packets=32, steps=10),
        # one Adam step of the surrogate at its usual batch
        dict(name="train 2048", kind="train", batch=2048),
        # surrogate inference on a bundle: descriptors of every orbital, then the network
        dict(name="infer 3420", kind="infer", side=3, mono=10),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve64", "solve", "fermi", "md", "batch", "labels", "spmm", "spmm", "wave", "train", "infer"])
    if kind == "solve64":
        s = log(5, 100)
        return dict(kind="solve", sites=s, shifts=rng.randint(1, 96), eta=rng.uniform(0.1, 0.4), cols=log(1, 4 * s),
                    tol=rng.choice([1e-10, 1e-11, 1e-12]), prec="fp64")
    if kind == "solve":
        m = log(2, 20)
        return dict(kind="solve", mono=m, shifts=rng.randint(1, 160), eta=rng.uniform(0.2, 0.5), cols=log(1, 38 * m),
                    tol=1e-10, prec=rng.choice(["mixed", "mixed", "fp64"]))
    if kind == "fermi":
        return dict(kind="fermi", mono=log(2, 15), shifts=rng.randint(64, 128), eta=rng.uniform(0.25, 0.4),
                    kT=rng.uniform(0.1, 0.3), tol=1e-10)
    if kind == "md":
        return dict(kind="md", mono=log(2, 22), poles=rng.randint(24, 40), kT=rng.uniform(0.1, 0.2), tol=1e-10)
    if kind == "batch":
        return dict(kind="batch", systems=log(4, 90), max_mono=log(4, 28), cols=rng.randint(2, 8),
                    eta=rng.uniform(0.3, 0.5), tol=1e-10, prec=rng.choice(["mixed", "mixed", "fp64"]))
    if kind == "labels":
        return dict(kind="labels", systems=rng.randint(1, 2), side=2, mono=rng.randint(1, 3), shifts=rng.randint(16, 48),
                    eta=rng.uniform(0.4, 0.6), tol=1e-10)
    if kind == "spmm":
        return dict(kind="spmm", side=rng.randint(2, 6), mono=rng.randint(3, 30), which=rng.randint(0, 1),
                    w=rng.choice([1, 1, 2, 4, 8, 16, 32, 64, 3, 12]), prec=rng.choice(["fp32", "fp32", "fp64"]))
    if kind == "wave":
        return dict(kind="wave", mono=log(4, 50), packets=log(1, 32), steps=rng.randint(1, 10))
    if kind == "train":
        return dict(kind="train", batch=log(64, 4096))
    return dict(kind="infer", side=rng.randint(1, 4), mono=rng.randint(4, 12))


def _build(case, seed):
    """Host inputs of a case: the same for prepare() and exact()."""
    rng = np.random.default_rng([seed, 1603])
    k = case["kind"]
    c = SimpleNamespace(rng=rng)
    if k == "solve":
        c.sys = _fill(_chain4(case["sites"]) if "sites" in case else _ppv(case["mono"]), rng)
        c.z = _grid(case["shifts"], case["eta"], *((-12.0, 12.0) if "sites" in case else (-15.0, 10.0)))
        c.wr, c.we = _fermi(c.z)
        c.cols = _cols(c.sys.n, case["cols"])
    elif k == "fermi":
        c.sys = _fill(_ppv(case["mono"]), rng)
        c.z = _grid(case["shifts"], case["eta"])
        c.cols = np.arange(c.sys.n, dtype=np.int32)
        c.nel = 1.0 * c.sys.n
    elif k == "md":
        c.sys = _fill(_ppv(case["mono"]), rng)
        c.z, c.wr, c.we, c.a, c.b, c.c = _poles(case["poles"], case["kT"])
        c.cols = np.arange(c.sys.n, dtype=np.int32)
        c.gh, c.gs = _gradients(c.sys)
        c.atom_off = np.concatenate([[0], np.cumsum(c.sys.atom_norb)]).astype(np.int64)
    elif k in ("batch", "labels"):
        c.sys, c.prob = [], []
        size = np.random.default_rng(case["systems"])
        for q in range(case["systems"]):
            if k == "batch":
                s = _fill(_ppv(int(size.integers(2, case["max_mono"] + 1)), q), rng)
                z = _grid(int(size.integers(32, 257)), case["eta"])
                cols = _cols(s.n, case["cols"])
            else:
                s = _fill(_bundle(case["side"], case["mono"], q), rng)
                z = _grid(case["shifts"], case["eta"])
                cols = np.arange(s.n, dtype=np.int32)
            wr, we = _fermi(z)
            c.sys.append(s)
            c.prob.append(dict(z=z, cols=cols, w_rho=wr, w_edm=we, tol=case["tol"], maxit=6000))
    elif k == "spmm":
        c.sys = _fill(_bundle(case["side"], case["mono"]), rng)
        c.x = rng.standard_normal((c.sys.n, case["w"])) + 1j * rng.standard_normal((c.sys.n, case["w"]))
    elif k == "wave":
        c.sys = _fill(_ppv(case["mono"]), rng)
        x = rng.standard_normal((c.sys.n, case["packets"])) + 1j * rng.standard_normal((c.sys.n, case["packets"]))
        c.psi = x / np.sqrt((np.abs(x) ** 2).sum(0))
        c.tau = 0.1 / 0.6582119569  # 0.1 fs in hbar / eV
    elif k == "train":
        c.x = rng.standard_normal((case["batch"], 64)).astype(np.float32)
        c.t = (np.tanh(c.x[:, :2]) + 0.1 * rng.standard_normal((case["batch"], 2))).astype(np.float32)
    elif k == "infer":
        c.sys = _fill(_bundle(case["side"], case["mono"]), rng)
    return c


def prepare(case, seed):
    c = _build(case, seed)
    k = case["kind"]
    dev = torch.device("cuda")
    if k in ("solve", "fermi", "md", "spmm", "wave", "infer"):
        c.mat = gbg.Matrix(c.sys)
    if k in ("batch", "labels"):
        c.mats = [gbg.Matrix(s) for s in c.sys]
    if k == "spmm":
        c.x = torch.as_tensor(c.x, device=dev).to(torch.complex64 if case["prec"] == "fp32" else torch.complex128)
    if k == "md":
        c.gh, c.gs = torch.as_tensor(c.gh, device=dev), torch.as_tensor(c.gs, device=dev)
    if k == "wave":
        lam = _modes(c.sys)[0]
        c.lo, c.hi = float(lam[0]) - 0.2, float(lam[-1]) + 0.2
        c.psi = torch.as_tensor(c.psi, device=dev)
    if k == "train":
        c.net = sg.MLP(seed=int(seed) % 1000)
        c.x, c.t = torch.as_tensor(c.x, device=dev), torch.as_tensor(c.t, device=dev)
    if k == "infer":
        # standardisation as a fit on this kind of data leaves it
        c.sur = sg.Surrogate(seed=int(seed) % 1000)
        x = torch.as_tensor(_descriptors(c.sys), device=dev)
        m, s = x.mean(0), x.std(0)
        s = torch.where(s > 1e-3, s, torch.ones_like(s))
        c.sur.x_scale, c.sur.x_shift = (1 / s).float(), (-m / s).float()
        c.sur.y_scale, c.sur.y_shift = torch.tensor([0.3, 0.7], device=dev), torch.tensor([1.0, -1.5], device=dev)
    c.case = case
    return c


_OUT = ("ldos", "rho", "edm", "q", "e_loc", "converged")


def run(c):
    k, case = c.case["kind"], c.case
    if k == "solve":
        r = gbg.shifted_solve(c.mat, c.z, c.cols, tol=case["tol"], maxit=6000, prec=case["prec"], w_rho=c.wr, w_edm=c.we)
        return {f: r[f] for f in _OUT}
    if k == "fermi":
        r = gbg.shifted_solve(c.mat, c.z, c.cols, tol=case["tol"], maxit=4000, prec="mixed", want_g=True)
        d = gbg.fermi_density(c.mat, c.z, c.cols, r, c.nel, case["kT"])
        return dict(g=r["g_proj"], ldos=r["ldos"], converged=r["converged"], mu=d["mu"],
                    **{f: d[f] for f in ("rho", "edm", "q", "e_loc")})
    if k == "md":
        r = gbg.shifted_solve(c.mat, c.z, c.cols, tol=case["tol"], maxit=4000, prec="mixed", w_rho=c.wr, w_edm=c.we)
        gbg.add_sinv_terms(c.mat, c.cols, r, c.a, c.b, c.c)
        f = gbg.forces(c.mat, c.cols, r["rho"], r["edm"], c.gh, c.gs, c.atom_off)
        return dict(forces=f, **{x: r[x] for x in ("rho", "edm", "q", "e_loc", "converged")})
    if k in ("batch", "labels"):
        res, _ = gbg.shifted_solve_batched(c.mats, c.prob, prec=case.get("prec", "mixed"))
        return {f: torch.cat([r[f].reshape(-1) for r in res]) for f in _OUT}
    if k == "spmm":
        return c.mat.spmm(case["which"], c.x, prec=case["prec"])
    if k == "wave":
        return gbg.wavepacket(c.mat, c.psi.clone(), case["steps"], c.tau, c.lo, c.hi)[0]
    if k == "train":
        loss = c.net.train_step(c.x, c.t, lr=2e-3)
        return dict(loss=loss.sum(), w=c.net.w, b=c.net.b, gw=c.net.gw, gb=c.net.gb)
    x = sg.descriptors(c.mat, c.sys)
    return dict(x=x, y=c.sur.predict(x))


# ------------------------------------------------------------------ least work
def _sizes(case):
    """Orbitals and pattern entries of one system, near enough."""
    if "sites" in case:
        n = 4 * case["sites"]
        return n, 28 * n
    mono = case.get("mono", case.get("max_mono", 2) // 2 + 1)
    side = case.get("side", 1)
    n = 38 * mono * side * side
    return n, (42 if case["kind"] not in ("spmm", "labels", "infer") else 130 if side > 3 else 95) * n


def work(case):
    k = case["kind"]
    if k == "train":
        p, b = 64 * 128 + 2 * 128 * 128 + 128 * 2, case["batch"]
        return dict(bytes=4.0 * b * 66 + 32.0 * p, flops=6.0 * b * p)
    n, nnz = _sizes(case)
    if k == "spmm":
        v = 4 if case["prec"] == "fp32" else 8
        return dict(bytes=float((v + 4) * nnz + 4 * v * n * case["w"]), flops=4.0 * nnz * case["w"])
    if k == "infer":
        return dict(bytes=20.0 * nnz + 4.0 * n * 66, flops=2.0 * n * 41216 + 60.0 * nnz)
    band = 55  # half-bandwidth of S on the chains
    if k == "wave":  # per term: one product with H and one factor solve
        terms = 26 * case["steps"] * case["packets"]
        return dict(bytes=32.0 * n * case["packets"] + 16.0 * nnz, flops=terms * (4.0 * nnz + 8.0 * n * band))
    systems = case.get("systems", 1)
    cols = n if k in ("fermi", "md", "labels") else min(case["cols"], n)
    shifts = case.get("shifts", case.get("poles", 128))
    eta = case.get("eta", math.pi * case.get("kT", 0.1))
    # the Krylov space a column needs: half the spectrum's width over eta, per e-fold of the residual
    its = min(float(n), 8.0 / eta * math.log(1.0 / case["tol"]))
    inner = 2.0 * nnz * 10 if k == "labels" else 4.0 * n * min(band, n)
    return dict(bytes=systems * (20.0 * nnz + 8.0 * cols * (shifts + 2 * nnz / n)),
                flops=systems * cols * its * (2.0 * nnz + inner + 8.0 * n + 10.0 * shifts))


# ------------------------------------------------------------------ the same answers in 64 bits
def _dense(s):
    rows = np.repeat(np.arange(s.n), np.diff(s.row_ptr))
    h, o = np.zeros((s.n, s.n)), np.zeros((s.n, s.n))
    h[rows, s.col_idx], o[rows, s.col_idx] = s.h_val, s.s_val
    return torch.as_tensor(h), torch.as_tensor(o)


def _modes(s):
    """Generalized eigenvalues and S-orthonormal vectors of H y = lambda S y."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    h, o = (t.to(dev) for t in _dense(s))
    c = torch.linalg.cholesky(o)
    a = torch.linalg.solve_triangular(c, torch.linalg.solve_triangular(c, h, upper=False).T, upper=False)
    lam, q = torch.linalg.eigh(0.5 * (a + a.T))
    return lam.cpu().numpy(), torch.linalg.solve_triangular(c.T, q, upper=True).cpu().numpy()


def _entries(s, cols):
    """(orbital i, column j, CSR position) of the packed pattern entries of the columns."""
    m = s.row_ptr[cols + 1] - s.row_ptr[cols]
    e = np.arange(int(m.sum())) - np.repeat(np.cumsum(m) - m, m) + np.repeat(s.row_ptr[cols], m)
    return s.col_idx[e], np.repeat(cols, m), e, np.repeat(np.arange(len(cols)), m)


def _pattern(y, i, j, f):
    """sum_l y_il y_jl f_l(.) for each pattern entry; f: [modes] or [modes, k]."""
    out = [(y[i[a:a + 16384]] * y[j[a:a + 16384]]) @ f for a in range(0, len(i), 16384)]
    return np.concatenate(out)


def _local(s, cols, rho):
    _, _, e, at = _entries(s, cols)
    return np.bincount(at, rho * s.s_val[e], len(cols)), np.bincount(at, rho * s.h_val[e], len(cols))


def _outputs(s, z, cols, wr, we):
    lam, y = _modes(s)
    i, j, e, at = _entries(s, cols)
    g = 1.0 / (z[None, :] - lam[:, None])
    rho, edm = _pattern(y, i, j, np.stack([(g @ wr).imag, (g @ we).imag], 1)).T
    sy = np.stack([np.bincount(at, s.s_val[e] * y[i, l], len(cols)) for l in range(s.n)], 1)  # (S y_l)_j
    ldos = -(sy * y[cols] @ g.imag).T / np.pi
    q, el = _local(s, cols, rho)
    return dict(ldos=ldos, rho=rho, edm=edm, q=q, e_loc=el)


def _descriptors(s):
    """The 64 environment features of every orbital, in 64 bits."""
    n, rp = s.n, s.row_ptr
    j = np.repeat(np.arange(n), np.diff(rp))
    i = s.col_idx.astype(np.int64)
    first = np.concatenate([[0], np.cumsum(s.atom_norb)])[:-1]
    h, o = s.h_val, s.s_val
    pos = s.positions.astype(np.float32).astype(np.float64)
    dg = np.zeros(n)
    dg[j[i == j]] = h[i == j]
    sd = np.zeros(n)
    sd[j[i == j]] = o[i == j]
    f = np.zeros((n, 64))
    nb = i != j
    J, hji, sji, hii = j[nb], h[nb], o[nb], dg[i[nb]]
    add = lambda w, at=J: np.bincount(at, w, n)  # noqa: E731
    f[:, 46], f[:, 47] = dg, sd
    for t in range(8):
        f[:, 48 + t] = add(hji ** 2 * np.exp(-((hii - (-3.0 + 6.0 * t / 7.0)) / 0.75) ** 2))
    f[:, 56], f[:, 57], f[:, 58], f[:, 59] = add(hji ** 2), add(sji ** 2), add(hji * sji), add(hji ** 2 * hii)
    f[:, 60], f[:, 62] = add(np.abs(hji)), add(sji * hii)
    a, b = s.orb_atom[j], s.orb_atom[i]
    d = pos[b] - pos[a]
    r = np.sqrt((d * d).sum(1))
    k = (a != b) & (i == first[b]) & (r > 1e-6) & (r < 0.5)
    J, r, u, hyd = j[k], r[k], d[k] / r[k][:, None], (s.atom_norb[b[k]] == 1)
    w = 0.5 * (np.cos(np.pi * r / 0.5) + 1.0)
    for t in range(16):
        g = w * np.exp(-((r - (0.1 + 0.4 * t / 15.0)) / 0.03) ** 2)
        f[:, t], f[:, 16 + t] = add(g * ~hyd, J), add(g * hyd, J)
    sh = np.minimum(3, (r / 0.125).astype(int))
    for q in range(4):
        m = w * (sh == q)
        f[:, 32 + 2 * q] = sum(add(m * u[:, x], J) ** 2 for x in range(3))
        f[:, 33 + 2 * q] = sum((1 if x == y else 2) * add(m * (u[:, x] * u[:, y] - (x == y) / 3.0), J) ** 2
                               for x in range(3) for y in range(x, 3))
    at = s.orb_atom
    f[np.arange(n), 40 + (s.atom_norb[at] == 1)] = 1.0
    f[np.arange(n), 42 + np.minimum(3, np.arange(n) - first[at])] = 1.0
    f[:, 61] = np.diff(rp) / 100.0
    f[:, 63] = 1.0
    return f


def _net(seed, dims=(64, 128, 128, 128, 2)):
    rng = np.random.default_rng(seed)
    return [torch.as_tensor(rng.normal(0.0, np.sqrt((2.0 if l < 3 else 1.0) / dims[l]),
                                       (dims[l + 1], dims[l])).astype(np.float32)) for l in range(4)]


def exact(case, seed):
    k = case["kind"]
    c = _build(case, seed)
    if k == "solve":
        return dict(_outputs(c.sys, c.z, c.cols, c.wr, c.we), converged=None)
    if k == "fermi":
        lam, y = _modes(c.sys)
        i, j, e, at = _entries(c.sys, c.cols)
        g = 1.0 / (c.z[None, :] - lam[:, None])
        G = (_pattern(y, i, j, g.real) + 1j * _pattern(y, i, j, g.imag)).T
        ldos = np.stack([np.bincount(at, -row * c.sys.s_val[e] / np.pi, c.sys.n) for row in G.imag])
        eps, d, kT = c.z.real, (c.z.real[-1] - c.z.real[0]) / (len(c.z) - 1), case["kT"]
        dos = ldos.sum(1)
        fermi = lambda mu: 0.5 * (1.0 - np.tanh((eps - mu) / (2 * kT)))  # noqa: E731
        lo, hi = eps[0] - 40 * kT, eps[-1] + 40 * kT
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if (2.0 * d * fermi(mid) * dos).sum() < c.nel else (lo, mid)
        mu = 0.5 * (lo + hi)
        w = -(2.0 / np.pi) * fermi(mu) * d
        rho, edm = w @ G.imag, (eps * w) @ G.imag
        q, el = _local(c.sys, c.cols, rho)
        return dict(g=G, ldos=ldos, converged=None, mu=mu, rho=rho, edm=edm, q=q, e_loc=el)
    if k == "md":
        lam, y = _modes(c.sys)
        i, j, e, _ = _entries(c.sys, c.cols)
        g = 1.0 / (c.z[None, :] - lam[:, None])
        rho, edm = _pattern(y, i, j, np.stack([(g @ c.wr).imag + c.a, (g @ c.we).imag + c.b + c.c * lam], 1)).T
        q, el = _local(c.sys, c.cols, rho)
        s = c.sys  # every column in order: the packed entries are the CSR's, both orders of an element are equal
        inter = s.orb_atom[i] != s.orb_atom[j]
        f = [np.bincount(s.orb_atom[j], inter * (2 * edm * c.gs[x] - 2 * rho * c.gh[x])) for x in range(3)]
        return dict(forces=np.stack(f, 1), rho=rho, edm=edm, q=q, e_loc=el, converged=None)
    if k in ("batch", "labels"):
        out = [_outputs(s, p["z"], p["cols"], p["w_rho"], p["w_edm"]) for s, p in zip(c.sys, c.prob)]
        return dict({f: np.concatenate([o[f].reshape(-1) for o in out]) for f in _OUT[:-1]}, converged=None)
    if k == "spmm":
        rows = np.repeat(np.arange(c.sys.n), np.diff(c.sys.row_ptr))
        v = c.sys.s_val if case["which"] else c.sys.h_val
        x = c.x.astype(np.complex64).astype(np.complex128) if case["prec"] == "fp32" else c.x
        y = np.empty_like(x)
        for q in range(case["w"]):
            xq = x[c.sys.col_idx, q]
            y[:, q] = np.bincount(rows, v * xq.real, c.sys.n) + 1j * np.bincount(rows, v * xq.imag, c.sys.n)
        return y
    if k == "wave":
        lam, y = _modes(c.sys)
        _, s = _dense(c.sys)
        return y @ (np.exp(-1j * lam * c.tau * case["steps"])[:, None] * (y.T @ (s.numpy() @ c.psi)))
    if k == "train":
        w32 = _net(int(seed) % 1000)
        w = [t.to(torch.bfloat16).double().requires_grad_() for t in w32]
        b = [torch.zeros(t.shape[0], dtype=torch.float64, requires_grad=True) for t in w32]
        a, t = torch.as_tensor(c.x).double(), torch.as_tensor(c.t).double()
        for l in range(4):
            a = a @ w[l].T + b[l]
            a = torch.nn.functional.gelu(a) if l < 3 else a
        loss = ((a - t) ** 2).mean()
        loss.backward()
        step = lambda p, g: p - 2e-3 * g / (g.abs() + 1e-8)  # noqa: E731  (Adam's first step)
        return dict(loss=loss.detach(), w=[step(p.double(), q.grad) for p, q in zip(w32, w)],
                    b=[step(q.detach(), q.grad) for q in b], gw=[q.grad for q in w], gb=[q.grad for q in b])
    x = torch.as_tensor(_descriptors(c.sys))
    m, s = x.mean(0), x.std(0)
    s = torch.where(s > 1e-3, s, torch.ones_like(s))
    a = x * (1 / s).float().double() + (-m / s).float().double()
    for l, w in enumerate(_net(int(seed) % 1000)):
        a = a @ w.to(torch.bfloat16).double().T
        a = torch.nn.functional.gelu(a) if l < 3 else a
    return dict(x=x, y=a * torch.tensor([0.3, 0.7]).double() + torch.tensor([1.0, -1.5]).double())
