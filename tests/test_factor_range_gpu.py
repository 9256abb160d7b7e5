"""The mixed path's factor solve where S's factor does not fit FP16's range: a basis that is
not normalised (orbitals scaled by up to 1e4, alternating or half against half), and a wide
band of mixed signs whose bounds on the solution's growth multiply from block to block while
the solution does not grow.

One solve, in the norm of the normalised basis: 5.7e-6 of the largest entry (the bound of
test_factor_passes_gpu.py) times the condition number of the normalised S.  Full solves: a
pair that reports convergence has a true residual of at most twice tol (the recursive
residual's own rounding).
"""
import numpy as np
import pytest

from synth import TBSystem, chain_4orb, ppv_chain, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


def rescaled(system, d):
    f = d[np.repeat(np.arange(system.n), np.diff(system.row_ptr))] * d[system.col_idx]
    system.h_val, system.s_val = system.h_val * f, system.s_val * f
    return system


def every_third(system, c):
    return rescaled(system, np.where(np.arange(system.n) % 3 == 0, float(c), 1.0))


def half(system, c):
    return rescaled(system, np.where(np.arange(system.n) < system.n // 2, float(c), 1.0))


def random_band(n, bw, lam_min, seed):
    """Unit diagonal, random elements of either sign, S's lowest eigenvalue lam_min."""
    rng = np.random.default_rng(seed)
    i, j = np.indices((n, n))
    band = np.abs(i - j) <= bw
    A = np.where(band, rng.standard_normal((n, n)), 0.0)
    A = A + A.T - np.diag(np.diag(A + A.T))
    S = np.eye(n) + A * (lam_min - 1.0) / np.linalg.eigvalsh(A)[0]
    H = np.where(band, rng.standard_normal((n, n)), 0.0) * 0.2
    H = H + H.T
    r, c = np.nonzero(band)
    ptr = np.concatenate([[0], np.cumsum(band.sum(1))]).astype(np.int64)
    return TBSystem(n=n, row_ptr=ptr, col_idx=c.astype(np.int32), h_val=H[r, c], s_val=S[r, c],
                    orb_atom=np.zeros(n, np.int32))


SYSTEMS = {
    "third 4": lambda: every_third(ppv_chain(5, seed=1), 4),  # the FP16 tiles' last
    "third 30": lambda: every_third(ppv_chain(5, seed=1), 30),
    "third 1e3": lambda: every_third(ppv_chain(5, seed=1), 1e3),
    "third 1e4": lambda: every_third(chain_4orb(40, seed=1), 1e4),
    "half 1e-3": lambda: half(ppv_chain(12, seed=2), 1e-3),
    "band": lambda: random_band(1500, 63, 0.05, 1),
}


@pytest.mark.parametrize("w", [1, 8, 32])
@pytest.mark.parametrize("name", SYSTEMS)
def test_one_solve(name, w):
    system = SYSTEMS[name]()
    _, S = system.dense()
    d = np.sqrt(np.diag(S))
    rng = np.random.default_rng(w)
    x = (rng.standard_normal((system.n, w)) + 1j * rng.standard_normal((system.n, w))).astype(np.complex64)
    x[:, w // 2:] *= d[:, None]
    mat = gbg.Matrix(system)
    y = mat.apply_sinv(torch.from_numpy(x).cuda(), prec="fp32").cpu().numpy()
    mat.close()
    Sn = S / d[:, None] / d[None]
    want = np.linalg.solve(Sn, x.astype(np.complex128) / d[:, None])  # D S^-1 x
    tol = 5.7e-6 * np.linalg.cond(Sn)
    for got, ref in ((y.real, want.real), (y.imag, want.imag)):
        err = np.abs(got * d[:, None] - ref).max(0)
        assert (err <= tol * np.abs(ref).max(0)).all(), err


@pytest.mark.parametrize("tol", [1e-6, 1e-8])
@pytest.mark.parametrize("name", SYSTEMS)
def test_converged_pairs_have_their_residual(name, tol):
    system = SYSTEMS[name]()
    cols = np.unique(np.linspace(0, system.n - 1, 6).astype(np.int32))
    z = shift_grid(-4.0, 4.0, 6, 0.5 if name == "band" else 0.05)
    mat = gbg.Matrix(system)
    out = gbg.shifted_solve(mat, z, cols, tol=tol, maxit=20000, prec="mixed")
    assert out["converged"].all()
    true = gbg.true_residual(mat, z, cols, np.arange(len(cols)), tol=tol, maxit=20000, prec="mixed").cpu().numpy()
    mat.close()
    assert (true <= 2 * tol).all(), true.max()


def test_batch_of_both():
    """A batch that holds such a system and an ordinary one gives what each gives alone."""
    systems = [SYSTEMS["third 1e3"](), ppv_chain(3, seed=4)]
    z = shift_grid(-4.0, 4.0, 6, 0.3)
    mats = [gbg.Matrix(s) for s in systems]
    problems = [dict(z=z, cols=np.arange(0, s.n, 23, dtype=np.int32), tol=1e-8, maxit=20000) for s in systems]
    res, info = gbg.shifted_solve_batched(mats, problems, prec="mixed", want_g=True)
    assert info["status"] == 0
    for s, m, p, r in zip(systems, mats, problems, res):
        H, S = s.dense()
        lam = np.linalg.eigvalsh(S)[0]
        one = gbg.shifted_solve(m, z, p["cols"], tol=1e-8, maxit=20000, prec="mixed", want_g=True)
        m.close()
        assert (r["g_proj"] - one["g_proj"]).abs().max().item() <= 2 * 1e-8 / (0.3 * lam)
