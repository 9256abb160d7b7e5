"""The dense inverse's refinement where a level gains little (every orbital coupled to every
other one: a level leaves 1e-3 of the residual), and an overlap that the dense inverse
refuses.

Three levels (tol 1e-9) leave the cube of a level's factor, four (tol 1e-10) its fourth power
down to the residual's own rounding: with 1e-3 a level, at least ten times less.  The refused
overlap is solved by iteration: a converged pair has a true residual of at most twice tol.
"""
import numpy as np
import pytest

from synth import TBSystem, chain_4orb, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


def solve(mat, tol):
    z, cols = shift_grid(-3.0, 3.0, 5, 0.5), np.array([0, mat.system.n // 2, mat.system.n - 1], np.int32)
    kw = dict(tol=tol, maxit=2000, prec="mixed")
    plan = gbg.solve_plan(mat, z, cols, **kw)
    out = gbg.shifted_solve(mat, z, cols, **kw)
    assert out["converged"].all()
    return plan["inner"], gbg.true_residual(mat, z, cols, np.arange(3), **kw).max().item()


def test_needed_level_is_run():
    n, a = 400, 0.9
    rng = np.random.default_rng(n)
    S = np.full((n, n), a) + (1.0 - a) * np.eye(n)
    L = np.linalg.cholesky(S)
    A = rng.standard_normal((n, n)) / np.sqrt(n)
    H = L @ (A + A.T) @ L.T
    H = 0.5 * (H + H.T)
    mat = gbg.Matrix(TBSystem(n=n, row_ptr=np.arange(n + 1, dtype=np.int64) * n,
                              col_idx=np.tile(np.arange(n, dtype=np.int32), n), h_val=H.ravel(), s_val=S.ravel(),
                              orb_atom=np.zeros(n, np.int32)))
    (inner3, three), (inner4, four) = solve(mat, 1e-9), solve(mat, 1e-10)
    mat.close()
    assert inner3 == inner4 == "inverse"
    assert four <= 0.1 * three


@pytest.mark.parametrize("tol", [1e-6, 1e-8, 1e-10])
def test_refused_overlap(tol):
    c = chain_4orb(60, seed=3)  # in random order, every third orbital scaled by 10
    new = np.random.default_rng(4).permutation(c.n)
    r, k = new[np.repeat(np.arange(c.n), np.diff(c.row_ptr))], new[c.col_idx]
    o = np.lexsort((k, r))
    d = np.where(np.arange(c.n) % 3 == 0, 10.0, 1.0)
    f = (d[r] * d[k])[o]
    ptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=c.n))]).astype(np.int64)
    mat = gbg.Matrix(TBSystem(n=c.n, row_ptr=ptr, col_idx=k[o].astype(np.int32), h_val=c.h_val[o] * f,
                              s_val=c.s_val[o] * f, orb_atom=np.zeros(c.n, np.int32)))
    inner, true = solve(mat, tol)
    mat.close()
    assert inner == "chebyshev"
    assert true <= 2 * tol
