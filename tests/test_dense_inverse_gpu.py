"""The mixed path's inner solve by the dense inverse, where S has no banded factor:
shuffled chains at the edges of its range (the fewest orbitals an unbanded S can
have, ragged last tiles, the largest kept and one more) and every panel width.

Tolerance: a converged pair has a residual of at most tol for a unit right-hand
side, so an entry of its solution is off by at most tol / (eta lambda_min(S));
twice that leaves room for the recursive residual's own rounding.
"""
import numpy as np
import pytest

import oracle
from synth import TBSystem, chain_4orb, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


def shuffled(n, scale):
    """Leading n orbitals of a chain in random order, the first and the last one coupled."""
    c = chain_4orb((n + 3) // 4, seed=n)
    rng = np.random.default_rng(n)
    rows = np.repeat(np.arange(c.n), np.diff(c.row_ptr))
    new = rng.permutation(n)
    j = int(c.col_idx[c.row_ptr[n // 2]:c.row_ptr[n // 2 + 1]][0])  # a neighbour of orbital n // 2
    assert j != n // 2
    for place, orb in ((0, n // 2), (n - 1, j)):
        at = int(np.flatnonzero(new == place)[0])
        new[at], new[orb] = new[orb], place
    keep = np.flatnonzero((rows < n) & (c.col_idx < n))
    r, k = new[rows[keep]], new[c.col_idx[keep]]
    order = np.lexsort((k, r))
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=ptr[1:])
    return TBSystem(n=n, row_ptr=ptr, col_idx=k[order].astype(np.int32), h_val=c.h_val[keep][order],
                    s_val=c.s_val[keep][order] * scale, orb_atom=np.zeros(n, np.int32))


@pytest.mark.parametrize("n,scale,panel", [(66, 1.0, 4), (67, 1e4, 8), (129, 1.0, 16), (130, 1e-4, 32), (456, 1.0, 0),
                                           (1021, 1.0, 32), (1024, 1.0, 8), (1025, 1.0, 8)])
def test_dense_inverse_solves(n, scale, panel):
    system = shuffled(n, scale)
    H, S = system.dense()
    eta, tol = 0.4 / scale, 1e-10
    z = shift_grid(-6.0 / scale, 6.0 / scale, 9, eta)
    cols = np.unique(np.linspace(0, n - 1, 37).astype(np.int32))
    mat = gbg.Matrix(system)
    plan = gbg.solve_plan(mat, z, cols, tol=tol, prec="mixed", panel=panel)
    assert plan["inner"] == ("inverse" if n <= 1024 else "chebyshev")
    out = gbg.shifted_solve(mat, z, cols, tol=tol, maxit=4000, prec="mixed", panel=panel, want_g=True)
    assert out["converged"].all()
    G = oracle.green_columns(H, S, z, cols)
    want = oracle.project_columns(system, G, cols)
    err = np.abs(out["g_proj"].cpu().numpy() - want).max()
    mat.close()
    assert err <= 2 * tol / (eta * np.linalg.eigvalsh(S)[0])


def test_badly_scaled_overlap_iterates():
    # S and H scaled by 10 on every third orbital: max |S| max |S^-1| is above 64
    system = shuffled(200, 1.0)
    d = np.where(np.arange(system.n) % 3 == 0, 10.0, 1.0)
    f = d[np.repeat(np.arange(system.n), np.diff(system.row_ptr))] * d[system.col_idx]
    system.h_val, system.s_val = system.h_val * f, system.s_val * f
    mat = gbg.Matrix(system)
    plan = gbg.solve_plan(mat, shift_grid(-6.0, 6.0, 9, 0.4), np.arange(8), prec="mixed")
    mat.close()
    assert plan["inner"] == "chebyshev"
