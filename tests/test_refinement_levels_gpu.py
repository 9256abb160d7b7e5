"""The mixed path's inner solve at tol 1e-10 on both sides of its rule for the fourth
refinement level: a well-conditioned S, which leaves it out, and one close to singular,
which needs it, against the oracle.  Tolerance: a converged pair's residual is at most
tol, so an entry is off by at most tol / (eta lambda_min(S)), doubled for the recursive
residual's own rounding."""
import numpy as np
import pytest

import oracle
from synth import ppv_chain, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("lam_min", [None, 0.01])
def test_levels(lam_min):
    system = ppv_chain(3, seed=5)
    H, S = system.dense()
    if lam_min is not None:  # stretch the couplings until S's lowest eigenvalue is lam_min
        off = system.col_idx != np.repeat(np.arange(system.n), np.diff(system.row_ptr))
        low = np.linalg.eigvalsh(S - np.diag(np.diag(S)))[0]
        assert np.allclose(np.diag(S), 1.0)
        system.s_val = np.where(off, system.s_val * (lam_min - 1.0) / low, system.s_val)
        H, S = system.dense()
    eta, tol = 0.4, 1e-10
    z = shift_grid(-8.0, 4.0, 5, eta)
    cols = np.array([0, 57], np.int32)
    mat = gbg.Matrix(system)
    out = gbg.shifted_solve(mat, z, cols, tol=tol, maxit=20000, prec="mixed", want_g=True)
    mat.close()
    assert out["converged"].all()
    want = oracle.project_columns(system, oracle.green_columns(H, S, z, cols), cols)
    err = np.abs(out["g_proj"].cpu().numpy() - want).max()
    assert err <= 2 * tol / (eta * np.linalg.eigvalsh(S)[0])
