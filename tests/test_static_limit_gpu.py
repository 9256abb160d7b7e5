"""The allocation-free solve near its scratch's 32 MiB: what one column's records fit is
solved, in panels as wide as fit, and what does not is refused.

Tolerance: a converged pair has a residual of at most tol for a unit right-hand side, so an
entry of its solution is off by at most tol / (eta lambda_min(S)); twice that for the
recursive residual's own rounding.
"""
import numpy as np
import pytest

import oracle
from synth import chain_4orb, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("ncol,maxit", [(1, 16000), (24, 16000), (24, 9000), (24, 4000)])
def test_narrow_panels_fit(ncol, maxit, prec):
    system = chain_4orb(120, seed=6)
    H, S = system.dense()
    eta, tol = 0.3, 1e-10
    z = shift_grid(-5.0, 5.0, 64, eta)
    cols = np.linspace(0, system.n - 1, ncol).astype(np.int32)
    mat = gbg.Matrix(system)
    out = gbg.shifted_solve_static(mat, z, cols, tol=tol, maxit=maxit, prec=prec, want_g=True)
    mat.close()
    assert out["status"] == 0, out["message"]
    want = oracle.project_columns(system, oracle.green_columns(H, S, z, cols), cols)
    err = np.abs(out["g_proj"].cpu().numpy() - want).max()
    assert err <= 2 * tol / (eta * np.linalg.eigvalsh(S)[0])


def test_too_large_is_refused():
    mat = gbg.Matrix(chain_4orb(120, seed=6))
    z = shift_grid(-5.0, 5.0, 64, 0.3)
    for cols, kw in (([0], dict(maxit=32000)), (np.arange(24), dict(maxit=16000, panel=8))):
        out = gbg.shifted_solve_static(mat, z, np.asarray(cols, np.int32), prec="fp64", want_g=True, **kw)
        assert out["status"] == gbg._binding.GB_ENOMEM
    mat.close()
