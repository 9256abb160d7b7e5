"""The automatic panel width of a mixed batch: unequal chains whose panels are narrowed
(more panels than SMs, on wide teams), equal ones whose panels are not, more systems of
eight columns than SMs, a few, each against the oracle.  Tolerance: a converged pair's
residual is at most tol, so an entry is off by at most tol / (eta lambda_min(S)), doubled
for the recursive residual's own rounding."""
import numpy as np
import pytest

import oracle
from synth import ppv_chain, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("sizes", [[7] * 10 + [1, 2] * 45, [3] * 100, [1] * 160, [2] * 3])
def test_batch_width(sizes):
    eta, tol = 0.4, 1e-10
    z = shift_grid(-8.0, 4.0, 3, eta)
    systems = [ppv_chain(m, seed=i) for i, m in enumerate(sizes)]
    cols = [np.linspace(0, s.n - 1, 8).astype(np.int32) for s in systems]
    mats = [gbg.Matrix(s) for s in systems]
    res, _ = gbg.shifted_solve_batched(mats, [dict(z=z, cols=c, tol=tol, maxit=4000) for c in cols], want_g=True)
    for s, c, r, m in zip(systems, cols, res, mats):
        H, S = s.dense()
        want = oracle.project_columns(s, oracle.green_columns(H, S, z, c), c)
        assert r["converged"].all()
        assert np.abs(r["g_proj"].cpu().numpy() - want).max() <= 2 * tol / (eta * np.linalg.eigvalsh(S)[0])
        m.close()
