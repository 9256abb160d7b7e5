"""The FP64 factor solve at the sizes where its row pairs and slices can go wrong:
a few orbitals, one ragged block, a ragged last block, narrow and wide bands, every
number of column chunks.

Tolerance: the four products (two triangular, two band) add at most 64 terms an
element, 64 x 2^-53 of the absolute sum, and the absolute row sums of the factor's
inverse stay below 8 for these systems: 4 x 64 x 2^-53 x 8 = 2.3e-13 of a column's
largest entry.
"""
import numpy as np
import pytest

from synth import chain_4orb, ppv_chain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("w", [1, 2, 8, 16, 32])
@pytest.mark.parametrize("maker", [lambda: chain_4orb(2, seed=1), lambda: chain_4orb(33, seed=2),
                                   lambda: ppv_chain(1, seed=3), lambda: ppv_chain(9, seed=4)])
def test_factor_solve_fp64(maker, w):
    system = maker()
    mat = gbg.Matrix(system)
    _, S = system.dense()
    rng = np.random.default_rng(w)
    x = rng.standard_normal((system.n, w)) + 1j * rng.standard_normal((system.n, w))
    y = mat.apply_sinv(torch.from_numpy(x).cuda(), prec="fp64").cpu().numpy()
    mat.close()
    want = np.linalg.solve(S, x)
    assert (np.abs(y - want).max(0) <= 2.3e-13 * np.abs(want).max(0)).all()
