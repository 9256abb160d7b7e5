"""The mixed path's factor solve (FP16 head / tail tensor-core passes) at the
sizes and ranges where it can go wrong: one block, a ragged last block, bands of
one and of four 16-column steps, every panel width, columns whose magnitudes span
the FP32 range, an S far from unit scale.

Tolerance: the operands keep 22 bits and the dropped tail products are 2^-22
relative, three times per product; the absolute row sums of the factor's inverse
stay below 8 for these systems, so a column's error is below
3 x 2^-22 x 8 = 5.7e-6 of its largest entry.
"""
import numpy as np
import pytest

from synth import chain_4orb, ppv_chain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("w", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("maker,scale", [(lambda: chain_4orb(4, seed=1), 1.0), (lambda: chain_4orb(33, seed=2), 1e8),
                                         (lambda: ppv_chain(2, seed=3), 1e-7), (lambda: ppv_chain(9, seed=4), 1.0)])
def test_factor_solve_ranges(maker, scale, w):
    system = maker()
    system.s_val = system.s_val * scale
    mat = gbg.Matrix(system)
    _, S = system.dense()
    rng = np.random.default_rng(w)
    x = rng.standard_normal((system.n, w)) + 1j * rng.standard_normal((system.n, w))
    x = (x * 10.0 ** rng.integers(-12, 12, w)).astype(np.complex64)
    x[:, 0] *= np.arange(system.n) % 7 == 0  # zeros between
    if w > 1:
        x[:, 1] = 0.0
    y = mat.apply_sinv(torch.from_numpy(x).cuda(), prec="fp32").cpu().numpy()
    mat.close()
    ref = np.linalg.solve(S, x.astype(np.complex128))
    for part, want in ((y.real, ref.real), (y.imag, ref.imag)):
        err = np.abs(part - want).max(0)
        assert (err <= 5.7e-6 * np.abs(want).max(0)).all(), err
