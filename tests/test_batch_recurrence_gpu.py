"""A batch runs every system by the recurrence and the inner solve that the system's own
parameters name, whatever its neighbours name, so that gb_true_residual with those parameters
checks the solve that ran: systems that name a seed shift, or panels of one column, beside
ones that do not, with and without a banded overlap.

Each system of the batch is compared with its solve alone: the counts of outer and inner
iterations may differ by what rounding decides at the end (two in a hundred), where the other
recurrence's inner solve of an unbanded overlap takes ten times the steps; entries agree
within the residual bound of both.  The inner steps are compared in the mixed path, where an
application takes the same number whatever the panel's width (the FP64 path's CG goes on until
a panel's last column is done).
"""
import ctypes as C

import numpy as np
import pytest

from synth import TBSystem, chain_4orb, shift_grid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")
from paper_1603_09616_gb300 import _binding as gb  # noqa: E402


def unbanded(n):
    """A chain in random order."""
    c = chain_4orb(n // 4, seed=n)
    new = np.random.default_rng(n).permutation(n)
    r, k = new[np.repeat(np.arange(n), np.diff(c.row_ptr))], new[c.col_idx]
    o = np.lexsort((k, r))
    ptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    return TBSystem(n=n, row_ptr=ptr, col_idx=k[o].astype(np.int32), h_val=c.h_val[o], s_val=c.s_val[o],
                    orb_atom=np.zeros(n, np.int32))


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("batch_panel", [1, 4, 8])
def test_own_parameters_choose(prec, batch_panel):
    eta, tol = 0.3, 1e-9
    z = shift_grid(-5.0, 5.0, 7, eta)
    # (system, its seed shift, its panel)
    cases = [(chain_4orb(30, seed=1), 2, 0), (unbanded(300), -1, 0), (chain_4orb(41, seed=2), -1, 8),
             (unbanded(200), -1, 1)]
    mats = [gbg.Matrix(s) for s, _, _ in cases]
    keep, dev, nsys = [], torch.device("cuda", 0), len(cases)
    cols = [np.arange(0, s.n, 29, dtype=np.int32) for s, _, _ in cases]
    params, outs, res = (gb.SolveParams * nsys)(), (gb.Outputs * nsys)(), []
    for i, (s, seed, panel) in enumerate(cases):
        params[i] = gb._params(z, cols[i], tol, 4000, prec, None, None, 0.0, panel, seed, keep, 0)
        r, outs[i] = gb._alloc_outputs(mats[i], len(z), cols[i], None, None, True, dev)
        res.append(r)
    handles = (C.c_void_p * nsys)(*[m.handle.value for m in mats])
    lib = gbg.load()
    need = lib.gb_batched_workspace_size(nsys, handles, params, batch_panel, 1)
    assert need > 0
    ws = torch.empty(int(need), dtype=torch.uint8, device=dev)
    assert lib.gb_shifted_solve_batched(nsys, handles, params, outs, batch_panel, C.c_void_p(ws.data_ptr()),
                                        C.c_size_t(int(need)), gb._stream_handle(None)) == 0
    for i, (s, seed, panel) in enumerate(cases):
        one = gbg.shifted_solve(mats[i], z, cols[i], tol=tol, maxit=4000, prec=prec, seed_shift=seed, panel=panel,
                                want_g=True)
        both = [(r["iters"].max().item(), r["inner_iters"].max().item()) for r in (res[i], one)]
        for a, b in list(zip(*both))[:2 if prec == "mixed" else 1]:
            assert abs(a - b) <= 0.02 * max(a, b) + 4, (i, both)
        lam = np.linalg.eigvalsh(s.dense()[1])[0]
        assert (res[i]["g_proj"] - one["g_proj"]).abs().max().item() <= 4 * tol / (eta * lam)
        true = gbg.true_residual(mats[i], z, cols[i], np.arange(len(cols[i])), tol=tol, maxit=4000, prec=prec,
                                 seed_shift=seed, panel=panel).cpu().numpy()
        assert (true <= 2 * tol).all()
        mats[i].close()
