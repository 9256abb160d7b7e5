"""Wavepackets shared by clusters of teams: chains from less than one factor block to
more blocks than a cluster has teams, narrow and wide bands, and packet counts on both
sides of each change of the cluster's size (a lone packet up to one team each), against
the oracle's generalized spectral sum."""
import numpy as np
import pytest
import scipy.linalg as sla

from oracle import wavepacket as owp
from synth import chain_4orb, ppv_chain

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")


@pytest.mark.parametrize("packets", [1, 19, 20, 38, 39, 76, 77])
@pytest.mark.parametrize("maker", [lambda: ppv_chain(1, seed=1), lambda: ppv_chain(4, seed=2),
                                   lambda: chain_4orb(171, seed=3), lambda: ppv_chain(23, seed=4)])
def test_cluster_packets(maker, packets):
    system = maker()
    H, S = system.dense()
    lam = sla.eigh(H, S, eigvals_only=True)
    rng = np.random.default_rng(packets)
    c0 = rng.standard_normal((system.n, packets)) + 1j * rng.standard_normal((system.n, packets))
    tau, steps = 0.15, 4
    mat = gbg.Matrix(system)
    psi, _ = gbg.wavepacket(mat, torch.from_numpy(c0).cuda(), steps, tau, lam[0] - 0.1, lam[-1] + 0.1)
    got = psi.cpu().numpy()
    mat.close()
    ref = owp.propagate(system, c0, steps * tau)
    # as the one-team test: 1e-10 of the largest element
    assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()
