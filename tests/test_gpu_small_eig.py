"""Davidson's Rayleigh-Ritz solve at every kind of subspace size (odd, even, the smallest and the
largest allowed) and with a near-degenerate lowest pair: the converged energies are the exact ones."""
import numpy as np
import pytest

import workloads as wl
from oracle import exact
from tests._gpu import engine_for, load_mps

pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _ed(mpo):
    from tests._helpers import mpo_to_matrix
    return float(np.linalg.eigvalsh(mpo_to_matrix(mpo))[0])


@pytest.mark.parametrize("kmax", [2, 3, 8, 31, 32])
def test_energy_at_every_subspace_size(kmax):
    """Heisenberg chain L = 10, untruncated: the variational minimum is the ED energy to the
    residual squared (1e-10) and rounding."""
    mpo = wl.heisenberg_chain(10)
    eng = engine_for(pd, mpo, kmax=kmax)
    load_mps(eng, wl.random_mps(10, mpo.site.qn, 0, 32, seed=2), list(mpo.site.qn))
    for _ in range(2):
        g = eng.sweep(32, dav_max_iter=300)
    assert abs(g["energy"] - _ed(mpo)) <= 1e-10
    eng.close()


def test_energy_with_nearly_degenerate_ground_states():
    """Ferromagnetic transverse-field Ising chain, h = 0.05: the two lowest energies differ by about
    h^L, far below what FP32 resolves."""
    L, h = 10, 0.05
    mpo = wl.tfim_chain(L, 1.0, h)
    eng = engine_for(pd, mpo)
    load_mps(eng, wl.random_mps(L, mpo.site.qn, 0, 32, seed=2), list(mpo.site.qn))
    for _ in range(2):
        g = eng.sweep(32)
    assert abs(g["energy"] - exact.tfim_energy(L, 1.0, h)) <= 1e-9
    eng.close()
