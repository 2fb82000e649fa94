"""Davidson's fused vector launches at the edges of their grid: vectors below one CTA, a few CTAs, and
longer than one pass of the whole grid (128 x 608 elements), with subspaces of one and several groups of
eight vectors, restarts included.  The converged energy is the exact one (bound as in the other exact
comparisons, 1e-9)."""
import pytest

import workloads as wl
from oracle import exact
from tests._gpu import engine_for, load_mps

pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


@pytest.mark.parametrize("L,m,kmax", [(4, 4, 8), (10, 32, 3), (10, 32, 17), (18, 200, 8), (18, 200, 20)])
def test_energy_at_every_vector_length(L, m, kmax):
    mpo = wl.tfim_chain(L, 1.0, 1.3)
    eng = engine_for(pd, mpo, kmax=kmax)
    load_mps(eng, wl.random_mps(L, mpo.site.qn, 0, m, seed=2), list(mpo.site.qn))
    for _ in range(2):
        g = eng.sweep(m, dav_max_iter=40)
    assert abs(g["energy"] - exact.tfim_energy(L, 1.0, 1.3)) <= 1e-9
    eng.close()
