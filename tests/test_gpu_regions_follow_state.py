"""Real-space sweeps follow the state that is loaded: from other states other first-sweep energies, and an
engine that has swept one state gives the next one the energies that a new engine gives it (nothing of
an earlier state, its environments or its regions is kept).

Two Davidson iterations a step from random 16-state matrices leave the first sweep some 1e-2 above the
ground state, by an amount of the start's own; the bf16 arithmetic repeats to about 1e-6."""
import numpy as np
import pytest

import workloads as wl
from tests._gpu import load_mps

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")

SWEEP = dict(dav_tol=1e-9, dav_max_iter=2, refine_iters=1)


@pytest.mark.parametrize("schedule", [0, 1, 2])
def test_energies_follow_the_loaded_state(schedule):
    mpo = wl.field_square_cylinder(6, 4, seed=3)
    qn = list(mpo.site.qn)
    W, flux, D = wl.pack_mpo(mpo)

    def new():
        return pd.Engine(W, flux, D, qn, mpo.qtot, "bf16", 8, fp64_emulation=True, accurate_edges=2)

    def first_sweeps(eng, seed):
        load_mps(eng, wl.random_mps(mpo.L, qn, 0, 16, seed=seed), qn)
        eng.setup_regions(4, 0, 48, serial_regions=schedule, **SWEEP)
        return np.array([eng.sweep(48, serial_regions=schedule, **SWEEP)["energy"] for _ in range(2)])

    kept = new()
    first = {}
    for seed in (1, 2, 1):
        fresh = new()
        want = first_sweeps(fresh, seed)
        fresh.close()
        assert np.abs(first_sweeps(kept, seed) - want).max() <= 1e-5
        first[seed] = want[0]
    kept.close()
    assert abs(first[1] - first[2]) >= 1e-3
