"""FP64 emulation inside an engine: fp64_emulation = 2 sends every batch through it, so these runs
(matvecs, environments, splits and their polish, gauge moves, measurements, merges) meet the emulated
arithmetic at any size; and one plan keeps one arithmetic however often it runs."""
import numpy as np
import pytest

import workloads as wl
from oracle import icmps as IC
from tests._gpu import load_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _engine(mpo, emu, precision="fp64", **more):
    W, flux, D = wl.pack_mpo(mpo)
    return pd.Engine(W, flux, D, list(mpo.site.qn), mpo.qtot, precision, 8, fp64_emulation=emu, **more)


@pytest.mark.parametrize("L,regions,plain", [(12, 0, False), (12, 0, True), (24, 4, False)])
def test_engine_follows_the_fp64_units(L, regions, plain):
    """Sweep by sweep the same energies as on the FP64 units (converged to 1e-10 residuals)."""
    mpo = wl.heisenberg_chain(L)
    qn = list(mpo.site.qn)
    got = []
    for emu in (0, 2):
        eng = _engine(mpo, emu, svd_plain_jacobi=plain)
        load_mps(eng, wl.random_mps(L, qn, 0, 8, seed=3), qn)
        pd.profile_reset()
        if regions:
            eng.setup_regions(regions, 2, 32)
        got.append([eng.sweep(m)["energy"] for m in (16, 32, 48)])
        ran = pd.profile_read()["emu_batches"]
        assert (ran > 0) == (emu == 2), ran
        eng.close()
    a, b = map(np.array, got)
    assert np.abs(a - b).max() <= 1e-9 * np.abs(a).max()


def test_mixed_engine_with_fp64_edges():
    """bf16 regions with FP64-accurate environments, edge solves and splits: the energy of a converged
    sweep agrees with the FP64 engine to the mixed mode's 1e-5."""
    L = 24
    mpo = wl.heisenberg_chain(L)
    qn = list(mpo.site.qn)
    mps = wl.random_mps(L, qn, 0, 16, seed=0)
    ref = _engine(mpo, 0)
    load_mps(ref, mps, qn)
    e = [ref.sweep(m)["energy"] for m in (32, 48, 48, 48)][-1]
    ref.close()
    eng = _engine(mpo, 2, "bf16", env_fp64=True, accurate_edges=2)
    load_mps(eng, mps, qn)
    pd.profile_reset()
    dav = dict(dav_tol=1e-9, dav_max_iter=12, refine_iters=6, serial_regions=1)
    eng.setup_regions(3, 1, 32, **dav)
    g = [eng.sweep(m, **dav) for m in (32, 48, 48, 48, 48)][-1]
    assert pd.profile_read()["emu_batches"] > 0
    assert abs(g["energy"] - e) <= 1e-5 * abs(e)
    eng.close()


def test_local_expectations_match_oracle():
    mpo = wl.heisenberg_square_cylinder(6, 4)
    qn = list(mpo.site.qn)
    eng = _engine(mpo, 2)
    load_mps(eng, wl.random_mps(mpo.L, qn, 0, 90, seed=4), qn)
    bonds, data, _ = eng.state()
    sites, off = [], 0
    for j in range(mpo.L):
        n = sum(bonds[j][q] * bonds[j + 1][q + s] for q in bonds[j] for s in qn if q + s in bonds[j + 1])
        sites.append(wl.unpack_site(data[off: off + n], bonds[j], bonds[j + 1], qn))
        off += n
    psi_o, V_o, _ = IC.inverse_canonical(sites, bonds, qn)
    eng.inverse_canonical()
    Sz, Sp, Sm = (mpo.site.op(x) for x in ("Sz", "Sp", "Sm"))
    ops1, ops2 = [Sz, Sz @ Sz], [np.kron(Sz, Sz), np.kron(Sp, Sm)]
    e1_o, e2_o = IC.all_expectations(psi_o, V_o, qn, ops1, ops2)
    pd.profile_reset()
    e1, e2, _ = eng.local_expectations(ops1, ops2)
    assert pd.profile_read()["emu_batches"] == 1                  # the Theta batch
    assert np.abs(e1 - e1_o).max() <= 1e-12
    assert np.abs(e2 - e2_o).max() <= 1e-12
    eng.close()


def test_a_repeated_measurement_repeats_its_bits():
    """A Theta batch of 1 to 6 GFLOP, where first and repeated runs of one plan cost differently: the
    arithmetic is the plan's, from its first run on."""
    L = 32
    mpo = wl.heisenberg_chain(L)
    qn = list(mpo.site.qn)
    eng = _engine(mpo, True)
    load_mps(eng, wl.random_mps(L, qn, 0, 600, seed=6, sigma=1.5), qn)
    eng.inverse_canonical()
    b = [eng.icmps_bond(j) for j in range(L + 1)]
    fl = sum(2.0 * b[j][q] * b[j + 1][q + s1] * b[j + 2][q + s1 + s2] for j in range(L - 1) for q in b[j]
             for s1 in qn for s2 in qn if q + s1 in b[j + 1] and q + s1 + s2 in b[j + 2])
    assert 1e9 <= fl < 6e9
    Sz = mpo.site.op("Sz")
    pd.profile_reset()
    got = [eng.local_expectations([Sz], [np.kron(Sz, Sz)])[:2] for _ in range(4)]
    ran = pd.profile_read()["emu_batches"]
    for e1, e2 in got[1:]:
        assert np.array_equal(e1, got[0][0]) and np.array_equal(e2, got[0][1])
    assert ran == 4
    eng.close()
