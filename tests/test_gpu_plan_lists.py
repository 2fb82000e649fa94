"""Host plans of the matvec, its backward and the environment updates over the forms their lists take:
irregular sectors (gaps in the charges, one-state sectors, sectors without partner), three local
states, many MPO channels, a window next to the chain's end; against the oracle element by element
(1e-12 of the largest element, the bound of the single-operation parity tests)."""
import numpy as np
import pytest

import workloads as wl
from oracle import dmrg as O
from oracle import grad as G
from tests import _layout as LY

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _case(kind):
    if kind == "gaps":
        mpo, j = wl.heisenberg_chain(12), 5
        bl, bm, br = {-5: 3, -1: 7, 1: 1, 3: 20}, {-4: 2, 0: 9, 2: 5, 4: 3}, {-3: 4, -1: 2, 1: 17, 5: 1}
    elif kind == "one":
        mpo, j = wl.heisenberg_chain(12), 5
        bl, bm, br = {1: 1}, {0: 1, 2: 1}, {1: 1}
    elif kind == "spin1":
        mpo, j = wl.aklt_chain(8), 3
        bl, bm, br = {-2: 4, 0: 9, 2: 5}, {-4: 3, -2: 6, 0: 8, 2: 4}, {-2: 7, 0: 3, 4: 2}
    elif kind == "jq2":
        mpo, j = wl.jq2_cylinder(4, 4)[0], 7
        bonds = wl.bond_sectors(mpo.L, list(mpo.site.qn), 0, 40, sigma=3.0)
        bl, bm, br = bonds[j], bonds[j + 1], bonds[j + 2]
    else:                                   # "end": the last two sites
        mpo, j = wl.heisenberg_square_cylinder(3, 2), 4
        bonds = wl.bond_sectors(mpo.L, list(mpo.site.qn), 0, 64)
        bl, bm, br = bonds[j], bonds[j + 1], bonds[j + 2]
    return mpo, list(mpo.site.qn), j, bl, bm, br


def _close(got, want, tol=1e-12):
    scale = max([1.0] + [np.abs(v).max() for v in want.values()])
    for k in got:
        assert np.abs(got[k] - want.get(k, np.zeros_like(got[k]))).max() <= tol * scale, k


@pytest.mark.parametrize("kind", ["gaps", "one", "spin1", "jq2", "end"])
def test_plans_against_oracle(kind):
    mpo, qn, j, bl, bm, br = _case(kind)
    rng = np.random.default_rng(3)
    W1, W2 = mpo.W[j], mpo.W[j + 1]
    f0, f1, f2 = mpo.flux[j], mpo.flux[j + 1], mpo.flux[j + 2]
    L, R = LY.random_env(bl, f0, rng), LY.random_env(br, f2, rng)
    keys = LY.psi_keys(bl, br, qn)
    x = {k: rng.standard_normal((bl[k[0]], br[k[0] + qn[k[1]] + qn[k[2]]])) for k in keys}
    yb = {k: rng.standard_normal(v.shape) for k, v in x.items()}
    bond = pd.Bond(qn, bl, br, W1, f0, f1, W2, f2)
    Ld, Rd = _dev(LY.pack_env(L, bl, f0)), _dev(LY.pack_env(R, br, f2))
    xd, ybd = _dev(LY.pack_psi(x, bl, br, qn)), _dev(LY.pack_psi(yb, bl, br, qn))
    y = torch.full_like(xd, float("nan"))
    pd.heff_apply(bond, pd.FP64, Ld.data_ptr(), Rd.data_ptr(), xd.data_ptr(), y.data_ptr())
    _close(LY.unpack_psi(y.cpu().numpy(), bl, br, qn), O.heff_apply(L, W1, f0, W2, f2, R, x, qn))
    xb, Lb, Rb = (torch.full_like(t, float("nan")) for t in (xd, Ld, Rd))
    W1b, W2b = pd.heff_backward(bond, Ld.data_ptr(), Rd.data_ptr(), xd.data_ptr(), ybd.data_ptr(), xb.data_ptr(),
                                Lb.data_ptr(), Rb.data_ptr())
    ref = G.heff_backward(L, W1, f0, W2, f2, R, x, yb, qn)
    _close(LY.unpack_psi(xb.cpu().numpy(), bl, br, qn), ref[0])
    _close(LY.unpack_env(Lb.cpu().numpy(), bl, f0), ref[1])
    _close(LY.unpack_env(Rb.cpu().numpy(), br, f2), ref[2])
    _close({0: W1b, 1: W2b}, {0: ref[3], 1: ref[4]})
    # environment updates through the left site
    A = {k: rng.standard_normal((bl[k[0]], bm[k[0] + qn[k[1]]])) for k in LY.site_keys(bl, bm, qn)}
    Rm = LY.random_env(bm, f1, rng)
    site = pd.Bond(qn, bl, bm, W1, f0, f1)
    Ad, Rmd = _dev(LY.pack_site(A, bl, bm, qn)), _dev(LY.pack_env(Rm, bm, f1))
    out_l = torch.full((sum(bm[q] * bm[q - int(f1[w])] for q, w in LY.env_keys(bm, f1)),), float("nan"),
                       dtype=torch.float64, device="cuda")
    out_r = torch.full((sum(bl[q] * bl[q - int(f0[w])] for q, w in LY.env_keys(bl, f0)),), float("nan"),
                       dtype=torch.float64, device="cuda")
    pd.env_left(site, pd.FP64, Ld.data_ptr(), Ad.data_ptr(), out_l.data_ptr())
    pd.env_right(site, pd.FP64, Rmd.data_ptr(), Ad.data_ptr(), out_r.data_ptr())
    _close(LY.unpack_env(out_l.cpu().numpy(), bm, f1), O.env_left(L, A, W1, f0, f1, qn))
    _close(LY.unpack_env(out_r.cpu().numpy(), bl, f0), O.env_right(Rm, A, W1, f0, f1, qn))
