"""FP32 grouped GEMM at the edges of its 64 x 64 tiles and 16-deep chunks, through the mixed-mode
environment updates: sectors of 1, 15, 16, 17, 63, 64, 65 and 130 states against the FP64 oracle.

Bound per element: the inputs are rounded to FP32 and the two contractions are FMA chains of at most
K1 and K2 terms around an MPO mix of n terms, so the error stays within (K1 + K2 + n + 4) 2^-24 times
the same update of absolute values."""
import numpy as np
import pytest

import workloads as wl
from oracle import dmrg as O
from tests import _layout as LY

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")

SECTORS = [({-1: 1, 1: 64, 3: 17}, {-2: 65, 0: 16, 2: 130, 4: 1}), ({-1: 63, 1: 65}, {0: 130, 2: 15}),
           ({1: 130}, {0: 64, 2: 63}), ({-3: 16, -1: 15, 1: 1, 3: 64}, {-2: 1, 0: 17, 2: 65})]


@pytest.mark.parametrize("prec", [pd.TF32, pd.BF16])
@pytest.mark.parametrize("case", range(len(SECTORS)))
def test_environment_update_fp32_edges(case, prec):
    bl, bm = SECTORS[case]
    mpo, j = wl.heisenberg_square_cylinder(4, 3), 5
    qn, W = list(mpo.site.qn), mpo.W[5]
    f0, f1 = mpo.flux[j], mpo.flux[j + 1]
    rng = np.random.default_rng(case)
    A = {k: rng.standard_normal((bl[k[0]], bm[k[0] + qn[k[1]]])) for k in LY.site_keys(bl, bm, qn)}
    ab = lambda t: {k: np.abs(v) for k, v in t.items()}  # noqa: E731
    bond = pd.Bond(qn, bl, bm, W, f0, f1)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    Ad = dev(LY.pack_site(A, bl, bm, qn))
    factor = (max(bl.values()) + max(bm.values()) + 2 * sum(W.shape) + 4) * 2.0 ** -24
    for side, b0, b1, g0, g1, step, ref in (("left", bl, bm, f0, f1, pd.env_left, O.env_left),
                                            ("right", bm, bl, f1, f0, pd.env_right, O.env_right)):
        E = LY.random_env(b0, g0, rng)
        out = torch.full((sum(b1[q] * b1[q - int(g1[w])] for q, w in LY.env_keys(b1, g1)),), float("nan"),
                         dtype=torch.float64, device="cuda")
        Ed = dev(LY.pack_env(E, b0, g0))
        step(bond, prec, Ed.data_ptr(), Ad.data_ptr(), out.data_ptr())
        got = LY.unpack_env(out.cpu().numpy(), b1, g1)
        want, size = ref(E, A, W, f0, f1, qn), ref(ab(E), ab(A), np.abs(W), f0, f1, qn)
        for k in got:
            if k not in want:
                assert not np.any(got[k]), (side, k)
                continue
            # d (s, s') blocks of each kind meet in one element
            assert np.all(np.abs(got[k] - want[k]) <= 2 * factor * size[k] + 1e-300), (side, k)
