"""FP64 splits of spectra with equal and nearly equal singular values: equal ones settle in the
whole-matrix passes (no scalar Jacobi), isolated near-degenerate pairs too; a wide cluster goes to the
scalar Jacobi.  Bounds as for any split: 10 n eps, orthonormality 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _values(kind, k):
    i = np.arange(k)
    if kind == "two":                          # two values, each many times
        return np.where(i % 2, 1.0, 0.3)
    if kind == "fours":
        return 10.0 ** (-3.0 * (i // 4) / k)
    if kind == "near":                         # pairs 1e-8 apart
        return 10.0 ** (-3.0 * (i // 2) / k) * (1 + 1e-8 * (i % 2))
    return 1.0 + 1e-9 * i                      # "cluster"


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("p,n", [(3, 5), (8, 8), (16, 200), (17, 17), (64, 64), (200, 200), (1000, 50)])
@pytest.mark.parametrize("kind", ["two", "fours", "near", "cluster"])
def test_clustered_spectra(kind, p, n, mode):
    rng = np.random.default_rng(p + 31 * n)
    k = min(p, n)
    s = _values(kind, k)
    U, V = (np.linalg.qr(rng.standard_normal((x, k)))[0] for x in (p, n))
    M = (U * s) @ V.T
    ref = np.linalg.svd(M, compute_uv=False)
    bond = pd.Bond([0], {0: p}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.from_numpy(np.ascontiguousarray(M).ravel()).cuda()
    A, lam, B = (torch.zeros(size, dtype=torch.float64, device="cuda") for size in (p * k, k, k * n))
    pd.profile_reset()
    mid, trunc = pd.svd_split(bond, x.data_ptr(), 10 ** 9, mode, A.data_ptr(), lam.data_ptr(), B.data_ptr())
    scalar = pd.profile_read()["svd_scalar"]
    assert mid == {0: k}
    lam = lam.cpu().numpy()
    Ah, Bh = A.cpu().numpy().reshape(p, k), B.cpu().numpy().reshape(k, n)
    nrm, tol = np.sqrt(np.sum(ref ** 2)), 10 * max(p, n) * np.finfo(float).eps
    assert np.abs(lam - ref / nrm).max() <= tol
    assert np.abs((Ah * lam) @ Bh - M / nrm).max() <= tol
    assert max(np.abs(Ah.T @ Ah - np.eye(k)).max(), np.abs(Bh @ Bh.T - np.eye(k)).max()) <= 1e-12
    if kind != "cluster":
        assert scalar == 0
    elif k >= 8:
        assert scalar == 1
