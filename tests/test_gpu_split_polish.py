"""FP64 split of one p x n sector matrix over the spectra that decide which way its singular vectors
are finished (whole-matrix rotations, FP32 passes over the columns below FP32 resolution, scalar
Jacobi): graded over 13 decades, exactly degenerate, clustered at 1e-9, rank-deficient, of any scale.

Bounds: a one-sided Jacobi's backward error is a small multiple of n eps sigma_max (10 n eps here);
columns end orthogonal to 4 eps sqrt(p) and A's are normalised by their computed norms (1e-12)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _spectrum(kind, n):
    i = np.arange(n)
    if kind == "graded":
        return 10.0 ** (-11.5 * i / max(1, n - 1))
    if kind == "degenerate":
        return np.where(i < (n + 1) // 2, 1.0, 1e-3)
    if kind == "cluster":
        return 1.0 + 1e-9 * i
    if kind == "rank":
        return np.where(i < (n + 1) // 2, 0.9 ** i, 0.0)
    return 0.8 ** np.minimum(i, 60)          # "decay": ordinary


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("p,n", [(1, 1), (2, 2), (3, 5), (17, 17), (64, 33), (65, 64), (150, 131)])
@pytest.mark.parametrize("kind", ["graded", "degenerate", "cluster", "rank", "decay"])
def test_split_of_one_sector(kind, p, n, mode):
    rng = np.random.default_rng(p + 31 * n)
    k = min(p, n)
    s = _spectrum(kind, k)
    U = np.linalg.qr(rng.standard_normal((p, k)))[0]
    V = np.linalg.qr(rng.standard_normal((n, k)))[0]
    M = (U * s) @ V.T * (2.0 ** -40 if kind == "decay" else 1.0)
    ref = np.linalg.svd(M, compute_uv=False)
    bond = pd.Bond([0], {0: p}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.from_numpy(np.ascontiguousarray(M).ravel()).cuda()
    A, lam, B = (torch.zeros(size, dtype=torch.float64, device="cuda") for size in (p * k, k, k * n))
    mid, trunc = pd.svd_split(bond, x.data_ptr(), 10 ** 9, mode, A.data_ptr(), lam.data_ptr(), B.data_ptr())
    kept = mid[0]
    # values next to the 1e-12 cutoff may fall either way; none here but the zeros of "rank"
    want = int(np.sum(s > 1e-12 * s[0]))
    assert kept == want
    tol = 10 * max(p, n) * np.finfo(float).eps
    nrm = np.sqrt(np.sum(ref[:kept] ** 2))
    assert np.abs(lam.cpu().numpy()[:kept] - ref[:kept] / nrm).max() <= tol
    Ah = A.cpu().numpy()[: p * kept].reshape(p, kept)
    Bh = B.cpu().numpy()[: kept * n].reshape(kept, n)
    assert np.abs(Ah.T @ Ah - np.eye(kept)).max() <= 1e-12
    assert np.abs(Bh @ Bh.T - np.eye(kept)).max() <= 1e-12
    assert np.abs((Ah * lam.cpu().numpy()[:kept]) @ Bh - M / nrm).max() <= tol
    assert trunc <= 1e-20
