"""FP64 splits of exactly low-rank matrices and of matrices outside FP32's range: the null columns (bitwise
multiples of each other) neither keep the split busy nor spoil it, and columns below what FP32 holds are
scaled before they are converted.

Bounds as for any split: 10 n eps for values and the factorisation, 1e-12 for orthonormality; all are
finished by whole-matrix passes, at most 16 of them (a scalar Jacobi that does not converge reports 61)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "ones":
        return np.ones((n, n)), 1
    if kind in ("rank1", "rank3"):
        r = int(kind[4:])
        return (rng.integers(-5, 6, (n, r)) @ rng.integers(-5, 6, (r, n))).astype(float), r
    if kind == "twice":                       # every column two times
        return np.repeat(rng.standard_normal((n, n // 2)), 2, axis=1), n // 2
    U, V = (np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2))
    return (U * 0.9 ** np.arange(n)) @ V.T * {"small": 1e-60, "large": 1e60, "tiny": 1e-100, "huge": 1e80}[kind], n


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("kind,n", [("ones", 16), ("ones", 200), ("rank1", 20), ("rank3", 20), ("rank3", 200),
                                    ("twice", 200), ("small", 100), ("large", 100), ("tiny", 100), ("huge", 100)])
def test_null_columns_and_scales(kind, n, mode):
    M, rank = _matrix(kind, n)
    ref = np.linalg.svd(M, compute_uv=False)
    assert ref[rank - 1] > 1e-9 * ref[0]
    bond = pd.Bond([0], {0: n}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.from_numpy(np.ascontiguousarray(M).ravel()).cuda()
    A, lam, B = (torch.zeros(size, dtype=torch.float64, device="cuda") for size in (n * n, n, n * n))
    pd.profile_reset()
    pd.profile_enable()
    mid, trunc = pd.svd_split(bond, x.data_ptr(), 10 ** 9, mode, A.data_ptr(), lam.data_ptr(), B.data_ptr())
    prof = pd.profile_read()
    pd.profile_enable(False)
    assert mid == {0: rank}
    lam = lam.cpu().numpy()[:rank]
    Ah, Bh = A.cpu().numpy()[: n * rank].reshape(n, rank), B.cpu().numpy()[: n * rank].reshape(rank, n)
    nrm, tol = np.sqrt(np.sum(ref[:rank] ** 2)), 10 * n * np.finfo(float).eps
    assert np.abs(lam - ref[:rank] / nrm).max() <= tol
    assert np.abs((Ah * lam) @ Bh - M / nrm).max() <= tol
    assert max(np.abs(Ah.T @ Ah - np.eye(rank)).max(), np.abs(Bh @ Bh.T - np.eye(rank)).max()) <= 1e-12
    assert trunc <= 1e-20
    assert prof["svd_sweeps"] <= 16, prof["svd_sweeps"]


def test_rounding_noise_is_not_refined():
    """The accurate recursion on an exactly low-rank matrix: its noise is of low rank too, level after
    level, and nothing of it is kept, so mode 1 adds no decomposition (one takes well over 16 launches)."""
    n = 200
    x = torch.ones(n * n, dtype=torch.float64, device="cuda")
    bond = pd.Bond([0], {0: n}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    A, lam, B = (torch.zeros(size, dtype=torch.float64, device="cuda") for size in (n * n, n, n * n))
    launches = []
    for mode in (0, 1):
        pd.profile_reset()
        assert pd.svd_split(bond, x.data_ptr(), 10 ** 9, mode, A.data_ptr(), lam.data_ptr(), B.data_ptr())[0] == {0: 1}
        launches.append(pd.profile_read()["launches"])
    assert launches[1] <= launches[0] + 16, launches
