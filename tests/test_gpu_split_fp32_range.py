"""FP32 split (mode 2) near the top of FP32's range: squared column norms up to the largest FP32 number.

Bound: the factorisation to max(p, n) FP32 roundings of the largest value, the kept left vectors
orthonormal in FP64 (1e-12)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


@pytest.mark.parametrize("scale", [1.0, 1e19, 1.35e19, 1.6e19, 1.8e19])
@pytest.mark.parametrize("kind", ["decay", "flat", "rank1"])
@pytest.mark.parametrize("p,n", [(8, 8), (40, 33), (100, 64)])
def test_largest_columns(p, n, kind, scale):
    rng = np.random.default_rng(p + n)
    k = min(p, n)
    U, V = (np.linalg.qr(rng.standard_normal((x, k)))[0] for x in (p, n))
    if kind == "rank1":                            # two columns of nearly the largest norm, parallel
        U, s = U[:, :2], np.array([1.0, 1e-3])
        V = np.zeros((n, 2))
        V[[0, 1], 0] = np.sqrt(0.5)
        V[2, 1] = 1.0
    else:
        s = 0.8 ** np.arange(k) if kind == "decay" else np.linspace(1.0, 0.9, k)
    M = (U * s) @ V.T * scale
    assert np.sum(M ** 2, axis=0).max() < 3.4e38
    bond = pd.Bond([0], {0: p}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.from_numpy(np.ascontiguousarray(M).ravel()).cuda()
    A, lam, B = (torch.zeros(size, dtype=torch.float64, device="cuda") for size in (p * k, k, k * n))
    mid, _ = pd.svd_split(bond, x.data_ptr(), 10 ** 9, 2, A.data_ptr(), lam.data_ptr(), B.data_ptr())
    r = mid[0]
    Ah, Bh = A.cpu().numpy()[: p * r].reshape(p, r), B.cpu().numpy()[: r * n].reshape(r, n)
    got = (Ah * lam.cpu().numpy()[:r]) @ Bh
    want = M / np.linalg.norm(M)                   # (what the 1e-5 cutoff drops is below the bound squared)
    assert np.abs(got - want).max() <= max(p, n) * 2.0 ** -23 + 1e-5
    assert np.abs(Ah.T @ Ah - np.eye(r)).max() <= 1e-12
