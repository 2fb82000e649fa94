"""Orthonormality of a split's vectors where the finishing series takes over from Newton-Schulz steps and
the triangular products meet their 64-column tiles: spectra flat (rotations orthonormal to 1e-6), mild
and graded (1e-3 and worse).  The last step's own bound is 1e-13 (FP32 split, the left factor) and
1e-14 (FP64, the rotations); columns normalised by computed norms add rounding: 1e-12 for both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("p,n", [(1, 1), (63, 63), (64, 64), (65, 65), (130, 127), (300, 257)])
@pytest.mark.parametrize("decay", [1.0, 0.97, 0.8])
def test_vectors_are_orthonormal(decay, p, n, mode):
    rng = np.random.default_rng(n)
    U = np.linalg.qr(rng.standard_normal((p, n)))[0]
    V = np.linalg.qr(rng.standard_normal((n, n)))[0]
    s = np.maximum(decay ** np.arange(n), 1e-4) * (1 + 0.01 * rng.random(n))
    M = (U * s) @ V.T
    bond = pd.Bond([0], {0: p}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.from_numpy(np.ascontiguousarray(M).ravel()).cuda()
    A, lam, B = (torch.zeros(p * n + 16, dtype=torch.float64, device="cuda") for _ in range(3))
    mid, _ = pd.svd_split(bond, x.data_ptr(), 10 ** 9, mode, A.data_ptr(), lam.data_ptr(), B.data_ptr())
    k = mid[0]
    assert k == n
    Ah = A.cpu().numpy()[: p * k].reshape(p, k)
    assert np.abs(Ah.T @ Ah - np.eye(k)).max() <= 1e-12
    if mode == 0:
        Bh = B.cpu().numpy()[: k * n].reshape(k, n)
        assert np.abs(Bh @ Bh.T - np.eye(k)).max() <= 1e-12
