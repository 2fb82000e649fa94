"""Tensor-core grouped GEMM at the edges of its tiles (128 rows, 64/128/256 columns read in pieces of 16
or 32 by sixteen warps), with one to five segments a problem, one tile in all, and more tiles than three
rounds of the persistent grid.  Through the FP64-accurate emulation (dmrg_gemm64 mode 1), whose products are
exact sums of tensor-core GEMMs: error at most 8 K 2^-53 max|A| max|B| an element, plus an ulp."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


def _run(shapes):
    rng = np.random.default_rng(len(shapes))
    A, B, probs, segs, ref = [], [], [], [], []
    na = nb = nc = 0
    for i, (M, N, Ks) in enumerate(shapes):
        seg0, acc = len(segs), np.zeros((M, N))
        bound = np.zeros((M, N))
        a = [rng.standard_normal((M, K)) for K in Ks]
        b = [rng.standard_normal((N, K)) for K in Ks]
        ld = max(Ks)
        for x, y in zip(a, b):
            for buf, z in ((A, x), (B, y)):
                w = np.zeros((z.shape[0], ld))
                w[:, : z.shape[1]] = z
                buf.append(w.ravel())
            segs.append((na, nb, x.shape[1]))
            na, nb = na + M * ld, nb + N * ld
            acc += x @ y.T
        amax = np.max([np.abs(x).max(1) for x in a], 0)
        bmax = np.max([np.abs(y).max(1) for y in b], 0)
        probs.append((M, N, seg0, len(Ks), nc, ld, 1, ld, 1, 1, M, 0, 1.0))
        nc += M * N
        ref.append((acc, 8 * sum(Ks) * 2.0 ** -53 * np.outer(amax, bmax) + 2.0 ** -52 * np.abs(acc)))
    dA, dB = (torch.as_tensor(np.concatenate(z)).cuda() for z in (A, B))
    C = torch.full((nc,), float("nan"), dtype=torch.float64, device="cuda")
    pd.gemm64(probs, segs, dA.data_ptr(), dB.data_ptr(), C.data_ptr(), 1)
    c = C.cpu().numpy()
    for p, (acc, bound) in zip(probs, ref):
        M, N, off = p[0], p[1], p[4]
        assert np.all(np.abs(c[off: off + M * N].reshape(N, M).T - acc) <= bound), p


@pytest.mark.parametrize("N", [1, 15, 16, 17, 31, 33, 63, 64, 65, 97, 128, 129, 255, 256, 257])
def test_tile_edges(N):
    _run([(M, N, Ks) for M in (1, 31, 32, 33, 127, 128, 129) for Ks in ([1], [64], [65, 63], [7, 130, 1, 64, 65])])


def test_one_tile():
    _run([(40, 40, [40])])


def test_more_tiles_than_the_grid_takes_in_three_rounds():
    rng = np.random.default_rng(0)
    _run([(int(rng.integers(1, 200)), int(rng.integers(1, 200)), [int(k) for k in rng.integers(1, 150, rng.integers(1, 4))])
          for _ in range(700)])
