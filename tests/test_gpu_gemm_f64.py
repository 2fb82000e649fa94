"""Grouped FP64 GEMM on the FP64 units (dmrg_gemm64 mode 0) against numpy, at the edges of its tiles
and in each of its shapes (one warp per 16 x 16 tile; 4 or 16 warps sharing the K of one).

Bound: a K-term dot product in any order is within K 2^-53 sum |a||b| of the exact one (so is
numpy's), alpha and the accumulation add one rounding each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")


# (blocks of M x N, K of each segment, how many such problems): few tiles split K over 16 warps
# (K >= 256) or 4 (below), short K and large batches run one warp per tile
CASES = [([(1, 1)], [1], 1), ([(16, 16), (17, 15), (33, 8)], [64, 65], 2), ([(9, 3), (8, 4), (7, 5)], [200], 3),
         ([(31, 37), (2, 50)], [300, 7], 2), ([(31, 37)], [3, 1, 2], 5), ([(5, 19), (40, 2)], [5] * 80, 2), ([(15, 15)], [15], 40),
         ([(130, 67)], [41], 30), ([(321, 300)], [37, 2], 26)]


@pytest.mark.parametrize("order", ["kk", "mk", "km"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_gemm_f64_shapes(case, order):
    blocks, ks, reps = CASES[case]
    rng = np.random.default_rng(100 + case)
    probs, segs, A, B, want, bound = [], [], [], [], [], []
    na = nb = nc = 0
    C0 = []
    for rep in range(reps):
        for i, (M, N) in enumerate(blocks):
            acc, alpha = (rep + i) % 2, 1.0 if rep % 3 else -0.75
            seg0, ref, ab = len(segs), np.zeros((M, N)), np.zeros((M, N))
            for K in ks:
                a, b = rng.standard_normal((M, K)), rng.standard_normal((N, K))
                segs.append((na, nb, K))
                # leading dimensions are the problem's: pad every segment to the longest K
                pa = np.zeros((M, max(ks)))
                pa[:, :K] = a
                pb = np.zeros((N, max(ks)))
                pb[:, :K] = b
                A.append((pa if order[0] == "k" else pa.T).ravel())
                B.append((pb if order[1] == "k" else pb.T).ravel())
                na += pa.size
                nb += pb.size
                ref += a @ b.T
                ab += np.abs(a) @ np.abs(b).T
            sam, sak = (max(ks), 1) if order[0] == "k" else (1, M)
            sbn, sbk = (max(ks), 1) if order[1] == "k" else (1, N)
            c0 = rng.standard_normal((N, M))
            probs.append((M, N, seg0, len(ks), nc, sam, sak, sbn, sbk, 1, M, acc, alpha))
            C0.append(c0.ravel())
            nc += c0.size
            want.append((alpha * ref + acc * c0.T).T.ravel())
            bound.append((2.0 ** -53 * ((2 * sum(ks) + 2) * abs(alpha) * ab + 2 * acc * np.abs(c0.T))).T.ravel())
    dev = lambda parts: torch.from_numpy(np.concatenate(parts)).cuda()  # noqa: E731
    Ad, Bd, Cd = dev(A), dev(B), dev(C0)
    pd.gemm64(probs, segs, Ad.data_ptr(), Bd.data_ptr(), Cd.data_ptr(), mode=0)
    err = np.abs(Cd.cpu().numpy() - np.concatenate(want))
    assert np.all(err <= np.concatenate(bound)), float((err / np.concatenate(bound)).max())
