"""Device memory that the library keeps: given back by trim(), and by the last context that is closed."""
import numpy as np
import pytest

import workloads as wl
from tests._gpu import engine_for, load_mps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
pd = pytest.importorskip("paper_1301_3494_gb300")

SLACK = 8 << 20          # (pool granularity is 2 MiB; the rest of the process allocates nothing in between)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_trim_gives_back_what_single_operations_keep():
    n = 1500                                      # some ten work matrices of 18 MB
    x = torch.eye(n, dtype=torch.float64, device="cuda").ravel()
    A, lam, B = (torch.zeros(s, dtype=torch.float64, device="cuda") for s in (n * n, n, n * n))
    bond = pd.Bond([0], {0: n}, {0: n}, np.zeros((1, 1, 1, 1)), [0], [0])

    def split():
        pd.svd_split(bond, x.data_ptr(), 10 ** 9, 0, A.data_ptr(), lam.data_ptr(), B.data_ptr())

    split()                                       # (kernels loaded)
    pd.trim()
    base = _free()
    split()
    assert base - _free() <= (2 << 30) + SLACK
    pd.trim()
    assert _free() >= base - SLACK
    split()                                       # and goes on working
    pd.trim()


def test_the_last_context_gives_everything_back():
    mpo = wl.heisenberg_chain(16)
    qn = list(mpo.site.qn)

    def run(n):
        engs = [engine_for(pd, mpo) for _ in range(n)]
        for e in engs:
            load_mps(e, wl.random_mps(16, qn, 0, 128, seed=1), qn)
            e.sweep(128)
        for e in engs:
            e.close()

    run(1)
    base = _free()
    bond = pd.Bond([0], {0: 1500}, {0: 1500}, np.zeros((1, 1, 1, 1)), [0], [0])
    x = torch.eye(1500, dtype=torch.float64, device="cuda").ravel()
    out = [torch.zeros(s, dtype=torch.float64, device="cuda") for s in (1500 * 1500, 1500, 1500 * 1500)]
    own = base - _free()                          # the test's own buffers
    pd.svd_split(bond, x.data_ptr(), 10 ** 9, 0, *(t.data_ptr() for t in out))
    run(2)
    assert _free() >= base - own - SLACK
