"""GPU parity of the two forms of the Eq. (17) fit (in shared memory; on the state buffer
for larger tables) on planted cell tables: sizes around a warp, ranks without samples
inside a row, and the last number of fitted rows that fits in shared memory at n = 96 (72),
256 (26) and 512 (12) with the first that does not, against the oracle's fit of the same
table."""
import numpy as np
import pytest
import torch

from oracle import psw_oracle as P
from paper_2004_14696_gb300 import dbw

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n,m", [(1, 1), (2, 2), (3, 1), (8, 8), (31, 20), (32, 32), (33, 33), (65, 40), (96, 1),
                                 (96, 72), (96, 73), (256, 26), (256, 27), (512, 12), (512, 13)])
def test_fit_forms_on_planted_tables(n, m):
    rng = np.random.default_rng(100 * n + m)
    unit = 2.0 ** -32
    sums, cnts = np.zeros((n, n), np.uint64), np.zeros((n, n), np.int32)
    for h in sorted(rng.choice(np.arange(1, n + 1), size=m, replace=False).tolist()):
        M = int(rng.integers(h, n + 1))
        i = np.arange(M)
        # increasing in the rank, decreasing in h, and noise that the projections pool
        mean = max(20.0, 0.05 * n) + 0.3 * i - 0.05 * h + rng.uniform(0.0, 2.0, size=M)
        c = rng.integers(1, 5, size=M)
        c[(rng.random(M) < 0.1) & (i != h - 1)] = 0
        sums[h - 1, :M] = np.round(mean * c / unit).astype(np.uint64)
        cnts[h - 1, :M] = c
    psw, ps = dbw.new_psw(n), P.psw_init(n)
    ps.sums[1:, 1:], ps.cnts[1:, 1:] = sums.astype(np.float64) * unit, cnts
    hdr = dbw.PswHeader.from_buffer_copy(psw[:256].cpu().numpy().tobytes())
    psw[hdr.off_sum:hdr.off_sum + 8 * n * n] = torch.from_numpy(sums.view(np.uint8).ravel()).cuda()
    psw[hdr.off_cnt:hdr.off_cnt + 4 * n * n] = torch.from_numpy(cnts.view(np.uint8).ravel()).cuda()
    T = torch.empty(n, dtype=torch.float64, device="cuda")
    ref = np.array(P.time_estimates(ps, tol=1e-11))
    for _ in range(2):   # cold, then warm from its own dual variables
        dbw.dbw_psw_estimate(psw, n, T, 1e-6)
        torch.cuda.synchronize()
        got = T.cpu().numpy()
        assert not dbw.read_psw(psw, n)["flags"]
        assert np.all(np.abs(got - ref) <= 1e-5 * np.abs(ref)), float(np.max(np.abs(got - ref) / np.abs(ref)))
