"""GPU parity of the aggregation's wide form (columns in pieces of 2048 per CTA, rows
streamed through shared memory four at a time), which serves d >= 8,000,000: whole and
ragged last pieces, numbers of rows around the groups of four, with and without every
row's norm, against the oracle; and the shorter form just below the line."""
import numpy as np
import pytest
import torch

from oracle import dbw_oracle as O
from paper_2004_14696_gb300 import dbw
from gpu_util import RTOL_FP32, assert_close_rows, assert_close_scalar

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


CASES = [(1, 8_000_000, 1), (2, 8_001_537, 1), (3, 8_000_003, 2), (4, 8_001_536, 4), (5, 8_001_535, 3),
         (6, 8_003_585, 5), (9, 8_000_001, 9), (6, 7_999_999, 5)]


@pytest.mark.parametrize("n,d,k", CASES)
def test_aggregate_wide(n, d, k):
    g = torch.Generator(device="cuda").manual_seed(n + d)
    ld = -(-d // 4) * 4
    G = 0.3 + torch.randn((n, ld), generator=g, device="cuda")
    G[:, d:] = float("nan")
    w0 = torch.randn(d, generator=g, device="cuda")
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    mask[torch.randperm(n, generator=g, device="cuda")[:k]] = 1
    Gh, wh, mh = G.cpu().numpy()[:, :d].astype(np.float64), w0.cpu().numpy(), mask.cpu().numpy()
    gbar = O.aggregate(Gh, mh)
    SS, norms = O.deviation_sumsq(Gh, mh, gbar), np.einsum("ij,ij->i", Gh, Gh)
    got = []
    for flags in (0, dbw.ALL_ROW_NORMS):
        w, gb = w0.clone(), torch.empty(d, device="cuda")
        part = torch.empty(dbw.dbw_aggregate_partials_bytes(n, d), dtype=torch.uint8, device="cuda")
        dbw.dbw_aggregate_update(G, n, d, mask, 0.05, w, part, gb, flags=flags)
        state = dbw.new_state(n, 5)
        stats = torch.empty(dbw.STATS_LEN, dtype=torch.float64, device="cuda")
        rows = torch.empty(n, dtype=torch.float64, device="cuda")
        dbw.dbw_grad_stats(part, n, mask, torch.ones(n, device="cuda"),
                           torch.arange(n, dtype=torch.float64, device="cuda"), 0.05, state, stats, rows)
        torch.cuda.synchronize()
        assert_close_rows(gb.cpu().numpy(), gbar, RTOL_FP32, "g_t")
        assert_close_rows(w.cpu().numpy(), O.sgd_update(wh, gbar, 0.05), RTOL_FP32, "w")
        s, r = stats.cpu().numpy(), rows.cpu().numpy()
        assert_close_scalar(s[dbw.STAT_GBAR_SQ], float(gbar @ gbar), RTOL_FP32, "||g_t||^2")
        if k > 1:
            assert_close_scalar(s[dbw.STAT_SS], SS, RTOL_FP32, "SS")
        else:
            assert s[dbw.STAT_SS] == 0.0
        for j in range(n):
            if mh[j] or flags:
                assert_close_scalar(r[j], norms[j], RTOL_FP32, f"||g_{j}||^2")
            else:
                assert np.isnan(r[j])
        got.append((w, gb, s, r[mh == 1]))
    # the received rows go through the same arithmetic with and without the others
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][2], got[1][2], equal_nan=True) and np.array_equal(got[0][3], got[1][3])


@pytest.mark.parametrize("flags", [0, dbw.ALL_ROW_NORMS])
@pytest.mark.parametrize("d", [7_999_999, 8_000_003])   # either side of the line
def test_one_received_row_is_its_own_mean(d, flags):
    """k = 1: g_t is the row, infinities and NaN included, and no entry deviates from it."""
    n, ld, lr = 3, -(-d // 4) * 4, 0.05
    g = torch.Generator(device="cuda").manual_seed(d)
    G = torch.randn((n, ld), generator=g, device="cuda")
    row = G[1]
    row[0], row[d // 2], row[d // 2 + 1], row[d - 1] = float("inf"), -float("inf"), torch.finfo(torch.float32).min, float("inf")
    mask = torch.tensor([0, 1, 0], dtype=torch.uint8, device="cuda")
    for nan in (False, True):
        if nan:
            row[5] = float("nan")
        w0 = torch.randn(d, generator=g, device="cuda")
        w, gb = w0.clone(), torch.empty(d, device="cuda")
        part = torch.empty(dbw.dbw_aggregate_partials_bytes(n, d), dtype=torch.uint8, device="cuda")
        dbw.dbw_aggregate_update(G, n, d, mask, lr, w, part, gb, flags=flags)
        state, stats = dbw.new_state(n, 5), torch.empty(dbw.STATS_LEN, dtype=torch.float64, device="cuda")
        rows = torch.empty(n, dtype=torch.float64, device="cuda")
        dbw.dbw_grad_stats(part, n, mask, torch.ones(n, device="cuda"),
                           torch.arange(n, dtype=torch.float64, device="cuda"), lr, state, stats, rows)
        torch.cuda.synchronize()
        assert torch.equal(gb.nan_to_num(7.0, 8.0, 9.0), row[:d].nan_to_num(7.0, 8.0, 9.0))
        step = torch.addcmul(w0.double(), row[:d].double(), torch.tensor(-np.float32(lr), device="cuda").double())
        step = step.float()   # one rounding, as the kernel's fused multiply-add
        assert torch.equal(w.nan_to_num(7.0, 8.0, 9.0), step.nan_to_num(7.0, 8.0, 9.0))
        s, r = stats.cpu().numpy(), rows.cpu().numpy()
        assert s[dbw.STAT_SS] == 0.0
        assert np.isnan(s[dbw.STAT_GBAR_SQ]) if nan else np.isposinf(s[dbw.STAT_GBAR_SQ])
        assert np.isnan(r[1]) if nan else np.isposinf(r[1])
        assert np.isfinite(r[[0, 2]]).all() if flags else np.isnan(r[[0, 2]]).all()
