"""GPU test of the bounded-wait path of the tensor-core kernels and of the wide aggregation.

Every wait of a tensor-core kernel on a pipeline barrier is bounded.  When one runs
out the kernel raises bit 0 of the status word, stops, waits (bounded) for its own
copies still in flight, releases its tensor memory and returns.  The test makes one
wait run out without faulting anything: dbw_test_arm_wait_timeout keeps the first
CTA of the next weight-gradient launch from issuing one stage's TMA load (no copy is
then outstanding for that stage) and shortens the bound to 1 ms.  Then: the call
returns, the status word has bit 0 set, and the next normal call on the same process
(which allocates the same tensor memory again) gives the oracle's result.  A tiny
shape only.  The aggregation has no status word: the columns whose rows did not arrive
keep w and g_t, and dbw_grad_stats raises a flag of the state and records nothing."""
import numpy as np
import pytest
import torch

from oracle import dbw_oracle as O
from paper_2004_14696_gb300 import dbw, workloads
from paper_2004_14696_gb300.pipeline import Iteration
from gpu_util import RTOL_BF16, assert_worker_grads_match, gpu_active_sets

pytestmark = pytest.mark.gpu

TINY = workloads.Workload(key="wait_tiny", widths=(64, 32, 10), n=2, B=32, prec=workloads.PREC_BF16, S=200,
                          feature_dist="normal", time_model="shifted_exp", time_params={"shift": 1.0, "rate": 1.0},
                          lr=0.01, seed_offset=97)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _grads(it):
    wl = it.wl
    dbw.dbw_worker_grads(wl.widths, wl.prec, it.w, it.pool, it.labels, it.idx, wl.n, wl.B, it.G, it.loss, it.ws)
    torch.cuda.synchronize()
    return int(it.ws[:4].view(torch.int32).item())


def test_a_wait_that_runs_out_sets_the_status_and_the_next_call_is_exact():
    wl = TINY
    it = Iteration(wl, static_b=0)
    it.load_inputs(0)
    assert _grads(it) == 0
    dbw.dbw_test_arm_wait_timeout(0, 1.0)
    assert _grads(it) & 1, "the wait for the stage without its load did not run out"
    # armed once: the next call is a normal one, on the same process and tensor memory
    assert _grads(it) == 0
    w = it.w.cpu().numpy().astype(np.float64)
    idx, _ = it.host_inputs(0)
    pool, labels = it.pool.cpu().numpy(), it.labels.cpu().numpy()
    assert_worker_grads_match(it.G.cpu().numpy()[:, :wl.d], it.loss.cpu().numpy(), wl.widths, w, pool[idx],
                              labels[idx], wl.B, True, range(wl.n), RTOL_BF16,
                              gpu_active=gpu_active_sets(it.ws, wl.widths, wl.n, wl.B, wl.prec))


def test_arming_is_checked_and_can_be_undone():
    with pytest.raises(dbw.DbwError):
        dbw.dbw_test_arm_wait_timeout(0, 0.0)
    with pytest.raises(dbw.DbwError):
        dbw.dbw_test_arm_wait_timeout(0, 5000.0)
    dbw.dbw_test_arm_wait_timeout(0, 1.0)
    dbw.dbw_test_arm_wait_timeout(-1, 0.0)          # disarmed: the next call runs normally
    it = Iteration(TINY, static_b=0)
    it.load_inputs(0)
    assert _grads(it) == 0


@pytest.mark.parametrize("flags", [0, dbw.ALL_ROW_NORMS])
@pytest.mark.parametrize("stage", [0, 2, 3, 10])   # rows 0 and 2 of the first chunk of 3 rows, 0 of the 2nd, 1 of the 4th
def test_an_aggregation_that_loses_rows_takes_no_step_from_them(stage, flags):
    n, k, d, lr = 4, 3, 8_000_003, 0.05
    rows = n if flags else k
    g = torch.Generator(device="cuda").manual_seed(d)
    G = torch.randn((n, -(-d // 4) * 4), generator=g, device="cuda")
    w0 = torch.randn(d, generator=g, device="cuda")
    mask = torch.tensor([1, 0, 1, 1], dtype=torch.uint8, device="cuda")
    loss, times = torch.ones(n, device="cuda"), torch.arange(n, dtype=torch.float64, device="cuda")

    def call():
        w, gb = w0.clone(), torch.full((d,), 7.0, device="cuda")
        part = torch.zeros(dbw.dbw_aggregate_partials_bytes(n, d), dtype=torch.uint8, device="cuda")
        dbw.dbw_aggregate_update(G, n, d, mask, lr, w, part, gb, flags=flags)
        state = dbw.new_state(n, 5)
        stats = torch.full((dbw.STATS_LEN,), -1.0, dtype=torch.float64, device="cuda")
        norms = torch.zeros(n, dtype=torch.float64, device="cuda")
        dbw.dbw_grad_stats(part, n, mask, loss, times, lr, state, stats, norms)
        torch.cuda.synchronize()
        return w, gb, dbw.read_state(state), stats, norms, int(part[:32].view(torch.int64)[1])

    w1, g1, s1, stats1, norms1, blocks = call()
    assert s1.flags & dbw.FLAG_WAIT_TIMEOUT == 0 and s1.t == 1 and torch.isfinite(norms1[mask.bool()]).all()
    dbw.dbw_test_arm_wait_timeout(stage, 5.0)
    w, gb, s, stats, norms, _ = call()
    # the first block's chunks of 2048 columns, from the one that lost a row on
    col = torch.arange(d, device="cuda") // 2048
    lost = (col % blocks == 0) & (col // blocks >= stage // rows)
    assert torch.equal(w, torch.where(lost, w0, w1))
    assert torch.equal(gb, torch.where(lost, torch.full_like(g1, 7.0), g1))
    assert s.flags == dbw.FLAG_WAIT_TIMEOUT
    assert s.t == 0 and s.c == 0 and s.cntV == 0 and s.cntN == 0 and not any(s.S[:n]) and s.vclock == 0.0
    assert (stats == -1.0).all() and torch.isnan(norms).all()
    # armed once: the next call is a normal one
    w, gb, s, stats, norms, _ = call()
    assert torch.equal(w, w1) and torch.equal(gb, g1) and torch.equal(stats.nan_to_num(), stats1.nan_to_num())
    assert s.flags == s1.flags and torch.equal(norms.nan_to_num(), norms1.nan_to_num())
