"""GPU parity of the mean-gradient GEMM where it splits the K of its last tiles into ranges
(few tiles or a partial last round of them, K = k B long) and another kernel of the pass adds
the ranges: g_t, the step and ||g_t||^2 against the mean of the same workers' gradient rows from
the two-call form, which never splits."""
import pytest
import torch

from paper_2004_14696_gb300 import dbw, workloads
from paper_2004_14696_gb300.pipeline import Iteration

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


# (widths, n, B, b): one tile of eight ranges; one worker left (K too short to split); ragged
# tiles whose 32 x 128 blocks end inside or lie outside the matrix, rows off 16 bytes; 90 tiles
# (more than the pairs of SMs) of which the last 14 are split, whatever the count of pairs up
# to 89; the problem's tiles dealt around dX tiles of two layers
CASES = [((256, 96, 10), 32, 64, 0), ((256, 96, 10), 32, 64, 31), ((300, 301, 130, 7), 16, 128, 3),
         ((2560, 2052, 10), 64, 32, 0), ((512, 520, 264, 34), 48, 64, 16)]


@pytest.mark.parametrize("with_gbar", [True, False], ids=["gbar", "nogbar"])
@pytest.mark.parametrize("widths,n,B,b", CASES, ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_split_mean_gradient(widths, n, B, b, with_gbar):
    wl = workloads.Workload(key="rx_ranges", widths=widths, n=n, B=B, prec=workloads.PREC_BF16, S=500,
                            feature_dist="normal", time_model="shifted_exp",
                            time_params={"shift": 1.0, "rate": 1.0}, lr=0.01, seed_offset=120)
    it = Iteration(wl, static_b=b, received=True)
    it.load_inputs(0)
    mask = torch.ones(n, dtype=torch.uint8, device="cuda")
    mask[:b] = 0
    k = n - b
    two = Iteration(wl, static_b=b)
    dbw.dbw_worker_grads(widths, wl.prec, two.w, it.pool, it.labels, it.idx, n, B, two.G, two.loss, two.ws)
    rows = two.G[b:, :wl.d].double()
    ref, largest = rows.mean(0), rows.abs().max().item()
    w0 = it.w.clone()
    gbar = torch.full((wl.d,), float("nan"), device="cuda") if with_gbar else None
    it.ws.fill_(0xff)   # no result may rest on what the scratch held
    dbw.dbw_received_grads_update(widths, wl.prec, it.w, it.pool, it.labels, it.idx, n, B, mask, 0.5, it.loss,
                                  it.partials, it.ws, gbar)
    torch.cuda.synchronize()
    assert int(it.ws[:4].view(torch.int32).item()) == 0, "device status word set"
    # both forms round a running sum at most once per MMA (16 samples) and range, by 2^-24 of a
    # partial sum, and no partial sum of the mean is taken to exceed the largest entry of a worker's row
    tol = (k * B / 16 + 8 + B / 16) * 2.0 ** -24 * largest
    step = it.w.double() - (w0.double() - 0.5 * ref)
    assert step.abs().max().item() <= 0.5 * tol + 2.0 ** -24 * w0.abs().max().item()
    if with_gbar:
        assert (gbar.double() - ref).abs().max().item() <= tol
        sq = it.partials.view(torch.float64)[-1].item()   # the last quantity of the one block
        want = (gbar.double() ** 2).sum().item()
        # fp32 sums of at most 32 squares, added in fp64
        assert abs(sq - want) <= 32 * 2.0 ** -24 * want
