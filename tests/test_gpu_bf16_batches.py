"""GPU parity of the bf16 pass at minibatches off the 32- and 64-deep K blocks of the
weight-gradient kernel and off the 16-row steps of its MMAs, and at those that the FFMA
tiles serve (a ragged B below 96, or in a model of more than three layers): every worker's
gradient row and loss against the oracle.  On the tensor cores a worker's rows past its B
samples belong to the next worker (or lie past the buffer); the kernel has to read them as
zero.  The FFMA pass stores its rows unpadded, so odd widths start them on 2 bytes."""
import pytest
import torch

from paper_2004_14696_gb300 import dbw, workloads
from paper_2004_14696_gb300.pipeline import Iteration
from gpu_util import RTOL_BF16, assert_worker_grads_match, gpu_active_sets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


# (widths, n, B): B at and around the K blocks, M = n B at and around 32-, 128- and 256-row
# tiles; (36, 18, 10) stores its second layer with scalar stores (rows off 16 bytes)
CASES = [((68, 40, 10), 3, B) for B in (1, 16, 17, 33, 50, 95, 97, 100, 111, 113, 127, 129, 191,
                                                     193, 225)]
CASES += [((36, 18, 10), 2, 17), ((36, 18, 10), 3, 97), ((68, 40, 36, 34, 10), 3, 100),
          ((68, 40, 36, 10), 3, 161), ((200, 96, 10), 1, 1), ((260, 300, 7), 1, 129), ((256, 130, 34), 5, 51),
          ((256, 131, 33), 2, 51), ((64, 320), 1, 255)]


@pytest.mark.parametrize("widths,n,B", CASES, ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_bf16_gradients_at_any_batch(widths, n, B):
    wl = workloads.Workload(key="bf16_batch", widths=widths, n=n, B=B, prec=workloads.PREC_BF16, S=300,
                            feature_dist="normal", time_model="shifted_exp",
                            time_params={"shift": 1.0, "rate": 1.0}, lr=0.01, seed_offset=110)
    it = Iteration(wl, static_b=0)
    idx, _ = it.host_inputs(0)
    it.load_inputs(0)
    it.G.fill_(float("nan"))
    dbw.dbw_worker_grads(wl.widths, wl.prec, it.w, it.pool, it.labels, it.idx, n, B, it.G, it.loss, it.ws)
    torch.cuda.synchronize()
    assert int(it.ws[:4].view(torch.int32).item()) == 0, "device status word set"
    pool, labels, w = it.pool.cpu().numpy(), it.labels.cpu().numpy(), it.w.cpu().numpy()
    assert_worker_grads_match(it.G.cpu().numpy()[:, :wl.d], it.loss.cpu().numpy(), widths, w, pool[idx], labels[idx],
                              B, True, range(n), RTOL_BF16, gpu_active_sets(it.ws, widths, n, B, wl.prec))
