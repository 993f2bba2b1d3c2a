"""GPU parity of the loss and bias-gradient kernels at the edges of their splits: class
counts around the register forms (32, 128, 1024), minibatches around the rows of a CTA
and over many CTAs per worker, both precisions, against the oracle; and a poisoned
sample in a worker's later CTA."""
import numpy as np
import pytest
import torch

from paper_2004_14696_gb300 import dbw, workloads
from paper_2004_14696_gb300.pipeline import Iteration
from gpu_util import RTOL_BF16, RTOL_FP32, assert_worker_grads_match

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def make(C, B, prec, n=3):
    wl = workloads.Workload(key="loss_bias", widths=(20, C), n=n, B=B, prec=prec, S=400, feature_dist="normal",
                            time_model="shifted_exp", time_params={"shift": 1.0, "rate": 1.0}, lr=0.01,
                            seed_offset=111)
    it = Iteration(wl, static_b=0)
    it.load_inputs(0)
    return wl, it


def run(wl, it):
    dbw.dbw_worker_grads(wl.widths, wl.prec, it.w, it.pool, it.labels, it.idx, wl.n, wl.B, it.G, it.loss, it.ws)
    torch.cuda.synchronize()


@pytest.mark.parametrize("prec", [workloads.PREC_FP32, workloads.PREC_BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("C,B", [(2, 1), (2, 500), (10, 64), (10, 65), (31, 63), (32, 500), (33, 32), (33, 33),
                                 (128, 70), (129, 16), (129, 17), (1024, 40), (1025, 40), (7, 1100)])
def test_loss_and_bias_at_the_edges(C, B, prec):
    wl, it = make(C, B, prec)
    idx, _ = it.host_inputs(0)
    run(wl, it)
    pool, labels, w = it.pool.cpu().numpy(), it.labels.cpu().numpy(), it.w.cpu().numpy()
    bf16 = prec == workloads.PREC_BF16
    assert_worker_grads_match(it.G.cpu().numpy()[:, :wl.d], it.loss.cpu().numpy(), wl.widths, w, pool[idx], labels[idx],
                              B, bf16, range(wl.n), RTOL_BF16 if bf16 else RTOL_FP32)
    first = it.loss.clone()
    run(wl, it)   # the counters start from zero again
    assert torch.equal(first, it.loss)


@pytest.mark.parametrize("prec", [workloads.PREC_FP32, workloads.PREC_BF16], ids=["fp32", "bf16"])
def test_a_bad_sample_in_a_later_cta_poisons_its_worker(prec):
    wl, it = make(10, 300, prec)
    it.idx[300 + 290] = wl.S
    run(wl, it)
    loss, G = it.loss.cpu().numpy(), it.G.cpu().numpy()[:, :wl.d]
    assert np.isnan(loss[1]) and np.isfinite(loss[[0, 2]]).all()
    assert np.isnan(G[1]).all() and np.isfinite(G[[0, 2]]).all()
