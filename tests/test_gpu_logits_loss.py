"""GPU parity of the fp32 pass where the last layer's logits and the loss are one launch (at
most 16 outputs, 16-byte operand rows): output counts up to the limit and past it, the short and
the long row forms, a single layer (rows straight from the pool) and one above others, and
minibatches around the rows of a CTA; and a sample index outside the pool in a single layer."""
import numpy as np
import pytest
import torch

from paper_2004_14696_gb300 import dbw, workloads
from paper_2004_14696_gb300.pipeline import Iteration
from gpu_util import RTOL_FP32, assert_worker_grads_match, gpu_active_sets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def run(widths, n, B):
    wl = workloads.Workload(key="logits_loss", widths=widths, n=n, B=B, prec=workloads.PREC_FP32, S=400,
                            feature_dist="normal", time_model="shifted_exp",
                            time_params={"shift": 1.0, "rate": 1.0}, lr=0.01, seed_offset=130)
    it = Iteration(wl, static_b=0)
    it.load_inputs(0)
    it.G.fill_(float("nan"))

    def go():
        dbw.dbw_worker_grads(wl.widths, wl.prec, it.w, it.pool, it.labels, it.idx, n, B, it.G, it.loss, it.ws)
        torch.cuda.synchronize()
        return it.G.cpu().numpy()[:, :wl.d], it.loss.cpu().numpy()
    return wl, it, go


CASES = [((4, 2), 1, 1), ((784, 10), 3, 33), ((256, 16), 2, 5), ((260, 16), 2, 4), ((516, 3), 1, 130), ((128, 17), 2, 9),
         ((20, 24, 10), 3, 7), ((24, 300, 16), 2, 50), ((24, 30, 10), 2, 6), ((8, 7), 600, 17)]


@pytest.mark.parametrize("widths,n,B", CASES, ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_logits_and_loss(widths, n, B):
    wl, it, go = run(widths, n, B)
    idx, _ = it.host_inputs(0)
    G, loss = go()
    pool, labels, w = it.pool.cpu().numpy(), it.labels.cpu().numpy(), it.w.cpu().numpy()
    active = gpu_active_sets(it.ws, widths, n, B, wl.prec) if len(widths) > 2 else None
    assert_worker_grads_match(G, loss, widths, w, pool[idx], labels[idx], B, False, range(0, n, max(1, n // 8)), RTOL_FP32,
                              active)


def test_a_sample_outside_the_pool_poisons_its_worker_only():
    wl, it, go = run((784, 10), 3, 33)
    it.idx[33 + 20] = wl.S
    it.idx[2 * 33 + 1] = it.idx[2 * 33]
    G, loss = go()
    assert np.isnan(loss[1]) and np.isfinite(loss[[0, 2]]).all()
    assert np.isnan(G[1]).all() and np.isfinite(G[[0, 2]]).all()
