"""The loss mean of dbw_grad_stats is the fp64 sum over the received workers in increasing
worker order.  It is summed in parallel when the losses' exponents leave no rounding in
any order, else sequentially: both must give the sequential sum's bits, at the edge of
the exponent span, beyond it, and for zeros, subnormals, infinities and NaN."""
import numpy as np
import pytest
import torch

from paper_2004_14696_gb300 import dbw

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def losses(kind, n, rng):
    mant = (1.0 + rng.random(n)).astype(np.float32)
    sign = np.where(rng.random(n) < 0.3, -1.0, 1.0).astype(np.float32)
    if kind.startswith("span"):
        span = int(kind[4:])
        e = rng.integers(0, span + 1, n)
        e[0], e[-1] = 0, span
        return (sign * np.ldexp(mant, e - 7)).astype(np.float32)
    x = mant * sign
    if kind == "subnormal":
        x[::2] = np.float32(1e-42)
    elif kind == "all_subnormal":
        x = (rng.integers(-1000, 1000, n) * np.float32(1.4e-45)).astype(np.float32)
    elif kind == "zeros":
        x[::2] = 0.0
        x[1::4] = -0.0
    elif kind == "all_zero":
        x[:] = -0.0
    elif kind == "inf":
        x[n // 2] = np.inf
    elif kind == "nan":
        x[n // 2] = np.nan
    elif kind == "lowest":
        x[:] = -np.finfo(np.float32).max
    return x


@pytest.mark.parametrize("n", [1, 2, 33, 256, 1024])
@pytest.mark.parametrize("kind", ["span0", "span19", "span20", "span60", "subnormal", "all_subnormal", "zeros",
                                  "all_zero", "inf", "nan", "lowest"])
def test_loss_mean_is_the_sequential_sum(n, kind):
    rng = np.random.default_rng(n)
    x = losses(kind, n, rng)
    mask = (rng.random(n) < 0.8).astype(np.uint8)
    mask[n // 2] = 1
    acc = np.float64(0.0)
    for j in range(n):
        if mask[j]:
            acc = acc + np.float64(x[j])
    want = acc / np.float64(mask.sum())
    blocks = 3
    head = np.array([dbw.PARTIALS_MAGIC, blocks, n, 0], dtype=np.int64).view(np.uint8)
    vals = np.arange((n + 2) * blocks, dtype=np.float64)
    part = torch.from_numpy(np.concatenate([head, np.zeros(n + 2).view(np.uint8), vals.view(np.uint8)])).cuda()
    state = dbw.new_state(n, 5)
    stats = torch.zeros(dbw.STATS_LEN, dtype=torch.float64, device="cuda")
    rows = torch.zeros(n, dtype=torch.float64, device="cuda")
    dbw.dbw_grad_stats(part, n, torch.from_numpy(mask).cuda(), torch.from_numpy(x).cuda(),
                       torch.arange(n, dtype=torch.float64, device="cuda"), 0.1, state, stats, rows)
    torch.cuda.synchronize()
    got = np.float64(stats[dbw.STAT_F].item())
    assert got.tobytes() == want.tobytes() or (np.isnan(got) and np.isnan(want)), (got, want)
    sums = vals.reshape(n + 2, blocks).sum(1)
    assert stats[dbw.STAT_SS].item() == sums[n] and stats[dbw.STAT_GBAR_SQ].item() == sums[n + 1]
    r = rows.cpu().numpy()
    assert np.array_equal(r[mask == 1], sums[:n][mask == 1]) and np.isnan(r[mask == 0]).all()


def test_select_may_sort_in_place():
    times = np.random.default_rng(3).exponential(size=700)
    t = torch.from_numpy(times.copy()).cuda()
    order = torch.empty(700, dtype=torch.int32, device="cuda")
    mask = torch.empty(700, dtype=torch.uint8, device="cuda")
    dbw.dbw_select_fastest(t, torch.tensor([5], dtype=torch.int32, device="cuda"), order, mask, t)
    torch.cuda.synchronize()
    assert np.array_equal(t.cpu().numpy(), np.sort(times))
    assert np.array_equal(order.cpu().numpy(), np.argsort(times, kind="stable"))


@pytest.mark.parametrize("n", [9, 1000])
def test_select_may_leave_k_in_b(n):
    times = np.random.default_rng(n).exponential(size=n)
    b = torch.tensor([n // 3], dtype=torch.int32, device="cuda")
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    mask = torch.empty(n, dtype=torch.uint8, device="cuda")
    tsorted = torch.empty(n, dtype=torch.float64, device="cuda")
    dbw.dbw_select_fastest(torch.from_numpy(times).cuda(), b, order, mask, tsorted, b)
    torch.cuda.synchronize()
    want = np.zeros(n, np.uint8)
    want[np.argsort(times, kind="stable")[:n - n // 3]] = 1
    assert int(b.item()) == n - n // 3 and np.array_equal(mask.cpu().numpy(), want)
