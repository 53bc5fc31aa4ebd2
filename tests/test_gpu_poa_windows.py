"""PoA of Eq. (12) on sparse records: the records span far more 5-s windows
than they have rows (a slow Poisson client, long outputs), so every window the
records reach must get a slot.  The estimate of simulate_replicas, of
poa_estimate and of poa_estimate_noalloc must all equal the oracle's per
window (numerator, count, OPT) and in total."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2606_17081_gb300 import routesim as rs
from paper_2606_17081_gb300 import workloads as wk

from gpu_helpers import gpu_run, oracle_cfg, oracle_run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _sparse_trace(n, seed):
    spec = wk.TraceSpec(n_req=n, len_kind="uniform", len_min=16, len_max=600, n_groups=4,
                        prefix_min=32, prefix_max=200, zipf_s=None, out_kind="uniform",
                        out_min=1000, out_max=4000, rate=0.05)
    return wk.make_trace(spec, seed)


def _to_device(o, n, W):
    rec, t = rs.device_records(n, W)
    for f in ("worker", "completion", "ttft", "nbt"):
        t[f].copy_(torch.from_numpy(np.ascontiguousarray(o[f])))
    for f in ("n_frozen", "prefix"):
        t[f].copy_(torch.from_numpy(np.ascontiguousarray(o[f]).reshape(-1).view(np.int16)))
    return rec, t


@pytest.mark.parametrize("W,C", [(3, 4), (5, 64)])
def test_sparse_windows_match_oracle(W, C):
    tr = _sparse_trace(400, 60 + W)
    ctx = rs.Context(W=W, K=300)
    reps = [wk.Replica(0, C, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, tr.n_req)]
    st, g = gpu_run(ctx, [tr], reps)
    assert st == 0
    cfg = oracle_cfg(ctx)
    o = oracle_run(cfg, tr, reps[0])
    num, opt, cnt, tot = O.poa(cfg, o)
    assert num.size > 3 * (tr.n_req + 2)         # far more windows than rows
    res = g[0]["result"]
    assert res["n_windows"] == num.size
    assert abs(res["poa_total"] - tot) <= 1e-9 * tot
    rec, keep = _to_device(o, tr.n_req, W)
    gn, go, gc, gt, nw = rs.poa_estimate(ctx.h, rec, tr.n_req, num.size)
    assert nw == num.size and np.array_equal(gc, cnt)
    assert np.allclose(gn, num, rtol=1e-12, atol=0)
    assert np.allclose(go, opt, rtol=1e-12, atol=0)
    assert abs(gt - tot) <= 1e-12 * tot
    # the allocation-free entry point: the windows take what the rows leave
    cap = num.size
    dn = torch.full((cap,), -1.0, dtype=torch.float64, device="cuda")
    do = torch.full((cap,), -1.0, dtype=torch.float64, device="cuda")
    dc = torch.full((cap,), -1, dtype=torch.int64, device="cuda")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    dw = torch.zeros(1, dtype=torch.int64, device="cuda")
    rs.poa_estimate_noalloc(ctx.cfg, rec, tr.n_req, dn, do, dc, cap, dt, dw)
    torch.cuda.synchronize()
    assert int(dw.item()) == num.size
    assert np.array_equal(dc.cpu().numpy(), cnt)
    assert np.allclose(dn.cpu().numpy(), num, rtol=1e-12, atol=0)
    assert np.allclose(do.cpu().numpy(), opt, rtol=1e-12, atol=0)
    assert abs(dt.item() - tot) <= 1e-12 * tot


def test_windows_far_apart_and_empty_records():
    # three routed rows thousands of windows apart; and no routed row at all
    W = 2
    ctx = rs.Context(W=W, K=16)
    cfg = oracle_cfg(ctx)
    o = {"worker": np.array([0, -1, 1, 0], np.int32),
         "completion": np.array([1.0, 7.0, 52_345.5, 9_999_999.0]),
         "ttft": np.array([0.1, 0.2, 0.3, 0.4]),
         "nbt": np.array([4, 1, 8, 2], np.int32),
         "n_frozen": np.array([[1, 2], [3, 4], [5, 6], [7, 8]], np.uint16),
         "prefix": np.array([[0, 1], [0, 0], [8, 2], [1, 1]], np.uint16)}
    num, opt, cnt, tot = O.poa(cfg, o)
    assert num.size == 2_000_000
    rec, keep = _to_device(o, 4, W)
    gn, go, gc, gt, nw = rs.poa_estimate(ctx.h, rec, 4, num.size)
    assert nw == num.size and np.array_equal(gc, cnt)
    assert np.allclose(gn, num, rtol=1e-12, atol=0) and np.allclose(go, opt, rtol=1e-12, atol=0)
    assert abs(gt - tot) <= 1e-12 * tot
    o["worker"][:] = -1
    rec, keep = _to_device(o, 4, W)
    gn, go, gc, gt, nw = rs.poa_estimate(ctx.h, rec, 4, 4)
    assert nw == 0 and gt == 0.0


def _random_records(rng, n, W, span, tied, cap):
    """Records whose cheapest workers exceed their capacity: worker 0 is cheap for every row;
    `tied` makes many costs equal (few load levels, no prefixes)."""
    nbt = rng.integers(1, 60, n).astype(np.int32)
    nf = rng.integers(20, 23 if tied else 60, (n, W)).astype(np.uint16)
    nf[:, 0] = rng.integers(1, 3 if tied else 20, n)
    nf = np.minimum(nf, cap - 1)
    pre = np.zeros((n, W), np.uint16) if tied else \
        (rng.integers(0, 2, (n, W)) * rng.integers(0, 60, (n, W)) % (nbt[:, None] + 1)).astype(np.uint16)
    comp = rng.uniform(0.0, span, n)
    comp[-1] = span - 1e-3
    worker = rng.integers(-1, W, n).astype(np.int32)
    worker[-1] = 0
    return {"worker": worker, "completion": comp, "ttft": rng.uniform(0.01, 3.0, n), "nbt": nbt,
            "n_frozen": nf, "prefix": pre}


# windows up to the sort's table (11 264) and one past it; rows that end inside a warp's 32; solvers
# for W = 3, 6, up to 16 and wider, at capacities that bind (rows per window > C_j on worker 0); costs
# and rows of a window inside and past what the solvers keep in shared memory (W <= 16: 4096 costs,
# 1024 rows; wider: 4096 rows), one warp per window (400 windows) and a CTA per window; W > 16 with a
# C_j whose lists fit nowhere
@pytest.mark.parametrize("W,n,windows,tied,cap", [
    (2, 1, 1, False, 64), (3, 331, 2, True, 64), (6, 1537, 4, False, 64), (6, 1000, 11264, False, 64),
    (6, 1000, 11265, False, 64), (6, 4801, 400, False, 3), (6, 900, 1, True, 64),
    (3, 1500, 1, False, 64), (16, 900, 3, True, 64), (17, 801, 2, False, 64), (33, 700, 2, True, 64),
    (64, 1400, 2, False, 64), (17, 4500, 1, False, 64), (20, 700, 1, False, 300)])
def test_sort_and_solvers_at_their_edges(W, n, windows, tied, cap):
    ctx = rs.Context(W=W, K=64, cap=cap)
    o = _random_records(np.random.default_rng(W * n + windows), n, W, 5.0 * windows, tied, cap)
    num, opt, cnt, tot = O.poa(oracle_cfg(ctx, cap=cap), o)
    assert num.size == windows
    rec, keep = _to_device(o, n, W)
    gn, go, gc, gt, nw = rs.poa_estimate(ctx.h, rec, n, windows)
    assert nw == windows and np.array_equal(gc, cnt)
    # sums of at most 4500 rows of one sign: n 2^-53 relative (5e-13)
    assert np.allclose(gn, num, rtol=1e-12, atol=0) and np.allclose(go, opt, rtol=1e-12, atol=0)
    assert abs(gt - tot) <= 1e-12 * tot


# a few costs of 1000 among many below 0.1 (on workers that no optimum takes), past a capacity: narrow
# solver with a CTA and with a warp per window, costs in shared memory and in place; wide solver with its
# lists in shared memory, in the window's rows' place, and without lists
@pytest.mark.parametrize("W,n,windows,cap", [(6, 600, 2, 128), (6, 900, 1, 128), (3, 150 * 400, 400, 80), (16, 500, 1, 128),
                                             (17, 800, 1, 200), (33, 700, 2, 100), (17, 9000, 2, 64), (20, 900, 1, 512)])
def test_opt_keeps_the_costs_bits(W, n, windows, cap):
    d = 1000.0
    ctx = rs.Context(W=W, K=64, cap=cap, lat_d=d)
    rng = np.random.default_rng(W + n)
    o = _random_records(rng, n, W, 5.0 * windows, False, cap)
    o["n_frozen"][:, 1:][rng.random((n, W - 1)) < 0.05] = cap - 1
    rec, keep = _to_device(o, n, W)
    _, go, gc, _, nw = rs.poa_estimate(ctx.h, rec, n, windows)
    assert nw == windows
    nf, pre = o["n_frozen"].astype(np.float64), o["prefix"].astype(np.float64)
    cost = ((0.005 * nf + 0.020) + d / ((cap - nf) * (cap - nf))) - 0.015 * (pre / o["nbt"][:, None])
    win = np.floor(o["completion"] / 5.0).astype(int)
    bound = 0
    for w in list(range(windows))[:4]:
        c = cost[(win == w) & (o["worker"] >= 0)]
        m = c.shape[0]
        capw = max(cap, -(-m // W))
        bound += np.bincount(c.argmin(1)).max() > capw
        _, at = O.assign(c, capw, 0)
        mine = c[np.arange(m), at]
        # equal costs may differ by their own rounding: one of the largest cost's, per row
        assert abs(go[w] - math.fsum(mine)) <= m * 2.0 ** -53 * mine.max(), (w, go[w], math.fsum(mine))
    assert bound


@pytest.mark.parametrize("W,n", [(3, 180), (6, 380), (17, 1080), (20, 9000)])
def test_no_assignment_at_the_pole(W, n):
    # loads at the pole of Eq. (9) (n_frozen = cap: infinite cost).  Worker 0 is cheap for all; at worker 1 two rows of
    # three cannot be, and a third can only at nearly the largest cost, which the optimum must take: the capacities
    # leave little room.  A penalty for the pole in its place would be the better bargain.
    cap = 64
    ctx = rs.Context(W=W, K=64)
    rng = np.random.default_rng(W)
    nf = rng.integers(45, 55, (n, W))
    nf[:, 0] = rng.integers(1, 4, n)
    other = np.arange(n) % 3 == 0
    nf[other, 1:] = rng.integers(1, 4, (int(other.sum()), W - 1))
    nf[:, 1] = np.where(other, cap - 1, cap)
    o = {"worker": np.zeros(n, np.int32), "completion": rng.uniform(0.0, 5.0, n), "ttft": np.ones(n),
         "nbt": np.ones(n, np.int32), "n_frozen": nf.astype(np.uint16), "prefix": np.zeros((n, W), np.uint16)}
    _, opt, _, tot = O.poa(oracle_cfg(ctx), o)
    assert opt.size == 1 and np.isfinite(opt[0])
    rec, keep = _to_device(o, n, W)
    _, go, _, gt, _ = rs.poa_estimate(ctx.h, rec, n, 1)
    assert np.allclose(go, opt, rtol=1e-12, atol=0) and abs(gt - tot) <= 1e-12 * tot
    o["n_frozen"][:, 1:] = cap   # no way out of worker 0
    rec, keep = _to_device(o, n, W)
    _, go, _, gt, _ = rs.poa_estimate(ctx.h, rec, n, 1)
    assert go[0] == np.inf and gt == 0.0


def test_more_windows_than_are_staged():
    W, last = 2, 11_500_000.0   # 2.3 M windows (2^21 go through pinned memory)
    ctx = rs.Context(W=W, K=16)
    o = {"worker": np.array([1, 0, 0], np.int32), "completion": np.array([2.0, 10_600_001.0, last]),
         "ttft": np.array([0.5, 0.25, 0.125]), "nbt": np.array([4, 8, 2], np.int32),
         "n_frozen": np.array([[1, 2], [5, 6], [7, 8]], np.uint16), "prefix": np.array([[0, 1], [8, 2], [1, 1]], np.uint16)}
    num, opt, cnt, tot = O.poa(oracle_cfg(ctx), o)
    rec, keep = _to_device(o, 3, W)
    gn, go, gc, gt, nw = rs.poa_estimate(ctx.h, rec, 3, num.size)
    assert nw == num.size == 2_300_001 and np.array_equal(gc, cnt)
    assert np.allclose(gn, num, rtol=1e-12, atol=0) and np.allclose(go, opt, rtol=1e-12, atol=0)
    assert abs(gt - tot) <= 1e-12 * tot
    gn2, _, _, _, nw2 = rs.poa_estimate(ctx.h, rec, 3, 10)   # fewer entries than windows
    assert nw2 == nw and np.array_equal(gn2[:10], gn[:10])
