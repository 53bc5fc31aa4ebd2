"""The simulation on block ids against the simulation on hash tables
(RS_SIM_TABLES): the same records, results and final caches, bit for bit, over
the shapes at which the kernel on block ids changes its course: one worker, a
worker per update warp, more workers than update warps, the most workers;
enough replicas for the launch with two update warps; prompts with more
victims than the window of the log holds; caches with exact-sequence updates
and compactions of both ring sizes; slot arrays in global memory; block hashes
given by the caller; a prompt that repeats a block; a prompt longer than the
cache."""
import numpy as np
import pytest

from paper_2606_17081_gb300 import routesim as rs
from paper_2606_17081_gb300 import workloads as wk

from gpu_helpers import assert_replica_equal, gpu_run, oracle_cfg, oracle_run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

OWN_COUNTS = ("probes", "slow_path", "rebuilds", "reserved0")   # of each form's own operations


def _trace(n, seed, groups=12, lo=0, hi=3000, pre=(64, 1500), rate=None):
    return wk.make_trace(wk.TraceSpec(n_req=n, len_kind="uniform", len_min=lo, len_max=hi, n_groups=groups,
                                      prefix_min=pre[0], prefix_max=pre[1], zipf_s=0.8, out_kind="uniform",
                                      out_min=0, out_max=400, rate=rate), seed)


def _both(ctx, traces, reps, caches=()):
    out = []
    for flags in (0, rs.RS_SIM_TABLES):
        st, g = gpu_run(ctx, traces, reps, flags=flags)
        out.append((st, g, [rs.route_cache_dump(ctx.h, 1, r, j, ctx.K) for r, j in caches]))
    (sa, a, ca), (sb, b, cb) = out
    assert sa == sb
    for x, y in zip(a, b):
        for f in x:   # (of a replica that stopped, the rows it routed, the others as they were)
            if f != "result":
                assert np.array_equal(x[f], y[f]), f
        for f, v in x["result"].items():
            if f not in OWN_COUNTS:
                w = y["result"][f]
                if f in ("sum_ttft", "sum_e2e"):   # n summands, taken by 128 threads or 256
                    assert abs(v - w) <= x["result"]["n_routed"] * 2.0 ** -53 * abs(w), (f, v, w)
                    continue
                assert (list(v) == list(w)) if hasattr(v, "__len__") else v == w, (f, v, w)
    for x, y in zip(ca, cb):
        assert x.size and np.array_equal(x, y)
    return sa, a


@pytest.mark.parametrize("W,K,C,tau,policy,hi", [
    (1, 700, 9, 0.0, wk.POLICY_DYNAMO, 3000),
    (3, 190, 40, 0.7, wk.POLICY_DYNAMO, 3000),       # ring of 2 K: every update evicts
    (6, 511, 33, 0.0, wk.POLICY_LOADBAL, 7000),      # more victims than the window
    (6, 512, 33, 0.0, wk.POLICY_DYNAMO, 7000),       # ring of 4 K
    (2, 700, 20, 0.0, wk.POLICY_RANDOM, 11000),      # two updates pass more entries than the plans' ring holds
    (4, 60, 20, 0.0, wk.POLICY_DYNAMO, 950),         # compactions while the rings are being filled
    (7, 900, 64, 0.5, wk.POLICY_DYNAMO, 1040),      # past one worker per warp
    (24, 300, 200, 0.0, wk.POLICY_DYNAMO, 3000),
    (25, 300, 200, 1.0, wk.POLICY_P2C, 3000),
    (64, 400, 500, 0.3, wk.POLICY_DYNAMO, 3000),
    (33, 100, 5000, 0.0, wk.POLICY_RANDOM, 500),    # slot arrays in global memory
])
def test_ids_equal_tables(W, K, C, tau, policy, hi):
    tr = _trace(900, W + K, hi=hi)
    rep = wk.Replica(0, C, policy, int(tau > 0), 1.0, tau, 5, tr.n_req)
    st, g = _both(rs.Context(W=W, K=K), [tr], [rep], [(0, j) for j in range(0, W, 5)])
    assert st == rs.RS_OK and g[0]["result"]["evicted_blocks"] > 0
    if K < 100 and C < 4096:
        assert g[0]["result"]["rebuilds"] > 0


# more than 1024 in flight with the request slots in shared memory: completion times in more groups than lanes; requests
# queued behind full workers, and workers enough for all
@pytest.mark.parametrize("W,C,tau,nrep", [(3, 1100, 0.5, 1), (24, 1500, 0.0, 1), (40, 2300, 0.0, 1), (20, 1300, 0.3, 306)])
def test_ids_equal_tables_thousands_in_flight(W, C, tau, nrep):
    tr = _trace(2 * C, W, hi=400, pre=(64, 300))
    tr.out_len[:] = np.random.default_rng(C).integers(0, 3000, tr.n_req)
    reps = [wk.Replica(0, C - r % 7, wk.POLICY_DYNAMO, r % 2, 1.0, tau, r, tr.n_req) for r in range(nrep)]
    reps.append(wk.Replica(0, 64, wk.POLICY_LOADBAL, 1, 0.0, 0.0, 3, tr.n_req))   # a spike to C and back
    reps[-1].c_t1, reps[-1].c_t2, reps[-1].c_mid, reps[-1].c_end = 2.0, 30.0, C, 40
    st, g = _both(rs.Context(W=W, K=2000), [tr], reps, [(0, 0), (nrep, W - 1)])
    assert st == rs.RS_OK
    a, e = g[0]["arrival"], g[0]["completion"]
    assert max(int(((a <= t) & (e > t)).sum()) for t in a[::50]) > 1024
    o = oracle_run(oracle_cfg(W, 2000), tr, reps[0])
    assert_replica_equal(g[0], o, W)


def test_ids_equal_tables_many_replicas():
    # two update warps per replica, traces of unequal length, truncated replicas, an idle one
    trs = [_trace(150, 1), _trace(90, 2, groups=3, hi=900), _trace(40, 3, lo=0, hi=40)]
    reps = [wk.Replica(r % 3, 1 + r % 50, wk.POLICY_DYNAMO if r % 4 else wk.POLICY_LOADBAL, r % 2, 1.0,
                       0.25 * (r % 3), r, (trs[r % 3].n_req, 0, 30)[0 if r % 7 else r % 3]) for r in range(330)]
    st, _ = _both(rs.Context(W=5, K=600), trs, reps, [(1, 0), (329, 4)])
    assert st == rs.RS_OK


def test_ids_from_given_hashes_repeated_block_and_long_prompt():
    tr = _trace(300, 9, hi=900)
    ctx = rs.Context(W=3, K=200)
    d = rs.device_trace(tr)
    h = torch.zeros(int(tr.offsets[-1]) // 16 + 1, dtype=torch.int64, device="cuda")
    rs.route_hash_blocks(ctx.h, d.tokens, d.offsets, tr.n_req, h)

    def run(hashes, n, flags):
        t = d.desc()
        t.tokens, t.hashes = None, hashes.data_ptr()
        p = [rs.replica_params(wk.Replica(0, 8, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, n))]
        try:
            return rs.simulate_replicas(ctx.h, [t], rs.RS_MEM_DEVICE, p, None, flags)[0].as_dict()
        except rs.RoutesimError as e:
            return e.results[0].as_dict()

    mine = h.clone()
    a = run(mine, tr.n_req, 0)
    mine.zero_()   # the caches that the call left do not refer to the caller's array
    torch.cuda.synchronize()
    got = [rs.route_cache_dump(ctx.h, 1, 0, j, 200) for j in range(3)]
    b = run(h, tr.n_req, rs.RS_SIM_TABLES)
    assert a["status"] == b["status"] == 0 and a["hit_blocks"] == b["hit_blocks"] and a["sum_ttft"] == b["sum_ttft"]
    for j in range(3):
        assert np.array_equal(got[j], rs.route_cache_dump(ctx.h, 1, 0, j, 200))
    nb = np.diff(tr.offsets) // 16
    i = int(np.nonzero(nb >= 4)[0][40])
    base = int(tr.offsets[i]) // 16
    h[base + 3] = h[base + 1]
    for f in (0, rs.RS_SIM_TABLES):
        r = run(h, tr.n_req, f)
        assert r["status"] == rs.RS_ERR_COLLISION and r["n_routed"] == i + 1, f
    small = rs.Context(W=2, K=int(nb.max()) - 1)
    tr2 = wk.Replica(0, 8, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, tr.n_req)
    st, _ = _both(small, [tr], [tr2])
    assert st == rs.RS_ERR_CAPACITY


@pytest.mark.parametrize("W,C", [(2, 150), (8, 40), (40, 4096)])
def test_records_of_stopped_replicas(W, C):
    # a prompt longer than the cache after some hundred others: what was routed until then is recorded alike, TTFTs of the
    # services that have started among it, requests still queued (62 in service a worker at W = 2) not
    n = 379
    tr = _trace(400, 31, hi=900)
    lens = np.diff(tr.offsets)
    lens[n] = 16 * 59
    off = np.concatenate([[0], np.cumsum(lens)])
    tok = np.random.default_rng(1).integers(0, 32000, int(off[-1]) + 3).astype(np.int32)
    tok[:off[n]] = tr.tokens[:off[n]]
    tr = wk.Trace(tok, off, tr.release, np.full(400, 5000, np.int32), tr.group)
    ctx = rs.Context(W=W, K=57)
    reps = [wk.Replica(0, C, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, tr.n_req), wk.Replica(0, 3, wk.POLICY_LOADBAL, 1, 0.0, 0.0, 1, 100)]
    st, g = _both(ctx, [tr], reps)
    assert st == rs.RS_ERR_CAPACITY and g[0]["result"]["n_routed"] == n and g[1]["result"]["status"] == rs.RS_OK
    started = g[0]["first_token"][:n] > 0
    assert started.sum() > 100 and (W != 2 or started.sum() < n)
    assert np.array_equal(g[0]["ttft"][:n][started], (g[0]["first_token"] - g[0]["arrival"])[:n][started])
    assert not g[0]["ttft"][n:].any()


# exact sequences of one chunk of 32 blocks, of whole chunks and of one block more, up to the longest prompts: blocks of
# a prompt among the least recent entries, evicted before their turn
@pytest.mark.parametrize("W,K,n,nrep", [(2, 31, 400, 1), (3, 64, 300, 1), (8, 65, 300, 1), (2, 700, 150, 1), (7, 2100, 60, 1),
                                        (4, 129, 120, 306)])   # (two update warps)
def test_exact_sequences_against_the_oracle(W, K, n, nrep):
    tr = _trace(n, K, groups=3, lo=0, hi=16 * K + 15, pre=(8 * K, 16 * K))
    reps = [wk.Replica(0, 6, wk.POLICY_RANDOM, 0, 1.0, 0.0, r, n) for r in range(nrep)]
    ctx = rs.Context(W=W, K=K)
    ref = {r: oracle_run(oracle_cfg(ctx), tr, reps[r], want_cache=True) for r in {0, nrep - 1}}
    for flags in (0, rs.RS_SIM_TABLES):
        st, g = gpu_run(ctx, [tr], reps, flags=flags)
        assert st == rs.RS_OK and g[0]["result"]["slow_path"] > 0
        for r, o in ref.items():
            assert_replica_equal(g[r], o, W)
            for j in range(W):
                assert np.array_equal(rs.route_cache_dump(ctx.h, 1, r, j, K), o["cache"][j])


@pytest.mark.parametrize("W,C", [(3, 8), (7, 8), (3, 5000)])   # planned updates, not planned, slot arrays in global memory
def test_first_error_in_request_order(W, C):
    # a prompt that repeats a block, right before one longer than the cache: the replica stops at the former
    K, i = 200, 50
    lens = np.array([320] * i + [100, 16 * K + 16, 320])
    rng = np.random.default_rng(3)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tr = wk.Trace(rng.integers(0, 32000, int(off[-1]) + 3).astype(np.int32), off, np.zeros(lens.size),
                  np.full(lens.size, 20, np.int32), np.zeros(lens.size, np.int32))
    ctx = rs.Context(W=W, K=K)
    d = rs.device_trace(tr)
    h = torch.zeros(int(off[-1]) // 16 + 1, dtype=torch.int64, device="cuda")
    rs.route_hash_blocks(ctx.h, d.tokens, d.offsets, tr.n_req, h)
    b = int(off[i]) // 16
    h[b + 3] = h[b + 1]
    t = d.desc()
    t.tokens, t.hashes = None, h.data_ptr()
    p = [rs.replica_params(wk.Replica(0, C, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, tr.n_req))]
    for f in (0, rs.RS_SIM_TABLES):
        with pytest.raises(rs.RoutesimError) as e:
            rs.simulate_replicas(ctx.h, [t], rs.RS_MEM_DEVICE, p, None, f)
        r = e.value.results[0].as_dict()
        assert (r["status"], r["n_routed"]) == (rs.RS_ERR_COLLISION, i + 1), f


@pytest.mark.parametrize("W,K,nrep,hi,decay,fmax", [
    (3, 190, 4, 3000, 0.5, 64),       # ring of 2 K, frequencies that decay between requests
    (6, 900, 5, 7000, 50.0, 1 << 20),  # mostly hot: the sequence is replayed, hot victims
    (2, 120, 3, 1900, 5.0, 2),         # a request evicts its own blocks
    (33, 300, 2, 3000, 1.0, 8),
    (4, 400, 310, 1500, 2.0, 16),      # two update warps
])
def test_frequency_eviction_ids_equal_tables(W, K, nrep, hi, decay, fmax):
    tr = _trace(600 if nrep < 300 else 150, W + K, groups=6 if fmax > 64 else 12, hi=hi)
    reps = []
    for r in range(nrep):
        rep = wk.Replica(0, 40 + 9 * (r % 7), wk.POLICY_DYNAMO if r % 3 else wk.POLICY_LOADBAL, r % 2, 1.0, 0.3 * (r % 2),
                         r, tr.n_req)
        if r % 4 != 3:   # exact LRU replicas in the same launch
            rep.eviction, rep.freq_max, rep.decay_s = rs.RS_EVICT_FREQ, fmax, decay * (1 + r % 2)
        reps.append(rep)
    st, g = _both(rs.Context(W=W, K=K), [tr], reps, [(r, j) for r in (0, nrep - 1) for j in (0, W - 1)])
    assert st == rs.RS_OK and min(x["result"]["evicted_blocks"] for x in g) > 0
