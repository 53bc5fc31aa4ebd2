"""simulate_replicas calls that are refused or run out of device memory: what
they leave of the call before."""
import numpy as np
import pytest

from paper_2606_17081_gb300 import routesim as rs
from paper_2606_17081_gb300 import workloads as wk

from gpu_helpers import gpu_run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _trace(n, seed, hi=600):
    return wk.make_trace(wk.TraceSpec(n_req=n, len_kind="uniform", len_min=16, len_max=hi, n_groups=4, prefix_min=32,
                                      prefix_max=200, zipf_s=None, out_kind="uniform", out_min=1, out_max=100), seed)


def _rep(n, trace=0):
    return wk.Replica(trace, 8, wk.POLICY_DYNAMO, 0, 1.0, 0.0, 0, n)


def _claims(length, hashes=None):
    """A device trace of one prompt of `length` tokens whose tokens (or hashes) are not there: for calls that end before
    any of them is read."""
    t = rs.TraceBuffers(None if hashes is not None else torch.zeros(16, dtype=torch.int32, device="cuda"),
                        torch.tensor([0, length], dtype=torch.int64, device="cuda"),
                        torch.zeros(1, dtype=torch.float64, device="cuda"),
                        torch.ones(1, dtype=torch.int32, device="cuda"), 1, hashes)
    return t


def test_no_caches_after_a_call_without_memory():
    # the hashes of 2^45 tokens (2^44 bytes) cannot be had; the old buffer that the caches' hashes lay in is gone
    ctx = rs.Context(W=3, K=100)
    tr = _trace(80, 1)
    st, _ = gpu_run(ctx, [tr], [_rep(80)])
    assert st == rs.RS_OK and rs.route_cache_dump(ctx.h, 1, 0, 0, 100).size
    big = _claims(1 << 45)
    with pytest.raises(rs.RoutesimError) as e:
        rs.simulate_replicas(ctx.h, [big.desc()], rs.RS_MEM_DEVICE, [rs.replica_params(_rep(1))], None)
    assert e.value.status == rs.RS_ERR_OOM
    with pytest.raises(rs.RoutesimError) as e:
        rs.route_cache_dump(ctx.h, 1, 0, 0, 100)
    assert e.value.status == rs.RS_ERR_INVALID
    st, _ = gpu_run(ctx, [tr], [_rep(80)])   # the context stays usable
    assert st == rs.RS_OK and rs.route_cache_dump(ctx.h, 1, 0, 0, 100).size


def test_caches_stay_after_a_refused_host_call():
    # refused before anything of the last call is overwritten: a prompt too long for the kernels' shared memory
    ctx = rs.Context(W=3, K=20000)
    tr = _trace(60, 2)
    st, _ = gpu_run(ctx, [tr], [_rep(60)], trace_mem=rs.RS_MEM_HOST)
    assert st == rs.RS_OK
    before = [rs.route_cache_dump(ctx.h, 1, 0, j, 20000) for j in range(3)]
    n = 16 * 16000
    long = rs.TraceBuffers(torch.zeros(n, dtype=torch.int32), torch.tensor([0, n]), torch.zeros(1, dtype=torch.float64),
                           torch.ones(1, dtype=torch.int32), 1)
    with pytest.raises(rs.RoutesimError) as e:
        rs.simulate_replicas(ctx.h, [long.desc()], rs.RS_MEM_HOST, [rs.replica_params(_rep(1))], None)
    assert e.value.status == rs.RS_ERR_CAPACITY
    for j in range(3):
        assert np.array_equal(rs.route_cache_dump(ctx.h, 1, 0, j, 20000), before[j])


def test_device_hashes_that_cannot_be_copied():
    # forty traces whose hashes take 8.6 GB each: no room for copies of them beside what the hash tables need (of each,
    # one prompt of 16 blocks is routed; the second, longer than the cache, is not and its hashes are not there)
    ctx = rs.Context(W=2, K=64)
    h = torch.arange(2, 34, dtype=torch.int64, device="cuda")
    t = rs.TraceBuffers(None, torch.tensor([0, 256, (1 << 34) - 256], dtype=torch.int64, device="cuda"),
                        torch.zeros(2, dtype=torch.float64, device="cuda"), torch.ones(2, dtype=torch.int32, device="cuda"), 2, h)
    res = rs.simulate_replicas(ctx.h, [t.desc()] * 40, rs.RS_MEM_DEVICE, [rs.replica_params(_rep(1, k)) for k in range(40)], None)
    assert all(r.status == rs.RS_OK and r.n_routed == 1 and r.inserted_blocks == 16 for r in res)
    assert np.array_equal(rs.route_cache_dump(ctx.h, 1, 39, 0, 64), np.arange(2, 18))
