"""The live router where its kernel changes its course, against the oracle's
router bit for bit: slots kept by the probe (W nb <= 2048), rounds to the first
miss past that, prompts whose arrays leave no room for kept slots; caches that
evict and rebuild; batches of one request and of many.  (A prompt that repeats
a block's chained hash, which the router stops at, takes a 64-bit collision of
hashes that it computes itself: not tested.)"""
import numpy as np
import pytest

import oracle as O
from paper_2606_17081_gb300 import routesim as rs
from paper_2606_17081_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("W,K,n,hi,pre,tau", [
    (1, 150, 300, 2000, 900, 0.0),
    (6, 120, 400, 1500, 900, 0.5),         # rebuilds
    (8, 256, 200, 4096, 2000, 0.0),        # around W nb = 2048
    (64, 200, 150, 3000, 1500, 1.0),       # rounds
    (3, 4096, 24, 46400, 20000, 0.3),      # up to 2 800 blocks: no kept slots
])
def test_route_batch_forms(W, K, n, hi, pre, tau):
    spec = wk.TraceSpec(n_req=n, len_kind="uniform", len_min=0, len_max=hi, n_groups=6, prefix_min=pre // 4,
                        prefix_max=pre, zipf_s=0.8, out_kind="uniform", out_min=0, out_max=300)
    tr = wk.make_trace(spec, W + K)
    ctx = rs.Context(W=W, K=K, n_instances=1, tau=tau, omega=1.0, seed=5)
    ref = O.Router(O.OracleConfig(W=W, K=K), 1.0, tau, 5, n_instances=1)
    cut = [0, 1, 2, n // 2, n]
    for lo, hi_ in zip(cut[:-1], cut[1:]):
        sub = wk.Trace(tr.tokens, tr.offsets[lo:hi_ + 1], tr.release[lo:hi_], tr.out_len[lo:hi_], tr.group[lo:hi_])
        d = rs.device_trace(sub)
        m = hi_ - lo
        wo = torch.zeros(m, dtype=torch.int32, device="cuda")
        co = torch.zeros(m * W, dtype=torch.float32, device="cuda")
        po = torch.zeros(m * W, dtype=torch.int32, device="cuda")
        rs.route_batch(ctx.h, 0, d.tokens, d.offsets, m, d.out_len, wo, co, po)
        st, rw, rc, rp = ref.route(0, sub.tokens, sub.offsets, sub.out_len)
        assert st == 0
        assert np.array_equal(wo.cpu().numpy(), rw)
        assert np.array_equal(co.cpu().numpy().reshape(m, W), rc)
        assert np.array_equal(po.cpu().numpy().reshape(m, W), rp)
        assert np.array_equal(rs.route_active(ctx.h, 0, W), ref.active(0))
    for j in range(W):
        assert np.array_equal(rs.route_cache_dump(ctx.h, 0, 0, j, K), ref.cache(0, j))


# the longest prompts that 227 KB of shared memory hold, and one block more (refused, the state as it was)
@pytest.mark.parametrize("W,nb", [(1, 2904), (3, 2904), (6, 2902), (64, 2864)])
def test_route_batch_longest_prompt(W, nb):
    K = 3000
    ctx = rs.Context(W=W, K=K, n_instances=1, tau=0.0, omega=1.0, seed=5)
    ref = O.Router(O.OracleConfig(W=W, K=K), 1.0, 0.0, 5, n_instances=1)
    rng = np.random.default_rng(nb)
    long = rng.integers(0, 32000, 16 * (nb + 1)).astype(np.int32)
    for parts in ([long[:16 * nb + 15], long[:160], long[:16 * nb], long[16 * 50:]], [long]):
        off = np.concatenate([[0], np.cumsum([p.size for p in parts])]).astype(np.int64)
        tok = np.concatenate(parts + [np.zeros(-int(off[-1]) % 4, np.int32)])
        tr = wk.Trace(tok, off, np.zeros(len(parts)), np.full(len(parts), 7, np.int32), np.zeros(len(parts), np.int32))
        d = rs.device_trace(tr)
        wo = torch.zeros(tr.n_req, dtype=torch.int32, device="cuda")
        if len(parts) == 1:
            with pytest.raises(rs.RoutesimError) as e:
                rs.route_batch(ctx.h, 0, d.tokens, d.offsets, 1, d.out_len, wo)
            assert e.value.status == rs.RS_ERR_CAPACITY
        else:
            rs.route_batch(ctx.h, 0, d.tokens, d.offsets, tr.n_req, d.out_len, wo)
            st, rw, _, _ = ref.route(0, tr.tokens, tr.offsets, tr.out_len)
            assert st == 0 and np.array_equal(wo.cpu().numpy(), rw)
        assert np.array_equal(rs.route_active(ctx.h, 0, W), ref.active(0))
        for j in range(min(W, 4)):
            assert np.array_equal(rs.route_cache_dump(ctx.h, 0, 0, j, K), ref.cache(0, j))
