// Live routing (route_batch / route_release) on one router instance.
//
// One CTA routes a batch of requests of one instance in array order: for each
// request, the cached prefix of every worker, the Eq. (1) cost with the
// instance's active blocks, the Eq. (2) choice, and the chosen worker's cache
// and load update -- the same steps as a simulated arrival, without the
// event loop (completions are reported by the caller through route_release).
#include "sim_probe.cuh"

namespace rs {

// Per request (512 threads):
//   probe    every (worker, block) pair at once while W nb <= PROBE_CAP, its
//            slot kept for the update, else in rounds to each worker's first
//            miss; beside it the request's hashes go through the repeat
//            detector;
//   choose   the first warp, a lane per worker;
//   update   the chosen worker's cache, from the kept slots; meanwhile the
//            next request's hashes are copied into the other buffer.
// Bound by the latency of that chain on one SM: of 14 300 cycles a request
// (W = 6, tau = 0.5) the probe takes 4 600, the choice 3 000, the update's reads
// 2 600 and its writes 3 700.  With two lookups of every block of the chosen
// worker, the choice on one thread and each request's hashes loaded on arrival
// a call of 256 requests took 2.39 ms, now 1.81; 256 threads with two lookups
// each in flight take the same.
constexpr int NT_ROUTE = 512;

struct RouterShared {
  int warp_tot[NT_ROUTE / 32];
  uint32_t scan_pos;
  int status, dup, js, rebuild;
  uint32_t u24;   // the request's draw
  uint64_t ordinal;
};

static_assert(sizeof(RouterShared) + sizeof(SimScalars) + 64 <= ROUTE_OWN_SMEM, "the host's margin");

struct RouteLayout {
  size_t hbuf, dupset, pslot, pfree, A, meta, slot, pst, fslot, vslot, vt, owner, victim, wm, wabs,
      wcost, wopen, kind, evk, touched, total;
  uint32_t dupmask;
};

// lean: no kept slots and one hash buffer, for prompts whose arrays would not
// fit in shared memory otherwise.
__host__ __device__ inline RouteLayout make_route_layout(int W, int nbmax, bool lean) {
  RouteLayout L;
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1);
  size_t dup = 1, o = 0;
  while (dup < 2 * nb) dup <<= 1;
  L.dupmask = (uint32_t)(dup - 1);
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += (bytes + 15) & ~(size_t)15;
    return r;
  };
  L.hbuf = take((lean ? 1 : 2) * 8 * nb);
  L.dupset = take(8 * dup);
  const size_t cap = lean ? 0 : (size_t)W * nb < (size_t)PROBE_CAP ? (size_t)W * nb : (size_t)PROBE_CAP;
  L.pslot = take(4 * cap);
  L.pfree = take(4 * cap);
  L.A = take(8 * (size_t)W);
  L.meta = take(sizeof(CacheMeta) * (size_t)W);
  L.slot = take(4 * nb);
  L.pst = take(4 * nb);
  L.fslot = take(4 * nb);
  L.vslot = take(8 * nb);
  L.vt = take(8 * nb);
  L.owner = take(8 * nb);
  L.victim = take(8 * nb);
  L.wm = take(4 * (size_t)W);
  L.wabs = take(4 * (size_t)W);
  L.wcost = take(4 * (size_t)W);
  L.wopen = take((size_t)(NT_ROUTE / 32) * WMAX);
  L.kind = take(nb);
  L.evk = take(nb);
  L.touched = take(2 * nb);
  L.total = o;
  return L;
}

__global__ void __launch_bounds__(NT_ROUTE) k_route_batch(
    const __grid_constant__ SimBuffers b, const __grid_constant__ SimLaunch L, RouterState s,
    int32_t instance, const int64_t* __restrict__ offsets, const uint64_t* __restrict__ hashes,
    int32_t n_req, const int32_t* __restrict__ out_len, int32_t* __restrict__ worker_out,
    float* __restrict__ cost_out, int32_t* __restrict__ prefix_out, float omega, float tau,
    uint64_t seed, bool lean) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RouterShared R;
  __shared__ SimScalars S;
  const TableGeom& g = L.g;
  const int W = L.mc.W, nbmax = L.nbmax;
  const size_t nb_cap = (size_t)(nbmax > 0 ? nbmax : 1);
  const RouteLayout lay = make_route_layout(W, nbmax, lean);
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  SimCtx c;   // the tables are those of "replica" 0
  c.S = &S;
  c.b = &b;
  c.L = &L;
  c.sid = 0;
  c.pslot = reinterpret_cast<uint32_t*>(smem + lay.pslot);
  c.pfree = reinterpret_cast<uint32_t*>(smem + lay.pfree);
  c.wm = reinterpret_cast<int32_t*>(smem + lay.wm);
  c.wabs = reinterpret_cast<int32_t*>(smem + lay.wabs);
  c.wopen = smem + lay.wopen;
  UpdateScratch& sc = c.sc;
  sc.dupset = reinterpret_cast<uint64_t*>(smem + lay.dupset);
  sc.dupmask = lay.dupmask;
  sc.slot = reinterpret_cast<uint32_t*>(smem + lay.slot);
  sc.pst = reinterpret_cast<uint32_t*>(smem + lay.pst);
  sc.fslot = reinterpret_cast<uint32_t*>(smem + lay.fslot);
  sc.vslot = reinterpret_cast<uint32_t*>(smem + lay.vslot);
  sc.vt = reinterpret_cast<uint32_t*>(smem + lay.vt);
  sc.owner = reinterpret_cast<int32_t*>(smem + lay.owner);
  sc.victim = reinterpret_cast<int32_t*>(smem + lay.victim);
  sc.kind = smem + lay.kind;
  sc.evk = smem + lay.evk;
  sc.touched = smem + lay.touched;
  uint64_t* hbuf = reinterpret_cast<uint64_t*>(smem + lay.hbuf);   // [2][nb_cap]
  int64_t* A = reinterpret_cast<int64_t*>(smem + lay.A);
  CacheMeta* meta = reinterpret_cast<CacheMeta*>(smem + lay.meta);
  float* wc = reinterpret_cast<float*>(smem + lay.wcost);   // (every warp writes the same costs)

  // the first request's hashes, and its scalars in every thread
  int64_t o0 = offsets[0], o1 = offsets[1];
  int out = out_len[0];
  auto copy_hashes = [&](int64_t a, int64_t e, int buf) {
    const int64_t nb = (e - a) >> 4;
    if (nb <= (int64_t)nb_cap) {
      const uint64_t* src = hashes + (a >> 4);
      for (int k = tid; k < (int)nb; k += NT_ROUTE) cp_async8(hbuf + buf * nb_cap + k, src + k);
    }
  };
  copy_hashes(o0, o1, 0);
  for (uint32_t q = tid; q <= sc.dupmask; q += NT_ROUTE) sc.dupset[q] = 0ull;
  for (int j = tid; j < W; j += NT_ROUTE) {
    A[j] = s.active[j];
    meta[j] = s.meta[j];
  }
  if (tid == 0) {
    R.status = *s.status;
    R.ordinal = *s.ordinal;
    R.dup = 0;
    S.status = RS_OK;
    S.probes = 0;
    update_reset(&S.us);
    S.us.err = 0;
  }
  for (int32_t i = 0; i < n_req; i++) {
    const int64_t Lp = o1 - o0, nb64 = Lp >> 4;
    const bool fits = nb64 <= (int64_t)g.K && nb64 <= (int64_t)nbmax;
    const int nb = fits ? (int)nb64 : 0, nbt = (int)((Lp + 15) >> 4);
    const uint64_t* hb = hbuf + (lean ? 0 : (size_t)(i & 1) * nb_cap);
    for (int j = tid; j < W; j += NT_ROUTE) {
      c.wm[j] = nb;
      c.wabs[j] = 0;
    }
    cp_async_wait_all();
    __syncthreads();   // hashes in place, the last update done
    if (R.status != RS_OK) break;
    if (!fits) {
      __syncthreads();   // (every thread has read the status)
      if (tid == 0) R.status = RS_ERR_CAPACITY;
      __syncthreads();
      break;
    }
    // the next request: its scalars now, its hashes once they are known
    const bool more = i + 1 < n_req;
    int64_t o2 = 0;
    int outn = 0;
    if (more) {
      o2 = offsets[i + 2];
      outn = out_len[i + 1];
    }
    // cached prefix on every worker; repeats among the prompt's hashes
    const bool full = !lean && W * nb64 <= PROBE_CAP;
    int32_t claim0 = -1;   // set entry of this thread's first block
    int dup = 0;
    for (int k = tid; k < nb; k += NT_ROUTE) {
      const int32_t cl = dup_claim(sc, hb[k], &dup);
      if (k == tid) claim0 = cl; else sc.owner[k] = cl;
    }
    if (dup) R.dup = 1;
    if (full)
      probe_full<NT_ROUTE, 1>(c, hb, nb);
    else
      probe_prefixes<NT_ROUTE, 2>(c, hb, nb);
    if (tau > 0.0f && tid == NT_ROUTE - 1) R.u24 = draw_u24(seed, R.ordinal, (uint32_t)instance, TAG_ROUTE);
    if (more && !lean) copy_hashes(o1, o2, (i + 1) & 1);
    __syncthreads();
    // ---- Eq. (1) costs and the Eq. (2) choice, by the first warp
    if (warp == 0) {
      float bc = __int_as_float(0x7F800000);
      int bj = 0x7FFFFFFF;
      for (int j = lane; j < W; j += 32) {
        const float cj = router_cost(omega, (int64_t)nbt - c.wm[j], A[j]);
        wc[j] = cj;
        if (cost_out) cost_out[(size_t)i * W + j] = cj;
        if (prefix_out) prefix_out[(size_t)i * W + j] = c.wm[j];
        if (cj < bc || bj == 0x7FFFFFFF) {
          bc = cj;
          bj = j;
        }
      }
      argmin_warp(bc, bj);
      __syncwarp();
      const int j = select_worker_warp(wc, W, tau, R.u24, bj, nullptr, lane);
      if (lane == 0) {
        const CacheMeta mt = meta[j];
        const uint64_t span = (uint64_t)mt.T - mt.head + (uint64_t)nb;
        R.js = j;
        R.rebuild = span > g.R || mt.tombs > g.slots / 8 || (uint64_t)mt.T + nb > STAMP_LIMIT;
      }
    }
    // the detector's entries given back, before the update claims slots there
    for (int k = tid; k < nb; k += NT_ROUTE) {
      const int32_t cl = k == tid ? claim0 : sc.owner[k];
      if (cl >= 0) sc.dupset[cl] = 0ull;
    }
    __syncthreads();
    const int js = R.js, nabs = c.wabs[js];
    const bool rebuild = R.rebuild;
    if (R.dup || S.status != RS_OK) {
      __syncthreads();
      if (tid == 0) R.status = S.status != RS_OK ? S.status : RS_ERR_COLLISION;
      __syncthreads();
      break;
    }
    const TableView tv = c.table(js);
    if (rebuild) cache_rebuild<NT_ROUTE>(tv, &meta[js], g.K, s.tmp, R.warp_tot, &S.us);
    const bool captured = full && !rebuild;
    if (captured)
      cache_prepare_captured<NT_ROUTE>(tv, &meta[js], g.K, c.pslot + (size_t)js * nb,
                                     c.pfree + (size_t)js * nb, nb, nabs, sc, &S.us, R.warp_tot,
                                     &R.scan_pos);
    else
      cache_lookup_all<NT_ROUTE>(tv, hb, nb, sc, &S.us, &S.probes);
    cache_apply<NT_ROUTE>(tv, &meta[js], g.K, hb, nb, sc, &S.us, R.warp_tot, &R.scan_pos, captured);
    if (tid == 0) {
      if (S.us.err) R.status = S.us.err;
      update_reset(&S.us);
      A[js] += (Lp + out + 15) >> 4;
      worker_out[i] = js;
      R.ordinal++;
    }
    if (more && lean) {
      __syncthreads();   // the update has read its hashes
      copy_hashes(o1, o2, 0);
    }
    o0 = o1;
    o1 = o2;
    out = outn;
  }
  cp_async_wait_all();
  __syncthreads();
  for (int j = tid; j < W; j += NT_ROUTE) {
    s.active[j] = A[j];
    s.meta[j] = meta[j];
  }
  if (tid == 0) {
    *s.status = R.status;
    *s.ordinal = R.ordinal;
  }
}

size_t router_smem(int W, int nbmax, bool lean) { return make_route_layout(W, nbmax, lean).total; }

cudaError_t launch_route_batch(const RouterState& s, int32_t instance, const int64_t* offsets,
                               const uint64_t* hashes, int32_t n_req, const int32_t* out_len,
                               int32_t* worker_out, float* cost_out, int32_t* prefix_out,
                               int nbmax, const TableGeom& g, const ModelConsts& mc, float omega,
                               float tau, uint64_t seed, bool lean, cudaStream_t st) {
  if (n_req <= 0) return cudaSuccess;
  const size_t smem = router_smem(mc.W, nbmax, lean);
  cudaError_t e = cudaFuncSetAttribute(k_route_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  SimBuffers b{};
  b.keys = s.keys;
  b.stamp = s.stamp;
  b.log = s.log;
  SimLaunch L{};
  L.nsim = 1;
  L.nbmax = nbmax;
  L.g = g;
  L.mc = mc;
  k_route_batch<<<1, NT_ROUTE, smem, st>>>(b, L, s, instance, offsets, hashes, n_req, out_len,
                                         worker_out, cost_out, prefix_out, omega, tau, seed, lean);
  return cudaGetLastError();
}

// Completions: subtract, then clamp at zero (equal to clamping after every
// subtraction, since a release only subtracts).  Invalid workers are skipped
// and flagged in *bad.
__global__ void k_route_release(int64_t* active, const int32_t* __restrict__ worker,
                                const int32_t* __restrict__ blocks, int32_t n, int32_t W,
                                int32_t* status, int32_t* host) {
  int32_t* bad = status + 1;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
    const int w = worker[i];
    if (w < 0 || w >= W) {
      atomicExch(bad, 1);
      continue;
    }
    atomicAdd(reinterpret_cast<unsigned long long*>(active + w),
              (unsigned long long)(-(long long)blocks[i]));
  }
  __syncthreads();
  for (int j = threadIdx.x; j < W; j += blockDim.x)
    if (active[j] < 0) active[j] = 0;
  if (threadIdx.x == 0) {
    host[0] = status[0];
    host[1] = __ldcg(bad);   // (set by any thread of this CTA, through L2)
  }
}

cudaError_t launch_route_release(const RouterState& s, const int32_t* worker, const int32_t* blocks,
                                 int32_t n, int32_t W, int32_t* host, cudaStream_t st) {
  k_route_release<<<1, 256, 0, st>>>(s.active, worker, blocks, n, W, s.status, host);
  return cudaGetLastError();
}

__global__ void k_clear_tables(uint64_t* keys, uint32_t* stamp, size_t nslots, CacheMeta* meta,
                               size_t nmeta) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x; s < nslots; s += stride) {
    keys[s] = KEY_EMPTY;
    stamp[s] = STAMP_NONE;
  }
  for (size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x; s < nmeta; s += stride)
    meta[s] = CacheMeta{};
}

cudaError_t launch_clear_tables(uint64_t* keys, uint32_t* stamp, size_t nslots, CacheMeta* meta,
                                size_t nmeta, cudaStream_t st) {
  k_clear_tables<<<152 * 4, 256, 0, st>>>(keys, stamp, nslots, meta, nmeta);
  return cudaGetLastError();
}

// Batch probe (route_probe): the first-miss prefix m_ij of S2 for every
// (request, worker) pair against one snapshot of the tables (only read).
//
// A warp takes a request.  First its block 0 on every worker, a lane per
// worker (most pairs miss there); then, for the workers still open, chunks of
// 32 blocks, a lane per block: a chunk's hashes are loaded once and give the
// same home bucket in every worker's table, and two workers' buckets are
// requested before any is scanned.  A worker closes at its first absent block.
// Bound by the latency of the bucket loads and by issue.  20 000 requests at
// W = 64 (a call with its hashing): 443 us with a warp's 64 pairs walked together
// in steps of shared lookup slots (5 460 instructions per 64 pairs), 257 us so
// (294 before the hashing staged its chunks; then three or four workers' buckets
// in flight took 297 and 310 us: registers).
constexpr int PROBE_NT = 128;
constexpr int PROBE_ILP = 2;

// Whether h is in table t, its home bucket b already loaded in v.
__device__ __forceinline__ bool probe_present(const uint64_t* keys, uint32_t bmask,
                                              const uint64_t (&v)[BUCKET], uint32_t b, uint64_t h) {
  bool hit = false, empty = false;
#pragma unroll
  for (int q = 0; q < BUCKET; q++) {
    hit |= v[q] == h;
    empty |= v[q] == KEY_EMPTY;
  }
  if (hit || empty) return hit;
  // (rare at the tables' load) a bucket full of other keys: along the probe sequence
  TableView t{};
  t.keys = const_cast<uint64_t*>(keys);
  t.bmask = bmask;
  int err = 0;
  uint32_t fr = SLOT_NONE;
  return table_find_free_from(t, h, (b + 1) & bmask, &err, &fr) != SLOT_NONE;
}

__global__ void __launch_bounds__(PROBE_NT) k_probe_batch(const uint64_t* __restrict__ keys,
                                                          const int64_t* __restrict__ offsets,
                                                          const uint64_t* __restrict__ hashes,
                                                          int64_t n_req, int W, size_t slots,
                                                          uint32_t bmask,
                                                          int32_t* __restrict__ prefix_out) {
  const int lane = (int)(threadIdx.x & 31);
  const int64_t nw = ((int64_t)gridDim.x * PROBE_NT) >> 5;
  for (int64_t i = ((int64_t)blockIdx.x * PROBE_NT + threadIdx.x) >> 5; i < n_req; i += nw) {
    const int64_t o0 = __ldg(offsets + i);
    const int64_t nbl = (__ldg(offsets + i + 1) - o0) >> 4;
    const int nb = (int)(nbl < 0x7FFFFFFF ? nbl : 0x7FFFFFFF);
    const uint64_t* hp = hashes + (o0 >> 4);
    int m[2] = {0, 0};             // of workers lane, lane + 32
    unsigned long long open = 0;   // (uniform) workers with every block so far present
    if (nb > 0) {
      const uint64_t h = __ldg(hp);
      const uint32_t bk = home_bucket(h, bmask);
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const int j = lane + 32 * q;
        bool in = false;
        if (j < W) {
          const uint64_t* t = keys + (size_t)j * slots;
          uint64_t v[BUCKET];
          ld_bucket(t, bk, v);
          in = probe_present(t, bmask, v, bk, h);
        }
        open |= (unsigned long long)__ballot_sync(FULL_MASK, in) << (32 * q);
      }
    }
    for (int k0 = 1; open != 0ull; k0 += 32) {
      const int k = k0 + lane;
      const bool past = k >= nb;   // the prompt's end closes a walk like a miss
      uint64_t h = 0;
      if (!past) h = __ldg(hp + k);
      const uint32_t bk = home_bucket(h, bmask);
      unsigned long long left = open;
      while (left != 0ull) {
        int jj[PROBE_ILP];
        uint64_t v[PROBE_ILP][BUCKET];
#pragma unroll
        for (int r = 0; r < PROBE_ILP; r++) {
          jj[r] = left != 0ull ? __ffsll((long long)left) - 1 : -1;
          left &= left - 1ull;
          if (jj[r] >= 0 && !past) ld_bucket(keys + (size_t)jj[r] * slots, bk, v[r]);
        }
#pragma unroll
        for (int r = 0; r < PROBE_ILP; r++) {
          if (jj[r] < 0) continue;
          const bool miss = past || !probe_present(keys + (size_t)jj[r] * slots, bmask, v[r], bk, h);
          const unsigned mm = __ballot_sync(FULL_MASK, miss);
          if (mm) {
            const int mj = k0 + __ffs(mm) - 1;
            if (lane == (jj[r] & 31)) {
              if (jj[r] < 32) m[0] = mj; else m[1] = mj;
            }
            open &= ~(1ull << jj[r]);
          }
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 2; q++)
      if (lane + 32 * q < W) prefix_out[i * W + lane + 32 * q] = m[q];
  }
}

cudaError_t launch_probe_batch(const RouterState& s, const int64_t* offsets, const uint64_t* hashes,
                               int64_t n_req, int W, const TableGeom& g, int32_t* prefix_out,
                               cudaStream_t st) {
  if (n_req <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // a warp per request, as short CTAs: walks differ in length
  int64_t nblk = (n_req + PROBE_NT / 32 - 1) / (PROBE_NT / 32);
  if (nblk > (int64_t)sms * 256) nblk = (int64_t)sms * 256;
  k_probe_batch<<<(unsigned)nblk, PROBE_NT, 0, st>>>(s.keys, offsets, hashes, n_req, W, g.slots,
                                                     g.bmask, prefix_out);
  return cudaGetLastError();
}

}  // namespace rs
