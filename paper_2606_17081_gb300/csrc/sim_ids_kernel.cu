// Closed-loop routing simulation on block ids: the simulation of sim_kernel.cu
// (same events, choices and LRU caches, same results) without hash tables.
//
// A call's traces are known before the first request is routed, so every
// block of a trace gets a number first (launch_block_ids): blocks whose hash
// occurs once in the trace ("single": most prompts' tails) and blocks that
// occur again (numbered 0 .. nre-1).  Two facts make the caches small:
//   - the first occurrence of a hash ("fresh") is in no cache, so it is never
//     looked up;
//   - a single block is never looked up at all.
// A worker's cache is then one stamp per reusable block (its time of last
// touch, STAMP_NONE when absent: 20 KB for a trace of 64 prefix groups) and
// the log ring of what was appended, in stamp order.  A log entry of a
// reusable block is live iff the block still carries that stamp; a single
// block's entry (SINGLE_FLAG | its position in the trace) is live as long as
// it is at or past the head.  A lookup is a 4-byte load of a stamp, 32
// consecutive blocks of a prompt usually one or two cache lines; nothing is
// inserted, probed or rehashed.
//
// One CTA per replica; NU update warps, a control warp, a staging warp, joined
// by one CTA barrier per request.  Between the joins of requests i and i+1:
//   update   the choice, request i's cache update on the chosen worker, then
//            request i+1's cached prefix on every worker;
//   control  the choice, request i's load and service start, then completions
//            and controller samples up to request i+1's arrival, whose loads
//            it publishes for the next choice;
//   staging  the choice, request i's records and statistics, then request
//            i+3's scalars and block ids.
// What the groups hand one another at the join is double-buffered by the
// request's parity, so no other barrier is shared.  The choice is computed by
// every warp alike.
#include <algorithm>

#include "sim_common.cuh"

namespace rs {

constexpr uint32_t CODE_FRESH = 0x80000000u;    // first occurrence in the trace
constexpr uint32_t CODE_SINGLE = 0x7FFFFFFFu;   // (low bits) occurs once
constexpr uint32_t SINGLE_FLAG = 0x80000000u;   // log entry: a single block's position

// ------------------------------------------------------------ block ids

// Passes over all blocks of the launch's traces, one warp per request.
// Pass 1: every hash into its trace's open-addressing set (keys 0 = empty),
// the least position holding it kept beside it; ids[pos] = the set's slot.
__global__ void __launch_bounds__(256) k_ids_insert(const IdJob* __restrict__ jobs, int njobs,
                                                    int64_t total_req) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total_req; r += nw) {
    int jb = 0;
    while (jb + 1 < njobs && r >= jobs[jb + 1].req_base) jb++;
    const IdJob& J = jobs[jb];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i), base = o0 >> 4;
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    for (int64_t k = lane; k < nb; k += 32) {
      const unsigned long long h = __ldg(J.hashes + base + k);
      const uint32_t pos = (uint32_t)(base + k);
      uint32_t d = (uint32_t)mix64(h) & J.tmask;
      for (;;) {   // ends: the set has at least twice as many slots as blocks
        unsigned long long cur = __ldcg(J.keys + d);
        if (cur == 0ull) cur = atomicCAS(J.keys + d, 0ull, h);
        if (cur == 0ull || cur == h) break;
        d = (d + 1) & J.tmask;
      }
      if (__ldcg(J.first + d) > pos) atomicMin(J.first + d, pos);
      J.ids[base + k] = d;
    }
  }
}

// Pass 2: slots whose hash occurs at a second position get bit 31 of `first`.
__global__ void __launch_bounds__(256) k_ids_again(const IdJob* __restrict__ jobs, int njobs,
                                                   int64_t total_req) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total_req; r += nw) {
    int jb = 0;
    while (jb + 1 < njobs && r >= jobs[jb + 1].req_base) jb++;
    const IdJob& J = jobs[jb];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i), base = o0 >> 4;
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    for (int64_t k = lane; k < nb; k += 32) {
      const uint32_t d = J.ids[base + k], f = __ldcg(J.first + d);
      if (f != (uint32_t)(base + k) && !(f >> 31) &&
          (f & 0x7FFFFFFFu) != (uint32_t)(base + k))
        J.first[d] = f | 0x80000000u;   // (every writer writes the same word)
    }
  }
}

// Pass 3: the reusable blocks' numbers, consecutive along the request that
// holds their first occurrences.
__global__ void __launch_bounds__(256) k_ids_number(const IdJob* __restrict__ jobs, int njobs,
                                                    int64_t total_req) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total_req; r += nw) {
    int jb = 0;
    while (jb + 1 < njobs && r >= jobs[jb + 1].req_base) jb++;
    const IdJob& J = jobs[jb];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i), base = o0 >> 4;
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    int cnt = 0;
    for (int64_t k0 = 0; k0 < nb; k0 += 32) {
      const int64_t k = k0 + lane;
      const bool mine =
          k < nb && J.first[J.ids[base + k]] == ((uint32_t)(base + k) | 0x80000000u);
      cnt += __popc(__ballot_sync(FULL_MASK, mine));
    }
    if (cnt == 0) continue;
    uint32_t next = 0;
    if (lane == 0) next = atomicAdd(J.count, (uint32_t)cnt);
    next = __shfl_sync(FULL_MASK, next, 0);
    for (int64_t k0 = 0; k0 < nb; k0 += 32) {
      const int64_t k = k0 + lane;
      const uint32_t d = k < nb ? J.ids[base + k] : 0u;
      const bool mine = k < nb && J.first[d] == ((uint32_t)(base + k) | 0x80000000u);
      const unsigned m = __ballot_sync(FULL_MASK, mine);
      if (mine) J.num[d] = next + __popc(m & ((1u << lane) - 1u));
      next += __popc(m);
    }
  }
}

// Pass 4: ids[pos] = CODE_FRESH (first occurrence) | the block's number or
// CODE_SINGLE; nz[i] = blocks of request i up to its last one that is not
// fresh.
__global__ void __launch_bounds__(256) k_ids_write(const IdJob* __restrict__ jobs, int njobs,
                                                   int64_t total_req) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total_req; r += nw) {
    int jb = 0;
    while (jb + 1 < njobs && r >= jobs[jb + 1].req_base) jb++;
    const IdJob& J = jobs[jb];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i), base = o0 >> 4;
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    int64_t last = 0;
    for (int64_t k0 = 0; k0 < nb; k0 += 32) {
      const int64_t k = k0 + lane;
      bool seen = false;
      if (k < nb) {
        const uint32_t d = J.ids[base + k], f = J.first[d];
        const bool fresh = (f & 0x7FFFFFFFu) == (uint32_t)(base + k);
        const uint32_t x = f >> 31 ? J.num[d] : CODE_SINGLE;
        J.ids[base + k] = fresh ? x | CODE_FRESH : x;
        seen = !fresh;
      }
      const unsigned m = __ballot_sync(FULL_MASK, seen);
      if (m) last = k0 + 32 - __clz(m);
    }
    if (lane == 0) J.nz[i] = (int32_t)last;
  }
}

cudaError_t launch_block_ids(const IdJob* jobs_dev, int njobs, int64_t total_req, cudaStream_t st) {
  if (total_req <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t nblk = std::min<int64_t>((total_req + 7) / 8, (int64_t)sms * 32);
  k_ids_insert<<<(unsigned)nblk, 256, 0, st>>>(jobs_dev, njobs, total_req);
  k_ids_again<<<(unsigned)nblk, 256, 0, st>>>(jobs_dev, njobs, total_req);
  k_ids_number<<<(unsigned)nblk, 256, 0, st>>>(jobs_dev, njobs, total_req);
  k_ids_write<<<(unsigned)nblk, 256, 0, st>>>(jobs_dev, njobs, total_req);
  return cudaGetLastError();
}

// ------------------------------------------------------------ the replica's state

constexpr int IDS_RING = 4;   // requests staged at once (i .. i+3)

// A staged request: what the loop needs beside its block ids.
struct IdsReq : ReqState {
  int64_t pos0;        // position of its first block in the trace
  double inv;          // 1 / nbt, rounded (0 for an empty prompt)
  uint32_t dx, dy;     // words 0 and 1 of its Philox block
  int32_t nz, pad;
};

// What the control warp publishes of a request's arrival.
struct IdsArrival {
  double a;
  float tau, omega;
};

struct IdsShared {
  IdsReq q[IDS_RING];
  IdsArrival pub[2];
  int stat[2];                 // by parity: an error seen before that join
  int hist[256];
  alignas(16) uint4 red[8];    // per update warp: absent blocks, least stamp, live entries
  int warp_tot[8];
  int err;                     // of the update
  int bad, nvic, nins;
};

struct IdsLayout {
  size_t ftab, f_oitl, f_a, f_o, h_k, wA, codes, meta, f_req, f_worker, f_blk, f_next, h_f,
      freestk, winserv, wqh, wqt, wm, act, nfz, whead, wlen, win;
  size_t total, slot_bytes;
};

__host__ __device__ inline IdsLayout make_ids_layout(int W, int nbmax, int cmax, int nft, int ntu,
                                                     bool slots_global) {
  IdsLayout L;
  size_t o = 0, og = 0;
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1), C = (size_t)(cmax > 0 ? cmax : 1);
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += (bytes + 15) & ~(size_t)15;
    return r;
  };
  auto slots = [&](size_t bytes) {
    if (!slots_global) return take(bytes);
    const size_t r = og;
    og += (bytes + 15) & ~(size_t)15;
    return r;
  };
  L.ftab = take(8 * (size_t)(nft > 0 ? nft : 1));
  L.f_oitl = slots(8 * C);
  L.f_a = slots(8 * C);
  L.f_o = slots(8 * C);
  L.h_k = slots(8 * C);
  L.wA = take(8 * (size_t)W);
  L.codes = take(4 * nb * IDS_RING);
  L.meta = take(sizeof(CacheMeta) * (size_t)W);
  L.f_req = slots(4 * C);
  L.f_worker = slots(4 * C);
  L.f_blk = slots(4 * C);
  L.f_next = slots(4 * C);
  L.h_f = slots(4 * C);
  L.freestk = slots(4 * C);
  L.winserv = take(4 * (size_t)W);
  L.wqh = take(4 * (size_t)W);
  L.wqt = take(4 * (size_t)W);
  L.wm = take(4 * 2 * (size_t)W);
  L.act = take(4 * 2 * (size_t)W);
  L.nfz = take(4 * 2 * (size_t)W);
  L.whead = take(4 * (size_t)W);
  L.wlen = take(4 * (size_t)W);
  L.win = take(4 * (size_t)W * ntu);
  L.total = o;
  L.slot_bytes = (og + 255) & ~(size_t)255;
  return L;
}

size_t sim_ids_smem_bytes(int W, int nbmax, int cmax, int cap, int ntu, bool slots_global) {
  return make_ids_layout(W, nbmax, cmax, ftab_size(cap), ntu, slots_global).total;
}

// Global scratch of one replica for the updates that need the exact sequence.
struct IdsScratch {
  uint32_t *vent, *vt, *pst;    // [2 nb] live entries and positions, [nb] stamps
  int32_t *owner, *victim;      // [2 nb]
  uint8_t *touched, *kind, *evk;   // [2 nb], [nb], [nb]
};

__host__ __device__ inline size_t ids_scratch_bytes(int nbmax) {
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1);
  return (40 * nb + 255) & ~(size_t)255;
}

size_t sim_ids_scratch_bytes(int nbmax) { return ids_scratch_bytes(nbmax); }

__device__ __forceinline__ IdsScratch ids_scratch(unsigned char* p, int nbmax) {
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1);
  IdsScratch s;
  s.vent = reinterpret_cast<uint32_t*>(p);
  s.vt = s.vent + 2 * nb;
  s.owner = reinterpret_cast<int32_t*>(s.vt + 2 * nb);
  s.victim = s.owner + 2 * nb;
  s.pst = reinterpret_cast<uint32_t*>(s.victim + 2 * nb);
  s.touched = reinterpret_cast<uint8_t*>(s.pst + nb);
  s.kind = s.touched + 2 * nb;
  s.evk = s.kind + nb;
  return s;
}

// One worker's cache.
struct IdsTable {
  uint32_t* st;    // [nre] stamps
  uint32_t* log;   // [rmask + 1]
  uint32_t rmask;
};

// 4-byte global -> shared copy in the background.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}

template <int NT>
__device__ __forceinline__ void join_cta() {
  asm volatile("barrier.sync 0, %0;" ::"n"(NT) : "memory");
}

// ------------------------------------------------------------ probe

// Leading blocks of the prompt found in one worker's cache from block k0 on,
// at most nz (a warp; four stamps per lane in flight).
__device__ __forceinline__ int ids_prefix(const uint32_t* st, const uint32_t* cd, int k0, int nz,
                                          unsigned& cnt) {
  const int lane = (int)(threadIdx.x & 31);
  for (int k = k0; k < nz; k += 128) {
    uint32_t v[4];
    bool in[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int kk = k + 32 * r + lane;
      in[r] = kk < nz;
      const uint32_t c = in[r] ? cd[kk] : CODE_FRESH;
      v[r] = STAMP_NONE;
      if (!(c >> 31)) {
        v[r] = st[c];
        cnt++;
      }
    }
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const unsigned m = __ballot_sync(FULL_MASK, in[r] && v[r] == STAMP_NONE);
      if (m) return k + 32 * r + __ffs(m) - 1;
    }
  }
  return nz;
}

// m_j of every worker (the NU update warps); wm[j] = m_j.  Up to NU workers:
// a warp each.  More: a warp walks four workers at a time, two chunks of 32
// blocks of each in flight, until each has its first miss.
template <int NU>
__device__ __forceinline__ void ids_probe(const uint32_t* stamps, size_t nre, const uint32_t* cd,
                                          int nz, int W, int* wm, unsigned& cnt) {
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  if (W <= NU) {
    if (warp < W) {
      const int m = ids_prefix(stamps + warp * nre, cd, 0, nz, cnt);
      if (lane == 0) wm[warp] = m;
    }
    return;
  }
  for (int j0 = warp; j0 < W; j0 += 4 * NU) {
    unsigned open = 0;   // (uniform) bit q: worker j0 + q NU still all present
    int m[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      m[q] = nz;
      open |= (unsigned)(j0 + q * NU < W) << q;
    }
    for (int k = 0; k < nz && open; k += 64) {
      const int ka = k + lane, kb = ka + 32;
      const uint32_t ca = ka < nz ? cd[ka] : CODE_FRESH, cb = kb < nz ? cd[kb] : CODE_FRESH;
      uint32_t va[4], vb[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const uint32_t* st = stamps + (size_t)(j0 + q * NU) * nre;
        va[q] = vb[q] = STAMP_NONE;
        if ((open >> q) & 1u) {
          if (!(ca >> 31)) {
            va[q] = st[ca];
            cnt++;
          }
          if (!(cb >> 31)) {
            vb[q] = st[cb];
            cnt++;
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const unsigned ma = __ballot_sync(FULL_MASK, ka < nz && va[q] == STAMP_NONE);
        const unsigned mb = __ballot_sync(FULL_MASK, kb < nz && vb[q] == STAMP_NONE);
        if (((open >> q) & 1u) && (ma | mb)) {
          m[q] = ma ? k + __ffs(ma) - 1 : k + 32 + __ffs(mb) - 1;
          open &= ~(1u << q);
        }
      }
    }
    if (lane < 4 && j0 + lane * NU < W)
      wm[j0 + lane * NU] = lane == 0 ? m[0] : (lane == 1 ? m[1] : (lane == 2 ? m[2] : m[3]));
  }
}

// ------------------------------------------------------------ choice

// Eq. (1) costs of workers lane and lane + 32 and the chosen worker (a warp;
// every warp the same).  Costs are >= +0, so their bit patterns order them.
struct IdsChoice {
  float c[2], best;
  int bj, js;
  float target, S, lo, hi;   // where an Eq. (2) draw fell
};

__device__ __forceinline__ IdsChoice ids_choice(const SimDesc& d, const IdsReq& q,
                                                const IdsArrival& ar, const int* wm,
                                                const float* act, int W, int64_t i, int lane) {
  IdsChoice r;
  const float om = ar.omega, tau = ar.tau;
  const float inf = __int_as_float(0x7F800000);
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int j = lane + 32 * h;
    r.c[h] = inf;
    if (j < W) r.c[h] = __fadd_rn(__fmul_rn(om, __int2float_rn(q.nbt - wm[j])), act[j]);
  }
  const unsigned mn = __reduce_min_sync(FULL_MASK, min(__float_as_uint(r.c[0]), __float_as_uint(r.c[1])));
  // the lowest index among the minima: workers 0-31 first
  const unsigned e0 =
      __ballot_sync(FULL_MASK, lane < W && __float_as_uint(r.c[0]) == mn);
  const unsigned e1 =
      W > 32 ? __ballot_sync(FULL_MASK, lane + 32 < W && __float_as_uint(r.c[1]) == mn) : 0u;
  r.bj = e0 ? __ffs(e0) - 1 : 32 + __ffs(e1) - 1;
  r.best = __uint_as_float(mn);
  r.js = r.bj;
  if (d.policy != RS_POLICY_DYNAMO && d.policy != RS_POLICY_LOADBAL) {
    // the static policies (as static_policy_worker)
    if (d.policy == RS_POLICY_ROUNDROBIN) {
      r.js = (int)((uint64_t)i % (uint64_t)W);
    } else {
      const int j1 = (int)(((uint64_t)(q.dx >> 8) * (uint64_t)W) >> 24);
      r.js = j1;
      if (d.policy == RS_POLICY_P2C && W >= 2) {
        int j2 = (int)(((uint64_t)(q.dy >> 8) * (uint64_t)(W - 1)) >> 24);
        if (j2 >= j1) j2++;
        const int lo = j1 < j2 ? j1 : j2, hi = j1 < j2 ? j2 : j1;
        const float cl0 = __shfl_sync(FULL_MASK, r.c[0], lo & 31);
        const float cl1 = __shfl_sync(FULL_MASK, r.c[1], lo & 31);
        const float ch0 = __shfl_sync(FULL_MASK, r.c[0], hi & 31);
        const float ch1 = __shfl_sync(FULL_MASK, r.c[1], hi & 31);
        r.js = (hi < 32 ? ch0 : ch1) < (lo < 32 ? cl0 : cl1) ? hi : lo;
      }
    }
  } else if (tau > 0.0f) {
    // Eq. (2), as select_worker_warp: one weight per lane, sums in worker order
    float e[2];
#pragma unroll
    for (int h = 0; h < 2; h++)
      e[h] = lane + 32 * h < W ? exp_sm(-__fdiv_rn(__fsub_rn(r.c[h], r.best), tau)) : 0.0f;
    float S = 0.0f;
    for (int j = 0; j < W; j++)
      S = __fadd_rn(S, __shfl_sync(FULL_MASK, j < 32 ? e[0] : e[1], j & 31));
    r.target = __fmul_rn(__fmul_rn((float)(q.dx >> 8), 0x1p-24f), S);
    r.S = S;
    const float qnan = __int_as_float(0x7FC00000);
    float cum = 0.0f;
    r.lo = r.hi = qnan;
    int pick = -1, last = r.bj;
    for (int j = 0; j < W; j++) {
      const float ej = __shfl_sync(FULL_MASK, j < 32 ? e[0] : e[1], j & 31);
      cum = __fadd_rn(cum, ej);
      if (ej > 0.0f) last = j;
      if (pick < 0 && r.target < cum) {
        pick = j;
        r.hi = cum;
      }
      if (!(r.target < cum)) r.lo = cum;
    }
    r.js = pick >= 0 ? pick : last;
  }
  return r;
}

// ------------------------------------------------------------ cache update (update warps)

// Position of the n-th (0-based) set bit of x; x has more than n set bits.
__device__ __forceinline__ int nth_set_bit32(unsigned x, int n) {
  int pos = 0;
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const int c = __popc(x & ((1u << w) - 1u));
    if (n >= c) {
      n -= c;
      x >>= w;
      pos += w;
    }
  }
  return pos;
}

// Whether log entry x at position p is live.
__device__ __forceinline__ bool ids_live(const IdsTable& t, uint32_t x, uint32_t p) {
  return (x & SINGLE_FLAG) || t.st[x] == p;
}

// Moves the live entries of the log down to the head, in order, and renumbers
// stamps by a multiple of the ring's length (so ring places stay), in place:
// an entry never moves up.
template <int NT>
__device__ __forceinline__ void ids_compact(const IdsTable& t, CacheMeta* meta, int* warp_tot,
                                            int* err) {
  const uint32_t head = meta->head, T = meta->T, size = meta->size;
  const uint32_t d = head & ~t.rmask;
  constexpr int PER = 4;
  uint32_t base = 0;
  for (uint32_t p0 = head; p0 < T; p0 += NT * PER) {
    const uint32_t pb = p0 + threadIdx.x * PER;
    uint32_t x[PER];
    bool live[PER];
    int cnt = 0;
#pragma unroll
    for (int e = 0; e < PER; e++) x[e] = pb + e < T ? t.log[(pb + e) & t.rmask] : 0u;
#pragma unroll
    for (int e = 0; e < PER; e++) {
      live[e] = pb + e < T && ids_live(t, x[e], pb + e);
      cnt += live[e];
    }
    int tot;
    uint32_t np = head + base + (uint32_t)grp_excl_scan<NT>(cnt, warp_tot, &tot);
#pragma unroll
    for (int e = 0; e < PER; e++)
      if (live[e]) {
        t.log[np & t.rmask] = x[e];
        if (!(x[e] & SINGLE_FLAG)) t.st[x[e]] = np - d;
        np++;
      }
    base += (uint32_t)tot;
    grp_bar<NT>();
  }
  if (threadIdx.x == 0) {
    if (base != size) *err = RS_ERR_TIMEOUT;
    meta->head = head - d;
    meta->T = head - d + base;
  }
  grp_bar<NT>();
}

// The first `want` live entries from the head into vent / vt; returns how many.
template <int NT>
__device__ __forceinline__ uint32_t ids_gather(const IdsTable& t, uint32_t head, uint32_t T,
                                               uint32_t want, const IdsScratch& sc, int* warp_tot) {
  uint32_t have = 0;
  for (uint32_t p0 = head; have < want && p0 < T; p0 += NT) {
    const uint32_t p = p0 + threadIdx.x;
    uint32_t x = 0;
    bool live = false;
    if (p < T) {
      x = t.log[p & t.rmask];
      live = ids_live(t, x, p);
    }
    int tot;
    const int r = cta_rank<NT>(live, warp_tot, &tot);
    if (live && have + r < want) {
      sc.vent[have + r] = x;
      sc.vt[have + r] = p;
    }
    have = min(want, have + (uint32_t)tot);
  }
  grp_bar<NT>();
  return have;
}

// Place of stamp st among the n increasing positions vt (n: none at or past it).
__device__ __forceinline__ uint32_t ids_place(const uint32_t* vt, uint32_t n, uint32_t st) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (vt[mid] < st) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// An update whose victims the window does not settle: more victims than it
// holds, or a present block among the least recent entries, which the exact
// sequence (one thread, over the first 2 nb live entries) decides.  Evicts;
// returns the head past the last victim, victims in *E, insertions in *nins.
template <int NT>
__device__ __forceinline__ uint32_t ids_evict_general(const IdsTable& t, const CacheMeta& m,
                                                      uint32_t K, const uint32_t* cd, int nb,
                                                      uint32_t E0, uint32_t pmin, int nabs,
                                                      const IdsScratch& sc, IdsShared& S,
                                                      int64_t* slow, uint32_t* E, int* nins) {
  uint32_t G = ids_gather<NT>(t, m.head, m.T, E0, sc, S.warp_tot);
  *E = 0;
  *nins = nabs;
  if (G < E0) {   // fewer live entries than the size says
    if (threadIdx.x == 0) S.err = RS_ERR_TIMEOUT;
    return m.head;
  }
  if (pmin > sc.vt[E0 - 1]) {   // (also pmin = STAMP_NONE: no block present)
    for (uint32_t v = threadIdx.x; v < E0; v += NT)
      if (!(sc.vent[v] & SINGLE_FLAG)) t.st[sc.vent[v]] = STAMP_NONE;
    *E = E0;
    return sc.vt[E0 - 1] + 1;
  }
  grp_bar<NT>();
  G = ids_gather<NT>(t, m.head, m.T, min(m.size, 2u * (uint32_t)nb), sc, S.warp_tot);
  for (uint32_t p = threadIdx.x; p < G; p += NT) {
    sc.owner[p] = -1;
    sc.touched[p] = 0;
  }
  grp_bar<NT>();
  const uint32_t last = G ? sc.vt[G - 1] : 0u;
  for (int k = threadIdx.x; k < nb; k += NT) {
    const uint32_t c = cd[k];
    const uint32_t st = c >> 31 ? STAMP_NONE : t.st[c];
    sc.pst[k] = st;
    sc.evk[k] = 0;
    if (st != STAMP_NONE && G && st <= last) sc.owner[ids_place(sc.vt, G, st)] = k;
  }
  grp_bar<NT>();
  if (threadIdx.x == 0) {
    uint32_t ptr = 0, sz = m.size;
    int e = 0, ni = 0;
    for (int k = 0; k < nb; k++) {
      const uint32_t st = sc.pst[k];
      if (st != STAMP_NONE && !sc.evk[k]) {
        if (G && st <= last) sc.touched[ids_place(sc.vt, G, st)] = 1;
        continue;
      }
      ni++;
      if (sz < K) {
        sz++;
        continue;
      }
      while (ptr < G && sc.touched[ptr]) ptr++;
      if (ptr >= G) {
        S.err = RS_ERR_TIMEOUT;
        break;
      }
      sc.victim[e++] = (int32_t)ptr;
      if (sc.owner[ptr] >= 0) sc.evk[sc.owner[ptr]] = 1;
      ptr++;
    }
    S.nvic = e;
    S.nins = ni;
    ++*slow;
  }
  grp_bar<NT>();
  const int e = S.nvic;
  for (int v = threadIdx.x; v < e; v += NT) {
    const uint32_t x = sc.vent[sc.victim[v]];
    if (!(x & SINGLE_FLAG)) t.st[x] = STAMP_NONE;
  }
  *E = (uint32_t)e;
  *nins = S.nins;
  const uint32_t nh = e > 0 ? sc.vt[sc.victim[e - 1]] + 1 : m.head;
  grp_bar<NT>();   // a victim may be a block of this request: its new stamp comes after
  return nh;
}

// Request i's blocks touched in order on the chosen worker's cache (exact
// LRU), by the update warps.  The window win holds the log entries from
// whead on (copied in the background after the worker's last update), so the
// common update makes one round of stamp loads and one barrier: every thread
// reads the stamp of one block of the prompt and of one window entry; the
// live entries before the oldest present block are the candidates, and the
// first E0 = absent - free of them are the victims.
template <int NT>
__device__ __forceinline__ void ids_update(SimCtx& c, IdsShared& S, const IdsTable& t,
                                           CacheMeta* meta, const uint32_t* cd, const IdsReq& q,
                                           const IdsScratch& sc, uint32_t* win, uint32_t* whead,
                                           uint32_t* wlen, int64_t i) {
  constexpr int NW = NT / 32;
  const uint32_t K = c.L->g.K;
  const int nb = q.nb, nz = q.nz, tid = (int)threadIdx.x, lane = tid & 31;
  cp_async_wait_all();   // this thread's window entries
  if ((uint64_t)meta->T - meta->head + (uint64_t)nb > (uint64_t)t.rmask + 1 ||
      (uint64_t)meta->T + nb > STAMP_LIMIT) {
    grp_bar<NT>();
    ids_compact<NT>(t, meta, S.warp_tot, &S.err);
    if (tid == 0) {
      c.S->rebuilds++;
      *wlen = 0;
    }
    grp_bar<NT>();
  }
  const CacheMeta m = *meta;
  const bool full = m.size + (uint32_t)nb > K;   // a victim may be needed
  // stamps of the prompt's blocks, of the window's entries
  int nabs = 0;
  uint32_t pmin = STAMP_NONE;
  for (int k = tid; k < nz; k += NT) {
    const uint32_t x = cd[k];
    const uint32_t st = x >> 31 ? STAMP_NONE : t.st[x];
    nabs += st == STAMP_NONE;
    pmin = min(pmin, st);
  }
  uint32_t x = 0;
  bool live = false;
  if (full) {
    const uint32_t p = m.head + tid;
    if (p < m.T) {
      x = *whead == m.head && (uint32_t)tid < *wlen ? win[tid] : t.log[p & t.rmask];
      live = ids_live(t, x, p);
    }
  }
  {
    const int a = (int)__reduce_add_sync(FULL_MASK, (unsigned)nabs);
    const uint32_t pm = __reduce_min_sync(FULL_MASK, pmin);
    const unsigned lv = __ballot_sync(FULL_MASK, live);
    if (lane == 0) S.red[tid >> 5] = make_uint4((unsigned)a, pm, lv, 0u);
  }
  grp_bar<NT>();
  nabs = nb - nz;   // past nz every block is fresh
  pmin = STAMP_NONE;
  unsigned lv[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) {
    const uint4 r = S.red[w];
    nabs += (int)r.x;
    pmin = min(pmin, r.y);
    lv[w] = r.z;
  }
  const uint32_t freeb = K - m.size;
  const uint32_t E0 = (uint32_t)nabs > freeb ? (uint32_t)nabs - freeb : 0u;
  uint32_t E = E0, nh = m.head;
  int nins = nabs;
  if (E0 > 0) {
    // candidates: live entries before the oldest present block
    const uint32_t lim = pmin - m.head;   // window places below lim qualify
    uint32_t have = 0;
    int last = -1;
#pragma unroll
    for (int w = 0; w < NW; w++) {
      const uint32_t l0 = 32u * w;
      const unsigned mk = lim >= l0 + 32u ? FULL_MASK : (lim > l0 ? (1u << (lim - l0)) - 1u : 0u);
      const unsigned b = lv[w] & mk;
      const uint32_t n = (uint32_t)__popc(b);
      if (have < E0 && have + n >= E0) last = (int)l0 + nth_set_bit32(b, (int)(E0 - have) - 1);
      have += n;
    }
    if (last >= 0) {
      if (live && tid <= last && !(x & SINGLE_FLAG)) t.st[x] = STAMP_NONE;
      nh = m.head + (uint32_t)last + 1u;
    } else {
      nh = ids_evict_general<NT>(t, m, K, cd, nb, E0, pmin, nabs, sc, S, &c.S->slow, &E, &nins);
    }
  }
  // every block of the prompt is now the most recent, in order
  for (int k = tid; k < nb; k += NT) {
    const uint32_t b = cd[k] & CODE_SINGLE, pos = m.T + (uint32_t)k;
    if (b != CODE_SINGLE) t.st[b] = pos;
    t.log[pos & t.rmask] = b != CODE_SINGLE ? b : SINGLE_FLAG | (uint32_t)(q.pos0 + k);
  }
  const uint32_t size = m.size + (uint32_t)nins - E;
  // the window of this worker's next update: entries written before this one
  // (all threads have read the old window: the barrier above)
  if (size + (uint32_t)c.L->nbmax > K) {
    const uint32_t p = nh + tid;
    if (p < m.T) cp_async4(win + tid, t.log + (p & t.rmask));
    if (tid == 0) {
      *whead = nh;
      *wlen = m.T > nh ? min((uint32_t)NT, m.T - nh) : 0u;
    }
  }
  if (tid == 0) {
    meta->size = size;
    meta->head = nh;
    meta->T = m.T + (uint32_t)nb;
    SimScalars& R = *c.S;
    R.inserted += nins;
    R.evicted += E;
    if (E > 0 && R.first_evict_i < 0) {
      // the first update that evicted; resident blocks = inserted - evicted
      R.first_evict_i = i;
      R.first_live = R.inserted - R.evicted;
    }
  }
}

// ------------------------------------------------------------ control warp

// A controller sample with a non-empty window (as the CTA-wide tick of the
// table kernel, by one warp): the window's nearest-rank P99 by an exact radix
// selection, from the highest byte in which its TTFTs differ.
__device__ __forceinline__ void ids_tick(SimCtx& c, IdsShared& Sh, int lane) {
  SimScalars& S = *c.S;
  const int cur = S.pend_cur;
  const int64_t np = S.np;
  const double* sft = c.pend_ft(cur);
  const double* stt = c.pend_tt(cur);
  double* dft = c.pend_ft(cur ^ 1);
  double* dtt = c.pend_tt(cur ^ 1);
  const uint64_t ktt = tkey(S.tick_t);
  int64_t nkeep = 0, nwin = 0;
  uint64_t mft = KEY_INF, all1 = ~0ull, any1 = 0ull;
  for (int64_t p0 = 0; p0 < np; p0 += 32) {
    const int64_t p = p0 + lane;
    double f = 0.0, v = 0.0;
    bool inwin = false;
    if (p < np) {
      f = sft[p];
      v = stt[p];
      inwin = tkey(f) < ktt;
    }
    const bool keep = p < np && !inwin;
    const unsigned mk = __ballot_sync(FULL_MASK, keep), mw = __ballot_sync(FULL_MASK, inwin);
    const unsigned below = (1u << lane) - 1u;
    if (keep) {
      dft[nkeep + __popc(mk & below)] = f;
      dtt[nkeep + __popc(mk & below)] = v;
      const uint64_t kf = tkey(f);
      mft = kf < mft ? kf : mft;
    }
    if (inwin) {
      c.pend_win[nwin + __popc(mw & below)] = v;
      const uint64_t bits = (uint64_t)__double_as_longlong(v);
      all1 &= bits;
      any1 |= bits;
    }
    nkeep += __popc(mk);
    nwin += __popc(mw);
  }
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t v = __shfl_xor_sync(FULL_MASK, mft, o);
    mft = v < mft ? v : mft;
    all1 &= __shfl_xor_sync(FULL_MASK, all1, o);
    any1 |= __shfl_xor_sync(FULL_MASK, any1, o);
  }
  __syncwarp();
  double L = 0.0;
  if (nwin > 0) {
    int kk = (int)((99 * nwin + 99) / 100);   // 1-based rank
    const uint64_t diff = all1 ^ any1;
    int shift = diff ? (63 - __clzll((long long)diff)) & ~7 : -8;
    uint64_t pre = shift < 0 ? all1 : (shift == 56 ? 0ull : all1 & (~0ull << (shift + 8)));
    for (; shift >= 0; shift -= 8) {
      for (int q = lane; q < 256; q += 32) Sh.hist[q] = 0;
      __syncwarp();
      const uint64_t mhi = shift == 56 ? 0ull : (~0ull << (shift + 8));
      for (int64_t p = lane; p < nwin; p += 32) {
        const uint64_t bits = (uint64_t)__double_as_longlong(c.pend_win[p]);
        if ((bits & mhi) == (pre & mhi)) atomicAdd(&Sh.hist[(bits >> shift) & 255], 1);
      }
      __syncwarp();
      // lane l holds bins 8 l .. 8 l + 7
      int sum = 0;
#pragma unroll
      for (int e = 0; e < 8; e++) sum += Sh.hist[8 * lane + e];
      int inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, inc, o);
        if (lane >= o) inc += y;
      }
      const unsigned hit = __ballot_sync(FULL_MASK, inc >= kk);
      const int ls = __ffs(hit) - 1;
      int dg = 0, cum = inc - sum;
      if (lane == ls)
        for (dg = 8 * lane; dg < 8 * lane + 7; dg++) {
          if (cum + Sh.hist[dg] >= kk) break;
          cum += Sh.hist[dg];
        }
      dg = __shfl_sync(FULL_MASK, dg, ls);
      kk -= __shfl_sync(FULL_MASK, cum, ls);
      pre |= (uint64_t)dg << shift;
      __syncwarp();
    }
    L = __longlong_as_double((long long)pre);
  }
  if (lane == 0) {
    S.np = nkeep;
    S.pend_cur = cur ^ 1;
    S.min_ft = tval(mft);
    ctl_sample(c, nwin > 0, L);
  }
  __syncwarp();
}

// Request i's arrival: every event before it, then what its choice needs.
__device__ __forceinline__ void ids_arrive(SimCtx& c, IdsShared& Sh, int64_t i, float* act,
                                           int* nfz, int lane) {
  SimScalars& S = *c.S;
  IdsReq& q = Sh.q[i & (IDS_RING - 1)];
  const int p = (int)(i & 1), W = c.L->mc.W;
  if (q.nb > (int)c.L->g.K) {
    if (lane == 0) Sh.stat[p] = S.status = RS_ERR_CAPACITY;
    return;
  }
  for (;;) {
    int ev = 0;
    if (lane == 0) ev = events_advance(c, q);
    if (!__shfl_sync(FULL_MASK, ev, 0)) break;
    ids_tick(c, Sh, lane);
  }
  if (lane == 0) {
    regime_params<false>(c, q);
    Sh.pub[p].a = q.a;
    Sh.pub[p].tau = q.tau;
    Sh.pub[p].omega = q.omega;
    if (S.status != RS_OK) Sh.stat[p] = S.status;
  }
  __syncwarp();
  for (int j = lane; j < W; j += 32) {
    act[p * W + j] = __int2float_rn((int)c.wA[j]);
    nfz[p * W + j] = min(c.winserv[j] + 1, c.L->mc.cap - 1);
  }
}

// ------------------------------------------------------------ staging warp

// Request i's scalars as read from the trace (issued a request ahead).
struct IdsRaw {
  int64_t o0, o1;
  double rel;
  int O, nz, dup;
};

__device__ __forceinline__ IdsRaw ids_read(const SimDesc& d, int64_t i) {
  IdsRaw r;
  r.o0 = d.offsets[i];
  r.o1 = d.offsets[i + 1];
  r.rel = d.release[i];
  r.O = d.out_len[i];
  r.nz = d.nz[i];
  r.dup = d.dupflag[i] == 1;
  return r;
}

// Starts the copy of request i's ids and writes its scalars (a warp).
__device__ __forceinline__ void ids_stage(const SimCtx& c, IdsShared& Sh, const IdsRaw& r,
                                          int64_t i, uint32_t* codes, int nbcap, int lane) {
  const int e = (int)(i & (IDS_RING - 1));
  IdsReq& q = Sh.q[e];
  const int64_t L = r.o1 - r.o0, nb64 = L >> 4;
  const int nb = nb64 > 0x7FFFFFFF ? 0x7FFFFFFF : (int)nb64;
  if (nb <= (int)c.L->g.K) {   // (a longer prompt stops the replica)
    const uint32_t* src = c.d->ids + (r.o0 >> 4);
    uint32_t* dst = codes + (size_t)e * nbcap;
    for (int k = lane; k < nb; k += 32) cp_async4(dst + k, src + k);
  }
  if (lane == 0) {
    q.off0 = r.o0;
    q.pos0 = r.o0 >> 4;
    q.rel = r.rel;
    q.O = r.O;
    q.dup = r.dup;
    q.oitl = __dmul_rn((double)r.O, c.L->mc.itl);
    q.nb = nb;
    q.nz = r.nz;
    q.nbt = (int)((L + 15) >> 4);
    q.blk = (L + r.O + 15) >> 4;
    q.phase = 0;
    q.inv = q.nbt > 0 ? __ddiv_rn(1.0, (double)q.nbt) : 0.0;
    const uint4 x = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)((uint64_t)i >> 32), 0u, TAG_SIM),
                                  make_uint2((uint32_t)c.d->seed, (uint32_t)(c.d->seed >> 32)));
    q.dx = x.x;
    q.dy = x.y;
  }
}

// ------------------------------------------------------------ the kernel

template <int NU, int MINB, bool SG>
__global__ void __launch_bounds__((NU + 2) * 32, MINB)
    k_sim_ids(const SimDesc* __restrict__ descs, const __grid_constant__ SimBuffers b,
              const __grid_constant__ SimLaunch L) {
  constexpr int NT = (NU + 2) * 32, NTU = NU * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SimScalars S;
  __shared__ IdsShared Sh;
  const int sid = blockIdx.x;
  const SimDesc d = descs[sid];
  const ModelConsts& mc = L.mc;
  const int W = mc.W;
  const int nft = ftab_size(mc.cap);
  const int nbcap = L.nbmax > 0 ? L.nbmax : 1;
  const IdsLayout lay = make_ids_layout(W, L.nbmax, L.cmax, nft, NTU, SG);
  unsigned char* slotbase;
  if constexpr (SG)
    slotbase = b.slotmem + (size_t)sid * lay.slot_bytes;
  else
    slotbase = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  SimCtx c;
  c.S = &S;
  c.d = &d;
  c.b = &b;
  c.L = &L;
  c.sid = sid;
  c.ftab = reinterpret_cast<double*>(smem + lay.ftab);
  c.f_oitl = reinterpret_cast<double*>(slotbase + lay.f_oitl);
  c.f_a = reinterpret_cast<double*>(slotbase + lay.f_a);
  c.f_o = reinterpret_cast<double*>(slotbase + lay.f_o);
  c.h_k = reinterpret_cast<uint64_t*>(slotbase + lay.h_k);
  c.f_req = reinterpret_cast<int32_t*>(slotbase + lay.f_req);
  c.f_worker = reinterpret_cast<int32_t*>(slotbase + lay.f_worker);
  c.f_blk = reinterpret_cast<int32_t*>(slotbase + lay.f_blk);
  c.f_next = reinterpret_cast<int32_t*>(slotbase + lay.f_next);
  c.h_f = reinterpret_cast<int32_t*>(slotbase + lay.h_f);
  c.freestk = reinterpret_cast<int32_t*>(slotbase + lay.freestk);
  c.winserv = reinterpret_cast<int32_t*>(smem + lay.winserv);
  c.wqh = reinterpret_cast<int32_t*>(smem + lay.wqh);
  c.wqt = reinterpret_cast<int32_t*>(smem + lay.wqt);
  c.wA = reinterpret_cast<int64_t*>(smem + lay.wA);
  c.wmeta = reinterpret_cast<CacheMeta*>(smem + lay.meta);
  double* pend = b.pend + (size_t)sid * 5 * b.pend_cap;
  c.pend_ft0 = pend;
  c.pend_tt0 = pend + b.pend_cap;
  c.pend_ft1 = pend + 2 * b.pend_cap;
  c.pend_tt1 = pend + 3 * b.pend_cap;
  c.pend_win = pend + 4 * b.pend_cap;
  uint32_t* codes = reinterpret_cast<uint32_t*>(smem + lay.codes);   // [ring][nbcap]
  int* wm = reinterpret_cast<int*>(smem + lay.wm);                   // [2][W]
  float* act = reinterpret_cast<float*>(smem + lay.act);             // [2][W]
  int* nfz = reinterpret_cast<int*>(smem + lay.nfz);                 // [2][W]
  uint32_t* whead = reinterpret_cast<uint32_t*>(smem + lay.whead);
  uint32_t* wlen = reinterpret_cast<uint32_t*>(smem + lay.wlen);
  uint32_t* win = reinterpret_cast<uint32_t*>(smem + lay.win);       // [W][NTU]
  uint32_t* stamps = d.stamps;
  const size_t nre = d.nre;
  const int64_t n = d.n_req;

  // ---- initial state: empty caches, idle workers
  {
    const size_t nst = (size_t)W * nre;   // (nre: a multiple of 4)
    for (size_t s = threadIdx.x; s < nst / 4; s += NT)
      reinterpret_cast<uint4*>(stamps)[s] = make_uint4(STAMP_NONE, STAMP_NONE, STAMP_NONE, STAMP_NONE);
    for (int q = 1 + threadIdx.x; q < nft; q += NT) c.ftab[q] = latency_f(mc, q);
    const int cslots = max(d.C, max(d.c_mid, d.c_end));
    for (int p = threadIdx.x; p < cslots; p += NT) c.freestk[p] = cslots - 1 - p;
    for (int j = threadIdx.x; j < W; j += NT) {
      c.wmeta[j] = CacheMeta{};
      c.winserv[j] = 0;
      c.wA[j] = 0;
      c.wqh[j] = -1;
      c.wqt[j] = -1;
      whead[j] = 0;
      wlen[j] = 0;
    }
    if (threadIdx.x == 0) {
      memset(&S, 0, sizeof(SimScalars));
      S.min_ft = __longlong_as_double(0x7FF0000000000000ll);
      S.next_tick = 1;
      S.tick_t = mc.dt;
      S.nfree = cslots;
      S.first_switch_t = -1.0;
      S.first_evict_i = -1;
      Sh.stat[0] = Sh.stat[1] = RS_OK;
      Sh.err = 0;
    }
  }
  // ---- prologue: the first requests staged
  IdsRaw raw;   // (staging warp) the request after the last one staged
  if (warp == NU + 1) {
    for (int64_t i = 0; i < 3 && i < n; i++) {
      raw = ids_read(d, i);
      ids_stage(c, Sh, raw, i, codes, nbcap, lane);
    }
    if (n > 3) raw = ids_read(d, 3);
    cp_async_wait_all();
  }
  __syncthreads();

  if (warp < NU) {
    // ================ update warps
    const IdsScratch sc = ids_scratch(b.scratch + (size_t)sid * ids_scratch_bytes(L.nbmax), L.nbmax);
    unsigned cnt = 0;
    if (n > 0 && Sh.q[0].nb <= (int)L.g.K)
      ids_probe<NU>(stamps, nre, codes, Sh.q[0].nz, W, wm, cnt);
    for (int64_t i = 0; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      join_cta<NT>();
      if (Sh.stat[p] != RS_OK) break;
      const IdsReq& q = Sh.q[e];
      const int js = ids_choice(d, q, Sh.pub[p], wm + p * W, act + p * W, W, i, lane).js;
      if (q.dup) {
        // two blocks of the prompt with one chained hash (a 64-bit collision)
        if (threadIdx.x == 0) Sh.stat[p ^ 1] = RS_ERR_COLLISION;
      } else {
        IdsTable t;
        t.st = stamps + js * nre;
        t.log = b.log + ((size_t)sid * W + js) * L.g.R;
        t.rmask = L.ids_rmask;
        ids_update<NTU>(c, Sh, t, c.wmeta + js, codes + (size_t)e * nbcap, q, sc,
                        win + (size_t)js * NTU, whead + js, wlen + js, i);
        if (threadIdx.x == 0 && Sh.err) Sh.stat[p ^ 1] = Sh.err;
      }
      grp_bar<NTU>();   // the update's stamps, before the next probe
      if (i + 1 < n) {
        const int e1 = (int)((i + 1) & (IDS_RING - 1));
        const IdsReq& q1 = Sh.q[e1];
        if (q1.nb <= (int)L.g.K)
          ids_probe<NU>(stamps, nre, codes + (size_t)e1 * nbcap, q1.nz, W, wm + (p ^ 1) * W, cnt);
      }
    }
    cp_async_wait_all();
    cnt = __reduce_add_sync(FULL_MASK, cnt);
    if (lane == 0) atomicAdd(&S.probes, (unsigned long long)cnt);
  } else if (warp == NU) {
    // ================ control warp
    if (n > 0) ids_arrive(c, Sh, 0, act, nfz, lane);
    for (int64_t i = 0; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      join_cta<NT>();
      if (Sh.stat[p] != RS_OK) break;
      const IdsReq& q = Sh.q[e];
      // w_c o_ij of every worker: m / nbt correctly rounded from the rounded
      // reciprocal (one exact remainder and one correction: Markstein 1990)
      double wco[2];
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int j = lane + 32 * h;
        wco[h] = 0.0;
        if (j < W) {
          const double m = (double)wm[p * W + j], nd = (double)q.nbt;
          const double q0 = __dmul_rn(m, q.inv);
          const double r = __fma_rn(-q0, nd, m);
          wco[h] = __dmul_rn(mc.w_c, __fma_rn(r, q.inv, q0));
        }
      }
      const int js = ids_choice(d, q, Sh.pub[p], wm + p * W, act + p * W, W, i, lane).js;
      const double w0 = __shfl_sync(FULL_MASK, wco[0], js & 31);
      const double w1 = __shfl_sync(FULL_MASK, wco[1], js & 31);
      if (lane == 0) {
        S.jstar = js;
        book_request<false>(c, q, i, js < 32 ? w0 : w1);
      }
      __syncwarp();
      if (i + 1 < n) ids_arrive(c, Sh, i + 1, act, nfz, lane);
    }
    // drain: remaining completions start the queued requests
    if (lane == 0 && S.status == RS_OK && Sh.stat[0] == RS_OK && Sh.stat[1] == RS_OK)
      while (S.nheap > 0) {
        uint64_t k;
        int f;
        heap_pop(c, &k, &f);
        complete(c, f, tval(k));
      }
  } else {
    // ================ staging warp
    int64_t hit = 0, pbl = 0, hashed = 0, sampled = 0;
    const bool eq2 = d.policy == RS_POLICY_DYNAMO || d.policy == RS_POLICY_LOADBAL;
    for (int64_t i = 0; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      join_cta<NT>();
      if (Sh.stat[p] != RS_OK) break;
      // request i+3 first: its copies run beside the records
      if (i + 3 < n) {
        ids_stage(c, Sh, raw, i + 3, codes, nbcap, lane);
        if (i + 4 < n) raw = ids_read(d, i + 4);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const IdsReq& q = Sh.q[e];
      const IdsChoice ch = ids_choice(d, q, Sh.pub[p], wm + p * W, act + p * W, W, i, lane);
      const int64_t row = d.rec_base + i;
      int pb = 0;
      float c2 = __int_as_float(0x7F800000);
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int j = lane + 32 * h;
        if (j < W) {
          const int m = wm[p * W + j];
          b.rec.n_frozen[row * W + j] = (uint16_t)nfz[p * W + j];
          b.rec.prefix[row * W + j] = (uint16_t)m;
          if (mc.write_cost) b.rec.cost[row * W + j] = ch.c[h];
          pb += min(m + 1, q.nb);
          if (j != ch.bj && ch.c[h] < c2) c2 = ch.c[h];
        }
      }
      c2 = __uint_as_float(__reduce_min_sync(FULL_MASK, __float_as_uint(c2)));
      pb = (int)__reduce_add_sync(FULL_MASK, (unsigned)pb);
      if (lane == 0) {
        float* ds = b.dstat + row * 6;
        ds[0] = ch.best;
        ds[1] = c2;
        if (eq2 && Sh.pub[p].tau > 0.0f) {
          ds[2] = ch.target;
          ds[3] = ch.S;
          ds[4] = ch.lo;
          ds[5] = ch.hi;
          sampled++;
        } else {
          ds[3] = -1.0f;   // no Eq. (2) draw
        }
        b.rec.worker[row] = ch.js;
        b.rec.arrival[row] = Sh.pub[p].a;
        b.rec.nbt[row] = q.nbt;
        hit += wm[p * W + ch.js];
        pbl += pb;
        hashed += q.nb;
      }
      asm volatile("cp.async.wait_group 1;" ::: "memory");   // request i+2's ids have landed
    }
    cp_async_wait_all();
    if (lane == 0) {
      S.hit_blocks = hit;
      S.probe_blocks = pbl;
      S.hashed_blocks = hashed;
      S.sampled = sampled;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && S.status == RS_OK)
    S.status = Sh.stat[0] != RS_OK ? Sh.stat[0] : Sh.stat[1];
  __syncthreads();
  {
    double st = 0.0, se = 0.0, mk = 0.0;
    if (S.status == RS_OK)
      for (int64_t q = threadIdx.x; q < S.n_routed; q += NT) {
        const int64_t row = d.rec_base + q;
        const double ct = b.rec.completion[row];
        st = __dadd_rn(st, b.rec.ttft[row]);
        se = __dadd_rn(se, __dsub_rn(ct, b.rec.arrival[row]));
        mk = fmax(mk, ct);
      }
    for (int o = 16; o > 0; o >>= 1) {
      st = __dadd_rn(st, __shfl_xor_sync(FULL_MASK, st, o));
      se = __dadd_rn(se, __shfl_xor_sync(FULL_MASK, se, o));
      mk = fmax(mk, __shfl_xor_sync(FULL_MASK, mk, o));
    }
    __shared__ double red3[3][NT / 32];
    if (lane == 0) {
      red3[0][warp] = st;
      red3[1][warp] = se;
      red3[2][warp] = mk;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a0 = 0.0, a1 = 0.0, a2 = 0.0;
      for (int w = 0; w < NT / 32; w++) {
        a0 = __dadd_rn(a0, red3[0][w]);
        a1 = __dadd_rn(a1, red3[1][w]);
        a2 = fmax(a2, red3[2][w]);
      }
      S.sum_ttft = a0;
      S.sum_e2e = a1;
      S.makespan = a2;
      write_result(c);
    }
  }
  for (int j = threadIdx.x; j < W; j += NT) b.meta_out[(size_t)sid * W + j] = c.wmeta[j];
}

size_t sim_ids_slot_bytes(int cmax) { return make_ids_layout(1, 1, cmax, 1, 32, true).slot_bytes; }

// Update warps of a launch: six per replica while every SM holds at most two
// replicas, else two, so that more replicas are resident per SM.
int sim_ids_update_warps(int nsim, int sms) { return nsim <= 2 * sms ? 6 : 2; }

cudaError_t launch_sim_ids(const SimDesc* d_desc, const SimBuffers& b, const SimLaunch& L,
                           cudaStream_t st) {
  if (L.nsim <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int nu = sim_ids_update_warps(L.nsim, sms);
  const bool sg = L.slots_global != 0;
  const size_t smem = sim_ids_smem_bytes(L.mc.W, L.nbmax, L.cmax, L.mc.cap, 32 * nu, sg);
  void (*kern)(const SimDesc*, const SimBuffers, const SimLaunch);
  if (nu == 6)
    kern = sg ? k_sim_ids<6, 2, true> : k_sim_ids<6, 2, false>;
  else
    kern = sg ? k_sim_ids<2, 5, true> : k_sim_ids<2, 5, false>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<L.nsim, (nu + 2) * 32, smem, st>>>(d_desc, b, L);
  return cudaGetLastError();
}

}  // namespace rs
