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
//   staging  the choice (handed to the others at a second, named barrier), then
//            request i+3's scalars and block ids, request i's records;
//   control  meanwhile the times that a service start would have on each
//            worker; then request i's load and service start, and completions
//            and controller samples up to request i+1's arrival, whose loads
//            it publishes for the next choice;
//   update   request i's cache update on the chosen worker, then request i+1's
//            cached prefix on every worker (and, with a warp per worker, what
//            request i+1's update would do to each).
// What the groups hand one another at the join is double-buffered by the
// request's parity.  Between 5 and 7 cycles pass per instruction of a warp
// that has its SM sub-partition to itself, and with four replicas per SM
// they are 13, 1.7 of them waits for instruction fetch: the loop's code and its
// instruction count are what to keep small.
//
// Calls before (hash tables) and now: 64 replicas x 10 000 requests at W = 3
// 53.5 and 19.8 ms, 648 x 10 000 at W = 6 246 and 50.7 ms, 256 x 6 000 at
// W = 6 with controller and sampling 62.5 and 18.4 ms, 16 x 5 000 at W = 64
// 206 and 32.8 ms, 512 requests at W = 3 2.33 and 0.97 ms; under frequency
// eviction 64 x 10 000 at W = 3 59.8 and 22.8 ms.
#include <algorithm>
#include <type_traits>

#include "sim_common.cuh"

namespace rs {

constexpr uint32_t CODE_FRESH = 0x80000000u;    // first occurrence in the trace
constexpr uint32_t CODE_SINGLE = 0x7FFFFFFFu;   // (low bits) occurs once
constexpr uint32_t SINGLE_FLAG = 0x80000000u;   // log entry: a single block's position
constexpr uint32_t LOG_DEAD = 0x7FFFFFFFu;      // log entry: evicted before the head passed it

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

// A numbered block's hash: that of its first occurrence.
__global__ void __launch_bounds__(256) k_ids_hashes(const uint32_t* __restrict__ ids,
                                                    const uint64_t* __restrict__ hashes, int64_t blocks,
                                                    uint64_t* __restrict__ of, int64_t nre) {
  for (int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x; q < blocks; q += (int64_t)gridDim.x * 256) {
    const uint32_t x = ids[q], b = x & CODE_SINGLE;
    if ((x & CODE_FRESH) && (int64_t)b < nre) of[b] = hashes[q];   // (CODE_SINGLE: past every number)
  }
}

__global__ void __launch_bounds__(256) k_ids_entries(const uint64_t* __restrict__ hashes,
                                                     const uint64_t* __restrict__ of, int64_t nre,
                                                     const uint32_t* __restrict__ stamps,
                                                     const uint32_t* __restrict__ log, uint32_t rmask,
                                                     uint32_t head, uint32_t n, uint64_t* __restrict__ out) {
  for (uint32_t q = blockIdx.x * 256 + threadIdx.x; q < n; q += gridDim.x * 256) {
    const uint32_t t = head + q, x = log[t & rmask];
    uint64_t h = 0;
    if (x & SINGLE_FLAG)
      h = hashes[x & ~SINGLE_FLAG];
    else if ((int64_t)x < nre && stamps[x] == t)   // (else dead)
      h = of[x];
    out[q] = h;
  }
}

// A dump of one worker's cache: a pass over the trace's ids and one over the log
// (on the host, with the arrays copied there first, 51 million blocks took 60 ms).
cudaError_t launch_ids_dump(const uint32_t* ids, const uint64_t* hashes, int64_t blocks, uint64_t* of,
                            int64_t nre, const uint32_t* stamps, const uint32_t* log, uint32_t rmask,
                            uint32_t head, uint32_t T, uint64_t* out, cudaStream_t st) {
  if (blocks > 0)
    k_ids_hashes<<<(unsigned)std::min<int64_t>((blocks + 255) / 256, 152 * 16), 256, 0, st>>>(ids, hashes, blocks,
                                                                                            of, nre);
  const uint32_t n = T - head;
  if (n > 0)
    k_ids_entries<<<std::min<uint32_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(hashes, of, nre, stamps, log,
                                                                                 rmask, head, n, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------ the replica's state

constexpr int IDS_RING = 4;   // requests staged at once (i .. i+3)

// A staged request: what the loop needs beside its block ids.
struct IdsReq : ReqState {
  int64_t pos0;        // position of its first block in the trace
  double inv;          // 1 / nbt, rounded (0 for an empty prompt; without the w_c o table)
  uint32_t dx, dy;     // words 0 and 1 of its Philox block
  int32_t nz, pad;
};

// What the control warp publishes of a request's arrival.
struct IdsArrival {
  double a;
  float tau, omega;
  uint32_t D;          // decay step (frequency eviction)
};

// What a worker's cache update will do, worked out before the choice
// (launches with an update warp per worker).
constexpr int IDS_WRING = 512;        // log entries kept ahead of the head (power of two)
constexpr uint32_t IDS_GENERAL = 0xFFFFFFFFu;
constexpr int IDS_WIN = 192;          // log entries an update examines that was not planned
struct IdsPlan {
  uint32_t nabs, E, step, pad;        // absent blocks, victims, log entries passed (or IDS_GENERAL)
  uint32_t vic[IDS_WRING / 32];       // victims among the entries from the head on, as bits
};

struct IdsShared {
  IdsReq q[IDS_RING];
  alignas(16) IdsPlan plan[8];

  IdsArrival pub[2];
  int2 stat[2];                // by parity: errors seen before that join, of the events (x) and of
                               // the update (y: of the request before, so it comes first)
  alignas(16) uint2 red[8];    // per update warp: absent blocks, least stamp
  unsigned livew[IDS_WIN / 32];   // live entries of the window (frequency eviction: cold ones)
  uint2 hot[8];                // per update warp: least e and position of the hot entries passed
  FreqShared fs;
  FreqMeta fnew;
  int warp_tot[8];
  int err;                     // of the update
  int nvic, nins, changed;
  uint32_t nh;
  int js;                      // the chosen worker
  uint32_t* lru_bits;          // of lru_exact
};

struct IdsLayout {
  size_t ftab, f_oitl, f_a, f_o, h_k, srec, gk, gf, wA, codes, meta, f_req, f_worker, f_blk, f_next, h_f,
      freestk, winserv, wqh, wqt, wm, act, nfz, whead, wlen, win, wfreq, lru;
  size_t total, slot_bytes;
};

__host__ __device__ inline IdsLayout make_ids_layout(int W, int nbmax, int cmax, int nft, int ntu,
                                                     bool slots_global, bool freq = false) {
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
  // by request slot: of IdsEvents in shared memory, or the heap's in global
  const size_t G = (C + 31) / 32;
  L.f_oitl = slots(8 * C);
  L.f_a = slots(8 * C);
  L.f_o = slots(8 * C);
  L.h_k = slots(8 * 32 * G);
  L.srec = L.gk = L.gf = 0;
  if (!slots_global) {
    L.srec = take(16 * 32 * G);   // (whole groups: read past the slots for no completion)
    if (G > 32) {
      L.gk = take(8 * G);
      L.gf = take(4 * G);
    }
  }
  L.wA = take(8 * (size_t)W);
  L.codes = take(4 * nb * IDS_RING);
  L.meta = take(sizeof(CacheMeta) * (size_t)W);
  L.f_req = L.f_worker = L.f_blk = L.f_next = L.h_f = 0;
  if (slots_global) {
    L.f_req = slots(4 * C);
    L.f_worker = slots(4 * C);
    L.f_blk = slots(4 * C);
    L.f_next = slots(4 * C);
    L.h_f = slots(4 * C);
  }
  L.freestk = slots(4 * C);
  L.winserv = take(4 * (size_t)W);
  L.wqh = take(4 * (size_t)W);
  L.wqt = take(4 * (size_t)W);
  L.wm = take(4 * 2 * (size_t)W);
  L.act = take(4 * 2 * (size_t)W);
  L.nfz = take(4 * 2 * (size_t)W);
  L.whead = take(4 * (size_t)W);
  L.wlen = take(4 * (size_t)W);
  const int nu = ntu / 32;
  L.win = take(4 * (size_t)W * (!freq && W <= nu ? IDS_WRING : IDS_WIN));
  L.wfreq = take(freq ? sizeof(FreqMeta) * (size_t)W : 0);
  L.lru = take(8 * ((2 * nb + 31) / 32));
  L.total = o;
  L.slot_bytes = (og + 255) & ~(size_t)255;
  return L;
}

size_t sim_ids_smem_bytes(int W, int nbmax, int cmax, int cap, int ntu, bool slots_global, bool freq) {
  return make_ids_layout(W, nbmax, cmax, ftab_size(cap), ntu, slots_global, freq).total;
}

// Global scratch of one replica for the updates that need the exact sequence.
struct IdsScratch {
  uint32_t *vent, *vt;   // [2 nb] live entries and their positions
  int32_t *owner, *w;    // [2 nb] the prompt's block holding an entry or -1, [nb] see lru_exact
  // frequency eviction: [2 nb] hot entries (position << 32 | id), [2 nb] victims,
  // [nb] stamps and e, [2 nb] touched entries, [nb] kinds, [nb] evicted early
  uint64_t* hot;
  int32_t* victim;
  uint32_t *pst, *e;
  uint8_t *touched, *kind, *evk;
};

__host__ __device__ inline size_t ids_scratch_bytes(int nbmax) {
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1);
  return (64 * nb + 255) & ~(size_t)255;
}

size_t sim_ids_scratch_bytes(int nbmax) { return ids_scratch_bytes(nbmax); }

__device__ __forceinline__ IdsScratch ids_scratch(unsigned char* p, int nbmax) {
  const size_t nb = (size_t)(nbmax > 0 ? nbmax : 1);
  IdsScratch s;
  s.hot = reinterpret_cast<uint64_t*>(p);
  s.vent = reinterpret_cast<uint32_t*>(s.hot + 2 * nb);
  s.vt = s.vent + 2 * nb;
  s.owner = reinterpret_cast<int32_t*>(s.vt + 2 * nb);
  s.w = s.owner + 2 * nb;
  s.victim = s.w + nb;
  s.pst = reinterpret_cast<uint32_t*>(s.victim + 2 * nb);
  s.e = s.pst + nb;
  s.touched = reinterpret_cast<uint8_t*>(s.e + nb);
  s.kind = s.touched + 2 * nb;
  s.evk = s.kind + nb;
  return s;
}

// One worker's cache.
struct IdsTable {
  uint32_t* st;    // [nre] stamps
  uint32_t* fe;    // [nre] frequency eviction: e, the decay step from which a block is cold
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

// Whether an error before the join of parity p stops the replica.
__device__ __forceinline__ bool ids_stopped(const IdsShared& Sh, int p) {
  const int2 s = Sh.stat[p];
  return (s.x | s.y) != RS_OK;
}

// The choice of request i: made by the staging warp (Sh.js written), waited
// for by the others.  (Every warp computing it alike took a third of all
// instructions and three copies of its code.)
template <int NT>
__device__ __forceinline__ void choice_made() {
  __syncwarp();
  asm volatile("barrier.arrive 2, %0;" ::"n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ void choice_wait() {
  asm volatile("barrier.sync 2, %0;" ::"n"(NT) : "memory");
}

// ------------------------------------------------------------ probe

// Leading blocks of the prompt found in one worker's cache from block k0 on,
// at most nz (a warp; four stamps per lane in flight).
__device__ __forceinline__ int ids_prefix(const uint32_t* st, const uint32_t* cd, int k0, int nz,
                                          unsigned& cnt) {
  const int lane = (int)(threadIdx.x & 31);
#pragma unroll 1
  for (int k = k0; k < nz; k += 128) {
    uint32_t v[4];
    bool in[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int kk = k + 32 * r + lane;
      in[r] = kk < nz;
      const uint32_t c = in[r] ? cd[kk] : CODE_FRESH;
      v[r] = STAMP_NONE;
      if (!(c >> 31)) {   // (without the branch, as in ids_prefixes: 760 -> 980 cycles at W = 3)
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

// The same for the workers j[q] of the set bits of `open`, Q at a time, 64
// blocks of each in flight, until each has its first miss.  Straight-line loads:
// with a branch around each, and the window's in ids_update, a call on the grid
// (648 replicas x 10 000 requests, W = 6, three workers a warp) took 61.4 ms,
// 54.3 so, and 52.1 with Q = 3 there instead of 4.
template <int Q>
__device__ __forceinline__ void ids_prefixes(const uint32_t* stamps, size_t nre, const int (&j)[Q],
                                            unsigned open, const uint32_t* cd, int k0, int nz,
                                            int (&m)[Q], unsigned& cnt) {
  const int lane = (int)(threadIdx.x & 31);
  const uint32_t* st[Q];
#pragma unroll
  for (int q = 0; q < Q; q++) {
    m[q] = nz;
    st[q] = stamps + (size_t)((open >> q) & 1u ? j[q] : j[0]) * nre;   // (bit 0 of open is set)
  }
#pragma unroll 1
  for (int k = k0; k < nz && open; k += 64) {
    const int ka = k + lane, kb = ka + 32;
    const uint32_t ca = cd[min(ka, nz - 1)], cb = cd[min(kb, nz - 1)];
    const bool ia = ka < nz, ib = kb < nz, oa = ia && !(ca >> 31), ob = ib && !(cb >> 31);
    const uint32_t xa = ca >> 31 ? 0u : ca, xb = cb >> 31 ? 0u : cb;
    uint32_t va[Q], vb[Q];
#pragma unroll
    for (int q = 0; q < Q; q++) {   // (no branch per load: what is not looked up reads a stamp not used)
      va[q] = st[q][xa];
      vb[q] = st[q][xb];
    }
    cnt += (unsigned)__popc(open) * ((unsigned)oa + (unsigned)ob);
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const unsigned ma = __ballot_sync(FULL_MASK, ia && !(oa && va[q] != STAMP_NONE));
      const unsigned mb = __ballot_sync(FULL_MASK, ib && !(ob && vb[q] != STAMP_NONE));
      if (((open >> q) & 1u) && (ma | mb)) {
        m[q] = ma ? k + __ffs(ma) - 1 : k + 32 + __ffs(mb) - 1;
        open &= ~(1u << q);
      }
    }
  }
}

// m_j of every worker (the NU update warps); wm[j] = m_j.  Up to NU workers: a
// warp each.  Up to 4 NU: a warp walks its workers together.  More: a warp
// looks up the first 32 blocks of B workers at once (most workers miss among
// them: one round of loads for all), then walks those where all are present,
// four together.  At W = 64 walks from block 0 on take 7 300 SM cycles a
// request; at W = 6 and NU = 2 the round of first blocks takes 5 200 against
// 3 200 for the walk.
template <int NU>
__device__ __forceinline__ void ids_probe(const uint32_t* stamps, size_t nre, const uint32_t* cd,
                                          int nz, int W, int* wm, unsigned& cnt) {
  constexpr int B = NU >= 6 ? 11 : 8;
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  if (W <= NU) {
    if (warp < W) {
      const int m = ids_prefix(stamps + warp * nre, cd, 0, nz, cnt);
      if (lane == 0) wm[warp] = m;
    }
    return;
  }
  auto together = [&](auto n) {   // n workers per warp
    constexpr int Q = decltype(n)::value;
    int j[Q], m[Q];
    unsigned open = 0;
#pragma unroll
    for (int q = 0; q < Q; q++) {
      j[q] = warp + q * NU;
      open |= (unsigned)(j[q] < W) << q;
    }
    ids_prefixes<Q>(stamps, nre, j, open, cd, 0, nz, m, cnt);
#pragma unroll
    for (int q = 0; q < Q; q++)
      if (lane == q && j[q] < W) wm[j[q]] = m[q];
  };
  if (W <= 3 * NU) return together(std::integral_constant<int, 3>());
  if (W <= 4 * NU) return together(std::integral_constant<int, 4>());
  int j[4], m[4];
  const uint32_t c = lane < nz ? cd[lane] : CODE_FRESH;
  const bool old = !(c >> 31);
  const uint32_t x = old ? c : 0u;
#pragma unroll 1
  for (int j0 = warp; j0 < W; j0 += B * NU) {
    uint32_t v[B];
#pragma unroll
    for (int q = 0; q < B; q++)
      v[q] = j0 + q * NU < W ? stamps[(size_t)(j0 + q * NU) * nre + x] : STAMP_NONE;
    int mine = nz;       // lane q: m of worker j0 + q NU
    unsigned open = 0;   // (uniform) bit q: its first 32 blocks are all present
#pragma unroll
    for (int q = 0; q < B; q++) {
      const unsigned ms = __ballot_sync(FULL_MASK, lane < nz && (!old || v[q] == STAMP_NONE));
      if (lane == q && ms) mine = __ffs(ms) - 1;
      if (!ms && j0 + q * NU < W) open |= 1u << q;
    }
    if (old) cnt += (unsigned)min(B, (W - j0 + NU - 1) / NU);
    if (nz <= 32) open = 0;
#pragma unroll 1
    while (open) {
      int w[4];
      unsigned some = 0;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        w[q] = open ? __ffs(open) - 1 : 0;
        some |= (unsigned)(open != 0) << q;
        open &= open - 1u;
        j[q] = j0 + w[q] * NU;
      }
      ids_prefixes<4>(stamps, nre, j, some, cd, 32, nz, m, cnt);
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (((some >> q) & 1u) && lane == w[q]) mine = m[q];
    }
    if (lane < B && j0 + lane * NU < W) wm[j0 + lane * NU] = mine;
  }
}

// ------------------------------------------------------------ choice

// Eq. (1) costs of workers lane and lane + 32 and the chosen worker (a warp).
// Costs are >= +0, so their bit patterns order them.
struct IdsChoice {
  float c[2], best;
  int bj, js;
  float target, S, lo, hi;   // where an Eq. (2) draw fell
};

template <bool WIDE>
__device__ __forceinline__ IdsChoice ids_choice(int policy, const IdsReq& q,
                                                const IdsArrival& ar, const int* wm,
                                                const float* act, int W, int64_t i, int lane) {
  IdsChoice r;
  const float om = ar.omega, tau = ar.tau;
  const float inf = __int_as_float(0x7F800000);
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int j = lane + 32 * h;
    r.c[h] = inf;
    if ((h == 0 || WIDE) && j < W) r.c[h] = __fadd_rn(__fmul_rn(om, __int2float_rn(q.nbt - wm[j])), act[j]);
  }
  const unsigned mn = __reduce_min_sync(FULL_MASK, min(__float_as_uint(r.c[0]), __float_as_uint(r.c[1])));
  // the lowest index among the minima: workers 0-31 first
  const unsigned e0 =
      __ballot_sync(FULL_MASK, lane < W && __float_as_uint(r.c[0]) == mn);
  const unsigned e1 =
      WIDE ? __ballot_sync(FULL_MASK, lane + 32 < W && __float_as_uint(r.c[1]) == mn) : 0u;
  r.bj = e0 ? __ffs(e0) - 1 : 32 + __ffs(e1) - 1;
  r.best = __uint_as_float(mn);
  r.js = r.bj;
  if (policy != RS_POLICY_DYNAMO && policy != RS_POLICY_LOADBAL) {
    // the static policies (as static_policy_worker)
    if (policy == RS_POLICY_ROUNDROBIN) {
      r.js = (int)((uint64_t)i % (uint64_t)W);
    } else {
      const int j1 = (int)(((uint64_t)(q.dx >> 8) * (uint64_t)W) >> 24);
      r.js = j1;
      if (policy == RS_POLICY_P2C && W >= 2) {
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
    // Eq. (2), as select_worker_warp: one weight per lane, summed in worker
    // order; each lane keeps the sum at its worker, so one pass gives S, the
    // worker where the draw falls and the sums around it
    float e[2], at[2] = {0.0f, 0.0f};
#pragma unroll
    for (int h = 0; h < 2; h++)
      e[h] = (h == 0 || WIDE) && lane + 32 * h < W ? exp_sm(-__fdiv_rn(__fsub_rn(r.c[h], r.best), tau)) : 0.0f;
    float cum = 0.0f;
#pragma unroll 4
    for (int j = 0; j < W; j++) {
      cum = __fadd_rn(cum, __shfl_sync(FULL_MASK, !WIDE || j < 32 ? e[0] : e[1], j & 31));
      if (lane == (j & 31)) at[!WIDE || j < 32 ? 0 : 1] = cum;
    }
    r.S = cum;
    r.target = __fmul_rn(__fmul_rn((float)(q.dx >> 8), 0x1p-24f), cum);
    unsigned long long past = __ballot_sync(FULL_MASK, lane < W && r.target < at[0]);
    unsigned long long some = __ballot_sync(FULL_MASK, e[0] > 0.0f);
    if (WIDE) {
      past |= (unsigned long long)__ballot_sync(FULL_MASK, lane + 32 < W && r.target < at[1]) << 32;
      some |= (unsigned long long)__ballot_sync(FULL_MASK, e[1] > 0.0f) << 32;
    }
    const int pick = past ? __ffsll((long long)past) - 1 : -1;
    const int last = some ? 63 - __clzll((long long)some) : r.bj;
    // the sums do not decrease: those at or below the target come before pick
    auto sum_at = [&](int j) {
      float x = __shfl_sync(FULL_MASK, at[0], j & 31);
      if (WIDE) {
        const float y = __shfl_sync(FULL_MASK, at[1], j & 31);
        if (j >= 32) x = y;
      }
      return x;
    };
    const float qnan = __int_as_float(0x7FC00000);
    const int below = (pick >= 0 ? pick : W) - 1;
    const float lo = sum_at(below >= 0 ? below : 0), hi = sum_at(pick >= 0 ? pick : 0);
    r.lo = below >= 0 ? lo : qnan;
    r.hi = pick >= 0 ? hi : qnan;
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
  return (x & SINGLE_FLAG) || (x != LOG_DEAD && t.st[x] == p);
}

// Moves the live entries of the log down to the head, in order, and renumbers
// stamps by a multiple of the ring's length (so ring places stay), in place:
// an entry never moves up.
template <int NT>
__device__ __noinline__ void ids_compact(IdsTable t, CacheMeta* meta, int* warp_tot, int* err) {
  const uint32_t head = meta->head, T = meta->T, size = meta->size;
  const uint32_t d = head & ~t.rmask;
  constexpr int PER = 4;
  uint32_t base = 0;
#pragma unroll 1
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
#pragma unroll 1
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
// holds, or a present block among the least recent entries (lru_exact over the
// first 2 nb live entries).  Evicts;
// returns the head past the last victim; victims in S.nvic, insertions in
// S.nins.  (Rare, and out of line: the loop's hot code has to stay small, its
// warps wait for instructions otherwise.)
template <int NT>
__device__ __noinline__ uint32_t ids_evict_general(IdsTable t, CacheMeta m, uint32_t K,
                                                   const uint32_t* cd, int nb, uint32_t E0,
                                                   uint32_t pmin, int nabs, unsigned char* scratch,
                                                   int nbmax, IdsShared& S, int64_t* slow) {
  const IdsScratch sc = ids_scratch(scratch, nbmax);
  if (threadIdx.x == 0) {
    S.nvic = 0;
    S.nins = nabs;
  }
  uint32_t G = ids_gather<NT>(t, m.head, m.T, E0, sc, S.warp_tot);
  if (G < E0) {   // fewer live entries than the size says
    if (threadIdx.x == 0) S.err = RS_ERR_TIMEOUT;
    return m.head;
  }
  if (pmin > sc.vt[E0 - 1]) {   // (also pmin = STAMP_NONE: no block present)
    for (uint32_t v = threadIdx.x; v < E0; v += NT)
      if (!(sc.vent[v] & SINGLE_FLAG)) t.st[sc.vent[v]] = STAMP_NONE;
    if (threadIdx.x == 0) S.nvic = (int)E0;
    grp_bar<NT>();
    return sc.vt[E0 - 1] + 1;
  }
  grp_bar<NT>();
  G = ids_gather<NT>(t, m.head, m.T, min(m.size, 2u * (uint32_t)nb), sc, S.warp_tot);
  for (uint32_t p = threadIdx.x; p < G; p += NT) sc.owner[p] = -1;
  grp_bar<NT>();
  const uint32_t last = G ? sc.vt[G - 1] : 0u;
  const int freeb = (int)(K - m.size);
  for (int k = threadIdx.x; k < nb; k += NT) {
    const uint32_t c = cd[k];
    const uint32_t st = c >> 31 ? STAMP_NONE : t.st[c];
    int v = st == STAMP_NONE ? LRU_ABSENT : LRU_FAR;
    if (v == LRU_FAR && G && st <= last) {
      v = (int)ids_place(sc.vt, G, st);
      sc.owner[v] = k;
    }
    sc.w[k] = v;
  }
  if (threadIdx.x == 0) S.nins = 0;
  lru_exact<NT>(sc.w, nb, freeb, (int)G, S.lru_bits);
  int ni = 0;
  for (int k = threadIdx.x; k < nb; k += NT) ni += sc.w[k] == LRU_ABSENT || sc.w[k] >= LRU_EVICTED;
  ni = (int)__reduce_add_sync(FULL_MASK, (unsigned)ni);
  if ((threadIdx.x & 31) == 0 && ni) atomicAdd(&S.nins, ni);
  grp_bar<NT>();
  const int E = max(0, S.nins - freeb);
  if (threadIdx.x == 0) {
    S.nvic = E;
    S.nh = m.head;
    ++*slow;
  }
  grp_bar<NT>();
  // the victims: the first entries that are not touched before their turn
  int have = 0;
  for (uint32_t p0 = 0; p0 < G && have < E; p0 += NT) {
    const uint32_t p = p0 + threadIdx.x;
    bool v = p < G;
    if (v) {
      const int k = sc.owner[p];
      v = k < 0 || sc.w[k] >= LRU_EVICTED;
    }
    int tot;
    const int r = have + cta_rank<NT>(v, S.warp_tot, &tot);
    if (v && r < E) {
      const uint32_t x = sc.vent[p];
      if (!(x & SINGLE_FLAG)) t.st[x] = STAMP_NONE;
      if (r == E - 1) S.nh = sc.vt[p] + 1;
    }
    have += tot;
  }
  if (have < E && threadIdx.x == 0) S.err = RS_ERR_TIMEOUT;
  grp_bar<NT>();   // (a victim may be a block of this request: its new stamp comes after)
  return S.nh;
}

// m_j of one worker and its update's plan, by its warp.  The worker's log
// entries from the head on come from a ring of IDS_WRING entries in shared
// memory, copied in the background two or more updates ahead; [head, safe) are
// known to have landed.  Loads: a stamp per block and per window entry, all in
// flight together.  Planning every worker before the choice takes the update's
// loads, its reductions and its barrier off the path between the choice and
// the next probe: 1 960 + 760 SM cycles a request for update and probe with
// the update's reads after the choice (64 replicas, W = 3).
__device__ __forceinline__ int ids_plan(const IdsTable& t, const CacheMeta& m, uint32_t K,
                                        const uint32_t* cd, int nb, int nz, uint32_t* ring,
                                        uint32_t safe, IdsPlan& P, unsigned& cnt) {
  const int lane = (int)(threadIdx.x & 31);
  const bool full = m.size + (uint32_t)nb > K;   // a victim may be needed
  // four words of the window (128 log entries): entries, then their stamps.
  // Loads take no branch: a place past the log or a single block reads a
  // stamp that is not used.
  auto entries = [&](int w0, uint32_t (&x)[4], uint32_t (&v)[4]) {
    const uint32_t p0 = m.head + 32 * w0 + lane;
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = ring[(p0 + 32 * r) & (IDS_WRING - 1)];
    if (p0 + 96 >= safe) {
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const uint32_t p = p0 + 32 * r;
        if (p >= safe) {
          x[r] = p < m.T ? t.log[p & t.rmask] : SINGLE_FLAG;
          ring[p & (IDS_WRING - 1)] = x[r];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; r++) v[r] = t.st[(x[r] & SINGLE_FLAG) ? 0u : x[r]];
  };
  uint32_t x[4], v[4];
  if (full) entries(0, x, v);
  int mj = nz, nabs = nb - nz;   // past nz every block is fresh
  uint32_t pmin = STAMP_NONE;
#pragma unroll 1
  for (int k = 0; k < nz; k += 128) {
    uint32_t u[4], cc[4];
#pragma unroll
    for (int r = 0; r < 4; r++) cc[r] = cd[min(k + 32 * r + lane, nz - 1)];
#pragma unroll
    for (int r = 0; r < 4; r++) u[r] = t.st[cc[r] >> 31 ? 0u : cc[r]];
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const bool in = k + 32 * r + lane < nz, old = in && !(cc[r] >> 31);
      cnt += old;
      if (!old) u[r] = STAMP_NONE;
      const unsigned ab = __ballot_sync(FULL_MASK, in && u[r] == STAMP_NONE);
      nabs += __popc(ab);
      if (ab && mj == nz) mj = k + 32 * r + __ffs(ab) - 1;
      pmin = min(pmin, u[r]);
    }
  }
  const uint32_t freeb = K - m.size;
  const uint32_t E = (uint32_t)nabs > freeb ? (uint32_t)nabs - freeb : 0u;
  uint32_t step = 0, bits = 0;   // lane w: victims among entries 32 w .. 32 w + 31
  if (E > 0) {
    // the first E live entries, all before the oldest present block
    const uint32_t end = min(__reduce_min_sync(FULL_MASK, pmin), m.T);
    uint32_t have = 0;
#pragma unroll 1
    for (int w0 = 0;;) {
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const uint32_t p = m.head + 32 * (w0 + r) + lane;
        unsigned b = __ballot_sync(FULL_MASK, p < end && ((x[r] & SINGLE_FLAG) || v[r] == p));
        const uint32_t n = (uint32_t)__popc(b);
        if (have < E) {
          if (have + n >= E) {
            const int q = nth_set_bit32(b, (int)(E - have) - 1);
            b &= q == 31 ? FULL_MASK : (2u << q) - 1u;
            step = 32u * (w0 + r) + (uint32_t)q + 1u;
          }
          if (lane == w0 + r) bits = b;
          have += n;
        }
      }
      w0 += 4;
      if (have >= E || w0 == IDS_WRING / 32 || m.head + 32 * w0 >= end) break;
      entries(w0, x, v);
    }
    if (have < E) step = IDS_GENERAL;
  }
  if ((uint64_t)m.T - m.head + (uint64_t)nb > (uint64_t)t.rmask + 1 ||
      (uint64_t)m.T + nb > STAMP_LIMIT)
    step = IDS_GENERAL;   // a compaction first
  if (lane == 0) {
    P.nabs = (uint32_t)nabs;
    P.E = E;
    P.step = step;
  }
  if (lane < IDS_WRING / 32) P.vic[lane] = bits;
  return mj;
}

// The planned update of the chosen worker, by the update warps.
template <int NT>
__device__ __forceinline__ void ids_apply(const IdsTable& t, CacheMeta* meta, const IdsPlan& P, const uint32_t* ring,
                                          const uint32_t* cd, const IdsReq& q) {
  const CacheMeta m = *meta;
  const uint32_t step = P.step;
  const int tid = (int)threadIdx.x;
#pragma unroll 1
  for (uint32_t w = tid; w < step; w += NT)
    if ((P.vic[w >> 5] >> (w & 31)) & 1u) {
      const uint32_t x = ring[(m.head + w) & (IDS_WRING - 1)];
      if (!(x & SINGLE_FLAG)) t.st[x] = STAMP_NONE;
    }
  // every block of the prompt is now the most recent, in order
  const int nb = q.nb;
#pragma unroll 1
  for (int k = tid; k < nb; k += NT) {
    const uint32_t b = cd[k] & CODE_SINGLE, pos = m.T + (uint32_t)k;
    if (b != CODE_SINGLE) t.st[b] = pos;
    t.log[pos & t.rmask] = b != CODE_SINGLE ? b : SINGLE_FLAG | (uint32_t)(q.pos0 + k);
  }
}

// Request i's blocks touched in order on the chosen worker's cache (exact
// LRU), by the update warps.  WINDOW: the window win holds the log entries from
// whead on (copied in the background after the worker's last update), so the
// common update makes one round of stamp loads and one barrier: every thread
// reads the stamp of one block of the prompt and of one window entry; the
// live entries before the oldest present block are the candidates, and the
// first E0 = absent - free of them are the victims.  Without: the course that
// a plan leaves to the whole group.
template <int NT, bool WINDOW>
__device__ __forceinline__ void ids_update(SimScalars& A, IdsShared& S, uint32_t K, int nbmax,
                                           const IdsTable& t, CacheMeta* meta, const uint32_t* cd,
                                           const IdsReq& q, unsigned char* scratch, uint32_t* win,
                                           uint32_t* whead, uint32_t* wlen, int64_t i) {
  constexpr int R = IDS_WIN / NT, NW = IDS_WIN / 32;   // window entries per thread, words
  static_assert(R * NT == IDS_WIN, "whole window entries per thread");
  const int nb = q.nb, nz = q.nz, tid = (int)threadIdx.x, lane = tid & 31;
  if (WINDOW) cp_async_wait_all();   // this thread's window entries
  if ((uint64_t)meta->T - meta->head + (uint64_t)nb > (uint64_t)t.rmask + 1 ||
      (uint64_t)meta->T + nb > STAMP_LIMIT) {
    if (!WINDOW) cp_async_wait_all();   // this thread's copies of the log into the rings
    grp_bar<NT>();
    ids_compact<NT>(t, meta, S.warp_tot, &S.err);
    if (tid == 0) {
      A.rebuilds++;
      *wlen = 0;
    }
    grp_bar<NT>();
  }
  const CacheMeta m = *meta;
  const bool full = m.size + (uint32_t)nb > K;   // a victim may be needed
  // stamps of the prompt's blocks, of the window's entries
  int nabs = 0;
  uint32_t pmin = STAMP_NONE;
#pragma unroll 1
  for (int k = tid; k < nz; k += NT) {
    const uint32_t x = cd[k], v = t.st[x >> 31 ? 0u : x];
    const uint32_t st = x >> 31 ? STAMP_NONE : v;
    nabs += st == STAMP_NONE;
    pmin = min(pmin, st);
  }
  uint32_t x[R];
  bool live[R];
  if (full) {
    const uint32_t have_win = WINDOW && *whead == m.head ? *wlen : 0u;
    uint32_t v[R];
#pragma unroll
    for (int r = 0; r < R; r++) x[r] = WINDOW ? win[r * NT + tid] : LOG_DEAD;
    if (have_win < (uint32_t)IDS_WIN) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        const uint32_t w = (uint32_t)(r * NT + tid), p = m.head + w;
        if (w >= have_win) x[r] = p < m.T ? t.log[p & t.rmask] : LOG_DEAD;
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = t.st[x[r] >= LOG_DEAD ? 0u : x[r]];
#pragma unroll
    for (int r = 0; r < R; r++) {
      live[r] = x[r] >= SINGLE_FLAG || (x[r] != LOG_DEAD && v[r] == m.head + (uint32_t)(r * NT + tid));
      const unsigned lv = __ballot_sync(FULL_MASK, live[r]);
      if (lane == 0) S.livew[r * (NT / 32) + (tid >> 5)] = lv;
    }
  }
  {
    const int a = (int)__reduce_add_sync(FULL_MASK, (unsigned)nabs);
    const uint32_t pm = __reduce_min_sync(FULL_MASK, pmin);
    if (lane == 0) S.red[tid >> 5] = make_uint2((unsigned)a, pm);
  }
  grp_bar<NT>();
  nabs = nb - nz;   // past nz every block is fresh
  pmin = STAMP_NONE;
#pragma unroll
  for (int w = 0; w < NT / 32; w++) {
    const uint2 r = S.red[w];
    nabs += (int)r.x;
    pmin = min(pmin, r.y);
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
      const unsigned b = S.livew[w] & mk;
      const uint32_t n = (uint32_t)__popc(b);
      if (have < E0 && have + n >= E0) last = (int)l0 + nth_set_bit32(b, (int)(E0 - have) - 1);
      have += n;
    }
    if (last >= 0) {
#pragma unroll
      for (int r = 0; r < R; r++)
        if (live[r] && r * NT + tid <= last && !(x[r] & SINGLE_FLAG)) t.st[x[r]] = STAMP_NONE;
      nh = m.head + (uint32_t)last + 1u;
    } else {
      nh = ids_evict_general<NT>(t, m, K, cd, nb, E0, pmin, nabs, scratch, nbmax, S, &A.slow);
      E = (uint32_t)S.nvic;
      nins = S.nins;
    }
  }
  // every block of the prompt is now the most recent, in order
#pragma unroll 1
  for (int k = tid; k < nb; k += NT) {
    const uint32_t b = cd[k] & CODE_SINGLE, pos = m.T + (uint32_t)k;
    if (b != CODE_SINGLE) t.st[b] = pos;
    t.log[pos & t.rmask] = b != CODE_SINGLE ? b : SINGLE_FLAG | (uint32_t)(q.pos0 + k);
  }
  const uint32_t size = m.size + (uint32_t)nins - E;
  // the window of this worker's next update: entries written before this one
  // (all threads have read the old window: the barrier above)
  if (WINDOW && size + (uint32_t)nbmax > K) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t p = nh + (uint32_t)(r * NT + tid);
      if (p < m.T) cp_async4(win + r * NT + tid, t.log + (p & t.rmask));
    }
    if (tid == 0) {
      *whead = nh;
      *wlen = m.T > nh ? min((uint32_t)IDS_WIN, m.T - nh) : 0u;
    }
  }
  if (tid == 0) {
    meta->size = size;
    meta->head = nh;
    meta->T = m.T + (uint32_t)nb;
    A.inserted += nins;
    A.evicted += E;
    if (E > 0 && A.first_evict_i < 0) {
      // the first update that evicted; resident blocks = inserted - evicted
      A.first_evict_i = i;
      A.first_live = A.inserted - A.evicted;
    }
  }
}

// The same out of line, for updates that a plan leaves to the whole group.
template <int NT>
__device__ __noinline__ void ids_update_unplanned(SimScalars& A, IdsShared& S, uint32_t K, int nbmax,
                                                  IdsTable t, CacheMeta* meta, const uint32_t* cd,
                                                  const IdsReq& q, unsigned char* scratch,
                                                  uint32_t* wlen, int64_t i) {
  ids_update<NT, false>(A, S, K, nbmax, t, meta, cd, q, scratch, nullptr, nullptr, wlen, i);
}

// ------------------------------------------------------------ frequency eviction
//
// The KV Block Manager's rule as in rs_device.cuh (a block is cold iff e <= D;
// e = D on insertion, raised on a hit).  A single block is never hit, so it is
// cold for good.  Victims beyond hot entries leave the head where it is: a
// single one's log entry becomes LOG_DEAD.

// The first `want` live cold entries from `start` on into vent / vt (hot ones
// passed lower S.fs); returns how many.
template <int NT>
__device__ __forceinline__ uint32_t ids_gather_cold(const IdsTable& t, uint32_t start, uint32_t T,
                                                    uint32_t want, uint32_t D, const IdsScratch& sc,
                                                    IdsShared& S) {
  uint32_t have = 0, he = 0xFFFFFFFFu, hp = 0xFFFFFFFFu;
#pragma unroll 1
  for (uint32_t p0 = start; have < want && p0 < T; p0 += NT) {
    const uint32_t p = p0 + threadIdx.x;
    uint32_t x = 0;
    bool cold = false;
    if (p < T) {
      x = t.log[p & t.rmask];
      cold = ids_live(t, x, p);
      if (cold && !(x & SINGLE_FLAG)) {
        const uint32_t e = t.fe[x];
        if (e > D) {
          cold = false;
          he = min(he, e);
          hp = min(hp, p);
        }
      }
    }
    int tot;
    const int r = cta_rank<NT>(cold, S.warp_tot, &tot);
    if (cold && have + r < want) {
      sc.vent[have + r] = x;
      sc.vt[have + r] = p;
    }
    have = min(want, have + (uint32_t)tot);
  }
  he = __reduce_min_sync(FULL_MASK, he);
  hp = __reduce_min_sync(FULL_MASK, hp);
  if ((threadIdx.x & 31) == 0) {
    if (he != 0xFFFFFFFFu) atomicMin(&S.fs.femin, he);
    if (hp != 0xFFFFFFFFu) atomicMin(&S.fs.fhot, hp);
  }
  grp_bar<NT>();
  return have;
}

// An update that the window does not settle.  With enough cold entries before
// the oldest present cold block, those are the victims; else one thread replays
// the sequence over the first 2 nb cold entries, the first 2 nb hot ones (only
// when the cold ones run out) and the prompt's own blocks.  Evicts; kinds in
// sc.kind (0 touched, 1 inserted, 2 / 3 inserted / touched and evicted again),
// victims in S.nvic, insertions in S.nins, S.changed = 1 when replayed, S.nh =
// one past the last victim otherwise.
template <int NT>
__device__ __noinline__ void ids_freq_general(IdsTable t, CacheMeta m, uint32_t start, uint32_t K,
                                              const uint32_t* cd, int nb, uint32_t E0, uint32_t pmin,
                                              int nabs, uint32_t D, uint32_t fmax,
                                              unsigned char* scratch, int nbmax, IdsShared& S,
                                              int64_t* slow) {
  const IdsScratch sc = ids_scratch(scratch, nbmax);
  if (threadIdx.x == 0) {
    S.fs.femin = S.fs.fhot = 0xFFFFFFFFu;
    S.changed = 0;
  }
  grp_bar<NT>();
  uint32_t G = ids_gather_cold<NT>(t, start, m.T, E0, D, sc, S);
  for (int k = threadIdx.x; k < nb; k += NT) {
    const uint32_t c = cd[k];
    const uint32_t st = c >> 31 ? STAMP_NONE : t.st[c];
    sc.pst[k] = st;
    sc.e[k] = st == STAMP_NONE ? 0u : t.fe[c];
    sc.evk[k] = 0;
    sc.kind[k] = st == STAMP_NONE;
  }
  grp_bar<NT>();
  if (G >= E0 && pmin > sc.vt[E0 - 1]) {
    for (uint32_t v = threadIdx.x; v < E0; v += NT) {
      const uint32_t x = sc.vent[v];
      if (x & SINGLE_FLAG) t.log[sc.vt[v] & t.rmask] = LOG_DEAD; else t.st[x] = STAMP_NONE;
    }
    if (threadIdx.x == 0) {
      S.nvic = (int)E0;
      S.nins = nabs;
      S.nh = sc.vt[E0 - 1] + 1;
    }
    grp_bar<NT>();
    return;
  }
  grp_bar<NT>();
  const uint32_t want = min(m.size, 2u * (uint32_t)nb);
  G = ids_gather_cold<NT>(t, start, m.T, want, D, sc, S);
  // hot entries, when the cold ones run out
  uint32_t GB = 0;
  if (G < want) {
#pragma unroll 1
    for (uint32_t p0 = m.head; GB < want && p0 < m.T; p0 += NT) {
      const uint32_t p = p0 + threadIdx.x;
      uint32_t x = 0;
      bool hot = false;
      if (p < m.T) {
        x = t.log[p & t.rmask];
        hot = !(x & SINGLE_FLAG) && ids_live(t, x, p) && t.fe[x] > D;
      }
      int tot;
      const int r = cta_rank<NT>(hot, S.warp_tot, &tot);
      if (hot && GB + r < want) sc.hot[GB + r] = ((uint64_t)p << 32) | x;
      GB = min(want, GB + (uint32_t)tot);
    }
  }
  for (uint32_t q = threadIdx.x; q < G; q += NT) {
    sc.owner[q] = -1;
    sc.touched[q] = 0;
  }
  grp_bar<NT>();
  const uint32_t last = G ? sc.vt[G - 1] : 0u;
  for (int k = threadIdx.x; k < nb; k += NT) {
    const uint32_t st = sc.pst[k];
    if (st != STAMP_NONE && G && st <= last && sc.e[k] <= D) {
      const uint32_t lo = ids_place(sc.vt, G, st);
      if (lo < G && sc.vt[lo] == st) sc.owner[lo] = k;
    }
  }
  grp_bar<NT>();
  if (threadIdx.x == 0) {
    const bool hits_cold = fmax < 2u;   // a hit at cap 1 leaves the block cold
    uint32_t pa = 0, pb = 0, sz = m.size;
    int qc = 0, qh = 0, E = 0, ni = 0;
    for (int k = 0; k < nb; k++) {
      if (sc.pst[k] != STAMP_NONE && !sc.evk[k]) {
        sc.kind[k] = 0;
        const uint32_t st = sc.pst[k];
        if (sc.e[k] <= D) {   // a cold entry: in the list if old enough
          if (G && st <= last) {
            const uint32_t lo = ids_place(sc.vt, G, st);
            if (lo < G && sc.vt[lo] == st) sc.touched[lo] = 1;
          }
        } else if (GB) {      // a hot entry: in the hot list if old enough
          uint32_t lo = 0, hi = GB;
          while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if ((uint32_t)(sc.hot[mid] >> 32) < st) lo = mid + 1; else hi = mid;
          }
          if (lo < GB && (uint32_t)(sc.hot[lo] >> 32) == st) sc.hot[lo] |= 0x80000000ull;   // touched
        }
        continue;
      }
      sc.kind[k] = 1;
      ni++;
      if (sz < K) {
        sz++;
        continue;
      }
      // the victim: old cold, own cold, old hot, own hot -- each oldest first
      while (pa < G && sc.touched[pa]) pa++;
      if (pa < G) {
        sc.victim[E++] = (int32_t)pa;
        if (sc.owner[pa] >= 0) sc.evk[sc.owner[pa]] = 1;   // evicted before its turn
        pa++;
        continue;
      }
      while (qc < k && !(sc.kind[qc] == 1 || (hits_cold && sc.kind[qc] == 0))) qc++;
      if (qc < k) {
        if (sc.kind[qc] == 1) {
          sc.kind[qc] = 2;
          sc.victim[E++] = VICTIM_OWN_INSERT;
        } else {
          sc.kind[qc] = 3;
          sc.victim[E++] = -(int32_t)(cd[qc] & CODE_SINGLE) - 2;
        }
        qc++;
        continue;
      }
      while (pb < GB && (sc.hot[pb] & 0x80000000ull)) pb++;
      if (pb < GB) {
        const uint32_t x = (uint32_t)sc.hot[pb];
        sc.victim[E++] = -(int32_t)x - 2;
        for (int k2 = k + 1; k2 < nb; k2++)   // a present hot block evicted before its turn
          if (cd[k2] == x && !sc.evk[k2]) sc.evk[k2] = 1;
        pb++;
        continue;
      }
      while (qh < k && sc.kind[qh] != 0) qh++;
      if (qh < k) {
        sc.kind[qh] = 3;
        sc.victim[E++] = -(int32_t)(cd[qh] & CODE_SINGLE) - 2;
        qh++;
        continue;
      }
      S.err = RS_ERR_TIMEOUT;   // nothing to evict: inconsistent state
      break;
    }
    S.nvic = E;
    S.nins = ni;
    S.changed = 1;
    ++*slow;
  }
  grp_bar<NT>();
  const int E = S.nvic;
  for (int v = threadIdx.x; v < E; v += NT) {
    const int32_t iv = sc.victim[v];
    if (iv == VICTIM_OWN_INSERT) continue;
    if (iv >= 0) {
      const uint32_t x = sc.vent[iv];
      if (x & SINGLE_FLAG) t.log[sc.vt[iv] & t.rmask] = LOG_DEAD; else t.st[x] = STAMP_NONE;
    } else {
      t.st[(uint32_t)(-(iv + 2))] = STAMP_NONE;
    }
  }
  grp_bar<NT>();   // (a victim may be a block of this request: its new stamp comes after)
}

// As ids_update under the frequency rule at decay step D (known with the
// arrival, so nothing is planned before the choice).  The window starts where
// the last search ended while the hot entries passed there are still hot.
template <int NT>
__device__ __forceinline__ void ids_update_freq(SimScalars& A, IdsShared& S, uint32_t K, int nbmax,
                                                const IdsTable& t, CacheMeta* meta, FreqMeta* fm,
                                                const uint32_t* cd, const IdsReq& q, uint32_t D,
                                                uint32_t fmax, unsigned char* scratch, uint32_t* win,
                                                uint32_t* whead, uint32_t* wlen, int64_t i) {
  constexpr int R = IDS_WIN / NT, NW = IDS_WIN / 32;
  const int nb = q.nb, nz = q.nz, tid = (int)threadIdx.x, lane = tid & 31;
  cp_async_wait_all();
  if ((uint64_t)meta->T - meta->head + (uint64_t)nb > (uint64_t)t.rmask + 1 ||
      (uint64_t)meta->T + nb > STAMP_LIMIT) {
    grp_bar<NT>();
    ids_compact<NT>(t, meta, S.warp_tot, &S.err);
    if (tid == 0) {
      A.rebuilds++;
      *wlen = 0;
      *fm = FreqMeta{0u, 0u};
    }
    grp_bar<NT>();
  }
  const CacheMeta m = *meta;
  const FreqMeta f = *fm;
  const uint32_t start = D < f.fmin ? f.fscan : m.head;
  const bool full = m.size + (uint32_t)nb > K;
  int nabs = 0;
  uint32_t pmin = STAMP_NONE;   // least stamp of a present cold block
#pragma unroll 1
  for (int k = tid; k < nz; k += NT) {
    const uint32_t x = cd[k], id = x >> 31 ? 0u : x;
    const uint32_t v = t.st[id], e = t.fe[id];
    const uint32_t st = x >> 31 ? STAMP_NONE : v;
    nabs += st == STAMP_NONE;
    if (e <= D) pmin = min(pmin, st);   // (an absent block's is STAMP_NONE)
  }
  uint32_t x[R], he = 0xFFFFFFFFu, hp = 0xFFFFFFFFu;
  bool cold[R];
#pragma unroll
  for (int r = 0; r < R; r++) cold[r] = false;
  if (full) {
    const uint32_t have_win = *whead == start ? *wlen : 0u;
    uint32_t v[R], e[R];
#pragma unroll
    for (int r = 0; r < R; r++) x[r] = win[r * NT + tid];
    if (have_win < (uint32_t)IDS_WIN) {
#pragma unroll
      for (int r = 0; r < R; r++) {
        const uint32_t w = (uint32_t)(r * NT + tid), p = start + w;
        if (w >= have_win) x[r] = p < m.T ? t.log[p & t.rmask] : LOG_DEAD;
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t id = x[r] >= LOG_DEAD ? 0u : x[r];
      v[r] = t.st[id];
      e[r] = t.fe[id];
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t p = start + (uint32_t)(r * NT + tid);
      const bool held = x[r] < LOG_DEAD && v[r] == p;
      cold[r] = x[r] >= SINGLE_FLAG || (held && e[r] <= D);
      if (held && e[r] > D) {
        he = min(he, e[r]);
        hp = min(hp, p);
      }
    }
  }
  {
    const int a = (int)__reduce_add_sync(FULL_MASK, (unsigned)nabs);
    const uint32_t pm = __reduce_min_sync(FULL_MASK, pmin);
    he = __reduce_min_sync(FULL_MASK, he);
    hp = __reduce_min_sync(FULL_MASK, hp);
    if (lane == 0) {
      S.red[tid >> 5] = make_uint2((unsigned)a, pm);
      S.hot[tid >> 5] = make_uint2(he, hp);
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
      const unsigned cv = __ballot_sync(FULL_MASK, cold[r]);
      if (lane == 0) S.livew[r * (NT / 32) + (tid >> 5)] = cv;
    }
  }
  grp_bar<NT>();
  nabs = nb - nz;   // past nz every block is fresh
  pmin = he = hp = 0xFFFFFFFFu;
#pragma unroll
  for (int w = 0; w < NT / 32; w++) {
    nabs += (int)S.red[w].x;
    pmin = min(pmin, S.red[w].y);
    he = min(he, S.hot[w].x);
    hp = min(hp, S.hot[w].y);
  }
  const uint32_t freeb = K - m.size;
  const uint32_t E0 = (uint32_t)nabs > freeb ? (uint32_t)nabs - freeb : 0u;
  uint32_t E = E0, next = start;
  int nins = nabs;
  bool general = false, replayed = false;
  if (E0 > 0) {
    // the first E0 cold entries, all before the oldest present cold block
    const uint32_t lim = pmin > start ? pmin - start : 0u;
    uint32_t have = 0;
    int last = -1;
#pragma unroll
    for (int w = 0; w < NW; w++) {
      const uint32_t l0 = 32u * w;
      const unsigned mk = lim >= l0 + 32u ? FULL_MASK : (lim > l0 ? (1u << (lim - l0)) - 1u : 0u);
      const unsigned b = S.livew[w] & mk;
      const uint32_t n = (uint32_t)__popc(b);
      if (have < E0 && have + n >= E0) last = (int)l0 + nth_set_bit32(b, (int)(E0 - have) - 1);
      have += n;
    }
    if (last >= 0) {
#pragma unroll
      for (int r = 0; r < R; r++)
        if (cold[r] && r * NT + tid <= last) {
          if (x[r] & SINGLE_FLAG)
            t.log[(start + (uint32_t)(r * NT + tid)) & t.rmask] = LOG_DEAD;
          else
            t.st[x[r]] = STAMP_NONE;
        }
      next = start + (uint32_t)last + 1u;
    } else {
      ids_freq_general<NT>(t, m, start, K, cd, nb, E0, pmin, nabs, D, fmax, scratch, nbmax, S, &A.slow);
      general = true;
      replayed = S.changed != 0;
      E = (uint32_t)S.nvic;
      nins = S.nins;
      next = S.nh;
      he = S.fs.femin;
      hp = S.fs.fhot;
    }
  }
  const IdsScratch sc = ids_scratch(scratch, nbmax);
#pragma unroll 1
  for (int k = tid; k < nb; k += NT) {
    const uint32_t b = cd[k] & CODE_SINGLE, pos = m.T + (uint32_t)k;
    const int kind = general ? sc.kind[k] : -1;
    if (kind >= 2) {   // evicted within this request
      t.log[pos & t.rmask] = LOG_DEAD;
      continue;
    }
    if (b != CODE_SINGLE) {
      const bool ins = kind >= 0 ? kind == 1 : (cd[k] >> 31) != 0u || t.st[b] == STAMP_NONE;
      t.fe[b] = ins ? D : freq_hit(t.fe[b], D, fmax);
      t.st[b] = pos;
    }
    t.log[pos & t.rmask] = b != CODE_SINGLE ? b : SINGLE_FLAG | (uint32_t)(q.pos0 + k);
  }
  const uint32_t size = m.size + (uint32_t)nins - E;
  FreqMeta fn = f;
  uint32_t nh = m.head;
  if (replayed) {
    fn = FreqMeta{m.head, 0u};   // the next search starts at the head
  } else if (E > 0) {
    if (start == m.head) {
      nh = min(hp, next);
      fn.fmin = he;
    } else {
      fn.fmin = min(f.fmin, he);
    }
    fn.fscan = next;
  }
  // the window of this worker's next update, from where its search will start
  const uint32_t ws = fn.fmin > D ? fn.fscan : nh;
  const bool refresh = size + (uint32_t)nbmax > K && !replayed;
  if (refresh) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t p = ws + (uint32_t)(r * NT + tid);
      if (p < m.T) cp_async4(win + r * NT + tid, t.log + (p & t.rmask));
    }
  }
  grp_bar<NT>();   // (every thread has read the old state)
  if (tid == 0) {
    // (a window that starts before this update's victims would miss their marks)
    *whead = ws;
    *wlen = refresh && ws >= next && m.T > ws ? min((uint32_t)IDS_WIN, m.T - ws) : 0u;
    *fm = fn;
    meta->size = size;
    meta->head = nh;
    meta->T = m.T + (uint32_t)nb;
    A.inserted += nins;
    A.evicted += E;
    if (E > 0 && A.first_evict_i < 0) {
      A.first_evict_i = i;
      A.first_live = A.inserted - A.evicted;
    }
  }
}

// ------------------------------------------------------------ control warp

// A controller sample with a non-empty window (as the CTA-wide tick of the
// table kernel, by one warp): the window's nearest-rank P99 by an exact radix
// selection, from the highest byte in which its TTFTs differ.
__device__ __noinline__ void ids_tick(SimScalars& S, const SimLaunch& L, double* pend,
                                      int64_t pend_cap, int lane) {
  SimCtx c;
  c.S = &S;
  c.L = &L;
  c.pend_ft0 = pend;
  c.pend_tt0 = pend + pend_cap;
  c.pend_ft1 = pend + 2 * pend_cap;
  c.pend_tt1 = pend + 3 * pend_cap;
  c.pend_win = pend + 4 * pend_cap;
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
  double p99 = 0.0;
  if (nwin > 0) {
    int kk = (int)((99 * nwin + 99) / 100);   // 1-based rank
    const uint64_t diff = all1 ^ any1;
    int shift = diff ? (63 - __clzll((long long)diff)) & ~7 : -8;
    uint64_t pre = shift < 0 ? all1 : (shift == 56 ? 0ull : all1 & (~0ull << (shift + 8)));
    for (; shift >= 0; shift -= 8) {
      for (int q = lane; q < 256; q += 32) c.S->hist[q] = 0;
      __syncwarp();
      const uint64_t mhi = shift == 56 ? 0ull : (~0ull << (shift + 8));
      for (int64_t p = lane; p < nwin; p += 32) {
        const uint64_t bits = (uint64_t)__double_as_longlong(c.pend_win[p]);
        if ((bits & mhi) == (pre & mhi)) atomicAdd(&c.S->hist[(bits >> shift) & 255], 1);
      }
      __syncwarp();
      // lane l holds bins 8 l .. 8 l + 7
      int sum = 0;
#pragma unroll
      for (int e = 0; e < 8; e++) sum += c.S->hist[8 * lane + e];
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
          if (cum + c.S->hist[dg] >= kk) break;
          cum += c.S->hist[dg];
        }
      dg = __shfl_sync(FULL_MASK, dg, ls);
      kk -= __shfl_sync(FULL_MASK, cum, ls);
      pre |= (uint64_t)dg << shift;
      __syncwarp();
    }
    p99 = __longlong_as_double((long long)pre);
  }
  if (lane == 0) {
    S.np = nkeep;
    S.pend_cur = cur ^ 1;
    S.min_ft = tval(mft);
    ctl_sample(c, nwin > 0, p99);
  }
  __syncwarp();
}

// A controller sample without a window.
__device__ __noinline__ void ids_tick_empty(SimScalars& S, const SimLaunch& L, int lane) {
  SimCtx c;
  c.S = &S;
  c.L = &L;
  if (lane == 0) ctl_sample(c, false, 0.0);
  __syncwarp();
}

// Request i's arrival: every event before it, then what its choice needs (dup as
// in ev_arrive; one thread and a heap: for concurrencies whose slots are in global memory).
__device__ __forceinline__ void ids_arrive(SimCtx& c, IdsShared& Sh, int64_t i, bool dup, float* act,
                                           int* nfz, int lane) {
  SimScalars& S = *c.S;
  IdsReq& q = Sh.q[i & (IDS_RING - 1)];
  const int p = (int)(i & 1), W = c.L->mc.W;
  if (dup || q.nb > (int)c.L->g.K) {
    if (lane == 0) Sh.stat[p].x = S.status = dup ? RS_ERR_COLLISION : RS_ERR_CAPACITY;
    __syncwarp();
    return;
  }
  for (;;) {
    int ev = 0;
    if (lane == 0) ev = events_advance(c, q);
    if (!__shfl_sync(FULL_MASK, ev, 0)) break;
    ids_tick(S, *c.L, c.pend_ft0, c.b->pend_cap, lane);
  }
  if (lane == 0) {
    regime_params<false>(c, q);
    Sh.pub[p].a = q.a;
    Sh.pub[p].tau = q.tau;
    Sh.pub[p].omega = q.omega;
    if (S.status != RS_OK) Sh.stat[p].x = S.status;
  }
  __syncwarp();
  for (int j = lane; j < W; j += 32) {
    act[p * W + j] = __int2float_rn((int)c.wA[j]);
    nfz[p * W + j] = min(c.winserv[j] + 1, c.L->mc.cap - 1);
  }
}

// ------------------------------------------------------------ events (control warp)

// The closed-loop client's events with their state in the control warp's
// registers, every lane running the same course: lane j holds workers j and
// (WIDE) j + 32: active blocks, requests in service, queue ends.  Completion
// times lie by request slot in groups of 32; lane g keeps the earliest of
// group g (and of groups g + 32, ...), so an insertion is one comparison and a
// removal one load across the warp and two pairs of warp minima, whatever the
// concurrency.
//
// This warp is the replica's critical path at one or two replicas per SM.  An
// FP64 instruction holds its SM sub-partition's unit for 63 cycles whatever
// the number of lanes, dependent or not, so the times that a service start
// would have are computed for every worker at once, one lane each, from loads
// issued before the choice; nothing that the next event does not need is computed here (TTFT is
// left to the pass over the records).  On one thread with a heap in shared
// memory and the FP64 chain after the choice, the booking took 1 150 SM cycles
// a request and the events 3 000 (64 replicas, W = 3).
constexpr uint64_t KEY_NONE = ~0ull;   // no completion (above every time's key)

template <bool WIDE>
struct IdsEvents {
  static constexpr int H = WIDE ? 2 : 1;
  uint64_t lk, kc;   // earliest completion of this lane's groups, of all
  int lf, fc;        // their slots
  int4 cr;           // srec[fc]
  int fnext;         // the free slot taken next
  int A[H], serv[H], qh[H], qt[H];
  int inflight, nfree, np, cur, ng;
  uint64_t mft, tick;   // keys: earliest pending first token, next controller sample
  uint64_t pk;       // key of the last arrival
  double prev;       // the last arrival
  int conc, ctl, spike, regimes;   // C, controller on, load-spike schedule, the policy takes regimes
  int64_t row0;           // first record row
  uint64_t dhi;           // (frequency eviction) key up to which the decay step is surely D
  uint32_t D;
  float tau, omega;       // in the Below regime
  uint64_t* skey;    // [32 ng] completion keys by slot
  int4* srec;        // [slots] worker, blocks, next in queue, request
  uint64_t* gk;      // [ng] earliest key of each group, and its slot (ng > 32)
  int* gf;
  double *sa, *so, *soitl;   // [slots] of queued requests: arrival, w_c o, O itl
  int* freestk;

  __device__ __forceinline__ int get(const int (&v)[H], int j) const {
    int x = __shfl_sync(FULL_MASK, v[0], j & 31);
    if (WIDE) {
      const int y = __shfl_sync(FULL_MASK, v[H - 1], j & 31);
      if (j >= 32) x = y;
    }
    return x;
  }
  __device__ __forceinline__ void add(int (&v)[H], int j, int x, int lane) {
#pragma unroll
    for (int h = 0; h < H; h++)
      if (lane + 32 * h == j) v[h] += x;
  }
  __device__ __forceinline__ void put(int (&v)[H], int j, int x, int lane) {
#pragma unroll
    for (int h = 0; h < H; h++)
      if (lane + 32 * h == j) v[h] = x;
  }
};

// f(n) of Eq. (9) past the table (rare: kept out of the loop's code).
__device__ __noinline__ double ids_latency(const ModelConsts& mc, int n) { return latency_f(mc, n); }

__device__ __forceinline__ double ev_f(const SimCtx& c, int n) {
  return n < FTAB_MAX ? c.ftab[n] : ids_latency(c.L->mc, n);
}

// The earliest of the warp's (key, slot) pairs, by (key, request).
template <bool WIDE>
__device__ __forceinline__ void ev_min(const IdsEvents<WIDE>& E, uint64_t k, int f, uint64_t& ko,
                                       int& fo) {
  const unsigned hi = __reduce_min_sync(FULL_MASK, (unsigned)(k >> 32));
  const unsigned lo =
      __reduce_min_sync(FULL_MASK, (unsigned)(k >> 32) == hi ? (unsigned)k : 0xFFFFFFFFu);
  ko = ((uint64_t)hi << 32) | lo;
  unsigned eq = __ballot_sync(FULL_MASK, k == ko);
  if ((eq & (eq - 1u)) && ko != KEY_NONE) {   // equal times: the earlier request first
    const unsigned rq = k == ko ? (unsigned)E.srec[f].w : 0xFFFFFFFFu;
    const unsigned mn = __reduce_min_sync(FULL_MASK, rq);
    eq = __ballot_sync(FULL_MASK, rq == mn);
  }
  fo = __shfl_sync(FULL_MASK, f, __ffs(eq) - 1);
}

// The request of record r, in slot f, completes at the time of key k.
template <bool WIDE>
__device__ __forceinline__ void ev_push(IdsEvents<WIDE>& E, int f, uint64_t k, const int4& r,
                                        int lane) {
  const int g = f >> 5;
  if (lane == (g & 31)) {
    E.skey[f] = k;
    if (E.ng > 32 && (k < E.gk[g] || (k == E.gk[g] && r.w < E.srec[E.gf[g]].w))) {
      E.gk[g] = k;
      E.gf[g] = f;
    }
    if (k < E.lk || (k == E.lk && r.w < E.srec[E.lf].w)) {
      E.lk = k;
      E.lf = f;
    }
  }
  if (k < E.kc || (k == E.kc && r.w < E.cr.w)) {
    E.kc = k;
    E.fc = f;
    E.cr = r;
  }
}

// A service's records, and its place in the controller's window (one lane).
template <bool WIDE>
__device__ __forceinline__ void ev_records(const SimCtx& c, const IdsEvents<WIDE>& E, int req,
                                           double t, double ft, double ct, double a) {
  const int64_t row = E.row0 + req;
  c.b->rec.start[row] = t;
  c.b->rec.first_token[row] = ft;
  c.b->rec.completion[row] = ct;
  if (E.ctl) {
    c.pend_ft(E.cur)[E.np] = ft;
    c.pend_tt(E.cur)[E.np] = __dsub_rn(ft, a);
  }
}

// Takes the earliest completion out and completes it: the slot is free, the
// worker's next queued request starts.
template <bool WIDE>
__device__ __forceinline__ void ev_complete(SimCtx& c, IdsEvents<WIDE>& E, int lane) {
  const int f = E.fc, g = f >> 5;
  const double t = tval(E.kc);
  const int4 r = E.cr;
  const int j = r.x;
  // the group without f, then the earliest of all groups
  const int s = 32 * g + lane;
  uint64_t k = E.skey[s];
  if (s == f) {
    k = KEY_NONE;
    E.skey[s] = KEY_NONE;
  }
  ev_min(E, k, s, E.kc, E.fc);
  if (E.ng > 1) {
    if (lane == (g & 31)) {
      E.lk = E.kc;
      E.lf = E.fc;
      if (E.ng > 32) {
        E.gk[g] = E.kc;
        E.gf[g] = E.fc;
        for (int q = lane; q < E.ng; q += 32) {
          const uint64_t kq = E.gk[q];
          if (kq < E.lk || (kq == E.lk && kq != KEY_NONE && E.srec[E.gf[q]].w < E.srec[E.lf].w)) {
            E.lk = kq;
            E.lf = E.gf[q];
          }
        }
      }
    }
    ev_min(E, E.lk, E.lf, E.kc, E.fc);
  } else if (lane == 0) {
    E.lk = E.kc;
    E.lf = E.fc;
  }
  E.cr = E.srec[E.fc];
  if (lane == 0) E.freestk[E.nfree] = f;
  E.nfree++;
  E.fnext = f;
  E.inflight--;
  E.add(E.A, j, -r.y, lane);
  const int f2 = E.get(E.qh, j);
  if (f2 < 0) {
    E.add(E.serv, j, -1, lane);
    __syncwarp();
  } else {   // (as many in service as before)
    const int4 r2 = E.srec[f2];
    E.put(E.qh, j, r2.z, lane);
    if (r2.z < 0) E.put(E.qt, j, -1, lane);
    const double ft = __dadd_rn(t, __dsub_rn(ev_f(c, E.get(E.serv, j)), E.so[f2]));
    const double ct = __dadd_rn(ft, E.soitl[f2]);
    ev_push(E, f2, tkey(ct), r2, lane);
    if (lane == 0) ev_records(c, E, r2.w, t, ft, ct, E.sa[f2]);
    if (E.ctl) {
      E.np++;
      E.mft = min(E.mft, tkey(ft));
    }
    __syncwarp();
  }
}

// A controller sample is due (at E.tick): with first tokens before it the
// window's P99, else none.
template <bool WIDE>
__device__ __forceinline__ void ev_sample(SimCtx& c, IdsEvents<WIDE>& E, int lane) {
  SimScalars& S = *c.S;
  if (E.mft >= E.tick) {
    ids_tick_empty(S, *c.L, lane);
  } else {
    if (lane == 0) {
      S.np = E.np;
      S.pend_cur = E.cur;
    }
    __syncwarp();
    ids_tick(S, *c.L, c.pend_ft0, c.b->pend_cap, lane);
    E.np = (int)S.np;
    E.cur = S.pend_cur;
    E.mft = tkey(S.min_ft);
  }
  E.tick = tkey(S.tick_t);
}

// Request i's arrival: every event before it in time order (completions,
// controller samples, steps of the load-spike schedule; ties in that order),
// then what its choice needs.  drain: past the last request, the completions
// that remain (they start the queued requests).  dup: two blocks of the request
// before have one chained hash (a 64-bit collision): that request is routed,
// its update cannot be made, and nothing after its arrival takes place.
template <bool WIDE, bool FREQ>
__device__ __forceinline__ void ev_arrive(SimCtx& c, IdsShared& Sh, IdsEvents<WIDE>& E, int64_t i,
                                          bool drain, bool dup, float* act, int* nfz, int lane) {
  SimScalars& S = *c.S;
  const IdsReq& q = Sh.q[i & (IDS_RING - 1)];
  const int p = (int)(i & 1), W = c.L->mc.W;
  if (dup || (!drain && q.nb > (int)c.L->g.K)) {
    if (lane == 0) Sh.stat[p].x = S.status = dup ? RS_ERR_COLLISION : RS_ERR_CAPACITY;
    return;
  }
  const uint64_t krel = tkey(q.rel);
  uint64_t ka = E.pk;              // while waiting: the time reached
  uint64_t lim = KEY_INF - 1;      // events up to here are due
  int conc = E.conc;
  bool wait = true, mid = false, step = false, ok = true;
  if (drain || !(E.ctl | E.spike)) {
    // no samples, one concurrency (or the end): completions alone, in a loop of
    // few branches (1 430 cycles a request at W = 3; 1 560 with the samples' test in it,
    // 1 730 in the loop below)
    if (drain) ka = KEY_NONE - 1;
    for (;;) {
      const bool w = !drain && E.inflight >= conc;
      if (!w && !drain && krel > ka) ka = krel;   // (a free place, once there, stays)
      if (E.kc > (w ? KEY_INF - 1 : ka)) {
        if (w && lane == 0) S.status = RS_ERR_TIMEOUT;   // cannot happen, as below
        ok = !w;
        break;
      }
      if (w && E.kc > ka) ka = E.kc;
      ev_complete(c, E, lane);
    }
  } else for (;;) {
    if (wait) {
      // closed-loop client (§7.4): until fewer than C(t) requests are in flight
      if (E.spike) {
        const SimDesc& d = *c.d;
        mid = ka >= tkey(d.c_t1);
        const bool end = ka >= tkey(d.c_t2);
        step = !end;
        conc = end ? d.c_end : (mid ? d.c_mid : d.C);
        lim = end ? KEY_INF - 1 : tkey(mid ? d.c_t2 : d.c_t1);
      }
      if (E.inflight < conc) {
        wait = false;
        if (krel > ka) ka = krel;
        lim = ka < KEY_INF ? ka : KEY_INF - 1;
      }
    }
    if (E.kc <= lim && E.kc <= E.tick) {
      if (wait && E.kc > ka) ka = E.kc;
      ev_complete(c, E, lane);
    } else if (E.tick <= lim) {
      ev_sample(c, E, lane);
      if (S.status != RS_OK) {
        ok = false;
        break;
      }
    } else if (!wait) {
      break;
    } else if (step) {
      ka = tkey(mid ? c.d->c_t2 : c.d->c_t1);   // the schedule steps
    } else {   // cannot happen: a request in flight is in service
      if (lane == 0) S.status = RS_ERR_TIMEOUT;
      ok = false;
      break;
    }
  }
  if (drain) return;
  E.pk = ka;
  E.prev = tval(ka);
  if (FREQ && ka >= E.dhi) {
    // decay step of the arrival, floor(a / decay_s); the division (650 cycles)
    // only where a has come near the next step (arrivals do not decrease)
    const double s = c.d->decay_s, fl = floor(__ddiv_rn(E.prev, s));
    E.D = fl < 2147483648.0 ? (uint32_t)fl : 2147483648u;
    E.dhi = fl < 2147483648.0 ? tkey(__dmul_rn(__dmul_rn(fl + 1.0, s), 1.0 - 0x1p-40)) : KEY_NONE;
  }
#pragma unroll
  for (int h = 0; h < IdsEvents<WIDE>::H; h++) {
    const int j = lane + 32 * h;
    if (j < W) {
      act[p * W + j] = __int2float_rn(E.A[h]);
      nfz[p * W + j] = min(E.serv[h] + 1, c.L->mc.cap - 1);
    }
  }
  if (lane == 0) {
    IdsArrival& ar = Sh.pub[p];
    ar.a = E.prev;
    if (FREQ) ar.D = E.D;
    if (E.ctl) {   // (else written once)
      const bool shift = E.regimes && S.regime > 0;
      ar.tau = shift ? c.L->mc.regime_tau[S.regime] : E.tau;
      ar.omega = shift ? c.L->mc.regime_omega[S.regime] : E.omega;
    }
    if (!ok) Sh.stat[p].x = S.status;
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
    if (!c.b->wco_tab) q.inv = q.nbt > 0 ? __ddiv_rn(1.0, (double)q.nbt) : 0.0;
    const uint4 x = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)((uint64_t)i >> 32), 0u, TAG_SIM),
                                  make_uint2((uint32_t)c.d->seed, (uint32_t)(c.d->seed >> 32)));
    q.dx = x.x;
    q.dy = x.y;
  }
}

// ------------------------------------------------------------ the kernel

// VAR 0: planned updates (a worker per update warp); 1: up to 32 workers; 2: up to 64.
// FREQ: launches that hold replicas which evict by frequency (not SG, not VAR 0).
template <int NU, int MINB, bool SG, int VAR, bool FREQ = false>
__global__ void __launch_bounds__((NU + 2) * 32, MINB)
    k_sim_ids(const SimDesc* __restrict__ descs, const __grid_constant__ SimBuffers b,
              const __grid_constant__ SimLaunch L) {
  constexpr int NT = (NU + 2) * 32, NTU = NU * 32;
  constexpr bool WIDE = VAR == 2, PLAN = VAR == 0;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SimScalars S;
  __shared__ IdsShared Sh;
  const int sid = blockIdx.x;
  const SimDesc d = descs[sid];
  const ModelConsts& mc = L.mc;
  const int W = mc.W;
  const int nft = ftab_size(mc.cap);
  const int nbcap = L.nbmax > 0 ? L.nbmax : 1;
  const IdsLayout lay = make_ids_layout(W, L.nbmax, L.cmax, nft, NTU, SG, FREQ);
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
  uint32_t* win = reinterpret_cast<uint32_t*>(smem + lay.win);       // [W][IDS_WIN or IDS_WRING]
  FreqMeta* wfreq = reinterpret_cast<FreqMeta*>(smem + lay.wfreq);
  // held in registers: the compiler would load them again from the descriptor
  // where they are used, on the path between two joins
  uint32_t* stamps = d.stamps;
  int64_t nre = d.nre, n = d.n_req;
  int policy = d.policy;
  asm volatile("" : "+r"(policy), "+l"(stamps), "+l"(nre), "+l"(n));

  // ---- initial state: empty caches, idle workers
  {
    const size_t nst = (size_t)W * nre;   // (nre: a multiple of 4)
    for (size_t s = threadIdx.x; s < nst / 4; s += NT)
      reinterpret_cast<uint4*>(stamps)[s] = make_uint4(STAMP_NONE, STAMP_NONE, STAMP_NONE, STAMP_NONE);
    for (int q = 1 + threadIdx.x; q < nft; q += NT) c.ftab[q] = latency_f(mc, q);
    for (int q = threadIdx.x; q < 2 * ((2 * nbcap + 31) / 32); q += NT)
      reinterpret_cast<uint32_t*>(smem + lay.lru)[q] = 0u;
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
      if (FREQ) wfreq[j] = FreqMeta{0u, 0u};
    }
    if (threadIdx.x == 0) {
      memset(&S, 0, sizeof(SimScalars));
      S.min_ft = __longlong_as_double(0x7FF0000000000000ll);
      S.next_tick = 1;
      S.tick_t = mc.dt;
      S.nfree = cslots;
      S.first_switch_t = -1.0;
      S.first_evict_i = -1;
      Sh.stat[0] = Sh.stat[1] = make_int2(RS_OK, RS_OK);
      Sh.err = 0;
      Sh.lru_bits = reinterpret_cast<uint32_t*>(smem + lay.lru);
    }
  }
  __syncthreads();

  if (warp < NU) {
    // ================ update warps
    unsigned char* scratch = b.scratch + (size_t)sid * ids_scratch_bytes(L.nbmax);
    unsigned cnt = 0;
    auto table = [&](int j) {
      IdsTable t;
      t.st = stamps + j * nre;
      t.fe = FREQ ? d.fexp + j * nre : nullptr;
      t.log = b.log + ((size_t)sid * W + j) * L.g.R;
      t.rmask = L.ids_rmask;
      return t;
    };
    // request k's cached prefix on every worker (parity pk), and the plans
    auto probe = [&](int64_t k, int pk) {
      const int ek = (int)(k & (IDS_RING - 1));
      const IdsReq& qk = Sh.q[ek];
      if (qk.nb > (int)L.g.K) return;
      const uint32_t* cd = codes + (size_t)ek * nbcap;
      if constexpr (PLAN) {
        // the ring's next entries, once a victim may be needed soon; those
        // copied the last time have landed before others are sent to their
        // places (copies in flight keep no order: after a compaction, or when
        // two updates together pass more entries than the ring holds, the same
        // place is written again)
        cp_async_wait_all();
        __syncwarp();
        if (warp < W) {
          const IdsTable t = table(warp);
          const CacheMeta m = c.wmeta[warp];
          uint32_t* ring = win + warp * IDS_WRING;
          const uint32_t safe = max(wlen[warp], m.head);   // (a compaction sets it to 0)
          const uint32_t to = min(m.T, m.head + IDS_WRING);
          const bool more = m.size + 2 * (uint32_t)L.nbmax > L.g.K && safe < to;
          __syncwarp();   // (every lane has read the last end)
          if (more) {
#pragma unroll 1
            for (uint32_t p = safe + lane; p < to; p += 32)
              cp_async4(ring + (p & (IDS_WRING - 1)), t.log + (p & L.ids_rmask));
          }
          if (lane == 0) wlen[warp] = more ? to : safe;
          const int mj = ids_plan(t, m, L.g.K, cd, qk.nb, qk.nz, ring, safe, Sh.plan[warp], cnt);
          if (lane == 0) wm[pk * W + warp] = mj;
        }
      } else {
        ids_probe<NU>(stamps, nre, cd, qk.nz, W, wm + pk * W, cnt);
      }
    };
    join_cta<NT>();   // the first requests are staged
#pragma unroll 1
    for (int64_t i = -1; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      if (i >= 0) {
        join_cta<NT>();
        if (ids_stopped(Sh, p)) break;
        const IdsReq& q = Sh.q[e];
        choice_wait<NT>();
        const int js = Sh.js;
        if (!q.dup) {   // (else the replica stops here: see ev_arrive)
          const IdsTable t = table(js);
          const uint32_t* cd = codes + (size_t)e * nbcap;
          if (PLAN && Sh.plan[js].step != IDS_GENERAL) {
            ids_apply<NTU>(t, c.wmeta + js, Sh.plan[js], win + js * IDS_WRING, cd, q);
          } else {
            if (FREQ && d.eviction == RS_EVICT_FREQ)
              ids_update_freq<NTU>(S, Sh, L.g.K, L.nbmax, t, c.wmeta + js, wfreq + js, cd, q, Sh.pub[p].D,
                                   (uint32_t)d.freq_max, scratch, win + (size_t)js * IDS_WIN, whead + js,
                                   wlen + js, i);
            else if constexpr (PLAN)
              ids_update_unplanned<NTU>(S, Sh, L.g.K, L.nbmax, t, c.wmeta + js, cd, q, scratch, wlen + js, i);
            else
              ids_update<NTU, true>(S, Sh, L.g.K, L.nbmax, t, c.wmeta + js, cd, q, scratch,
                                    win + (size_t)js * IDS_WIN, whead + js, wlen + js, i);
            if (threadIdx.x == 0 && Sh.err) Sh.stat[p ^ 1].y = Sh.err;
          }
        }
        grp_bar<NTU>();   // the update's stamps, before the next probe
        if (PLAN && warp == js % NU && Sh.plan[js].step != IDS_GENERAL && !q.dup) {
          // (every update warp has read the old state)
          if (lane == 0) {
            CacheMeta m = c.wmeta[js];
            const IdsPlan& P = Sh.plan[js];
            m.size += P.nabs - P.E;
            m.head += P.step;
            m.T += (uint32_t)q.nb;
            c.wmeta[js] = m;
            S.inserted += P.nabs;
            if (P.E > 0) {
              S.evicted += P.E;
              if (S.first_evict_i < 0) {
                // the first update that evicted; resident blocks = inserted - evicted
                S.first_evict_i = i;
                S.first_live = S.inserted - S.evicted;
              }
            }
          }
          __syncwarp();
        }
      }
      if (i + 1 < n) probe(i + 1, p ^ 1);
    }
    cp_async_wait_all();
    // (each lane its own: a lane makes one lookup per worker and 32 blocks, so
    // its 32 bits last for 10^8 requests; their sum over the warp would not)
    if (cnt) atomicAdd(&S.probes, (unsigned long long)cnt);
  } else if (warp == NU) {
    // ================ control warp
    IdsEvents<WIDE> E;
    if constexpr (!SG) {
      E.lk = E.kc = KEY_NONE;
      E.lf = E.fc = 0;
#pragma unroll
      for (int h = 0; h < E.H; h++) {
        E.A[h] = E.serv[h] = 0;
        E.qh[h] = E.qt[h] = -1;
      }
      E.inflight = E.np = E.cur = 0;
      E.nfree = max(d.C, max(d.c_mid, d.c_end));
      E.ng = (E.nfree + 31) >> 5;
      E.mft = KEY_INF;
      E.tick = d.controller ? tkey(mc.dt) : KEY_INF;
      E.prev = 0.0;
      E.pk = tkey(0.0);
      E.D = 0u;
      E.dhi = 0ull;
      // held in registers: a later load of the descriptor would be on the path
      E.conc = d.C;
      E.ctl = d.controller;
      E.spike = d.c_mid > 0;
      E.regimes = d.policy != RS_POLICY_LOADBAL;
      E.tau = d.policy == RS_POLICY_LOADBAL ? 0.0f : d.tau;
      E.omega = d.policy == RS_POLICY_LOADBAL ? 0.0f : d.omega;
      E.row0 = d.rec_base;
      asm volatile("" : "+r"(E.conc), "+r"(E.ctl), "+r"(E.spike), "+r"(E.regimes), "+f"(E.tau), "+f"(E.omega), "+l"(E.row0));
      E.skey = c.h_k;
      E.srec = reinterpret_cast<int4*>(smem + lay.srec);
      E.gk = reinterpret_cast<uint64_t*>(smem + lay.gk);
      E.gf = reinterpret_cast<int*>(smem + lay.gf);
      E.sa = c.f_a;
      E.so = c.f_o;
      E.soitl = c.f_oitl;
      E.freestk = c.freestk;
      E.cr = make_int4(0, 0, -1, 0);
      E.fnext = 0;   // (freestk[cslots - 1])
      if (lane < 2) {
        Sh.pub[lane].tau = E.tau;
        Sh.pub[lane].omega = E.omega;
        Sh.pub[lane].D = 0u;
      }
      for (int f = lane; f < 32 * E.ng; f += 32) E.skey[f] = KEY_NONE;
      if (E.ng > 32)
        for (int g = lane; g < E.ng; g += 32) {
          E.gk[g] = KEY_NONE;
          E.gf[g] = 0;
        }
      __syncwarp();
    }
    join_cta<NT>();   // the first requests are staged
#pragma unroll 1
    for (int64_t i = -1; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      bool dup = false;
      if (i >= 0) {
        join_cta<NT>();
        if (ids_stopped(Sh, p)) break;
        const IdsReq& q = Sh.q[e];
        // w_c o_ij of workers lane, lane + 32: from the table of every (nbt, m),
        // or m / nbt correctly rounded from the rounded reciprocal (one exact
        // remainder and one correction: Markstein 1990)
        constexpr int H = IdsEvents<WIDE>::H;
        double wco[H];
#pragma unroll
        for (int h = 0; h < H; h++) {
          const int j = lane + 32 * h;
          const int m = j < W ? wm[p * W + j] : 0;
          if (b.wco_tab) {
            wco[h] = __ldg(b.wco_tab + (size_t)q.nbt * b.wco_dim + m);
          } else {
            const double md = (double)m, nd = (double)q.nbt;
            const double q0 = __dmul_rn(md, q.inv);
            wco[h] = __dmul_rn(mc.w_c, __fma_rn(__fma_rn(-q0, nd, md), q.inv, q0));
          }
        }
        double ft[H], ct[H];
        uint64_t kt[H];
        unsigned can[H];   // workers below the service limit
        if constexpr (!SG) {
          // first token and completion of a service that starts on each worker now
#pragma unroll
          for (int h = 0; h < H; h++) {
            const int ns = min(E.serv[h] + 1, mc.cap - 1);
            ft[h] = __dadd_rn(E.prev, __dsub_rn(ev_f(c, ns), wco[h]));
            ct[h] = __dadd_rn(ft[h], q.oitl);
            kt[h] = tkey(ct[h]);
            can[h] = __ballot_sync(FULL_MASK, E.serv[h] < mc.cap - 1);
          }
        }
        const int blk = (int)q.blk;
        dup = q.dup != 0;
        choice_wait<NT>();
        const int js = Sh.js;
        auto of = [&](const double (&v)[H]) {
          double x = __shfl_sync(FULL_MASK, v[0], js & 31);
          if (WIDE) {
            const double y = __shfl_sync(FULL_MASK, v[H - 1], js & 31);
            if (js >= 32) x = y;
          }
          return x;
        };
        if constexpr (!SG) {
          // request i's load and service start on worker js
          const int f = E.fnext;
          E.inflight++;
          if (--E.nfree > 0) E.fnext = E.freestk[E.nfree - 1];
          const int4 r = make_int4(js, blk, -1, (int)i);
          if (lane == 0) E.srec[f] = r;
          const int hj = WIDE ? js >> 5 : 0;
          const bool mine = lane == (js & 31);
          if ((((WIDE && hj) ? can[H - 1] : can[0]) >> (js & 31)) & 1u) {
            const uint64_t kj = (WIDE && hj) ? kt[H - 1] : kt[0];
            const unsigned hi = __shfl_sync(FULL_MASK, (unsigned)(kj >> 32), js & 31);
            const unsigned lo = __shfl_sync(FULL_MASK, (unsigned)kj, js & 31);
            ev_push(E, f, ((uint64_t)hi << 32) | lo, r, lane);
#pragma unroll
            for (int h = 0; h < H; h++)
              if (mine && h == hj) {
                E.A[h] += blk;
                E.serv[h]++;
                ev_records(c, E, (int)i, E.prev, ft[h], ct[h], E.prev);
              }
            if (E.ctl) {
              E.np++;
              E.mft = min(E.mft, tkey(of(ft)));
            }
          } else {
            E.add(E.A, js, blk, lane);
            const int qt = E.get(E.qt, js);
            const double w = of(wco);
            if (lane == 0) {
              E.sa[f] = E.prev;
              E.so[f] = w;
              E.soitl[f] = q.oitl;
              if (qt >= 0) E.srec[qt].z = f;
            }
            if (qt < 0) E.put(E.qh, js, f, lane);
            E.put(E.qt, js, f, lane);
          }
          __syncwarp();
          if (lane == 0) S.n_routed = i + 1;
        } else {
          const double w = of(wco);
          if (lane == 0) {
            S.jstar = js;
            book_request<false>(c, q, i, w);
          }
          __syncwarp();
        }
      }
      if constexpr (!SG)
        ev_arrive<WIDE, FREQ>(c, Sh, E, i + 1, i + 1 == n, dup, act, nfz, lane);
      else if (i + 1 < n || dup)
        ids_arrive(c, Sh, i + 1, dup, act, nfz, lane);
    }
    if constexpr (!SG) {
      // each worker's first request still queued (none: past every request): a
      // queue is in request order, and nobody overtakes it
#pragma unroll
      for (int h = 0; h < IdsEvents<WIDE>::H; h++)
        if (lane + 32 * h < W)
          c.wqh[lane + 32 * h] = E.qh[h] >= 0 ? E.srec[E.qh[h]].w : 0x7FFFFFFF;
    }
    if constexpr (SG) {
      // drain: remaining completions start the queued requests
      if (lane == 0 && S.status == RS_OK)
        while (S.nheap > 0) {
          uint64_t k;
          int f;
          heap_pop(c, &k, &f);
          complete(c, f, tval(k));
        }
    }
  } else {
    // ================ staging warp
    int64_t hit = 0, pbl = 0, hashed = 0, sampled = 0;
    const bool eq2 = d.policy == RS_POLICY_DYNAMO || d.policy == RS_POLICY_LOADBAL;
    IdsRaw raw;   // the request after the last one staged
    if (n > 0) raw = ids_read(d, 0);
    // (from request 0 - 3: each turn stages three requests ahead)
#pragma unroll 1
    for (int64_t i = -3; i < n; i++) {
      const int p = (int)(i & 1), e = (int)(i & (IDS_RING - 1));
      const IdsReq& q = Sh.q[e];
      IdsChoice ch;
      if (i >= 0) {
        join_cta<NT>();
        if (ids_stopped(Sh, p)) break;
        ch = ids_choice<WIDE>(policy, q, Sh.pub[p], wm + p * W, act + p * W, W, i, lane);
        if (lane == 0) Sh.js = ch.js;
        choice_made<NT>();
      }
      if (i + 3 < n) {
        ids_stage(c, Sh, raw, i + 3, codes, nbcap, lane);
        if (i + 4 < n) raw = ids_read(d, i + 4);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (i < 0) {
        if (i == -1) {
          cp_async_wait_all();
          join_cta<NT>();
        }
        continue;
      }
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
  if (threadIdx.x == 0 && (Sh.stat[0].y | Sh.stat[1].y) != RS_OK)   // (at most one: the loop has ended there)
    S.status = Sh.stat[0].y | Sh.stat[1].y;
  __syncthreads();
  {
    double st = 0.0, se = 0.0, mk = 0.0;
    if (S.status == RS_OK)
      for (int64_t q = threadIdx.x; q < S.n_routed; q += NT) {
        const int64_t row = d.rec_base + q;
        const double ct = b.rec.completion[row], a = b.rec.arrival[row];
        const double tt = __dsub_rn(b.rec.first_token[row], a);
        b.rec.ttft[row] = tt;
        st = __dadd_rn(st, tt);
        se = __dadd_rn(se, __dsub_rn(ct, a));
        mk = fmax(mk, ct);
      }
    else if constexpr (!SG)   // (else written at the service starts)
      for (int64_t q = threadIdx.x; q < S.n_routed; q += NT) {
        const int64_t row = d.rec_base + q;
        if (q < c.wqh[b.rec.worker[row]])   // service has started
          b.rec.ttft[row] = __dsub_rn(b.rec.first_token[row], b.rec.arrival[row]);
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
  const bool freq = b.fexp != nullptr;
  if (freq && sg) return cudaErrorInvalidValue;   // (such launches use the tables)
  const size_t smem = sim_ids_smem_bytes(L.mc.W, L.nbmax, L.cmax, L.mc.cap, 32 * nu, sg, freq);
  void (*kern)(const SimDesc*, const SimBuffers, const SimLaunch);
  const int var = L.mc.W <= nu ? 0 : (L.mc.W <= 32 ? 1 : 2);
  if (freq)
    kern = nu == 6 ? (var == 2 ? k_sim_ids<6, 2, false, 2, true> : k_sim_ids<6, 2, false, 1, true>)
                   : (var == 2 ? k_sim_ids<2, 5, false, 2, true> : k_sim_ids<2, 5, false, 1, true>);
  else if (nu == 6)
    kern = var == 0 ? (sg ? k_sim_ids<6, 2, true, 0> : k_sim_ids<6, 2, false, 0>)
                    : (sg ? k_sim_ids<6, 2, true, 2>
                          : (var == 1 ? k_sim_ids<6, 2, false, 1> : k_sim_ids<6, 2, false, 2>));
  else
    kern = var == 0 ? (sg ? k_sim_ids<2, 5, true, 0> : k_sim_ids<2, 5, false, 0>)
                    : (sg ? k_sim_ids<2, 5, true, 2>
                          : (var == 1 ? k_sim_ids<2, 5, false, 1> : k_sim_ids<2, 5, false, 2>));
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<L.nsim, (nu + 2) * 32, smem, st>>>(d_desc, b, L);
  return cudaGetLastError();
}

}  // namespace rs
