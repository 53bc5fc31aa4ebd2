// Cached prefixes on every worker's hash table, by a CTA's thread group: the
// probes of the table simulation and of the live router, and the choice's argmin.
#pragma once

#include "sim_common.cuh"

namespace rs {

constexpr int PROBE_CAP = SIM_PROBE_CAP;   // W * nb up to which the probe captures every slot

// A warp's lookups sit at consecutive lanes; those of one worker cover
// consecutive blocks, the lane holding the window's position kw on the
// worker's span of `span` blocks.  The lanes of that span in this warp, as a
// mask: from lane - kw to lane - kw + span - 1, clipped to the warp.
__device__ __forceinline__ unsigned span_mask(int lane, int kw, int span) {
  const int lo = lane - kw > 0 ? lane - kw : 0;
  const int hi = lane - kw + span;   // one past the span's last lane
  const unsigned below_hi = hi >= 32 ? FULL_MASK : (hi > 0 ? (1u << hi) - 1u : 0u);
  return below_hi & ~((1u << lo) - 1u);
}

// Resolves ILP loaded home buckets: sl[r] the slot holding hh[r] or
// SLOT_NONE, fr[r] the first free slot of its probe path.  A bucket full of
// other keys (rare at the tables' load) continues along the probe sequence
// after all of them are scanned, so the common case runs straight through.
template <int ILP>
__device__ __forceinline__ void resolve_buckets(const SimCtx& c, const uint64_t (&v)[ILP][BUCKET],
                                                const uint32_t (&bk)[ILP],
                                                const uint64_t (&hh)[ILP], const int (&jj)[ILP],
                                                uint32_t (&sl)[ILP], uint32_t (&fr)[ILP],
                                                int* err) {
  bool cont[ILP], any = false;
#pragma unroll
  for (int r = 0; r < ILP; r++) {
    sl[r] = SLOT_NONE;
    fr[r] = SLOT_NONE;
    cont[r] = bucket_scan_masks(v[r], bk[r], hh[r], &sl[r], &fr[r]) < 0 && jj[r] >= 0;
    any |= cont[r];
  }
  if (any) {
#pragma unroll
    for (int r = 0; r < ILP; r++)
      if (cont[r]) {
        const TableView t = c.table(jj[r]);
        sl[r] = table_find_free_from(t, hh[r], (bk[r] + 1) & t.bmask, err, &fr[r]);
      }
  }
}

// m_j: leading blocks of the prompt found in worker j's cache, for every j
// (threads of the group), when W nb is too large to look every pair up at
// once.  Rounds over the workers still undecided: a round looks up the next
// `len` blocks of each open worker, with len = ILP NT / (open workers) so
// that a round is ILP lookups per thread (4 with one replica per SM under LRU,
// 1 within the two-per-SM register budget or under frequency eviction, whose
// heap leaves no registers for more), all issued before any is resolved;
// a worker is decided once a miss falls in its window.  Most workers miss at
// their first block, so the few left open after the first round get long
// windows.  Each warp lists the open workers for itself after the round's
// barrier: a miss of the next round lowers m_j only to a block at or past
// that round's start, so a worker's open state does not depend on when a
// warp reads it, and no second barrier is needed.
template <int NT, int ILP>
__device__ __forceinline__ void probe_prefixes(SimCtx& c, const uint64_t* hbuf, int nb) {
  SimScalars& S = *c.S;
  const int W = c.L->mc.W;
  const int lane = (int)(threadIdx.x & 31);
  uint8_t* wl = c.wopen + (threadIdx.x >> 5) * WMAX;   // this warp's open workers
  for (int j = lane; j < W; j += 32) wl[j] = (uint8_t)j;
  __syncwarp();
  int nopen = W;
  int c0 = 0;
  int err = 0;
  unsigned cnt = 0;
  for (;;) {
    int len = (ILP * NT) / nopen;
    if (len < 1) len = 1;
    if (len > nb - c0) len = nb - c0;   // (>= 1: the workers listed are open, so c0 < nb)
    const int total = nopen * len;      // <= ILP NT
    // open worker of lookup `it` = floor(it / len): (it + 0.5) / len lies at
    // least 0.5 / len from an integer and it < ILP NT, so the float product
    // truncates to it exactly
    const float inv_len = 1.0f / (float)len;
    int jj[ILP], kk[ILP], kw[ILP];
    uint64_t hh[ILP], v[ILP][BUCKET];
    uint32_t bk[ILP];
    // every lookup's home bucket requested before any is resolved; a thread
    // past the round's lookups repeats the round's last one (in bounds, unused)
#pragma unroll
    for (int r = 0; r < ILP; r++) {
      const int it0 = r * NT + (int)threadIdx.x;
      const int it = it0 < total ? it0 : total - 1;
      const int o = (int)(((float)it + 0.5f) * inv_len);
      const int j = wl[o];
      kw[r] = it - o * len;
      kk[r] = c0 + kw[r];
      jj[r] = it0 < total && kk[r] < c.wm[j] ? j : -1;   // (no miss known below k yet)
      hh[r] = hbuf[kk[r]];
      const TableView t = c.table(j);
      bk[r] = home_bucket(hh[r], t.bmask);
      ld_bucket(t.keys, bk[r], v[r]);
    }
    uint32_t sl[ILP], fr[ILP];
    resolve_buckets<ILP>(c, v, bk, hh, jj, sl, fr, &err);
#pragma unroll
    for (int r = 0; r < ILP; r++) {
      if (r > 0 && r * NT >= total) break;   // (uniform)
      cnt += jj[r] >= 0;
      // the first miss of the worker's window in this warp: its lanes rise
      // by one block each, so it is the window's lowest missing lane, and
      // the window's lowest lane here (kw = 0, or lane 0) records it
      const unsigned mb =
          __ballot_sync(FULL_MASK, jj[r] >= 0 && sl[r] == SLOT_NONE) & span_mask(lane, kw[r], len);
      if (jj[r] >= 0 && mb && (kw[r] == 0 || lane == 0))
        atomicMin(&c.wm[jj[r]], kk[r] + (__ffs(mb) - 1) - lane);
    }
    grp_bar<NT>();   // every miss of the round is in wm
    c0 += len;
    nopen = 0;
    for (int j0 = 0; j0 < W; j0 += 32) {
      const int j = j0 + lane;
      const bool op = c0 < nb && j < W && c.wm[j] >= c0;
      const unsigned bal = __ballot_sync(FULL_MASK, op);
      if (op) wl[nopen + __popc(bal & ((1u << lane) - 1u))] = (uint8_t)j;
      nopen += __popc(bal);
    }
    __syncwarp();
    if (nopen == 0) break;
  }
  cnt = __reduce_add_sync(FULL_MASK, cnt);
  if (lane == 0 && cnt) atomicAdd(&S.probes, (unsigned long long)cnt);
  if (err) S.status = RS_ERR_TIMEOUT;
}

// The same m_j with every (worker, block) pair looked up at once (W nb <=
// PROBE_CAP): each thread issues the first-bucket loads of ILP pairs
// before resolving them, and the slot found (or the first free slot of the
// probe path) is kept for the chosen worker's update.
// TIER: m_j counts the leading blocks in G1 (a found slot's stamp at or
// past the worker's b1); every pair's tier goes to ptier; the absent count
// is of blocks in no tier.
template <int NT, int ILP, bool TIER = false>
__device__ __forceinline__ void probe_full(SimCtx& c, const uint64_t* hbuf, int nb) {
  SimScalars& S = *c.S;
  const int W = c.L->mc.W;
  const int total = W * nb;
  const int lane = (int)(threadIdx.x & 31);
  // worker of pair `it` = floor(it / nb): (it + 0.5) / nb lies at least
  // 0.5 / nb from an integer, and with W nb <= PROBE_CAP the float product's
  // error stays far below that, so it truncates to the quotient exactly
  const float inv_nb = nb > 0 ? 1.0f / (float)nb : 0.0f;
  int err = 0;
  for (int base = 0; base < total; base += NT * ILP) {   // uniform
    int jj[ILP], kk[ILP];
    uint64_t hh[ILP], v[ILP][BUCKET];
    uint64_t stw[ILP][TIER ? 4 : 1];   // tiers: the home bucket's 8 stamps, beside its keys
    uint32_t bk[ILP];
    // every pair's home bucket requested before any is resolved; a thread
    // past the pairs repeats the last one (in bounds, unused)
#pragma unroll
    for (int r = 0; r < ILP; r++) {
      const int it0 = base + r * NT + (int)threadIdx.x;
      const int it = it0 < total ? it0 : total - 1;
      const int j = (int)(((float)it + 0.5f) * inv_nb);
      jj[r] = it0 < total ? j : -1;
      kk[r] = it - j * nb;
      hh[r] = hbuf[kk[r]];
      const TableView t = c.table(j);
      bk[r] = home_bucket(hh[r], t.bmask);
      ld_bucket(t.keys, bk[r], v[r]);
      if (TIER)   // one 32-byte sector: stamps are 4-byte, buckets of 8 start 32-byte aligned
        ld_keys4(reinterpret_cast<const uint64_t*>(t.stamp + (size_t)BUCKET * bk[r]), stw[r][0],
                 stw[r][TIER ? 1 : 0], stw[r][TIER ? 2 : 0], stw[r][TIER ? 3 : 0]);
    }
    uint32_t sl[ILP], fr[ILP];
    resolve_buckets<ILP>(c, v, bk, hh, jj, sl, fr, &err);
#pragma unroll
    for (int r = 0; r < ILP; r++) {
      const int it = base + r * NT + (int)threadIdx.x;
      bool miss = false, absent = false;
      if (jj[r] >= 0) {
        c.pslot[it] = sl[r];
        c.pfree[it] = fr[r];
        if (TIER) {
          int tier = 0;
          if (sl[r] != SLOT_NONE) {
            uint32_t st;
            if (sl[r] / BUCKET == bk[r]) {   // in the home bucket: its stamp came with the keys
              const uint32_t q = sl[r] % BUCKET;
              const uint64_t w2 = q < 2 ? stw[r][0]
                                        : (q < 4 ? stw[r][TIER ? 1 : 0]
                                                 : (q < 6 ? stw[r][TIER ? 2 : 0]
                                                          : stw[r][TIER ? 3 : 0]));
              st = (uint32_t)(q & 1u ? w2 >> 32 : w2);
            } else {
              st = __ldcg(c.table(jj[r]).stamp + sl[r]);
            }
            const TierMeta tm = c.wtier[jj[r]];
            tier = st >= tm.b1 ? 1 : (st >= tm.b2 ? 2 : 3);
          }
          c.ptier[it] = (uint8_t)tier;
          absent = sl[r] == SLOT_NONE;
          miss = tier != 1;
        } else {
          miss = sl[r] == SLOT_NONE;
        }
      }
      // per worker's lanes in this warp (blocks rise by one per lane): the
      // first miss and the absent count, recorded by the worker's lowest
      // lane here (block 0, or lane 0)
      const unsigned span = span_mask(lane, kk[r], nb);
      const unsigned mb = __ballot_sync(FULL_MASK, miss) & span;
      const unsigned nab = TIER ? __popc(__ballot_sync(FULL_MASK, absent) & span) : __popc(mb);
      // (tiers: a block below G1 ends the prefix though it is present)
      if (jj[r] >= 0 && (kk[r] == 0 || lane == 0) && (nab || (TIER && mb))) {
        if (mb) atomicMin(&c.wm[jj[r]], kk[r] + (__ffs(mb) - 1) - lane);
        if (nab) atomicAdd(&c.wabs[jj[r]], (int)nab);   // absent blocks, for the victim count
      }
    }
  }
  if (threadIdx.x == 0) S.probes += (unsigned long long)total;
  if (err) S.status = RS_ERR_TIMEOUT;
  // (the CTA barrier after the probe orders these results with their readers)
}

// Lowest-index argmin across a warp: each lane holds the minimum of its own
// elements (cost c >= +0, index j; no element: +inf and INT_MAX); every lane ends
// with the (cost, index) that is least in (cost, then index) order.  Bit
// patterns order such costs: two warp minima (21 cycles each) for five steps of
// two shuffles.
__device__ __forceinline__ void argmin_warp(float& c, int& j) {
  const unsigned m = __reduce_min_sync(FULL_MASK, __float_as_uint(c));
  j = (int)__reduce_min_sync(FULL_MASK, __float_as_uint(c) == m ? (unsigned)j : 0x7FFFFFFFu);
  c = __uint_as_float(m);
}

}  // namespace rs
