// PoA estimate of Eq. (12) (K4).
//
// k_poa_keys (rows of every problem over the whole grid): the window of every
// request, floor of its completion time over the window length, and the last
// window of each problem, from which the host sizes the window scratch.
//
// k_poa_sort (one CTA per replica, integers only): a stable bucket sort of the
// requests by window (request order kept inside a window).
//
// k_poa_solve / k_poa_solve_wide (windows handed to the warps / CTAs of the
// whole grid): the frozen costs c_ij = a n_ij + b + d/(C - n_ij)^2 - w_c o_ij of
// the §6.4 matrix, the window's sums, and OPT = the minimum-cost assignment of
// its requests to W workers of capacity max(C_j, ceil(n/W)) each (the
// replicated-column square matrix of §6.4).
//
// FP64 runs at two lanes per clock and SM here, so one CTA that computed a
// replica's costs was bound by its SM's FP64 pipe: the costs of 20 000 rows at
// W = 6 took 1.48 ms in one CTA, and the window divisions 97 us more.  The
// keys and the costs therefore run where the whole grid shares them, f(n) comes
// from a table, and a prefix of 0 needs no division.  What stays in one CTA,
// the sort, is integer work.
//
// OPT: every request first takes its cheapest worker; that is optimal unless a
// worker exceeds its capacity.  Otherwise the rows past the capacities move
// out one at a time, each along a shortest path from any worker over its
// capacity to one with room (successive shortest paths on the W worker nodes;
// edge j -> k = the cheapest move, min over the requests at j of c_qk - c_qj).
// The initial assignment is optimal for its own loads (every row sits at its
// minimum), and a shortest path keeps that, so the loads that respect the
// capacities end with the optimum.  The edge weights are kept across
// augmentations: a request that moves in lowers its worker's weights in O(W);
// only the weights whose minimum moved out are looked up again.
//
// The paths run on integers: a window's costs become multiples of 2^-s (s from
// the window's largest cost: 53 significant bits of it at W <= 16, 51 above),
// so sums and comparisons are exact, no cycle is negative by rounding, and the
// integer units carry the serial chain (a dependent FP64 add costs 64 cycles).
// The rounding, at most 2^-52 of the window's largest cost per request, is far
// below the 1e-12 below which a search on doubles must ignore gains.
// Measured: poa_estimate on 20 000 records, W = 6 (81 windows): 4.22 -> 0.61 ms
// a call (keys 97 -> 5 us, sort and costs 1480 -> 17 us, solver 2941 -> 578 us,
// total 19 -> 6 us); the estimate of 16 replicas x 5000 requests at W = 64,
// 126 -> 18 ms.
//
// k_poa_total (one warp per replica): the whole-run PoA, sum of observed
// latency over sum of OPT across the replica's windows; and the static
// counterfactual of §9, the realized assignment's frozen cost over OPT.
#include <climits>

#include "rs_device.cuh"

namespace rs {

// Eq. (9)'s part of a frozen cost.
__device__ __forceinline__ double frozen_f(const ModelConsts& mc, int nf) {
  const double t1 = __dmul_rn(mc.lat_a, (double)nf);
  const double t2 = __dadd_rn(t1, mc.lat_b);
  const double den = (double)(mc.cap - nf);
  return __dadd_rn(t2, __ddiv_rn(mc.lat_d, __dmul_rn(den, den)));
}

constexpr int POA_FTAB = 256;   // f(n) tabulated for n < POA_FTAB (a CTA's shared memory)

__device__ __forceinline__ void fill_ftab(const ModelConsts& mc, double* ftab) {
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  for (int q = threadIdx.x; q < nft; q += blockDim.x) ftab[q] = frozen_f(mc, q);
  __syncthreads();
}

// c_ij of §6.4; a prefix of 0 leaves f(n) - w_c 0 = f(n) without the division.
__device__ __forceinline__ double frozen_cost(const ModelConsts& mc, const double* ftab, int nft,
                                              int nf, int m, int nbt) {
  const double f = nf < nft ? ftab[nf] : frozen_f(mc, nf);
  if (m == 0 || nbt <= 0) return __dsub_rn(f, __dmul_rn(mc.w_c, 0.0));
  return __dsub_rn(f, __dmul_rn(mc.w_c, __ddiv_rn((double)m, (double)nbt)));
}

// Window of each row into wkey: -1 for a row that was not routed, KEY_BAD for
// a completion that is negative, not finite or past 2^31 - 2 windows.  maxw
// (nullable, -1 before the launch) becomes the largest floor(completion /
// window) of each problem's routed rows, negative and NaN ones left out,
// clamped at 2^62.  Grid (problems, row chunks).
constexpr int KEY_BAD = -2;

__global__ void __launch_bounds__(NT_POA) k_poa_keys(const PoaProblem* __restrict__ probs,
                                                     rs_records rec, double window,
                                                     int32_t* __restrict__ wkey,
                                                     long long* __restrict__ maxw) {
  __shared__ long long red[NT_POA / 32];
  const PoaProblem pr = probs[blockIdx.x];
  long long mx = -1;
  for (int64_t q = (int64_t)blockIdx.y * NT_POA + threadIdx.x; q < pr.n;
       q += (int64_t)gridDim.y * NT_POA) {
    const int64_t r = pr.rec_base + q;
    int key = -1;
    if (rec.worker[r] >= 0) {
      const double w = floor(__ddiv_rn(rec.completion[r], window));
      key = KEY_BAD;
      if (w >= 0.0) {
        const long long k = w < 4.611686018427387904e18 ? (long long)w : (1ll << 62);
        mx = k > mx ? k : mx;
        if (k <= (long long)INT_MAX - 2) key = (int)k;
      }
    }
    wkey[pr.scratch_base + q] = key;
  }
  if (!maxw) return;
  for (int o = 16; o > 0; o >>= 1) {
    const long long v = __shfl_xor_sync(FULL_MASK, mx, o);
    mx = v > mx ? v : mx;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long m = red[0];
    for (int w = 1; w < NT_POA / 32; w++) m = red[w] > m ? red[w] : m;
    if (m >= 0) atomicMax(maxw + blockIdx.x, m);
  }
}

// Stable bucket sort of a problem's rows by window.  The rows are cut into
// nseg consecutive segments, one per warp; each warp counts its segment's
// windows into its own column of a (window, segment) table in shared memory,
// one scan of the table in that order gives every (window, segment) its first
// position, and each warp walks its segment again and places its rows, 32 at a
// time, with no barrier between steps.  A problem whose windows do not fit the
// table (more than POA_SORT_TAB of them: records spread over more windows than
// they usually have rows) counts in global memory and is placed by one warp.
constexpr int POA_SORT_TAB = 11 * 1024;   // table entries (44 KB: no opt-in)
constexpr int POA_SORT_NT = 1024;         // most threads of a sorting CTA

__global__ void __launch_bounds__(POA_SORT_NT) k_poa_sort(const PoaProblem* __restrict__ probs,
                                                          PoaBuffers b, int W) {
  extern __shared__ uint32_t tab[];
  __shared__ long long s_warp[POA_SORT_NT / 32];
  __shared__ int s_max, s_bad;
  __shared__ long long s_carry;
  const PoaProblem pr = probs[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nt = blockDim.x, nwarps = nt >> 5;
  if (b.wprob)   // the owner of every window slot of this problem
    for (int64_t w = threadIdx.x; w < pr.win_cap; w += nt) b.wprob[pr.win_base + w] = blockIdx.x;
  if (threadIdx.x == 0) {
    s_max = -1;
    s_bad = 0;
    s_carry = 0;
  }
  __syncthreads();
  const int32_t* key = b.wkey + pr.scratch_base;
  int mx = -1, bad = 0;
  for (int64_t q = threadIdx.x; q < pr.n; q += nt) {
    const int k = key[q];
    mx = k > mx ? k : mx;
    bad |= k == KEY_BAD;
  }
  mx = __reduce_max_sync(FULL_MASK, mx);
  bad = __any_sync(FULL_MASK, bad);
  if (lane == 0) {
    if (mx >= 0) atomicMax(&s_max, mx);
    if (bad) s_bad = 1;
  }
  __syncthreads();
  const int64_t nw = (int64_t)s_max + 1;
  if (W > POA_WMAX_WIDE || s_bad || nw > pr.win_cap) {
    if (threadIdx.x == 0) b.nwin[blockIdx.x] = W > POA_WMAX_WIDE ? -2 : -1;
    return;
  }
  int64_t* cnt = b.wcnt + pr.win_base;
  int64_t* wst = b.wstart + pr.win_base + blockIdx.x;   // nw + 1 entries
  int32_t* order = b.order + pr.scratch_base;
  if (nw == 0) {
    if (threadIdx.x == 0) {
      wst[0] = 0;
      b.nwin[blockIdx.x] = 0;
    }
    return;
  }
  if (nw <= POA_SORT_TAB) {
    int nseg = (int)(POA_SORT_TAB / nw);
    if (nseg > nwarps) nseg = nwarps;
    const int total = (int)nw * nseg;
    for (int e = threadIdx.x; e < total; e += nt) tab[e] = 0;
    __syncthreads();
    const int64_t per = (pr.n + nseg - 1) / nseg;
    const int64_t q0 = (int64_t)warp * per;
    const int64_t q1 = warp < nseg ? (q0 + per < pr.n ? q0 + per : pr.n) : 0;
    for (int64_t q = q0; q < q1; q += 32) {   // warp-uniform
      const int k = q + lane < q1 ? key[q + lane] : -1;
      if (k >= 0) atomicAdd(tab + k * nseg + warp, 1u);
    }
    __syncthreads();
    // exclusive scan of the table in (window, segment) order
    const int chunk = (total + nt - 1) / nt;
    const int e0 = threadIdx.x * chunk < total ? threadIdx.x * chunk : total;
    const int e1 = e0 + chunk < total ? e0 + chunk : total;
    uint32_t sum = 0;
    for (int e = e0; e < e1; e++) sum += tab[e];
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL_MASK, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t off = x - sum;
    for (int i = 0; i < warp; i++) off += (uint32_t)s_warp[i];
    for (int e = e0; e < e1; e++) {
      const uint32_t v = tab[e];
      tab[e] = off;
      off += v;
    }
    if (threadIdx.x == nt - 1) {   // (its range ends the table)
      s_carry = off;
      wst[nw] = off;
    }
    __syncthreads();
    for (int w = threadIdx.x; w < (int)nw; w += nt) {
      const uint32_t a = tab[w * nseg];
      const uint32_t z = w + 1 < (int)nw ? tab[(w + 1) * nseg] : (uint32_t)s_carry;
      wst[w] = a;
      cnt[w] = z - a;
    }
    __syncthreads();
    for (int64_t q = q0; q < q1; q += 32) {
      const int k = q + lane < q1 ? key[q + lane] : -1;
      const unsigned peers = __match_any_sync(FULL_MASK, k);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      uint32_t pos = 0;
      if (k >= 0) pos = tab[k * nseg + warp];
      __syncwarp();
      if (k >= 0) {
        order[pos + rank] = (int32_t)(q + lane);
        if (rank == 0) tab[k * nseg + warp] = pos + __popc(peers);
      }
      __syncwarp();
    }
    if (threadIdx.x == 0) b.nwin[blockIdx.x] = nw;
    return;
  }
  // more windows than the table holds
  int64_t* fill = b.wfill + pr.win_base;
  for (int64_t w = threadIdx.x; w < nw; w += nt) cnt[w] = 0;
  __syncthreads();
  for (int64_t q = threadIdx.x; q < pr.n; q += nt) {
    const int k = key[q];
    if (k >= 0) atomicAdd(reinterpret_cast<unsigned long long*>(cnt + k), 1ull);
  }
  __syncthreads();
  for (int64_t w0 = 0; w0 < nw; w0 += nt) {
    const int64_t w = w0 + threadIdx.x;
    const long long v = w < nw ? (long long)__ldcg(cnt + w) : 0;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(FULL_MASK, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    long long off = s_carry;
    for (int i = 0; i < warp; i++) off += s_warp[i];
    if (w < nw) {
      wst[w] = off + x - v;
      fill[w] = off + x - v;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int i = 0; i < nwarps; i++) s_carry += s_warp[i];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    wst[nw] = s_carry;
    b.nwin[blockIdx.x] = nw;
  }
  if (warp != 0) return;
  for (int64_t q = 0; q < pr.n; q += 32) {
    const int k = q + lane < pr.n ? key[q + lane] : -1;
    const unsigned peers = __match_any_sync(FULL_MASK, k);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    int64_t pos = 0;
    if (k >= 0) pos = fill[k];
    __syncwarp();
    if (k >= 0) {
      order[pos + rank] = (int32_t)(q + lane);
      if (rank == 0) fill[k] = pos + __popc(peers);
    }
    __syncwarp();
  }
}

// Fixed-point costs of one window: value = cost * 2^s.  With BITS bits for the
// largest cost, |value| < 2^BITS, an edge weight is below 2^(BITS + 1) and the
// sum of a path's weights (at most W of them) below 2^59 < FX_INF / 4.
constexpr long long FX_INF = 1ll << 61;    // no path / no row
constexpr long long FX_REAL = 1ll << 60;   // every finite distance is below
constexpr int FX_BITS = 53;                // W <= 16
constexpr int FX_BITS_WIDE = 51;           // W <= 64

// Biased exponent of a finite cost (0 for one that is not finite).
__device__ __forceinline__ int cost_exp(double c) {
  const int e = (int)((uint64_t)__double_as_longlong(c) >> 52) & 0x7FF;
  return e < 0x7FF ? e : 0;
}
// The scale 2^s that puts costs of biased exponent emax below 2^bits, and
// 2^-s (s within the normal range: smaller costs than it covers round to 0).
__device__ __forceinline__ double fx_scale(int emax, int bits, double* inv) {
  int s = bits - (emax - 1022);
  s = s > 1000 ? 1000 : (s < -1000 ? -1000 : s);
  *inv = __longlong_as_double((long long)(1023 - s) << 52);
  return __longlong_as_double((long long)(1023 + s) << 52);
}
// A cost that is not finite counts as the largest magnitude.
__device__ __forceinline__ long long to_fx(double c, double scale, int bits) {
  const long long lim = 1ll << bits;
  if (!(fabs(c) < __longlong_as_double(0x7FF0000000000000ll))) return c < 0.0 ? -lim : lim;
  return __double2ll_rn(__dmul_rn(c, scale));
}

// Least (value, lowest lane) over the warp's lanes with `in` set; lane -1 if
// there is none.
__device__ __forceinline__ int warp_argmin(long long v, bool in, long long* best) {
  const unsigned hi = in ? (unsigned)((unsigned long long)v >> 32) ^ 0x80000000u : 0xFFFFFFFFu;
  const unsigned mh = __reduce_min_sync(FULL_MASK, hi);
  const bool c1 = in && hi == mh;
  const unsigned lo = c1 ? (unsigned)v : 0xFFFFFFFFu;
  const unsigned ml = __reduce_min_sync(FULL_MASK, lo);
  const unsigned who = __ballot_sync(FULL_MASK, c1 && lo == ml);
  *best = (long long)(((unsigned long long)(mh ^ 0x80000000u) << 32) | ml);
  return who ? __ffs(who) - 1 : -1;
}

constexpr int NT_SOLVE = 128;   // most threads of a narrow solver CTA (one window per warp)

struct PoaWarpShared {
  long long wmin[POA_WMAX][POA_WMAX];   // edge weights, FX_INF without a row
  int wrow[POA_WMAX][POA_WMAX];         // the request behind each
  int counts[POA_WMAX];
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

// Weights j -> k, for the columns k set in `need`, from the requests now at j:
// min of c_qk - c_qj, ties to the lowest row.  Rows go 128 at a time, four per
// lane in flight.
template <int WT>
__device__ __forceinline__ void poa_rescan(PoaWarpShared& S, const long long* cost,
                                           const int32_t* asg, int64_t m, int W, int j,
                                           unsigned need, int lane) {
  while (need) {   // (uniform)
    const int k = __ffs(need) - 1;
    need &= need - 1;
    long long best = FX_INF;
    int row = -1;
    for (int64_t r0 = lane; r0 < m; r0 += 128) {
      int at[4];
      long long v[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t r = r0 + 32 * u;
        at[u] = -1;
        v[u] = 0;
        if (r < m) {
          at[u] = asg[r];
          v[u] = cost[r * W + k] - cost[r * W + j];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (at[u] == j && v[u] < best) {
          best = v[u];
          row = (int)(r0 + 32 * u);
        }
    }
    long long least;
    warp_argmin(best, row >= 0, &least);
    const bool mine = row >= 0 && best == least;
    const unsigned rr = __reduce_min_sync(FULL_MASK, mine ? (unsigned)row : 0xFFFFFFFFu);
    if (lane == 0) {
      S.wmin[j][k] = rr != 0xFFFFFFFFu ? least : FX_INF;
      S.wrow[j][k] = (int)rr;   // (-1 without a row)
    }
  }
}

// The next window a solver takes: with b.wnext the solvers of the whole grid
// take window slots from the counter in order (a replica's windows spread over
// the GPU, so a few heavy replicas do not hold the end of the launch); without
// it the solvers of problem blockIdx.x stride over its windows (next, stride).
// One warp calls this alike; returns false when no window is left.
__device__ __forceinline__ bool poa_next(const PoaProblem* __restrict__ probs, const PoaBuffers& b,
                                         int lane, int64_t& next, int64_t stride, int* pi,
                                         int64_t* w) {
  for (;;) {
    if (b.wnext) {
      unsigned long long item = 0;
      if (lane == 0) item = atomicAdd(b.wnext, 1ull);
      item = __shfl_sync(FULL_MASK, item, 0);
      if ((int64_t)item >= b.nslots) return false;
      const int p = b.wprob[item];
      const int64_t ww = (int64_t)item - probs[p].win_base;
      const int64_t nw = b.nwin[p];
      if (nw < 0 || ww >= nw) continue;   // a spare slot, or a problem that overflowed
      *pi = p;
      *w = ww;
      return true;
    }
    const int64_t nw = b.nwin[blockIdx.x];
    const int64_t ww = next;
    next += stride;
    if (nw < 0 || ww >= nw) return false;
    *pi = (int)blockIdx.x;
    *w = ww;
    return true;
  }
}

// WT: a compile-time bound on W (the exact W for the common 3 and 6, else
// POA_WMAX), so that the unrolled per-worker loops hold no dead iterations:
// the solver's warps run different phases at once and its code must stay
// small for the instruction cache.
template <int WT>
__global__ void __launch_bounds__(NT_SOLVE) k_poa_solve(const PoaProblem* __restrict__ probs,
                                                        PoaBuffers b, ModelConsts mc) {
  __shared__ PoaWarpShared P[NT_SOLVE / 32];
  __shared__ double ftab[POA_FTAB];
  fill_ftab(mc, ftab);
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  const int W = mc.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpc = blockDim.x >> 5;
  PoaWarpShared& S = P[warp];
  int64_t next = (int64_t)blockIdx.y * wpc + warp;
  const int64_t stride = (int64_t)gridDim.y * wpc;
  int pi;
  int64_t w;
  // (a problem whose windows overflowed: k_poa_total reports it)
  while (poa_next(probs, b, lane, next, stride, &pi, &w)) {
    const PoaProblem pr = probs[pi];
    const int64_t* wst = b.wstart + pr.win_base + pi;
    const int64_t s0 = wst[w];
    const int64_t m = wst[w + 1] - s0;
    const int64_t base = pr.scratch_base + s0;   // window rows in order[], asg[]
    const int64_t slot = pr.win_base + w;
    if (m == 0) {
      if (lane == 0) {
        b.wnum[slot] = 0.0;
        b.wopt[slot] = 0.0;
        b.wstat[slot] = 0.0;
        b.wcnt[slot] = 0;
      }
      continue;
    }
    int64_t capw = (m + W - 1) / W;
    if (capw < mc.cap) capw = mc.cap;
    if (lane < W) S.counts[lane] = 0;
    __syncwarp();
    double* cost = b.cost + base * W;
    int32_t* asg = b.asg + base;
    double num = 0.0, nst = 0.0, opt = 0.0;
    int emax = 0;
    for (int64_t r = lane; r < m; r += 32) {
      const int64_t q = pr.rec_base + b.order[base + r];
      const int nbt = b.rec.nbt[q], wk = b.rec.worker[q];
      const uint16_t* nfr = b.rec.n_frozen + q * W;
      const uint16_t* pre = b.rec.prefix + q * W;
      double* cr = cost + r * W;
      double bc = 0.0, cw = 0.0;
      int best = 0;
#pragma unroll
      for (int j = 0; j < WT; j++) {
        if (j < W) {
          const double c = frozen_cost(mc, ftab, nft, nfr[j], pre[j], nbt);
          cr[j] = c;
          if (j == 0 || c < bc) { bc = c; best = j; }
          if (j == wk) cw = c;
          const int e = cost_exp(c);
          emax = e > emax ? e : emax;
        }
      }
      nst += cw;   // the realized assignment's frozen cost
      asg[r] = best;
      atomicAdd(&S.counts[best], 1);
      num += b.rec.ttft[q];
      opt += bc;
    }
    num = warp_sum(num);
    nst = warp_sum(nst);
    __syncwarp();
    int count = lane < W ? S.counts[lane] : 0;   // lane j keeps worker j's load
    if (__any_sync(FULL_MASK, lane < W && count > capw)) {
      emax = __reduce_max_sync(FULL_MASK, emax);
      double inv;
      const double scale = fx_scale(emax, FX_BITS, &inv);
      long long* fx = reinterpret_cast<long long*>(cost);   // in place
      for (int64_t e = lane; e < m * W; e += 32) fx[e] = to_fx(cost[e], scale, FX_BITS);
      __syncwarp();
      const unsigned wmask = (1u << W) - 1u;
      for (int j = 0; j < W; j++)
        poa_rescan<WT>(S, fx, asg, m, W, j, wmask & ~(1u << j), lane);
      if (lane < W) {
        S.wmin[lane][lane] = FX_INF;
        S.wrow[lane][lane] = -1;
      }
      __syncwarp();
      for (;;) {
        // distances from the workers over their capacity, in Jacobi rounds:
        // lane k < W owns target k and every round reads the previous one's
        // distances (shortest paths have at most W - 1 edges)
        const bool src = lane < W && count > capw;
        if (!__any_sync(FULL_MASK, src)) break;
        long long dk = src ? 0 : FX_INF;
        int pk = -1;
        long long wm[WT];
#pragma unroll
        for (int j = 0; j < WT; j++) wm[j] = j < W && lane < W ? S.wmin[j][lane] : FX_INF;
        for (int it = 0; it < W; it++) {
          long long bv = dk < FX_REAL ? dk : FX_REAL;
          int bj = -1;
#pragma unroll
          for (int j = 0; j < WT; j++) {
            const long long v = __shfl_sync(FULL_MASK, dk, j) + wm[j];   // (<= 2 FX_INF)
            if (v < bv) { bv = v; bj = j; }
          }
          if (bj >= 0) { dk = bv; pk = bj; }
          if (!__any_sync(FULL_MASK, bj >= 0)) break;
        }
        // target: the nearest worker with room (ties: lowest index)
        long long dt;
        const int tgt = warp_argmin(dk, lane < W && count < capw && dk < FX_REAL, &dt);
        if (tgt < 0) break;   // (cannot happen: W capw >= m)
        // walk the path back from its end: each edge j -> k moves the request
        // behind wrow[j][k] from j to k; lane t keeps step t
        int k = tgt, nmv = 0, mj = -1, mk = -1, mr = -1;
        for (; nmv < W; nmv++) {
          const int j = __shfl_sync(FULL_MASK, pk, k);
          if (j < 0) break;
          if (lane == nmv) {
            mj = j;
            mk = k;
            mr = S.wrow[j][k];
          }
          k = j;
        }
        if (lane == k) count--;
        if (lane == tgt) count++;
        if (lane < nmv) asg[mr] = mk;
        __syncwarp();
        // a worker that lost a request: the weights whose minimum it was
        for (int t = 0; t < nmv; t++) {
          const int j = __shfl_sync(FULL_MASK, mj, t), r = __shfl_sync(FULL_MASK, mr, t);
          const unsigned need = __ballot_sync(FULL_MASK, lane < W && lane != j && S.wrow[j][lane] == r);
          poa_rescan<WT>(S, fx, asg, m, W, j, need, lane);
        }
        __syncwarp();
        // requests that moved in lower their new worker's weights
        for (int t = 0; t < nmv; t++) {
          const int to = __shfl_sync(FULL_MASK, mk, t), r = __shfl_sync(FULL_MASK, mr, t);
          if (lane < W && lane != to) {
            const long long v = fx[(int64_t)r * W + lane] - fx[(int64_t)r * W + to];
            const long long o = S.wmin[to][lane];
            if (v < o || (v == o && r < S.wrow[to][lane])) {
              S.wmin[to][lane] = v;
              S.wrow[to][lane] = r;
            }
          }
        }
        __syncwarp();
      }
      const bool bad = __any_sync(FULL_MASK, lane < W && count > capw);
      opt = 0.0;
      for (int64_t r = lane; r < m; r += 32) opt += (double)fx[r * W + asg[r]] * inv;
      if (bad) opt = __longlong_as_double(0x7FF8000000000000ll);
    }
    opt = warp_sum(opt);
    if (lane == 0) {
      b.wnum[slot] = num;
      b.wstat[slot] = nst;
      b.wopt[slot] = opt;
      b.wcnt[slot] = m;
    }
    __syncwarp();
  }
}

// The same OPT for W > POA_WMAX workers, one CTA per window: few windows, each
// of hundreds to thousands of requests, so the latency of one augmentation is
// what counts.  Thread t owns the target worker t % 64 and a quarter t / 64 of
// the sources (or of a worker's requests) in every W x W step; the quarters
// meet in shared memory.
constexpr int NT_WIDE = 256;
constexpr int WIDE_G = NT_WIDE / POA_WMAX_WIDE;   // source groups

struct PoaWideShared {
  long long dist[POA_WMAX_WIDE];
  long long pv[WIDE_G][POA_WMAX_WIDE];   // per group: the best value of each target ...
  int pi[WIDE_G][POA_WMAX_WIDE];         // ... and its source (or request)
  double red[3][NT_WIDE / 32];
  double ftab[POA_FTAB];
  int pred[POA_WMAX_WIDE], counts[POA_WMAX_WIDE];
  int mv_j[POA_WMAX_WIDE], mv_k[POA_WMAX_WIDE], mv_r[POA_WMAX_WIDE];   // the last path's moves
  int dpos[POA_WMAX_WIDE];     // where a source's request list starts, -1: not rescanned
  int dfill[POA_WMAX_WIDE];
  int nmv, changed, emax, done, tgt, pi_next;
  int64_t w_next;
};

__host__ __device__ inline size_t poa_wide_smem(int W) {
  return (size_t)W * W * 12;   // weights and their requests; PoaWideShared is static
}

// Weights j -> k of every source with dpos[j] >= 0, for the columns whose
// minimum left (wrow[j][k] == lost[j]; every column when `all`), from the
// requests now at j.  list: scratch for the rescanned sources' requests.
__device__ __forceinline__ void wide_rescan(PoaWideShared& S, long long* wmin, int* wrow,
                                            const long long* fx, const int32_t* asg, int32_t* list,
                                            int64_t m, int W, int nsrc, const int* srcs,
                                            const int* lost, bool all) {
  const int k = threadIdx.x % POA_WMAX_WIDE, g = threadIdx.x / POA_WMAX_WIDE;
  // the rescanned sources' requests, gathered per source (any order: ties are
  // settled by the row)
  for (int64_t r = threadIdx.x; r < m; r += NT_WIDE) {
    const int j = asg[r];
    const int d = S.dpos[j];
    if (d >= 0) list[d + atomicAdd(&S.dfill[j], 1)] = (int32_t)r;
  }
  __syncthreads();
  for (int s = 0; s < nsrc; s++) {
    const int j = all ? s : srcs[s];
    const int n = S.dfill[j];
    const int32_t* rows = list + S.dpos[j];
    const bool need = k < W && k != j && (all || wrow[j * W + k] == lost[s]);
    long long best = FX_INF;
    int row = -1;
    if (need) {
      for (int t0 = g; t0 < n; t0 += 8 * WIDE_G) {
        long long v[8];
        int rr[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
          const int t = t0 + u * WIDE_G;
          rr[u] = t < n ? rows[t] : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; u++) {
          const long long* cr = fx + (int64_t)(rr[u] < 0 ? 0 : rr[u]) * W;
          v[u] = cr[k] - cr[j];
        }
#pragma unroll
        for (int u = 0; u < 8; u++)
          if (rr[u] >= 0 && (v[u] < best || (v[u] == best && rr[u] < row))) {
            best = v[u];
            row = rr[u];
          }
      }
    }
    S.pv[g][k] = best;
    S.pi[g][k] = row;
    __syncthreads();
    if (g == 0 && need) {
#pragma unroll
      for (int h = 1; h < WIDE_G; h++) {
        const long long v = S.pv[h][k];
        const int r = S.pi[h][k];
        if (r >= 0 && (v < best || (v == best && r < row))) {
          best = v;
          row = r;
        }
      }
      wmin[j * W + k] = row >= 0 ? best : FX_INF;
      wrow[j * W + k] = row;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(NT_WIDE) k_poa_solve_wide(const PoaProblem* __restrict__ probs,
                                                            PoaBuffers b, ModelConsts mc) {
  extern __shared__ __align__(16) unsigned char wsm[];
  __shared__ PoaWideShared S;
  const int W = mc.W;
  long long* wmin = reinterpret_cast<long long*>(wsm);
  int* wrow = reinterpret_cast<int*>(wmin + (size_t)W * W);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = threadIdx.x % POA_WMAX_WIDE, g = threadIdx.x / POA_WMAX_WIDE;
  fill_ftab(mc, S.ftab);
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  int64_t next = blockIdx.y;
  const int64_t stride = gridDim.y;
  for (;;) {
    if (warp == 0) {
      int pi;
      int64_t w;
      const bool any = poa_next(probs, b, lane, next, stride, &pi, &w);
      if (lane == 0) {
        S.pi_next = any ? pi : -1;
        S.w_next = any ? w : 0;
        S.emax = 0;
      }
    }
    for (int j = threadIdx.x; j < W; j += NT_WIDE) S.counts[j] = 0;
    __syncthreads();
    const int pi = S.pi_next;
    if (pi < 0) return;
    const int64_t w = S.w_next;
    const PoaProblem pr = probs[pi];
    const int64_t* wst = b.wstart + pr.win_base + pi;
    const int64_t s0 = wst[w];
    const int64_t m = wst[w + 1] - s0;
    const int64_t base = pr.scratch_base + s0;
    const int64_t slot = pr.win_base + w;
    int64_t capw = (m + W - 1) / W;
    if (capw < mc.cap) capw = mc.cap;
    double* cost = b.cost + base * W;
    int32_t* asg = b.asg + base;
    // costs and cheapest workers, one warp per request (lane: workers lane, lane + 32)
    double num = 0.0, nst = 0.0, opt = 0.0;
    int emax = 0;
    for (int64_t r = warp; r < m; r += NT_WIDE / 32) {
      const int64_t q = pr.rec_base + b.order[base + r];
      const int nbt = b.rec.nbt[q];
      double c[2];
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int j = lane + 32 * h;
        c[h] = 0.0;
        if (j < W) {
          c[h] = frozen_cost(mc, S.ftab, nft, b.rec.n_frozen[q * W + j], b.rec.prefix[q * W + j], nbt);
          cost[r * W + j] = c[h];
          const int e = cost_exp(c[h]);
          emax = e > emax ? e : emax;
        }
      }
      // the lowest-index cheapest worker (W > 32 or not: lane l's first is l)
      double bc = c[0];
      int best = lane;
      bool in = lane < W;
      if (lane + 32 < W && c[1] < bc) {
        bc = c[1];
        best = lane + 32;
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double oc = __shfl_xor_sync(FULL_MASK, bc, o);
        const int ob = __shfl_xor_sync(FULL_MASK, best, o);
        const bool oi = __shfl_xor_sync(FULL_MASK, in, o);
        if (oi && (!in || oc < bc || (oc == bc && ob < best))) {
          bc = oc;
          best = ob;
          in = true;
        }
      }
      const int wk = b.rec.worker[q];
      const double cw = __shfl_sync(FULL_MASK, wk < 32 ? c[0] : c[1], wk & 31);
      if (lane == 0) {
        asg[r] = best;
        atomicAdd(&S.counts[best], 1);
        num += b.rec.ttft[q];
        nst += cw;
        opt += bc;
      }
    }
    emax = __reduce_max_sync(FULL_MASK, emax);
    if (lane == 0) {
      atomicMax(&S.emax, emax);
      S.red[0][warp] = num;
      S.red[1][warp] = nst;
      S.red[2][warp] = opt;
    }
    __syncthreads();
    num = nst = opt = 0.0;
    for (int v = 0; v < NT_WIDE / 32; v++) {
      num += S.red[0][v];
      nst += S.red[1][v];
      opt += S.red[2][v];
    }
    if (__syncthreads_or(threadIdx.x < W && S.counts[threadIdx.x] > capw)) {
      double inv;
      const double scale = fx_scale(S.emax, FX_BITS_WIDE, &inv);
      long long* fx = reinterpret_cast<long long*>(cost);   // in place
      int32_t* list = b.wkey + base;   // (the keys are not needed past the sort)
      for (int64_t e = threadIdx.x; e < m * W; e += NT_WIDE)
        fx[e] = to_fx(cost[e], scale, FX_BITS_WIDE);
      if (threadIdx.x == 0) {
        int o = 0;
        for (int j = 0; j < W; j++) {
          S.dpos[j] = o;
          S.dfill[j] = 0;
          o += S.counts[j];
        }
      }
      for (int j = threadIdx.x; j < W; j += NT_WIDE) {
        wmin[j * W + j] = FX_INF;
        wrow[j * W + j] = -1;
      }
      __syncthreads();
      wide_rescan(S, wmin, wrow, fx, asg, list, m, W, W, nullptr, nullptr, true);
      for (;;) {
        // distances from the workers over their capacity, in Jacobi rounds
        const bool src = threadIdx.x < W && S.counts[threadIdx.x] > capw;
        if (threadIdx.x < W) {
          S.dist[threadIdx.x] = src ? 0 : FX_INF;
          S.pred[threadIdx.x] = -1;
        }
        if (!__syncthreads_or(src)) break;
        for (int it = 0; it < W; it++) {
          long long bv = FX_REAL;
          int bj = -1;
          if (k < W) {
#pragma unroll 4
            for (int j = g; j < W; j += WIDE_G) {
              const long long v = S.dist[j] + wmin[j * W + k];   // (<= 2 FX_INF)
              if (v < bv) {
                bv = v;
                bj = j;
              }
            }
          }
          S.pv[g][k] = bv;
          S.pi[g][k] = bj;
          __syncthreads();
          bool ch = false;
          if (g == 0 && k < W) {
            for (int h = 1; h < WIDE_G; h++)
              if (S.pv[h][k] < bv) {
                bv = S.pv[h][k];
                bj = S.pi[h][k];
              }
            if (bj >= 0 && bv < S.dist[k]) {
              S.dist[k] = bv;
              S.pred[k] = bj;
              ch = true;
            }
          }
          if (!__syncthreads_or(ch)) break;
        }
        if (warp == 0) {
          // target: the nearest worker with room (ties: lowest index)
          const bool r0 = lane < W && S.counts[lane] < capw && S.dist[lane] < FX_REAL;
          const bool r1 = lane + 32 < W && S.counts[lane + 32] < capw && S.dist[lane + 32] < FX_REAL;
          long long v0, v1;
          const int t0 = warp_argmin(r0 ? S.dist[lane] : 0, r0, &v0);
          const int t1 = warp_argmin(r1 ? S.dist[lane + 32] : 0, r1, &v1);
          const int tgt = t0 >= 0 && (t1 < 0 || v0 <= v1) ? t0 : (t1 >= 0 ? t1 + 32 : -1);
          for (int j = lane; j < W; j += 32) {
            S.dpos[j] = -1;
            S.dfill[j] = 0;
          }
          __syncwarp();
          if (lane == 0) {
            // walk the path back from its end: edge j -> kk moves the request
            // behind wrow[j][kk] from j to kk
            int kk = tgt, n = 0, o = 0;
            while (tgt >= 0 && n < W && S.pred[kk] >= 0) {
              const int j = S.pred[kk];
              const int r = wrow[j * W + kk];
              S.mv_j[n] = j;
              S.mv_k[n] = kk;
              S.mv_r[n++] = r;
              asg[r] = kk;
              kk = j;
            }
            if (n > 0) {
              S.counts[kk]--;
              S.counts[tgt]++;
            }
            for (int t = 0; t < n; t++) {   // (a path visits a worker once)
              const int j = S.mv_j[t];
              S.dpos[j] = o;
              o += S.counts[j];
            }
            S.nmv = n;
          }
        }
        __syncthreads();
        const int nmv = S.nmv;
        if (nmv == 0) break;   // (cannot happen: W capw >= m)
        wide_rescan(S, wmin, wrow, fx, asg, list, m, W, nmv, S.mv_j, S.mv_r, false);
        // requests that moved in lower their new worker's weights (a path
        // enters a worker once: the moves are independent)
        for (int t = g; t < nmv; t += WIDE_G) {
          const int to = S.mv_k[t], r = S.mv_r[t];
          if (k < W && k != to) {
            const long long v = fx[(int64_t)r * W + k] - fx[(int64_t)r * W + to];
            const long long o = wmin[to * W + k];
            if (v < o || (v == o && r < wrow[to * W + k])) {
              wmin[to * W + k] = v;
              wrow[to * W + k] = r;
            }
          }
        }
        __syncthreads();
      }
      const bool bad = __syncthreads_or(threadIdx.x < W && S.counts[threadIdx.x] > capw);
      opt = 0.0;
      for (int64_t r = threadIdx.x; r < m; r += NT_WIDE) opt += (double)fx[r * W + asg[r]] * inv;
      opt = warp_sum(opt);
      if (lane == 0) S.red[0][warp] = opt;
      __syncthreads();
      opt = 0.0;
      for (int v = 0; v < NT_WIDE / 32; v++) opt += S.red[0][v];
      if (bad) opt = __longlong_as_double(0x7FF8000000000000ll);
    }
    if (threadIdx.x == 0) {
      b.wnum[slot] = num;
      b.wstat[slot] = nst;
      b.wopt[slot] = opt;
      b.wcnt[slot] = m;
    }
    __syncthreads();   // (S is reused by the next window)
  }
}

// Whole-run PoA of every replica: one warp per replica, lane l summing windows
// l, l + 32, ... and the lanes' sums joined in a fixed order.
__global__ void __launch_bounds__(NT_POA) k_poa_total(int nprob, PoaBuffers b,
                                                      const PoaProblem* __restrict__ probs) {
  const int lane = threadIdx.x & 31;
  const int p = (int)(((int64_t)blockIdx.x * NT_POA + threadIdx.x) >> 5);
  if (p >= nprob) return;
  const PoaProblem pr = probs[p];
  const int64_t nw = b.nwin[p];
  double tn = 0.0, to = 0.0, ts = 0.0;
  for (int64_t w = lane; w < nw; w += 32) {
    tn += b.wnum[pr.win_base + w];
    to += b.wopt[pr.win_base + w];
    ts += b.wstat[pr.win_base + w];
  }
  tn = warp_sum(tn);
  to = warp_sum(to);
  ts = warp_sum(ts);
  if (lane != 0) return;
  double tot = __longlong_as_double(0x7FF8000000000000ll), tst = tot;
  if (nw >= 0) {
    tot = to > 0.0 ? tn / to : 0.0;
    tst = to > 0.0 ? ts / to : 0.0;
  }
  b.total[p] = tot;
  if (b.total_static) b.total_static[p] = tst;
  if (b.res) {
    b.res[p].poa_total = tot;
    b.res[p].poa_static = tst;
    b.res[p].n_windows = nw;
  }
}

static int sm_count() {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

cudaError_t launch_poa_keys(const PoaProblem* d_prob, int nprob, int64_t max_rows,
                            const rs_records& rec, double window, int32_t* wkey, long long* maxw,
                            cudaStream_t st) {
  if (nprob <= 0) return cudaSuccess;
  // as many row chunks as spread the problems over the whole GPU
  const int64_t chunks = (max_rows + NT_POA - 1) / NT_POA;
  int64_t split = (8 * sm_count() + nprob - 1) / nprob;
  split = split < chunks ? split : chunks;
  split = split < 1 ? 1 : (split > 65535 ? 65535 : split);
  if (maxw) {
    const cudaError_t e = cudaMemsetAsync(maxw, 0xFF, sizeof(long long) * (size_t)nprob, st);
    if (e != cudaSuccess) return e;
  }
  k_poa_keys<<<dim3(nprob, (unsigned)split), NT_POA, 0, st>>>(d_prob, rec, window, wkey, maxw);
  return cudaGetLastError();
}

cudaError_t launch_poa(const PoaProblem* d_prob, int nprob, const PoaBuffers& b,
                       const ModelConsts& mc, cudaStream_t st) {
  if (nprob <= 0) return cudaSuccess;
  const int sms = sm_count();
  // one large sorting CTA per SM while the problems do not fill the SMs
  const int nts = nprob <= sms ? POA_SORT_NT : 256;
  k_poa_sort<<<nprob, nts, POA_SORT_TAB * sizeof(uint32_t), st>>>(d_prob, b, mc.W);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  void (*kern)(const PoaProblem*, PoaBuffers, ModelConsts) =
      mc.W > POA_WMAX ? k_poa_solve_wide
      : mc.W == 3     ? k_poa_solve<3>
                      : (mc.W == 6 ? k_poa_solve<6> : k_poa_solve<POA_WMAX>);
  const bool wide = mc.W > POA_WMAX;
  const size_t smem = wide ? poa_wide_smem(mc.W) : 0;
  if (wide && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem)) != cudaSuccess)
    return e;
  if (b.wnext) {
    // one wave of CTAs that take the windows from the counter; few windows go
    // one to a CTA, so that each has an SM's integer and FP64 pipes to itself
    if ((e = cudaMemsetAsync(b.wnext, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
    const int nt = wide ? NT_WIDE : (b.nslots <= 4 * (int64_t)sms ? 32 : NT_SOLVE);
    const int wpc = wide ? 1 : nt / 32;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem)) != cudaSuccess)
      return e;
    int64_t gr = (b.nslots + wpc - 1) / wpc;
    const int64_t cap = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    gr = gr < cap ? gr : cap;
    kern<<<(unsigned)(gr > 0 ? gr : 1), nt, smem, st>>>(d_prob, b, mc);
  } else {
    // each problem's windows on its own CTAs, enough of them to fill the GPU
    int split = (4 * sms + nprob - 1) / nprob;
    kern<<<dim3(nprob, split), wide ? NT_WIDE : 32, smem, st>>>(d_prob, b, mc);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_poa_total<<<(nprob + NT_POA / 32 - 1) / (NT_POA / 32), NT_POA, 0, st>>>(nprob, b, d_prob);
  return cudaGetLastError();
}

}  // namespace rs
