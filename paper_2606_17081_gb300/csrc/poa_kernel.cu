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
// the window's largest cost: 55 significant bits of it at W <= 16, 53 above),
// so sums and comparisons are exact, no cycle is negative by rounding, and the
// integer units carry the serial chain (a dependent FP64 add costs 64 cycles).
// The assignment found is optimal for costs that differ from the window's by at
// most 2^-56 (2^-54) of its largest each.  OPT is the sum of that assignment's
// own costs, taken in two integer parts and rounded once (opt_add).
// Measured: poa_estimate on 20 000 records, W = 6 (81 windows): 4.22 -> 0.61 ms
// a call (keys 97 -> 5 us, sort and costs 1480 -> 17 us, solver 2941 -> 578 us,
// total 19 -> 6 us) with one warp per window, 0.42 ms with a CTA; the estimate
// of 16 replicas x 5000 requests at W = 64, 126 -> 10.7 ms.
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

// c_ij of §6.4; a prefix of 0 leaves f(n) - w_c 0 without the division (and,
// w_c being finite, f(n) itself).
__device__ __forceinline__ double frozen_cost(const ModelConsts& mc, const double* ftab, int nft,
                                              bool wc_finite, int nf, int m, int nbt) {
  const double f = nf < nft ? ftab[nf] : frozen_f(mc, nf);
  if (m == 0 || nbt <= 0) return wc_finite ? f : __dsub_rn(f, __dmul_rn(mc.w_c, 0.0));
  return __dsub_rn(f, __dmul_rn(mc.w_c, __ddiv_rn((double)m, (double)nbt)));
}

// Order-preserving map of a double onto int64 (NaN above all, -0 below +0): the
// comparisons run on the integer units.
__device__ __forceinline__ long long okey(double x) {
  const long long u = __double_as_longlong(x);
  return (u & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll ? 0x7FFFFFFFFFFFFFFFll
                                                            : u ^ ((u >> 63) & 0x7FFFFFFFFFFFFFFFll);
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
// largest cost, |value| <= 2^BITS, an edge weight is at most 2^(BITS + 1), and a
// path's weights (at most 15, or 63, of them) sum to less than FX_REAL.
constexpr long long FX_INF = 1ll << 61;    // no path / no row
constexpr long long FX_REAL = 1ll << 60;   // every finite distance is below
constexpr int FX_BITS = 55;                // W <= 16: 15 2^56 < 2^60
constexpr int FX_BITS_WIDE = 53;           // W <= 64: 63 2^54 < 2^60

// Biased exponent of a finite cost (0 for one that is not finite).
__device__ __forceinline__ int cost_exp(double c) {
  const int e = (int)((uint64_t)__double_as_longlong(c) >> 52) & 0x7FF;
  return e < 0x7FF ? e : 0;
}
// The scale 2^s that puts costs of biased exponent emax below 2^bits (s within
// the normal range: smaller costs than it covers round to 0).
__device__ __forceinline__ double fx_scale(int emax, int bits) {
  int s = bits - (emax - 1022);
  s = s > 1000 ? 1000 : (s < -1000 ? -1000 : s);
  return __longlong_as_double((long long)(1023 + s) << 52);
}
// A cost that is not finite: +infinity (a load at the pole of Eq. (9)) or NaN is
// FX_NONE, -infinity FX_NEG.  A row sits at its least cost first, so it is at an
// FX_NONE only if all its costs are, and has an FX_NEG only where it is at one; a
// move from a finite cost to an FX_NONE, or away from an FX_NEG, weighs more than
// FX_INF, that is, there is no such edge, and from like to like weighs 0.
constexpr long long FX_NONE = 1ll << 62;
constexpr long long FX_NEG = -(3ll << 60);

__device__ __forceinline__ long long to_fx(double c, double scale) {
  if (!(fabs(c) < __longlong_as_double(0x7FF0000000000000ll))) return c < 0.0 ? FX_NEG : FX_NONE;
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

// A row's cost at its worker in units of 2^(emax - 1084) (62 bits: emax is the
// largest biased exponent of the costs summed, all finite), rounded, in two
// parts of 31 bits: sums of either over a window's rows are exact.
__device__ __forceinline__ void opt_add(double c, int emax, long long& hi, long long& lo) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(c);
  const int e = (int)(u >> 52) & 0x7FF, sh = emax - (e ? e : 1);
  unsigned long long v = ((u & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull)) << 9;
  v = sh < 63 ? (v + (sh ? 1ull << (sh - 1) : 0ull)) >> sh : 0ull;
  const long long h = (long long)(v >> 31), l = (long long)(v & 0x7FFFFFFFull);
  hi += u >> 63 ? -h : h;
  lo += u >> 63 ? -l : l;
}

// The cost whose parts these are, with one rounding.
__device__ __forceinline__ double opt_value(long long hi, long long lo, int emax) {
  hi += lo >> 31;
  lo &= 0x7FFFFFFFll;
  const double d = (double)hi;
  const double r = d + ((double)(hi - (long long)d) + (double)lo * 0x1p-31);
  return scalbn(r, emax - 1084 + 31);
}

__device__ __forceinline__ long long warp_sum_int(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

constexpr int NT_SOLVE = 128;   // threads of a narrow solver CTA at one warp per window
constexpr int NW_SOLVE = 8;     // warps of a CTA that works on one window
constexpr int SOLVE_SROWS = 1024;   // rows whose assignment stays in shared memory
constexpr int SOLVE_SCOST = 4096;   // costs (rows x W) a CTA per window keeps there too (32 KB)

struct PoaWinShared {
  long long wmin[POA_WMAX][POA_WMAX];   // edge weights, FX_INF without a row
  int wrow[POA_WMAX][POA_WMAX];         // the request behind each
  int counts[POA_WMAX];
  int item[POA_WMAX * POA_WMAX];        // weights to look up again: 16 j + k
  int nitems, emax;
  uint8_t asg[SOLVE_SROWS];
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

// Weight j -> k from the requests now at j: min of c_qk - c_qj, ties to the
// lowest row (one warp).  fx is [W][m]: lanes over the rows read whole sectors.
// Rows go 256 at a time, eight per lane in flight.
__device__ __forceinline__ void poa_rescan(PoaWinShared& S, const long long* fx,
                                           const uint8_t* asg, int m, int j, int k, int lane) {
  constexpr int U = 8;
  const long long* ck = fx + (int64_t)k * m;
  const long long* cj = fx + (int64_t)j * m;
  long long best = FX_INF;
  int row = -1;
  for (int r0 = lane; r0 < m; r0 += 32 * U) {
    int at[U];
    long long v[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int r = r0 + 32 * u;
      at[u] = -1;
      v[u] = 0;
      if (r < m) {
        at[u] = asg[r];
        v[u] = ck[r] - cj[r];
      }
    }
#pragma unroll
    for (int u = 0; u < U; u++)
      if (at[u] == j && v[u] < best) {
        best = v[u];
        row = r0 + 32 * u;
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

// OPT of a solved window (a warp's or a CTA's): the sum of its rows' costs at their
// workers asg[r].  kept: those costs are still in b.cost; else they are computed
// again where the fixed point took their place.
template <int NWP>
__device__ __forceinline__ double narrow_opt(PoaWinShared& S, const PoaBuffers& b, const ModelConsts& mc,
                                          const double* ftab, bool wc_finite, double (*red)[NWP],
                                          int64_t rec_base, int64_t base, int m, const uint8_t* asg,
                                          bool kept) {
  constexpr int NT = 32 * NWP;
  const int lane = threadIdx.x & 31, ww = NWP == 1 ? 0 : (int)threadIdx.x >> 5, tid = 32 * ww + lane;
  const int W = mc.W, nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  double* cost = b.cost + base * W;   // [W][m]
  int ex = 1;
  for (int r = tid; r < m; r += NT) {
    const int j = asg[r];
    double* at = cost + (int64_t)j * m + r;
    if (!kept) {
      const int64_t q = rec_base + b.order[base + r];
      *at = frozen_cost(mc, ftab, nft, wc_finite, b.rec.n_frozen[q * W + j], b.rec.prefix[q * W + j],
                        b.rec.nbt[q]);
    }
    ex = max(ex, (int)(__double_as_longlong(*at) >> 52) & 0x7FF);
  }
  ex = __reduce_max_sync(FULL_MASK, ex);
  if (NWP > 1) {
    if (tid == 0) S.emax = 0;
    __syncthreads();
    if (lane == 0) atomicMax(&S.emax, ex);
    __syncthreads();
    ex = S.emax;
  }
  long long hi = 0, lo = 0;
  double opt = 0.0;
  for (int r = tid; r < m; r += NT) {
    const double c = cost[(int64_t)asg[r] * m + r];
    if (ex < 0x7FF) opt_add(c, ex, hi, lo); else opt += c;
  }
  hi = warp_sum_int(hi);
  lo = warp_sum_int(lo);
  if (ex == 0x7FF) opt = warp_sum(opt);
  if (NWP > 1) {
    if (lane == 0) {
      red[0][ww] = __longlong_as_double(hi);
      red[1][ww] = __longlong_as_double(lo);
      red[2][ww] = opt;
    }
    __syncthreads();
    hi = lo = 0;
    opt = 0.0;
    for (int q = 0; q < NWP; q++) {
      hi += __double_as_longlong(red[0][q]);
      lo += __double_as_longlong(red[1][q]);
      opt += red[2][q];
    }
    __syncthreads();
  }
  return ex < 0x7FF ? opt_value(hi, lo, ex) : opt;
}

// The same out of line, for a window per CTA: with it in the kernel's body the
// augmentations took 2% more time.
template <int NWP>
__device__ __noinline__ double narrow_opt_out(PoaWinShared& S, const PoaProblem* __restrict__ probs,
                                              const PoaBuffers& b, const ModelConsts& mc,
                                              const double* ftab, double (*red)[NWP], int pi, int64_t w,
                                              int m, const uint8_t* asg, bool kept) {
  const PoaProblem pr = probs[pi];
  const int64_t base = pr.scratch_base + b.wstart[pr.win_base + pi + w];
  return narrow_opt<NWP>(S, b, mc, ftab, __dmul_rn(mc.w_c, 0.0) == 0.0, red, pr.rec_base, base, m, asg,
                         kept);
}

// WT: a compile-time bound on W (the exact W for the common 3 and 6, else
// POA_WMAX), so that the unrolled per-worker loops hold no dead iterations:
// the solver's warps run different phases at once and its code must stay
// small for the instruction cache.
// NWP: warps working on a window.  One when there are windows enough to fill
// the GPU; NW_SOLVE (a CTA per window) when there are few and the launch waits
// for its longest chain of augmentations: the warps then share the rows and
// look up an augmentation's weights at the same time, while warp 0 runs the
// path, and the window's costs sit in shared memory.  (poa_estimate on 20 000
// records at W = 6, 81 windows of about 250 requests, 200 of them past a
// capacity: 0.61 ms a call at one warp per window, 0.43 ms so.)
template <int WT, int NWP>
__global__ void __launch_bounds__(NWP == 1 ? NT_SOLVE : 32 * NWP)
    k_poa_solve(const PoaProblem* __restrict__ probs, PoaBuffers b, ModelConsts mc) {
  constexpr int WPC = NWP == 1 ? NT_SOLVE / 32 : 1;   // windows of a CTA
  constexpr int NT = 32 * NWP;                        // threads of a window
  __shared__ PoaWinShared P[WPC];
  __shared__ long long s_fx[NWP == 1 ? 1 : SOLVE_SCOST];
  __shared__ double ftab[POA_FTAB];
  __shared__ double red[3][NWP];
  __shared__ int64_t s_w;
  __shared__ int s_pi;
  fill_ftab(mc, ftab);
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  const bool wc_finite = __dmul_rn(mc.w_c, 0.0) == 0.0;
  const int W = mc.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ww = NWP == 1 ? 0 : warp;                 // warp of the window
  const int tid = ww * 32 + lane;
  PoaWinShared& S = P[NWP == 1 ? warp : 0];
  auto sync = [] {
    if (NWP == 1) __syncwarp(); else __syncthreads();
  };
  // a sum over the window's threads, in a fixed order (every thread gets it)
  auto sum3 = [&](double& x, double& y, double& z) {
    x = warp_sum(x);
    y = warp_sum(y);
    z = warp_sum(z);
    if (NWP > 1) {
      if (lane == 0) { red[0][ww] = x; red[1][ww] = y; red[2][ww] = z; }
      __syncthreads();
      // (a tree again: three roundings instead of eight, a third of the FP64)
      static_assert((NWP & (NWP - 1)) == 0, "a power of two of warps");
      x = red[0][lane & (NWP - 1)];
      y = red[1][lane & (NWP - 1)];
      z = red[2][lane & (NWP - 1)];
#pragma unroll
      for (int o = NWP / 2; o > 0; o >>= 1) {
        x += __shfl_xor_sync(FULL_MASK, x, o);
        y += __shfl_xor_sync(FULL_MASK, y, o);
        z += __shfl_xor_sync(FULL_MASK, z, o);
      }
      __syncthreads();
    }
  };
  int64_t next = (int64_t)blockIdx.y * WPC + (NWP == 1 ? warp : 0);
  const int64_t stride = (int64_t)gridDim.y * WPC;
  for (;;) {
    // (a problem whose windows overflowed: k_poa_total reports it)
    int pi = -1;
    int64_t w = 0;
    if (ww == 0 && !poa_next(probs, b, lane, next, stride, &pi, &w)) pi = -1;
    if (NWP > 1) {
      if (threadIdx.x == 0) { s_pi = pi; s_w = w; }
      __syncthreads();
      pi = s_pi;
      w = s_w;
    }
    if (pi < 0) return;
    const PoaProblem pr = probs[pi];
    const int64_t* wst = b.wstart + pr.win_base + pi;
    const int64_t s0 = wst[w];
    const int m = (int)(wst[w + 1] - s0);
    const int64_t base = pr.scratch_base + s0;   // window rows in order[], asg[]
    const int64_t slot = pr.win_base + w;
    int capw = (m + W - 1) / W;
    if (capw < mc.cap) capw = mc.cap;
    if (tid < W) S.counts[tid] = 0;
    if (tid == 0) S.emax = 0;
    sync();
    double* cost = b.cost + base * W;   // [W][m]
    uint8_t* asg = m <= SOLVE_SROWS ? S.asg : reinterpret_cast<uint8_t*>(b.asg + base);
    double num = 0.0, nst = 0.0, opt = 0.0;
    int emax = 0;
    for (int r = tid; r < m; r += NT) {
      const int64_t q = pr.rec_base + b.order[base + r];
      const int nbt = b.rec.nbt[q], wk = b.rec.worker[q];
      const uint16_t* nfr = b.rec.n_frozen + q * W;
      const uint16_t* pre = b.rec.prefix + q * W;
      double bc = 0.0, cw = 0.0;
      long long bk = 0;
      int best = 0;
#pragma unroll
      for (int j = 0; j < WT; j++) {
        if (j < W) {
          const double c = frozen_cost(mc, ftab, nft, wc_finite, nfr[j], pre[j], nbt);
          const long long ck = okey(c);
          cost[(int64_t)j * m + r] = c;
          if (j == 0 || ck < bk) { bk = ck; bc = c; best = j; }
          if (j == wk) cw = c;
          const int e = cost_exp(c);
          emax = e > emax ? e : emax;
        }
      }
      nst += cw;   // the realized assignment's frozen cost
      asg[r] = (uint8_t)best;
      atomicAdd(&S.counts[best], 1);
      num += b.rec.ttft[q];
      opt += bc;
    }
    emax = __reduce_max_sync(FULL_MASK, emax);
    if (lane == 0) atomicMax(&S.emax, emax);
    sync();
    sum3(num, nst, opt);
    int count = lane < W ? S.counts[lane] : 0;   // lane j of warp 0 keeps worker j's load
    if (__any_sync(FULL_MASK, lane < W && count > capw)) {   // (every warp alike)
      const double scale = fx_scale(S.emax, FX_BITS);
      long long* fx = NWP > 1 && (int64_t)m * W <= SOLVE_SCOST ? s_fx
                                                                : reinterpret_cast<long long*>(cost);
      for (int64_t e = tid; e < (int64_t)m * W; e += NT) fx[e] = to_fx(cost[e], scale);
      if (tid < W) {
        S.wmin[tid][tid] = FX_INF;
        S.wrow[tid][tid] = -1;
      }
      sync();
      for (int e = ww; e < W * W; e += NWP)
        if (e / W != e % W) poa_rescan(S, fx, asg, m, e / W, e % W, lane);
      sync();
      for (;;) {
        int nmv = 0, mk = -1, mr = -1;
        if (ww == 0) {
          // distances from the workers over their capacity, in Jacobi rounds:
          // lane k < W owns target k and every round reads the previous one's
          // distances (shortest paths have at most W - 1 edges)
          const bool src = lane < W && count > capw;
          int pk = -1, tgt = -1;
          long long dk = src ? 0 : FX_INF, dt;
          if (__any_sync(FULL_MASK, src)) {
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
            tgt = warp_argmin(dk, lane < W && count < capw && dk < FX_REAL, &dt);
          }
          // walk the path back from its end: each edge j -> k moves the
          // request behind wrow[j][k] from j to k; lane t keeps step t.  A
          // worker that loses a request: the weights whose minimum it was go
          // to the list
          int k = tgt, ni = 0;
          for (; tgt >= 0 && nmv < W; nmv++) {
            const int j = __shfl_sync(FULL_MASK, pk, k);
            if (j < 0) break;
            const int r = S.wrow[j][k];
            if (lane == nmv) {
              mk = k;
              mr = r;
            }
            const bool need = lane < W && lane != j && S.wrow[j][lane] == r;
            const unsigned nm = __ballot_sync(FULL_MASK, need);
            if (need) S.item[ni + __popc(nm & ((1u << lane) - 1u))] = j * POA_WMAX + lane;
            ni += __popc(nm);
            k = j;
          }
          if (tgt >= 0 && lane == k) count--;
          if (tgt >= 0 && lane == tgt) count++;
          if (lane < nmv) asg[mr] = (uint8_t)mk;
          if (lane == 0) S.nitems = ni;
        }
        sync();
        const int ni = S.nitems;
        if (ni == 0) break;   // no worker over its capacity is left (a path has items)
        for (int e = ww; e < ni; e += NWP)
          poa_rescan(S, fx, asg, m, S.item[e] / POA_WMAX, S.item[e] % POA_WMAX, lane);
        sync();
        // requests that moved in lower their new worker's weights
        if (ww == 0) {
          for (int t = 0; t < nmv; t++) {
            const int to = __shfl_sync(FULL_MASK, mk, t), r = __shfl_sync(FULL_MASK, mr, t);
            if (lane < W && lane != to) {
              const long long v = fx[(int64_t)lane * m + r] - fx[(int64_t)to * m + r];
              const long long o = S.wmin[to][lane];
              if (v < o || (v == o && r < S.wrow[to][lane])) {
                S.wmin[to][lane] = v;
                S.wrow[to][lane] = r;
              }
            }
          }
          __syncwarp();
        }
      }
      // (W capw >= m: a load past its capacity is left only where every way out
      // costs infinity)
      const bool bad = ww == 0 && __any_sync(FULL_MASK, lane < W && count > capw);
      if constexpr (NWP > 1)
        opt = narrow_opt_out<NWP>(S, probs, b, mc, ftab, red, pi, w, m, asg, fx == s_fx);
      else
        opt = narrow_opt<NWP>(S, b, mc, ftab, wc_finite, red, pr.rec_base, base, m, asg, false);
      if (bad) opt = __longlong_as_double(0x7FF0000000000000ll);
    }
    if (tid == 0) {
      b.wnum[slot] = num;
      b.wstat[slot] = nst;
      b.wopt[slot] = opt;
      b.wcnt[slot] = m;
    }
    sync();   // (S is reused by the next window)
  }
}

// The same OPT for W > POA_WMAX workers, one CTA of 32 warps per window: few
// windows, each of hundreds to thousands of requests, so the latency of one
// augmentation is what counts, and a window's weights (52 KB), its requests by
// worker and each request's cost at its worker stay in shared memory.  Per
// augmentation: Jacobi rounds relax the edges out of the sources that changed
// in the round before, thread (g, k) those of sources 4 g .. 4 g + 3 into target
// k, and a thread per target joins the groups; warp 0 walks the path and moves
// its requests between the workers' lists; the weights that lost their minimum
// are listed, and a warp looks up one of them, or a part of one while there
// are fewer than warps, lanes over its worker's requests.  (16 replicas x 5000
// requests with 1024 in flight, windows of 950 to 1450 rows with 450 to 1070 to
// move: 10.6 ms; with 8 warps and a quarter of the sources per thread it took 2.6
// times as long.  A round costs about 500 cycles, of 6 per augmentation.)
constexpr int NT_WIDE = 1024;
constexpr int NW_WIDE = NT_WIDE / 32;
constexpr int WIDE_G = NT_WIDE / POA_WMAX_WIDE;            // source groups of a round
constexpr int WIDE_GS = POA_WMAX_WIDE / WIDE_G;            // sources of a group
constexpr int WIDE_SROWS = 4096;   // rows of a window whose lists fit in shared memory
// list entries then: every worker's list holds max(its first load, capacity)
// rows, in all at most rows + max(64 W, rows + W)
constexpr int WIDE_SLIST = 2 * WIDE_SROWS + POA_WMAX_WIDE;
static_assert(NW_WIDE == 32, "a lane per warp joins the warps' sums");

struct PoaWideShared {
  long long dist[POA_WMAX_WIDE];
  long long pv[WIDE_G][POA_WMAX_WIDE];   // a round: best way into each target from each group
  uint8_t pj[WIDE_G][POA_WMAX_WIDE];     // ... and its source
  long long part_v[NW_WIDE];             // a weight's parts
  int part_r[NW_WIDE];
  unsigned act[2];                       // sources that changed in the last round
  double red[3][NW_WIDE];
  double ftab[POA_FTAB];
  int32_t* list[POA_WMAX_WIDE];          // each worker's requests
  int pred[POA_WMAX_WIDE], counts[POA_WMAX_WIDE], fill[POA_WMAX_WIDE];
  int path[POA_WMAX_WIDE + 1];           // workers from the target back to the source
  int mv_r[POA_WMAX_WIDE];               // the request moved from path[t + 1] to path[t]
  int nmv, nitems, emax, pi_next, q_first, q_last;
  int64_t w_next;
};

// Row stride of the weights, stored [target][source] and odd: lanes over the
// sources of one target, or over the targets of one source, hit other banks.
__host__ __device__ inline int wide_ld(int W) { return W | 1; }
__host__ __device__ inline size_t poa_wide_smem(int W) {
  return (size_t)W * wide_ld(W) * 12 + (size_t)WIDE_SROWS * 12 + (size_t)WIDE_SLIST * 4 +
         (size_t)W * W * 2 + 8;
}

// Weight j -> k over part `part` of `parts` of worker j's n requests: min of
// c_qk - c_qj, ties to the lowest row (one warp; row -1: no request there).
// rows NULL: the requests r < n with pos[r] == j.  cur: the requests' costs at
// their workers, or NULL (then read from fx).
__device__ __forceinline__ void wide_weight(const int32_t* rows, const int32_t* pos, int n,
                                            const long long* fx, const long long* cur, int W, int j,
                                            int k, int part, int parts, int lane, long long* least,
                                            int* lrow) {
  constexpr int U = 4;
  long long best = FX_INF;
  int row = -1;
  for (int t0 = part * 32 * U + lane; t0 < n; t0 += parts * 32 * U) {
    int rr[U];
    long long v[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int t = t0 + 32 * u;
      rr[u] = -1;
      if (t < n) rr[u] = rows ? rows[t] : (pos[t] == j ? t : -1);
      v[u] = 0;
      if (rr[u] >= 0) {
        const long long* cr = fx + (int64_t)rr[u] * W;
        v[u] = cr[k] - (cur ? cur[rr[u]] : cr[j]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; u++)
      if (rr[u] >= 0 && (v[u] < best || (v[u] == best && rr[u] < row))) {
        best = v[u];
        row = rr[u];
      }
  }
  warp_argmin(best, row >= 0, least);
  const bool mine = row >= 0 && best == *least;
  *lrow = (int)__reduce_min_sync(FULL_MASK, mine ? (unsigned)row : 0xFFFFFFFFu);
  if (*lrow < 0) *least = FX_INF;
}

// OPT of a solved window: the sum of its rows' costs at their workers pos[r].  The
// costs are computed again where the fixed point took their place.  Out of line:
// with this in the kernel's body its loops took 5% more time.
// Where the lists took the place of the window's rows in order[], S.q_first ..
// S.q_last are the rows between its first and its last (else none).
__device__ __noinline__ double wide_opt(PoaWideShared& S, const PoaProblem* __restrict__ probs,
                                        const PoaBuffers& b, const ModelConsts& mc, int m,
                                        const int32_t* pos) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = mc.W;
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  const bool wc_finite = __dmul_rn(mc.w_c, 0.0) == 0.0;
  const int64_t rec_base = probs[S.pi_next].rec_base, w = S.w_next;
  const int64_t base = probs[S.pi_next].scratch_base + b.wstart[probs[S.pi_next].win_base + S.pi_next + w];
  double* cost = b.cost + base * W;   // [m][W]
  const int q_first = S.q_first, q_last = S.q_last;
  // those of them that complete in the window, in order
  int have = 0;
  for (int q0 = q_first; q0 <= q_last; q0 += NT_WIDE) {
    const int q = q0 + (int)threadIdx.x;
    bool in = q <= q_last;
    if (in) {
      const int64_t r = rec_base + q;
      in = b.rec.worker[r] >= 0 &&
           floor(__ddiv_rn(b.rec.completion[r], mc.poa_window)) == (double)w;
    }
    const unsigned mk = __ballot_sync(FULL_MASK, in);
    if (lane == 0) S.part_r[warp] = __popc(mk);
    __syncthreads();
    const int n = S.part_r[lane];
    const int below = (int)__reduce_add_sync(FULL_MASK, (unsigned)(lane < warp ? n : 0));
    if (in) b.order[base + have + below + __popc(mk & ((1u << lane) - 1u))] = q;
    have += (int)__reduce_add_sync(FULL_MASK, (unsigned)n);
    __syncthreads();
  }
  int ex = 1;
  for (int r = threadIdx.x; r < m; r += NT_WIDE) {
    const int64_t q = rec_base + b.order[base + r];
    const int j = pos[r];
    const double c = frozen_cost(mc, S.ftab, nft, wc_finite, b.rec.n_frozen[q * W + j],
                                 b.rec.prefix[q * W + j], b.rec.nbt[q]);
    cost[(int64_t)r * W + j] = c;
    ex = max(ex, (int)(__double_as_longlong(c) >> 52) & 0x7FF);
  }
  ex = __reduce_max_sync(FULL_MASK, ex);
  if (threadIdx.x == 0) S.emax = 0;
  __syncthreads();
  if (lane == 0) atomicMax(&S.emax, ex);
  __syncthreads();
  ex = S.emax;
  long long hi = 0, lo = 0;
  double opt = 0.0;
  for (int r = threadIdx.x; r < m; r += NT_WIDE) {
    const double c = cost[(int64_t)r * W + pos[r]];
    if (ex < 0x7FF) opt_add(c, ex, hi, lo); else opt += c;
  }
  hi = warp_sum_int(hi);
  lo = warp_sum_int(lo);
  opt = warp_sum(opt);
  if (lane == 0) {
    S.red[0][warp] = __longlong_as_double(hi);
    S.red[1][warp] = __longlong_as_double(lo);
    S.red[2][warp] = opt;
  }
  __syncthreads();
  hi = warp_sum_int(__double_as_longlong(S.red[0][lane]));
  lo = warp_sum_int(__double_as_longlong(S.red[1][lane]));
  return ex < 0x7FF ? opt_value(hi, lo, ex) : warp_sum(S.red[2][lane]);
}

__global__ void __launch_bounds__(NT_WIDE) k_poa_solve_wide(const PoaProblem* __restrict__ probs,
                                                            PoaBuffers b, ModelConsts mc) {
  extern __shared__ __align__(16) unsigned char wsm[];
  __shared__ PoaWideShared S;
  const int W = mc.W, ld = wide_ld(W);
  long long* wmin = reinterpret_cast<long long*>(wsm);               // [target][source]
  long long* s_cur = wmin + (size_t)W * ld;
  int* wrow = reinterpret_cast<int*>(s_cur + WIDE_SROWS);
  int32_t* s_pos = wrow + (size_t)W * ld;
  int32_t* s_list = s_pos + WIDE_SROWS;
  uint16_t* item = reinterpret_cast<uint16_t*>(s_list + WIDE_SLIST);   // 64 j + k
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  fill_ftab(mc, S.ftab);
  const int nft = mc.cap < POA_FTAB ? mc.cap : POA_FTAB;
  const bool wc_finite = __dmul_rn(mc.w_c, 0.0) == 0.0;
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
    if (threadIdx.x < W) S.counts[threadIdx.x] = 0;
    __syncthreads();
    const int pi = S.pi_next;
    if (pi < 0) return;
    const int64_t w = S.w_next;
    const PoaProblem pr = probs[pi];
    const int64_t* wst = b.wstart + pr.win_base + pi;
    const int64_t s0 = wst[w];
    const int m = (int)(wst[w + 1] - s0);
    const int64_t base = pr.scratch_base + s0;
    const int64_t slot = pr.win_base + w;
    int capw = (m + W - 1) / W;
    if (capw < mc.cap) capw = mc.cap;
    double* cost = b.cost + base * W;   // [m][W]
    const bool in_smem = m <= WIDE_SROWS && capw <= WIDE_SROWS / W;
    // lists fit: in shared memory, or in the window's order[] and wkey[], not
    // needed past the sums below (the full workers' lists, m rows at most, in
    // the one, the others' capacities in the other).  They do not when a large
    // C_j leaves the workers room for several times the window's rows; a
    // worker's requests are then found by scanning the rows
    const bool listed = in_smem || (int64_t)(W - 1) * capw <= m;
    // a row's worker; once the lists are built, its position in its list
    int32_t* pos = in_smem ? s_pos : b.asg + base;
    // costs and cheapest workers, one warp per request (lane: workers lane, lane + 32)
    double num = 0.0, nst = 0.0, opt = 0.0;
    int emax = 0;
    for (int r = warp; r < m; r += NW_WIDE) {
      const int64_t q = pr.rec_base + b.order[base + r];
      const int nbt = b.rec.nbt[q];
      double c[2];
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int j = lane + 32 * h;
        c[h] = 0.0;
        if (j < W) {
          c[h] = frozen_cost(mc, S.ftab, nft, wc_finite, b.rec.n_frozen[q * W + j],
                             b.rec.prefix[q * W + j], nbt);
          cost[(int64_t)r * W + j] = c[h];
          const int e = cost_exp(c[h]);
          emax = e > emax ? e : emax;
        }
      }
      // the lowest-index cheapest worker: the lower half's on a tie
      long long k0, k1;
      const int b0 = warp_argmin(okey(c[0]), lane < W, &k0);
      const int b1 = warp_argmin(okey(c[1]), lane + 32 < W, &k1);
      const int best = b1 >= 0 && k1 < k0 ? b1 + 32 : b0;
      const double bc = __shfl_sync(FULL_MASK, best < 32 ? c[0] : c[1], best & 31);
      const int wk = b.rec.worker[q];
      const double cw = __shfl_sync(FULL_MASK, wk < 32 ? c[0] : c[1], wk & 31);
      if (lane == 0) {
        pos[r] = best;
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
    num = warp_sum(S.red[0][lane]);   // (NW_WIDE == 32: a lane per warp)
    nst = warp_sum(S.red[1][lane]);
    opt = warp_sum(S.red[2][lane]);
    if (__syncthreads_or(threadIdx.x < W && S.counts[threadIdx.x] > capw)) {
      const double scale = fx_scale(S.emax, FX_BITS_WIDE);
      long long* fx = reinterpret_cast<long long*>(cost);   // in place
      if (threadIdx.x == 0) {
        S.q_first = listed && !in_smem ? b.order[base] : 0;
        S.q_last = listed && !in_smem ? b.order[base + m - 1] : -1;
      }
      for (int64_t e = threadIdx.x; e < (int64_t)m * W; e += NT_WIDE)
        fx[e] = to_fx(cost[e], scale);
      // room for a worker's first load or, below it, its capacity
      if (threadIdx.x == 0) {
        int32_t *over = in_smem ? s_list : b.order + base, *under = b.wkey + base;
        for (int j = 0; j < W; j++) {
          S.fill[j] = 0;
          if (in_smem || S.counts[j] >= capw) {
            S.list[j] = over;
            over += S.counts[j] > capw ? S.counts[j] : capw;
          } else {
            S.list[j] = under;
            under += capw;
          }
        }
      }
      if (threadIdx.x < W) {
        wmin[threadIdx.x * ld + threadIdx.x] = FX_INF;
        wrow[threadIdx.x * ld + threadIdx.x] = -1;
      }
      __syncthreads();
      long long* cur = in_smem ? s_cur : nullptr;
      for (int r = threadIdx.x; listed && r < m; r += NT_WIDE) {
        const int j = pos[r];
        const int p = atomicAdd(&S.fill[j], 1);
        S.list[j][p] = r;
        pos[r] = p;
        if (cur) cur[r] = fx[(int64_t)r * W + j];
      }
      __syncthreads();
      // every weight: a warp per worker, lanes over the targets
      for (int j = warp; j < W; j += NW_WIDE) {
        const int32_t* rows = S.list[j];
        const int n = listed ? S.counts[j] : m;
        long long best[2] = {FX_INF, FX_INF};
        int row[2] = {-1, -1};
        for (int t0 = 0; t0 < n; t0 += 4) {
          int rr[4];
          long long c[4][3];
#pragma unroll
          for (int u = 0; u < 4; u++) {
            rr[u] = -1;
            if (t0 + u < n) rr[u] = listed ? rows[t0 + u] : (pos[t0 + u] == j ? t0 + u : -1);
            const long long* cr = fx + (int64_t)(rr[u] < 0 ? 0 : rr[u]) * W;
            c[u][0] = lane < W ? cr[lane] : 0;
            c[u][1] = lane + 32 < W ? cr[lane + 32] : 0;
            c[u][2] = cr[j];
          }
#pragma unroll
          for (int u = 0; u < 4; u++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
              const long long v = c[u][h] - c[u][2];
              if (rr[u] >= 0 && (v < best[h] || (v == best[h] && rr[u] < row[h]))) {
                best[h] = v;
                row[h] = rr[u];
              }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int q = lane + 32 * h;
          if (q < W && q != j) {
            wmin[q * ld + j] = best[h];
            wrow[q * ld + j] = row[h];
          }
        }
      }
      for (;;) {
        // distances from the workers over their capacity, in Jacobi rounds:
        // every round reads the previous one's distances and relaxes the edges
        // out of the sources that changed in it (an edge out of another was
        // tested against a distance that has only fallen since)
        if (threadIdx.x < POA_WMAX_WIDE) {
          const bool src = threadIdx.x < W && S.counts[threadIdx.x] > capw;
          S.dist[threadIdx.x] = src ? 0 : FX_INF;
          S.pred[threadIdx.x] = -1;
          const unsigned bal = __ballot_sync(FULL_MASK, src);
          if (lane == 0) S.act[warp] = bal;
        }
        if (threadIdx.x == 0) S.nitems = 0;
        __syncthreads();
        uint64_t act = (uint64_t)S.act[0] | ((uint64_t)S.act[1] << 32);
        if (act == 0) break;
        const int k = threadIdx.x & (POA_WMAX_WIDE - 1), g = threadIdx.x / POA_WMAX_WIDE;
        for (int it = 0; it < W && act; it++) {
          const unsigned mine = (unsigned)(act >> (WIDE_GS * g)) & ((1u << WIDE_GS) - 1u);
          long long bv = FX_REAL;
          int bj = 0;
          if (mine && k < W) {   // (mine is alike in the warp)
            long long v[WIDE_GS];
#pragma unroll
            for (int q = 0; q < WIDE_GS; q++) {
              const int j = WIDE_GS * g + q < W ? WIDE_GS * g + q : W - 1;
              v[q] = S.dist[j] + wmin[k * ld + j];   // (<= 2 FX_INF)
            }
#pragma unroll
            for (int q = 0; q < WIDE_GS; q++)
              if ((mine >> q & 1u) && v[q] < bv) {
                bv = v[q];
                bj = WIDE_GS * g + q;
              }
          }
          S.pv[g][k] = bv;
          S.pj[g][k] = (uint8_t)bj;
          __syncthreads();
          if (threadIdx.x < POA_WMAX_WIDE) {
            // (sources in increasing order: ties keep the lowest)
            long long v[WIDE_G];
#pragma unroll
            for (int q = 0; q < WIDE_G; q++) v[q] = S.pv[q][k];
            const long long d = S.dist[k];
            long long nv = d < FX_REAL ? d : FX_REAL;
            int from = -1;
#pragma unroll
            for (int q = 0; q < WIDE_G; q++)
              if (v[q] < nv) {
                nv = v[q];
                from = q;
              }
            const bool ch = from >= 0 && k < W;
            if (ch) {
              S.dist[k] = nv;
              S.pred[k] = S.pj[from][k];
            }
            const unsigned bal = __ballot_sync(FULL_MASK, ch);
            if (lane == 0) S.act[warp] = bal;
          }
          __syncthreads();
          act = (uint64_t)S.act[0] | ((uint64_t)S.act[1] << 32);
        }
        if (warp == 0) {
          // target: the nearest worker with room (ties: lowest index)
          const long long d0 = lane < W ? S.dist[lane] : FX_INF;
          const long long d1 = lane + 32 < W ? S.dist[lane + 32] : FX_INF;
          const bool r0 = lane < W && S.counts[lane] < capw && d0 < FX_REAL;
          const bool r1 = lane + 32 < W && S.counts[lane + 32] < capw && d1 < FX_REAL;
          long long v0, v1;
          const int t0 = warp_argmin(d0, r0, &v0);
          const int t1 = warp_argmin(d1, r1, &v1);
          const int tgt = t0 >= 0 && (t1 < 0 || v0 <= v1) ? t0 : (t1 >= 0 ? t1 + 32 : -1);
          // the path back from its end (it visits a worker once)
          int at = tgt, n = 0;
          while (tgt >= 0 && n < W) {
            if (lane == 0) S.path[n] = at;
            const int j = S.pred[at];
            if (j < 0) break;
            n++;
            at = j;
          }
          __syncwarp();
          // step t moves the request behind the edge path[t + 1] -> path[t]
          for (int t = lane; t < n; t += 32) S.mv_r[t] = wrow[S.path[t] * ld + S.path[t + 1]];
          __syncwarp();
          // path[t], 0 < t < n, loses request mv_r[t - 1] and gains mv_r[t], which
          // takes the lost one's place; the source's last request fills its
          // gap; the target's list grows
          int sl[2] = {0, 0};
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const int t = lane + 32 * u;
            if (listed && t >= 1 && t <= n) sl[u] = pos[S.mv_r[t - 1]];
          }
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const int t = lane + 32 * u;
            if (n > 0 && t <= n) {
              const int j = S.path[t];
              int32_t* rows = S.list[j];
              if (!listed) {
                if (t < n) pos[S.mv_r[t]] = j;
                if (t == 0) S.counts[j]++;
                if (t == n) S.counts[j]--;
              } else if (t == n) {
                const int last = S.counts[j] - 1;
                const int x = rows[last];
                rows[sl[u]] = x;
                if (x != S.mv_r[t - 1]) pos[x] = sl[u];
                S.counts[j] = last;
              } else {
                const int x = S.mv_r[t];
                const int p = t == 0 ? S.counts[j] : sl[u];
                rows[p] = x;
                pos[x] = p;
                if (t == 0) S.counts[j] = p + 1;
              }
            }
          }
          if (lane == 0) S.nmv = n;
        }
        __syncthreads();
        const int nmv = S.nmv;
        if (nmv == 0) break;   // every way out costs infinity (W capw >= m)
        // warp t (and t + 32 on a longer path): the weights out of path[t + 1]
        // whose minimum moved away are listed; the moved request's costs beside
        // the one at its new worker are loaded for the end of the step
        long long in_v[2][2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int t = warp + 32 * u;
          if (t < nmv) {
            const int to = S.path[t], j = S.path[t + 1], r = S.mv_r[t];
            const long long ct = fx[(int64_t)r * W + to];
            if (cur && lane == 0) cur[r] = ct;
#pragma unroll
            for (int h = 0; h < 2; h++) {
              const int q = lane + 32 * h;
              in_v[u][h] = FX_INF;
              if (q < W) {
                if (q != to) in_v[u][h] = fx[(int64_t)r * W + q] - ct;
                if (q != j && wrow[q * ld + j] == r)
                  item[atomicAdd(&S.nitems, 1)] = (uint16_t)(j * POA_WMAX_WIDE + q);
              }
            }
          }
        }
        __syncthreads();
        const int ni = S.nitems;
        // fewer weights than warps: each in `parts` parts
        const int parts = ni <= NW_WIDE / 8 ? 8 : (ni <= NW_WIDE / 4 ? 4 : (ni <= NW_WIDE / 2 ? 2 : 1));
        for (int e = warp; e < ni * parts; e += NW_WIDE) {
          const int x = item[e / parts], j = x / POA_WMAX_WIDE, q = x % POA_WMAX_WIDE;
          long long v;
          int r;
          wide_weight(listed ? S.list[j] : nullptr, pos, listed ? S.counts[j] : m, fx, cur, W, j, q,
                      e % parts, parts, lane, &v, &r);
          if (lane == 0) {
            if (parts == 1) {
              wmin[q * ld + j] = v;
              wrow[q * ld + j] = r;
            } else {   // (one round: ni parts <= 32)
              S.part_v[e] = v;
              S.part_r[e] = r;
            }
          }
        }
        __syncthreads();
        if (parts > 1) {
          if (threadIdx.x < ni) {
            long long v = FX_INF;
            int r = -1;
            for (int p = 0; p < parts; p++) {
              const long long pv = S.part_v[threadIdx.x * parts + p];
              const int pr2 = S.part_r[threadIdx.x * parts + p];
              if (pr2 >= 0 && (r < 0 || pv < v || (pv == v && pr2 < r))) {
                v = pv;
                r = pr2;
              }
            }
            const int x = item[threadIdx.x], j = x / POA_WMAX_WIDE, q = x % POA_WMAX_WIDE;
            wmin[q * ld + j] = v;
            wrow[q * ld + j] = r;
          }
          __syncthreads();
        }
        // requests that moved in lower their new worker's weights (a path
        // enters a worker once: the moves are independent)
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int t = warp + 32 * u;
          if (t < nmv) {
            const int to = S.path[t], r = S.mv_r[t];
#pragma unroll
            for (int h = 0; h < 2; h++) {
              const int q = lane + 32 * h;
              const long long v = in_v[u][h];
              if (q < W && q != to) {
                const long long o = wmin[q * ld + to];
                if (v < o || (v == o && r < wrow[q * ld + to])) {
                  wmin[q * ld + to] = v;
                  wrow[q * ld + to] = r;
                }
              }
            }
          }
        }
        __syncthreads();
      }
      const bool bad = __syncthreads_or(threadIdx.x < W && S.counts[threadIdx.x] > capw);
      // each row's worker again
      for (int j = warp; listed && j < W; j += NW_WIDE)
        for (int t = lane; t < S.counts[j]; t += 32) pos[S.list[j][t]] = j;
      __syncthreads();
      opt = wide_opt(S, probs, b, mc, m, pos);
      if (bad) opt = __longlong_as_double(0x7FF0000000000000ll);
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
  // a CTA per window while they all fit on the GPU at about two to an SM
  const bool wide = mc.W > POA_WMAX;
  const bool few = b.wnext ? b.nslots <= 2 * (int64_t)sms : nprob <= sms;
  void (*kern)(const PoaProblem*, PoaBuffers, ModelConsts) = nullptr;
  if (wide)
    kern = k_poa_solve_wide;
  else if (few)
    kern = mc.W == 3 ? k_poa_solve<3, NW_SOLVE>
                     : (mc.W == 6 ? k_poa_solve<6, NW_SOLVE> : k_poa_solve<POA_WMAX, NW_SOLVE>);
  else
    kern = mc.W == 3 ? k_poa_solve<3, 1>
                     : (mc.W == 6 ? k_poa_solve<6, 1> : k_poa_solve<POA_WMAX, 1>);
  const size_t smem = wide ? poa_wide_smem(mc.W) : 0;
  if (wide && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem)) != cudaSuccess)
    return e;
  const int nt = wide ? NT_WIDE : (few ? 32 * NW_SOLVE : NT_SOLVE);
  const int wpc = wide || few ? 1 : NT_SOLVE / 32;   // windows of a CTA
  if (b.wnext) {
    // one wave of CTAs that take the windows from the counter
    if ((e = cudaMemsetAsync(b.wnext, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem)) != cudaSuccess)
      return e;
    int64_t gr = (b.nslots + wpc - 1) / wpc;
    const int64_t cap = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    gr = gr < cap ? gr : cap;
    kern<<<(unsigned)(gr > 0 ? gr : 1), nt, smem, st>>>(d_prob, b, mc);
  } else {
    // each problem's windows on its own CTAs, enough of them to fill the GPU
    const int split = (2 * sms + nprob - 1) / nprob;
    kern<<<dim3(nprob, split), nt, smem, st>>>(d_prob, b, mc);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_poa_total<<<(nprob + NT_POA / 32 - 1) / (NT_POA / 32), NT_POA, 0, st>>>(nprob, b, d_prob);
  return cudaGetLastError();
}

}  // namespace rs
