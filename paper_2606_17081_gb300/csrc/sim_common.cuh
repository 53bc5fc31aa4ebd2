// State and event machinery shared by the simulation kernels: the closed-loop
// client, the completions heap, service starts, controller samples and the
// result record of one replica.
#pragma once

#include "rs_device.cuh"

namespace rs {

constexpr int FTAB_MAX = 1024;           // f(n) tabulated for n < FTAB_MAX

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__host__ __device__ inline int ftab_size(int cap) { return cap < FTAB_MAX ? cap : FTAB_MAX; }

// One request as the loop sees it (two live at once: i and i+1).
struct ReqState {
  int64_t off0;
  double oitl;     // O * itl
  int64_t blk;     // ceil((L + O) / 16): active blocks while unfinished
  double a;        // arrival
  double rel;      // client release time
  double twait;    // while waiting for a free client slot: the time reached
  int nb, nbt, O, phase, full;   // phase 0 new, 2 waiting for a slot, 1 arrival known
  int dup;                       // two blocks of the prompt share a chained hash
  float tau, omega;
};

// Request i's scalars as read from the trace (control thread).
struct RawReq {
  int64_t o0, o1;
  double rel;
  int O, dup;
};

struct SimScalars {
  ReqState q[2];
  RawReq nraw;                 // the request after the next one to arrive, as read
  double prev_arrival, min_ft, tick_t, lastL, ewma, sum_ttft, sum_e2e, makespan, first_switch_t;
  int64_t first_evict_i, first_live;   // first evicting update: request, resident blocks after it
  int64_t next_tick, np;
  int64_t near_ties, exact_ties, sampled, near_bd, hit_blocks, inserted, evicted, slow, rebuilds;
  int64_t ticks, switches, tir[3], n_routed, probe_blocks, hashed_blocks;
  unsigned long long probes;
  uint64_t sel_prefix;
  int32_t in_flight, nheap, nfree, evres, status, jstar, regime, up_cnt, down_cnt;
  int32_t have_L, have_ewma, max_regime, pend_cur, sel_kk;
  uint32_t dclock;             // decay step of the request being updated (frequency eviction)
  int64_t kv[5];               // Game 2: own G1 / G2 / G3, remote, recompute blocks
  double kv_cost;              // summed Eq. kv-cost
  int kvacc[10];               // one request's Game 2 categories (update group)
  int64_t tier_out;            // blocks the last update pushed out of G1
  UpdateShared us;
  uint32_t scan_pos;
  int warp_tot[NT_SIM / 32];
  int hist[256];
  double red[NT_SIM / 32];
  FreqShared fs;               // the frequency update's scalars
};

// Everything a device helper needs, resolved once per CTA.
struct SimCtx {
  SimScalars* S;
  const SimDesc* d;
  const SimBuffers* b;
  const SimLaunch* L;
  int sid;
  double *f_a, *f_o, *ftab, *f_oitl;
  uint64_t* h_k;
  uint64_t *hbuf0, *hbuf1;
  int32_t *f_req, *f_worker, *f_blk, *f_next, *h_f, *freestk;
  CacheMeta* wmeta;
  FreqMeta* wfreq;
  TierMeta* wtier;    // Game 2 band boundaries per worker (tiered)
  uint8_t* ptier;     // [W][nb] tier of each (worker, block) pair, 0 = absent (tiered)
  int32_t *winserv, *wqh, *wqt, *wm, *wabs;
  uint8_t* wopen;     // [NT_SIM / 32][WMAX] each probing warp's open workers
  uint32_t *pslot, *pfree;
  int64_t* wA;
  float* wcost;
  UpdateScratch sc;
  double *pend_ft0, *pend_tt0, *pend_ft1, *pend_tt1, *pend_win;

  __device__ __forceinline__ uint64_t* hbuf(int p) const { return p ? hbuf1 : hbuf0; }
  __device__ __forceinline__ double* pend_ft(int p) const { return p ? pend_ft1 : pend_ft0; }
  __device__ __forceinline__ double* pend_tt(int p) const { return p ? pend_tt1 : pend_tt0; }

  __device__ __forceinline__ TableView table(int j) const {
    TableView t;
    const size_t wi = (size_t)sid * L->mc.W + j;
    t.keys = b->keys + wi * L->g.slots;
    t.stamp = b->stamp + wi * L->g.slots;
    t.log = b->log + wi * L->g.R;
    t.fexp = b->fexp ? b->fexp + wi * L->g.slots : nullptr;
    t.bmask = L->g.bmask;
    t.rmask = L->g.rmask;
    return t;
  }
};

// Monotone integer key of a float64 (same order as the float64 comparison
// for every non-NaN value) and its inverse.
__device__ __forceinline__ uint64_t tkey(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double tval(uint64_t k) {
  const uint64_t b = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
  return __longlong_as_double((long long)b);
}
constexpr uint64_t KEY_INF = 0xFFF0000000000000ull;   // tkey(+infinity)

// ------------------------------------------------------------ event machinery (control thread)

__device__ __forceinline__ bool ev_less(const SimCtx& c, uint64_t ka, int fa, uint64_t kb, int fb) {
  return ka < kb || (ka == kb && c.f_req[fa] < c.f_req[fb]);
}

// The completions heap: 4-ary (children of i at 4i+1 .. 4i+4), half the
// levels of a binary heap on the control thread's dependent chain; ev_less is
// a strict total order (time, then request), so the pops are the same events
// in the same order whatever the heap's shape.
constexpr int HEAP_D = 4;

__device__ __forceinline__ void heap_push(SimCtx& c, uint64_t k, int f) {
  int i = c.S->nheap++;
  while (i > 0) {
    const int p = (i - 1) / HEAP_D;
    if (!ev_less(c, k, f, c.h_k[p], c.h_f[p])) break;
    c.h_k[i] = c.h_k[p];
    c.h_f[i] = c.h_f[p];
    i = p;
  }
  c.h_k[i] = k;
  c.h_f[i] = f;
}

__device__ __forceinline__ void heap_pop(SimCtx& c, uint64_t* k, int* f) {
  *k = c.h_k[0];
  *f = c.h_f[0];
  const int n = --c.S->nheap;
  const uint64_t lk = c.h_k[n];
  const int lf = c.h_f[n];
  int i = 0;
  for (;;) {
    const int c0 = HEAP_D * i + 1;
    if (c0 >= n) break;
    const int c1 = min(c0 + HEAP_D, n);
    // the children's keys first (independent loads), then their minimum
    uint64_t kk[HEAP_D];
#pragma unroll
    for (int q = 0; q < HEAP_D; q++) kk[q] = c0 + q < c1 ? c.h_k[c0 + q] : KEY_INF;
    int s = c0;
    uint64_t ks = kk[0];
    int fs = c.h_f[c0];
#pragma unroll
    for (int q = 1; q < HEAP_D; q++) {
      if (c0 + q >= c1) break;
      const int fq = c.h_f[c0 + q];
      if (ev_less(c, kk[q], fq, ks, fs)) {
        s = c0 + q;
        ks = kk[q];
        fs = fq;
      }
    }
    if (!ev_less(c, ks, fs, lk, lf)) break;
    c.h_k[i] = ks;
    c.h_f[i] = fs;
    i = s;
  }
  c.h_k[i] = lk;
  c.h_f[i] = lf;
}

// Eq. (9) with beta = 2: f(n) = a n + b + d / (cap - n)^2
__device__ __forceinline__ double latency_f(const ModelConsts& mc, int n) {
  const double t1 = __dmul_rn(mc.lat_a, (double)n);
  const double t2 = __dadd_rn(t1, mc.lat_b);
  const double den = (double)(mc.cap - n);
  const double t3 = __ddiv_rn(mc.lat_d, __dmul_rn(den, den));
  return __dadd_rn(t2, t3);
}

// Service of slot f starts on worker j at time t: TTFT = wait + f(n) - w_c o.
__device__ __forceinline__ void start_service(SimCtx& c, int f, int j, double t) {
  SimScalars& S = *c.S;
  const ModelConsts& mc = c.L->mc;
  const int n = ++c.winserv[j];
  const double fv = n < FTAB_MAX ? c.ftab[n] : latency_f(mc, n);
  const double svc = __dsub_rn(fv, c.f_o[f]);          // f_o holds w_c * o
  const double ft = __dadd_rn(t, svc);
  const double tt = __dsub_rn(ft, c.f_a[f]);
  const double ct = __dadd_rn(ft, c.f_oitl[f]);         // O * itl
  const int64_t row = c.d->rec_base + c.f_req[f];
  c.b->rec.start[row] = t;
  c.b->rec.first_token[row] = ft;
  c.b->rec.ttft[row] = tt;
  c.b->rec.completion[row] = ct;
  heap_push(c, tkey(ct), f);
  if (c.d->controller) {
    const int cur = S.pend_cur;
    c.pend_ft(cur)[S.np] = ft;
    c.pend_tt(cur)[S.np] = tt;
    S.np++;
    if (tkey(ft) < tkey(S.min_ft)) S.min_ft = ft;
  }
}

__device__ __forceinline__ void complete(SimCtx& c, int f, double t) {
  SimScalars& S = *c.S;
  const int j = c.f_worker[f];
  c.winserv[j]--;
  c.wA[j] -= c.f_blk[f];
  S.in_flight--;
  c.freestk[S.nfree++] = f;
  const int f2 = c.wqh[j];
  if (f2 >= 0) {
    c.wqh[j] = c.f_next[f2];
    if (c.wqh[j] < 0) c.wqt[j] = -1;
    start_service(c, f2, j, t);
  }
}

// EWMA of Eq. (10) and the hysteretic regime of Eq. (11); one sample.
__device__ __forceinline__ void ctl_sample(SimCtx& c, bool has_window, double Lw) {
  SimScalars& S = *c.S;
  const ModelConsts& mc = c.L->mc;
  const int64_t sw0 = S.switches;
  double L = 0.0;
  if (has_window) {
    L = Lw;
    S.have_L = 1;
    S.lastL = L;
  } else if (S.have_L) {
    L = S.lastL;
  }
  if (S.have_L) {
    if (!S.have_ewma) {
      S.ewma = L;
      S.have_ewma = 1;
    } else {
      S.ewma = __dadd_rn(__dmul_rn(mc.alpha, L), __dmul_rn(__dsub_rn(1.0, mc.alpha), S.ewma));
    }
    bool up = false, down = false;
    if (S.regime == 0) up = S.ewma >= mc.theta1;
    if (S.regime == 1) {
      up = S.ewma >= mc.theta2;
      down = S.ewma < __dsub_rn(mc.theta1, __dmul_rn(mc.eps_frac, mc.theta1));
    }
    if (S.regime == 2) down = S.ewma < __dsub_rn(mc.theta2, __dmul_rn(mc.eps_frac, mc.theta2));
    S.up_cnt = up ? S.up_cnt + 1 : 0;
    S.down_cnt = down ? S.down_cnt + 1 : 0;
    if (S.up_cnt >= mc.hyst_k) {
      S.regime++;
      S.up_cnt = S.down_cnt = 0;
      S.switches++;
    } else if (S.down_cnt >= mc.hyst_k) {
      S.regime--;
      S.up_cnt = S.down_cnt = 0;
      S.switches++;
    }
    if (S.regime > S.max_regime) S.max_regime = S.regime;
  }
  if (sw0 == 0 && S.switches > 0) S.first_switch_t = S.tick_t;   // this sample's time
  S.tir[S.regime]++;
  S.ticks++;
  S.next_tick++;
  S.tick_t = __dmul_rn((double)S.next_tick, mc.dt);
  if (S.ticks >= TICK_LIMIT) S.status = RS_ERR_CAPACITY;
}

__device__ __forceinline__ uint64_t tick_key(const SimCtx& c) {
  return c.d->controller ? tkey(c.S->tick_t) : KEY_INF;
}

// Advances events for request q (control thread).  Returns 1 when a
// controller sample with a non-empty window is due (the CTA computes it), 0
// when the arrival time is known and every event up to it is processed.
__device__ __forceinline__ int events_advance(SimCtx& c, ReqState& q) {
  SimScalars& S = *c.S;
  if (q.phase == 0) {
    q.twait = S.prev_arrival;
    q.phase = 2;
  }
  if (q.phase == 2) {
    // closed-loop client (§7.4): wait until fewer than C(t) requests are in
    // flight; completions, controller samples and steps of the load-spike
    // schedule in time order (ties in that order)
    const SimDesc& d = *c.d;
    for (;;) {
      const uint64_t kw = tkey(q.twait);
      const bool mid = d.c_mid > 0 && kw >= tkey(d.c_t1);
      const bool end = d.c_mid > 0 && kw >= tkey(d.c_t2);
      const int conc = end ? d.c_end : (mid ? d.c_mid : d.C);
      if (S.in_flight < conc) break;
      if (S.status != RS_OK) return 0;
      const uint64_t kc = S.nheap > 0 ? c.h_k[0] : KEY_INF;
      const uint64_t kt = tick_key(c);
      const uint64_t ks = d.c_mid <= 0 || end ? KEY_INF : tkey(mid ? d.c_t2 : d.c_t1);
      if (kc == KEY_INF && ks == KEY_INF) {   // cannot happen: a request in flight is in service
        S.status = RS_ERR_TIMEOUT;
        return 0;
      }
      if (kc <= kt && kc <= ks) {
        uint64_t k;
        int f;
        heap_pop(c, &k, &f);
        const double t = tval(k);
        complete(c, f, t);
        if (k > kw) q.twait = t;
      } else if (kt <= ks) {
        if (tkey(S.min_ft) >= kt) { ctl_sample(c, false, 0.0); continue; }
        return 1;
      } else {
        q.twait = mid ? d.c_t2 : d.c_t1;   // the schedule steps
      }
    }
    q.a = tkey(q.rel) > tkey(q.twait) ? q.rel : q.twait;
    q.phase = 1;
  }
  const uint64_t ka = tkey(q.a);
  for (;;) {
    if (S.status != RS_OK) return 0;
    const uint64_t kc = S.nheap > 0 ? c.h_k[0] : KEY_INF;
    const uint64_t kt = tick_key(c);
    if (kc <= kt) {
      if (kc > ka) break;
      uint64_t k;
      int f;
      heap_pop(c, &k, &f);
      complete(c, f, tval(k));
    } else {
      if (kt > ka) break;
      if (tkey(S.min_ft) >= kt) { ctl_sample(c, false, 0.0); continue; }
      return 1;
    }
  }
  return 0;
}

// Request i's load, records and service start (control thread); wco: w_c *
// o_ij of the chosen worker.  REC: the decision's records are written here.
template <bool REC = true>
__device__ __forceinline__ void book_request(SimCtx& c, const ReqState& q, int64_t i, double wco) {
  SimScalars& S = *c.S;
  const ModelConsts& mc = c.L->mc;
  const int js = S.jstar;
  const int f = c.freestk[--S.nfree];
  c.f_req[f] = (int32_t)i;
  c.f_worker[f] = js;
  c.f_blk[f] = (int32_t)q.blk;
  c.f_a[f] = q.a;
  c.f_o[f] = wco;
  c.f_oitl[f] = q.oitl;
  c.wA[js] += q.blk;
  S.in_flight++;
  if (REC) {
    const int64_t row = c.d->rec_base + i;
    c.b->rec.worker[row] = js;
    c.b->rec.arrival[row] = q.a;
    c.b->rec.nbt[row] = q.nbt;
  }
  if (c.winserv[js] < mc.cap - 1) {
    start_service(c, f, js, q.a);
  } else {
    c.f_next[f] = -1;
    if (c.wqt[js] >= 0) c.f_next[c.wqt[js]] = f; else c.wqh[js] = f;
    c.wqt[js] = f;
  }
  S.prev_arrival = q.a;
  S.n_routed++;
}

// Algorithm 1: the router parameters of the current regime (control thread).
// Called once request q's arrival is known and its events are done; with
// frequency eviction it also sets the decay step of that arrival.
template <bool FREQ>
__device__ __forceinline__ void regime_params(const SimCtx& c, ReqState& q) {
  if (FREQ && c.d->eviction == RS_EVICT_FREQ) {   // decay step of the arrival
    const double t = floor(__ddiv_rn(q.a, c.d->decay_s));
    c.S->dclock = t < 2147483648.0 ? (uint32_t)t : 2147483648u;
  }
  float tau = c.d->tau, om = c.d->omega;
  if (c.d->policy == RS_POLICY_LOADBAL) {
    tau = 0.0f;
    om = 0.0f;
  } else if (c.d->controller && c.S->regime > 0) {
    tau = c.L->mc.regime_tau[c.S->regime];
    om = c.L->mc.regime_omega[c.S->regime];
  }
  q.tau = tau;
  q.omega = om;
}

// The replica's result from its final state (one thread).
__device__ __forceinline__ void write_result(const SimCtx& c) {
  const SimScalars& S = *c.S;
  rs_replica_result r;
  memset(&r, 0, sizeof r);
  r.status = S.status;
  r.final_regime = S.regime;
  r.n_routed = S.n_routed;
  r.sum_ttft = S.sum_ttft;
  r.sum_e2e = S.sum_e2e;
  r.makespan = S.makespan;
  r.near_ties = S.near_ties;
  r.exact_ties = S.exact_ties;
  r.sampled = S.sampled;
  r.near_boundary = S.near_bd;
  r.hit_blocks = S.hit_blocks;
  r.inserted_blocks = S.inserted;
  r.evicted_blocks = S.evicted;
  r.ticks = S.ticks;
  r.regime_switches = S.switches;
  r.max_regime = S.max_regime;
  r.ticks_in_regime[0] = S.tir[0];
  r.ticks_in_regime[1] = S.tir[1];
  r.ticks_in_regime[2] = S.tir[2];
  r.final_ewma = S.have_ewma ? S.ewma : -1.0;
  r.probes = (int64_t)S.probes;
  r.probe_blocks = S.probe_blocks;
  r.hashed_blocks = S.hashed_blocks;
  r.slow_path = S.slow;
  r.rebuilds = S.rebuilds;
  r.first_switch_t = S.first_switch_t;
  // KV-cache pressure: resident blocks of every tier over W K_G1
  // (resident = inserted - evicted)
  const double cap = __dmul_rn((double)c.L->mc.W, (double)c.L->k1);
  r.first_evict_t = -1.0;
  r.rho_first_evict = -1.0;
  if (S.first_evict_i >= 0) {
    r.first_evict_t = c.b->rec.arrival[c.d->rec_base + S.first_evict_i];
    r.rho_first_evict = __ddiv_rn((double)S.first_live, cap);
  }
  r.rho_end = __ddiv_rn((double)(S.inserted - S.evicted), cap);
  r.kv_g1 = S.kv[0];
  r.kv_g2 = S.kv[1];
  r.kv_g3 = S.kv[2];
  r.kv_remote = S.kv[3];
  r.kv_recompute = S.kv[4];
  r.kv_cost = S.kv_cost;
  c.b->res[c.sid] = r;
}

}  // namespace rs
