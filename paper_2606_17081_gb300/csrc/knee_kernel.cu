// Saturation knee of load sweeps (§5.1, the PoA-growth proposition, item 3:
// the second derivative of latency with respect to load above a threshold
// marks the onset of saturation; Experiment 2 takes difference quotients of
// TTFT P99 across a sweep of concurrency levels).
//
// k_replica_pct (one CTA per replica): the nearest-rank percentile of the
// replica's routed TTFTs by an exact selection on order-preserving 64-bit keys
// of the doubles.  The routed keys are packed into shared memory as the rows
// are read (up to PCT_ROWS; more rows are read again in each pass); a pass
// counts an 11-bit digit that starts at the highest bit in which the keys left
// differ, so a few milliseconds to seconds of latency spread over hundreds of
// bins at once, and once a bin holds at most PCT_LAST keys their ranks are
// counted directly: two or three passes in place of eight 8-bit digits from the
// top byte, each with a serial scan of its 256 bins (54 replicas x 6 000 rows:
// 152 -> 91 us a call with its eight copies, 55 with one in and one out).  Bound
// by the latency of its barriers.  The result is an element of the input, so it
// is bit-exact.
//
// k_sweep_knee (one warp per sweep; a sweep is a handful of levels): the
// neighbour difference quotients, the three-point second divided difference
// and the first interior level above the threshold, each operation rounded
// once in the order written; a lane per level, since a division takes 650
// cycles.
#include "rs_device.cuh"

namespace rs {

constexpr int NT_PCT = 1024;
constexpr int PCT_BINS = 2048, PCT_BITS = 11;
constexpr int PCT_ROWS = 24576;   // keys held in shared memory (192 KB)
constexpr int PCT_LAST = 256;

// ascending doubles <-> ascending unsigned keys (sign-magnitude to offset binary)
__device__ __forceinline__ uint64_t order_key(double v) {
  const uint64_t u = (uint64_t)__double_as_longlong(v);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__device__ __forceinline__ double key_value(uint64_t k) {
  const uint64_t u = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
  return __longlong_as_double((long long)u);
}

__global__ void __launch_bounds__(NT_PCT) k_replica_pct(const int32_t* __restrict__ worker,
                                                        const double* __restrict__ ttft,
                                                        const int64_t* __restrict__ row_start,
                                                        int pct, int cap,
                                                        double* __restrict__ stat,
                                                        double* __restrict__ d1,
                                                        double* __restrict__ d2) {
  extern __shared__ uint64_t keys[];   // [cap]
  __shared__ unsigned hist[PCT_BINS];
  __shared__ unsigned wsum[NT_PCT / 32];
  __shared__ uint64_t last[PCT_LAST];
  __shared__ unsigned long long s_n, s_and, s_or;
  __shared__ unsigned s_last, s_bin, s_cnt;
  __shared__ long long s_rank;
  const int r = blockIdx.x, tid = (int)threadIdx.x, lane = tid & 31;
  const int64_t a = row_start[r], b = row_start[r + 1];
  const bool held = b - a <= (int64_t)cap;
  if (tid == 0) {
    s_n = 0;
    s_and = ~0ull;
    s_or = 0;
    d1[r] = __longlong_as_double(0x7FF8000000000000ll);
    d2[r] = __longlong_as_double(0x7FF8000000000000ll);
  }
  __syncthreads();
  // the routed rows' keys, packed in any order; the bits they agree on
  uint64_t all1 = ~0ull, any1 = 0ull;
  for (int64_t i0 = a; i0 < b; i0 += NT_PCT) {
    const int64_t i = i0 + tid;
    const bool in = i < b && worker[i] >= 0;
    uint64_t k = 0;
    if (in) {
      k = order_key(ttft[i]);
      all1 &= k;
      any1 |= k;
    }
    const unsigned m = __ballot_sync(FULL_MASK, in);
    unsigned long long base = 0;
    if (lane == 0 && m) base = atomicAdd(&s_n, (unsigned long long)__popc(m));
    base = __shfl_sync(FULL_MASK, base, 0);
    if (in && held) keys[base + __popc(m & ((1u << lane) - 1u))] = k;
  }
  // the keys of the replica one after another: fn(key, whether there is one)
  auto each = [&](auto fn) {
    const int64_t n = held ? (int64_t)s_n : b - a;
    for (int64_t i0 = 0; i0 < n; i0 += NT_PCT) {
      const int64_t i = i0 + tid;
      bool in = i < n;
      uint64_t k = 0;
      if (held) {
        if (in) k = keys[i];
      } else if (in) {
        in = worker[a + i] >= 0;
        if (in) k = order_key(ttft[a + i]);
      }
      fn(k, in);
    }
  };
  uint64_t mask = 0, prefix = 0;   // the keys left agree with prefix on mask
  for (bool first = true;; first = false) {
    if (!first) {
      // the bits on which the keys left agree
      all1 = ~0ull;
      any1 = 0ull;
      each([&](uint64_t k, bool in) {
        if (in && (k & mask) == prefix) {
          all1 &= k;
          any1 |= k;
        }
      });
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      all1 &= __shfl_xor_sync(FULL_MASK, all1, o);
      any1 |= __shfl_xor_sync(FULL_MASK, any1, o);
    }
    if (lane == 0) {
      atomicAnd(&s_and, (unsigned long long)all1);
      atomicOr(&s_or, (unsigned long long)any1);
    }
    for (int q = tid; q < PCT_BINS; q += NT_PCT) hist[q] = 0;
    __syncthreads();
    const long long n = (long long)s_n;
    if (n == 0) {
      if (tid == 0) stat[r] = __longlong_as_double(0x7FF8000000000000ll);
      return;
    }
    if (first && tid == 0) s_rank = ((long long)pct * n + 99) / 100 - 1;   // 0-based ascending
    const uint64_t com = s_and, diff = com ^ s_or;
    if (diff == 0) {   // all equal
      if (tid == 0) stat[r] = key_value(com);
      return;
    }
    const int top = 63 - __clzll((long long)diff);
    const int shift = top >= PCT_BITS - 1 ? top - (PCT_BITS - 1) : 0;
    each([&](uint64_t k, bool in) {
      if (in && (k & mask) == prefix) atomicAdd(&hist[(unsigned)(k >> shift) & (PCT_BINS - 1)], 1u);
    });
    __syncthreads();
    // the bin that holds the rank: thread t sums bins 2 t and 2 t + 1
    const unsigned h0 = hist[2 * tid], h1 = hist[2 * tid + 1];
    unsigned inc = h0 + h1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(FULL_MASK, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[tid >> 5] = inc;
    __syncthreads();
    {
      unsigned w = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(FULL_MASK, w, o);
        if (lane >= o) w += y;
      }
      const int wi = tid >> 5;
      const unsigned below = __shfl_sync(FULL_MASK, w, wi > 0 ? wi - 1 : 0);
      const long long c1 = (long long)inc + (wi > 0 ? below : 0u);   // through bin 2 t + 1
      const long long c0 = c1 - h1, cb = c0 - h0;
      const long long k = s_rank;
      __syncthreads();   // (every thread has read the rank)
      if (k >= cb && k < c1) {
        const bool hi = k >= c0;
        s_bin = 2 * (unsigned)tid + hi;
        s_cnt = hi ? h1 : h0;
        s_rank = k - (hi ? c0 : cb);
        s_last = 0;
        s_and = ~0ull;
        s_or = 0;
      }
    }
    __syncthreads();
    // the keys left: those in that bin (the bits above the digit are common)
    mask = ~0ull << shift;
    prefix = (shift + PCT_BITS < 64 ? com & (~0ull << (shift + PCT_BITS)) : 0ull) |
             ((uint64_t)s_bin << shift);
    if (shift == 0) {   // every bit is decided
      if (tid == 0) stat[r] = key_value(prefix);
      return;
    }
    if (s_cnt <= PCT_LAST) {
      each([&](uint64_t k, bool in) {
        if (in && (k & mask) == prefix) last[atomicAdd(&s_last, 1u)] = k;
      });
      __syncthreads();
      const int c = (int)s_cnt;
      if (tid < c) {
        const uint64_t mine = last[tid];
        int less = 0;
        for (int q = 0; q < c; q++) less += last[q] < mine || (last[q] == mine && q < tid);
        if (less == (int)s_rank) stat[r] = key_value(mine);
      }
      return;
    }
  }
}

__global__ void k_sweep_knee(const double* __restrict__ load, const double* __restrict__ stat,
                             const int32_t* __restrict__ sweep_start, int n_sweeps, double theta,
                             double* d1, double* __restrict__ d2,
                             double* __restrict__ knee_load, int32_t* __restrict__ knee_index) {
  const int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = (int)(threadIdx.x & 31);
  if (s >= n_sweeps) return;
  const int a = sweep_start[s], b = sweep_start[s + 1];
  bool inc = true;
  for (int r = a + 1 + lane; r < b; r += 32) inc &= load[r] > load[r - 1];
  if (!__all_sync(FULL_MASK, inc)) {
    if (lane == 0) {
      knee_load[s] = __longlong_as_double(0x7FF8000000000000ll);
      knee_index[s] = -2;
    }
    return;
  }
  for (int r = a + lane; r + 1 < b; r += 32)
    d1[r] = __ddiv_rn(__dsub_rn(stat[r + 1], stat[r]), __dsub_rn(load[r + 1], load[r]));
  __syncwarp();   // (d1 is read back across the warp)
  int ki = -1;
  for (int r0 = a + 1; r0 + 1 < b; r0 += 32) {
    const int r = r0 + lane;
    bool over = false;
    if (r + 1 < b) {
      const double v = __ddiv_rn(__dmul_rn(2.0, __dsub_rn(d1[r], d1[r - 1])),
                                 __dsub_rn(load[r + 1], load[r - 1]));
      d2[r] = v;
      over = v > theta;
    }
    const unsigned m = __ballot_sync(FULL_MASK, over);
    if (ki < 0 && m) ki = r0 + __ffs(m) - 1;
  }
  if (lane == 0) {
    knee_load[s] = ki < 0 ? -1.0 : load[ki];
    knee_index[s] = ki;
  }
}

cudaError_t launch_sweep_knee(const int32_t* worker, const double* ttft, const int64_t* row_start,
                              int n_rep, int64_t max_rows, const double* load, const int32_t* sweep_start,
                              int n_sweeps, int pct, double theta, double* stat, double* d1,
                              double* d2, double* knee_load, int32_t* knee_index,
                              cudaStream_t st) {
  static_assert(PCT_BINS == 2 * NT_PCT && NT_PCT == 32 * 32, "two bins per thread, a warp of warp sums");
  if (n_rep > 0) {
    // (replicas past PCT_ROWS rows are read again in each pass)
    const int cap = (int)(max_rows < 1 ? 1 : (max_rows < PCT_ROWS ? max_rows : PCT_ROWS));
    cudaError_t ea = cudaFuncSetAttribute(k_replica_pct, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          8 * PCT_ROWS);
    if (ea != cudaSuccess) return ea;
    k_replica_pct<<<n_rep, NT_PCT, (size_t)8 * cap, st>>>(worker, ttft, row_start, pct, cap, stat, d1, d2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (n_sweeps > 0) {
    k_sweep_knee<<<(n_sweeps + 3) / 4, 128, 0, st>>>(load, stat, sweep_start, n_sweeps, theta,
                                                        d1, d2, knee_load, knee_index);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

}  // namespace rs
