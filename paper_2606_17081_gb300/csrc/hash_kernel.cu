// KV block hashing of prompts (K1): one fused pass over all traces of a call.
//
// One warp per request, lane l on block k0 + l of each 32-block chunk:
//  1. content: the block's 64 bytes, staged in shared memory, fold into g_k;
//  2. prefix: H_k = H_{k-1} P + g_k (mod 2^64) is an affine map per block, and
//     composing affine maps is associative, so the warp computes the chunk's
//     H values with a five-step shuffle scan (step s combines partials 2^s
//     blocks apart: a = a_prev P^(2^s) + a), then adds the carry H_{k0-1}
//     times P^(l+1);
//  3. the lane stores mix(H_k ^ k); lane 31's H carries to the next chunk.
// No serial chain per request remains: the pass streams tokens once (4 bytes
// per token in) and hashes once (8 bytes per block out), the HBM floor.
//
// A warp copies its chunks into shared memory in the background, two in
// flight, with coalesced 16-byte copies past L1; a block's row there is padded
// to 80 bytes, so the lanes' reads of their own blocks meet no bank conflict,
// and the word at which a prompt starts within its first vector selects one of
// four unrolled reads.  Loads straight from global memory touch 16 lines per
// instruction.  Bound by instruction issue (about 300 per 32 blocks, ragged
// ends included) and by the latency of short prompts.  60 000 requests of median
// 1 024 tokens (325 MB) 101 -> 82 us a call (105 -> 92 with a cold L2), 5 000 of
// 256 12.3 -> 8.3 (19.1 -> 10.9), 40 000 of 100 22.6 -> 18.6 (29.3 -> 23.2);
// three chunks in flight leave fewer warps: 96 us at best on the first.
#include <algorithm>
#include <climits>

#include "rs_device.cuh"

namespace rs {

constexpr int HASH_NT = 128;
constexpr int HASH_STAGES = 2;    // chunks of 32 blocks in flight per warp
constexpr int HASH_ROW = 5;       // 16-byte vectors per staged block: four and a pad (no bank conflicts)
constexpr int HASH_STAGE = 33 * HASH_ROW;   // a chunk, and the vector past its last block

// 16-byte global -> shared copy in the background, past L1.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// Content of the staged block at row whose 64 bytes start S words into it.
template <int S>
__device__ __forceinline__ uint64_t content_staged(const uint4* row) {
  const uint4 v0 = row[0], v1 = row[1], v2 = row[2], v3 = row[3];
  const uint4 v4 = S ? row[HASH_ROW] : make_uint4(0u, 0u, 0u, 0u);   // the next row's first
  const uint32_t a[20] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w, v2.x, v2.y,
                          v2.z, v2.w, v3.x, v3.y, v3.z, v3.w, v4.x, v4.y, v4.z, v4.w};
  uint32_t w[16];
#pragma unroll
  for (int j = 0; j < 16; j++) w[j] = a[j + S];
  return block_content16(w);
}

__device__ __forceinline__ int find_job(const HashJob* jobs, int njobs, int64_t r) {
  int j = 0;
  while (j + 1 < njobs && r >= jobs[j + 1].req_base) j++;
  return j;
}

// P^(2^s), s = 0..5, by repeated squaring (mod 2^64)
__host__ __device__ constexpr uint64_t p_pow2(int s) {
  uint64_t x = PREFIX_P;
  for (int i = 0; i < s; i++) x *= x;
  return x;
}

// jobs: device array of njobs traces, or NULL: the one trace `one`.
__global__ void __launch_bounds__(HASH_NT) k_block_hash(const HashJob* __restrict__ jobs,
                                                        const HashJob one, int njobs,
                                                        int64_t total_req,
                                                        uint64_t seed) {
  __shared__ HashJob s_jobs[HASH_MAX_JOBS];
  __shared__ uint4 s_stage[HASH_NT / 32][HASH_STAGES][HASH_STAGE];
  if (jobs) {
    for (int j = threadIdx.x; j < njobs; j += HASH_NT) s_jobs[j] = jobs[j];
  } else if (threadIdx.x == 0) {
    s_jobs[0] = one;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  // P^(lane + 1): the factor of the carry H_{k0-1} at this lane's block
  uint64_t plane = 1;
#pragma unroll
  for (int s = 0; s < 6; s++)
    if (((lane + 1) >> s) & 1) plane *= p_pow2(s);
  uint4* stage = s_stage[threadIdx.x >> 5][0];
  const int64_t warp0 = ((int64_t)blockIdx.x * HASH_NT + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * HASH_NT) >> 5;
  for (int64_t r = warp0; r < total_req; r += nwarps) {
    const HashJob& J = s_jobs[find_job(s_jobs, njobs, r)];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i);
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    const int shift = (int)(o0 & 3);
    const int4* q = reinterpret_cast<const int4*>(J.tokens) + (o0 >> 2);
    uint64_t* out = J.out + (o0 >> 4);
    const int nch = (int)((nb + 31) >> 5);
    // chunk c's vectors into its stage (one commit per call, empty past the prompt)
    auto fetch = [&](int c, int st) {
      if (c < nch) {
        const int64_t left = nb - 32 * (int64_t)c;
        const int nv = 4 * (int)(left < 32 ? left : 32) + (shift ? 1 : 0);
        const int4* src = q + 128 * (int64_t)c;
        uint4* dst = stage + st * HASH_STAGE;
#pragma unroll
        for (int t = 0; t < 4; t++) {
          const int v = lane + 32 * t;
          if (v < nv) cp_async16(dst + (v >> 2) * HASH_ROW + (v & 3), src + v);
        }
        if (lane == 0 && nv == 129) cp_async16(dst + 32 * HASH_ROW, src + 128);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int c = 0; c < HASH_STAGES; c++) fetch(c, c);
    uint64_t carry = seed;   // H_{k0 - 1}
    int st = 0;
    for (int c = 0; c < nch; c++) {
      asm volatile("cp.async.wait_group %0;" ::"n"(HASH_STAGES - 1) : "memory");
      __syncwarp();   // every lane's copies of chunk c have landed
      const int64_t k = 32 * (int64_t)c + lane;
      const bool valid = k < nb;
      const uint4* row = stage + st * HASH_STAGE + lane * HASH_ROW;
      uint64_t a = 0;   // g_k; blocks past the prompt add nothing to the ones before
      switch (shift) {   // (uniform)
        case 0: a = content_staged<0>(row); break;
        case 1: a = content_staged<1>(row); break;
        case 2: a = content_staged<2>(row); break;
        default: a = content_staged<3>(row);
      }
      if (!valid) a = 0;
      __syncwarp();   // the chunk has been read
      fetch(c + HASH_STAGES, st);
      st = st + 1 == HASH_STAGES ? 0 : st + 1;
      // inclusive scan: a = sum over j <= l of g_(32c+j) P^(l - j)
#pragma unroll
      for (int s = 0; s < 5; s++) {
        const int o = 1 << s;
        const uint64_t ap = __shfl_up_sync(FULL_MASK, a, o);
        if (lane >= o) a = ap * p_pow2(s) + a;
      }
      const uint64_t H = carry * plane + a;
      if (valid) out[k] = prefix_output(H, (uint64_t)k);
      carry = __shfl_sync(FULL_MASK, H, 31);
    }
  }
}

static cudaError_t hash_launch(const HashJob* jobs_dev, const HashJob& one, int njobs,
                               int64_t total_req, uint64_t seed, cudaStream_t st) {
  if (total_req <= 0) return cudaSuccess;
  if (njobs < 1 || njobs > HASH_MAX_JOBS) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // one warp per request, up to 48 CTAs per SM: prompt lengths vary, and short
  // CTAs leave a shorter tail than one wave with the tokens shared out (which
  // also spends a third more instructions on finding its work: 106 us against
  // 82 on 60 000 requests)
  int64_t nblk = (total_req + HASH_NT / 32 - 1) / (HASH_NT / 32);
  if (nblk > (int64_t)sms * 48) nblk = (int64_t)sms * 48;
  k_block_hash<<<(unsigned)nblk, HASH_NT, 0, st>>>(jobs_dev, one, njobs, total_req, seed);
  return cudaGetLastError();
}

cudaError_t launch_block_hash(const HashJob* jobs_dev, int njobs, int64_t total_req, uint64_t seed,
                              cudaStream_t st) {
  return hash_launch(jobs_dev, HashJob{}, njobs, total_req, seed, st);
}

cudaError_t launch_block_hash_one(const HashJob& job, uint64_t seed, cudaStream_t st) {
  return hash_launch(nullptr, job, 1, job.n_req, seed, st);
}

// A small batch's sizes, written to (pinned host) out: the longest prompt's
// full blocks and the end of the last prompt.  One CTA.
__global__ void __launch_bounds__(1024) k_batch_sizes(const int64_t* __restrict__ offsets, int n,
                                                      int64_t* out) {
  __shared__ long long s_max[32];
  long long m = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const long long nb = (offsets[i + 1] - offsets[i]) >> 4;
    m = nb > m ? nb : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long v = __shfl_xor_sync(FULL_MASK, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) m = s_max[w] > m ? s_max[w] : m;
    out[0] = m;
    out[1] = offsets[n];
  }
}

cudaError_t launch_batch_sizes(const int64_t* offsets, int n, int64_t* out, cudaStream_t st) {
  k_batch_sizes<<<1, n < 1024 ? (n + 31) / 32 * 32 : 1024, 0, st>>>(offsets, n, out);
  return cudaGetLastError();
}

// The largest number of full blocks of any request of the jobs (offsets
// only): atomicMax into *nbmax, which the caller clears.
__global__ void __launch_bounds__(256) k_nbmax(const HashJob* __restrict__ jobs, int njobs,
                                               int64_t total_req, int64_t* __restrict__ nbmax) {
  __shared__ HashJob s_jobs[HASH_MAX_JOBS];
  __shared__ int64_t s_max[8];
  for (int j = threadIdx.x; j < njobs; j += blockDim.x) s_jobs[j] = jobs[j];
  __syncthreads();
  int64_t m = 0;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < total_req;
       r += (int64_t)gridDim.x * blockDim.x) {
    const HashJob& J = s_jobs[find_job(s_jobs, njobs, r)];
    const int64_t i = r - J.req_base;
    const int64_t nb = (__ldg(J.offsets + i + 1) - __ldg(J.offsets + i)) >> 4;
    m = nb > m ? nb : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int64_t v = __shfl_xor_sync(FULL_MASK, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t x = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) x = s_max[w] > x ? s_max[w] : x;
    if (x > 0) atomicMax(reinterpret_cast<unsigned long long*>(nbmax), (unsigned long long)x);
  }
}

cudaError_t launch_nbmax(const HashJob* jobs_dev, int njobs, int64_t total_req, int64_t* nbmax,
                         cudaStream_t st) {
  if (total_req <= 0) return cudaSuccess;
  if (njobs < 1 || njobs > HASH_MAX_JOBS) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int64_t nblk = (total_req + 255) / 256;
  if (nblk > (int64_t)sms * 4) nblk = (int64_t)sms * 4;
  k_nbmax<<<(unsigned)nblk, 256, 0, st>>>(jobs_dev, njobs, total_req, nbmax);
  return cudaGetLastError();
}

// Duplicate block hashes within one prompt (a 64-bit collision, which the
// simulation reports as RS_ERR_COLLISION at that request): flags[r] = 1 when
// two blocks of request r share a chained hash, 0 when none do, 2 when the
// request has more than nbmax blocks (not checked; in the simulation such a
// prompt is longer than the cache and stops its replica for capacity before
// any update).  One warp per request, each warp with an open-addressing set
// of cap entries in shared memory (cap a power of two >= 2 nbmax; the set of
// a request uses the first power of two >= 2 nb of them).  Hashes are >= 2,
// so 0 marks an empty entry.
__global__ void __launch_bounds__(256) k_dup_flags(const HashJob* __restrict__ jobs, int njobs,
                                                   int64_t total_req, int64_t nbmax, uint32_t cap,
                                                   uint8_t* __restrict__ flags) {
  extern __shared__ unsigned long long dset[];
  __shared__ HashJob s_jobs[HASH_MAX_JOBS];
  for (int j = threadIdx.x; j < njobs; j += blockDim.x) s_jobs[j] = jobs[j];
  __syncthreads();
  const int lane = threadIdx.x & 31, wpc = (int)(blockDim.x >> 5);
  unsigned long long* set = dset + (size_t)(threadIdx.x >> 5) * cap;
  const int64_t nw = (int64_t)gridDim.x * wpc;
  for (int64_t r = (int64_t)blockIdx.x * wpc + (threadIdx.x >> 5); r < total_req; r += nw) {
    const HashJob& J = s_jobs[find_job(s_jobs, njobs, r)];
    const int64_t i = r - J.req_base;
    const int64_t o0 = __ldg(J.offsets + i);
    const int64_t nb = (__ldg(J.offsets + i + 1) - o0) >> 4;
    int dup = nb > nbmax ? 2 : 0;
    if (nb >= 2 && nb <= nbmax) {   // warp-uniform (2 nb <= cap)
      uint32_t m = 2;
      while (m < 2 * nb) m <<= 1;
      const uint32_t mask = m - 1;
      for (uint32_t e = lane; e < m; e += 32) set[e] = 0ull;
      __syncwarp();
      const uint64_t* h = J.out + (o0 >> 4);
      for (int64_t k = lane; k < nb; k += 32) {
        const unsigned long long x = __ldg(h + k);
        uint32_t d = (uint32_t)(x ^ (x >> 29)) & mask;
        for (uint32_t it = 0; it <= mask; it++) {
          const unsigned long long prev = atomicCAS(set + d, 0ull, x);
          if (prev == 0ull) break;
          if (prev == x) {
            dup = 1;
            break;
          }
          d = (d + 1) & mask;
        }
      }
      dup = __any_sync(FULL_MASK, dup);   // (every lane's claims are made before the next clear)
    }
    if (lane == 0) flags[r] = (uint8_t)dup;
  }
}

cudaError_t launch_dup_flags(const HashJob* jobs_dev, int njobs, int64_t total_req, int64_t nbmax,
                             uint8_t* flags, cudaStream_t st) {
  if (total_req <= 0) return cudaSuccess;
  if (njobs < 1 || njobs > HASH_MAX_JOBS || nbmax < 1) return cudaErrorInvalidValue;
  int dev = 0, sms = 0, maxsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  uint32_t cap = 2;
  while ((int64_t)cap < 2 * nbmax) cap <<= 1;
  // dynamic shared memory beside the static job table: up to the default
  // 48 KB per CTA without opting in, else one warp's set with the opt-in
  const size_t per_warp = (size_t)cap * 8;
  const size_t stat = sizeof(HashJob) * HASH_MAX_JOBS;
  const size_t room = (size_t)maxsm - stat, dflt = 48 * 1024 - stat;
  if (per_warp > room) return cudaErrorInvalidValue;
  int wpc = (int)std::min<size_t>(8, std::max<size_t>(1, dflt / per_warp));
  const size_t smem = per_warp * wpc;
  if (smem > dflt) {
    e = cudaFuncSetAttribute(k_dup_flags, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  int64_t nblk = (total_req + wpc - 1) / wpc;
  if (nblk > (int64_t)sms * 16) nblk = (int64_t)sms * 16;
  k_dup_flags<<<(unsigned)nblk, 32 * wpc, smem, st>>>(jobs_dev, njobs, total_req, nbmax, cap,
                                                     flags);
  return cudaGetLastError();
}

}  // namespace rs
