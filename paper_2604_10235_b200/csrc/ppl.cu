// Query-conditioned perplexity scores of chunks (Section 4.1): for every (chunk, query position)
// the negative log-likelihood of the query token, logsumexp(row) - row[target], from one
// streaming pass over the row of V logits, then the mean over the query positions, and the
// choice of the k chunks with the lowest score.
//
// The scoring kernel is bound by HBM: every logit is read once (V * 2 or 4 bytes per row, rows
// of several hundred KB), the arithmetic per element is one scale, one exponential and one add.
// A thread requests 128 bytes in 16-byte vectors before it uses the first, takes them in pairs as
// they arrive, and keeps a running (maximum, sum) in base 2 that is rescaled only when a pair
// raises the maximum; the threads' pairs are merged with shuffles.  With 2-byte logits the issue
// slots come close to the memory time, so scaling and sums are packed f32x2 operations, maxima of
// bf16 logits are taken on the packed words, and (POLY) one pair of exponentials in eight is evaluated
// on the FMA pipe.  32 x 64 rows of 128256 logits, replayed: bf16 85 us = 6.2 TB/s (scalar
// arithmetic: 3 us more), f32 150 us = 7.0 TB/s.  Keeping the loads of the next batch in flight during the
// arithmetic needs 64 registers and costs a resident CTA: slower for bf16 (97 us).
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include "cc_internal.cuh"
#include "exp2_poly.cuh"

namespace cg = cooperative_groups;

namespace cc {

namespace {

constexpr int kThreads = 512;
constexpr int kVecWidth = 8;              // logits a thread takes at a time
constexpr int kMeanThreads = 128;
constexpr int kRankThreads = 512;
constexpr int kMaxParts = 8;              // CTAs that share a row at most
constexpr int kCtasPerSm = 3;             // resident CTAs of ppl_nll_kernel per SM (40 registers)
constexpr int kPolyPairs = 8;             // one pair of exponentials in this many goes to the FMA pipe
constexpr int kGroup = 2;                 // vectors taken at a time
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// The maximum starts at the lowest finite value, not at -inf: while a thread has met only -inf (or
// values that scale to it: masked logits) the arguments x log2(e) - m are then -inf and not
// -inf + inf.  What the clamp of the FMA-pipe exponentials leaves in the sum meanwhile is multiplied by
// 0 when the maximum is raised or merged.
constexpr float kNoMax = -FLT_MAX;

struct Running {
  float m, s;       // maximum (base-2 units) and sum of 2^(x log2(e) - m)
  __device__ __forceinline__ void raise(float top) {
    const float vm = top * kLog2e;
    if (vm > m) {
      s *= ex2(m - vm);          // m = kNoMax at the start: the factor is 0
      m = vm;
    }
  }
  __device__ __forceinline__ void merge(float om, float os) {
    const float nm = fmaxf(m, om);
    s = s * ex2(m - nm) + os * ex2(om - nm);
    m = nm;
  }
};

// A streaming 16-byte load that the compiler keeps where it is written, so that the loads of a
// batch are all issued before the first of them is used.
__device__ __forceinline__ uint4 ld16(const void* p) {
  uint4 v;
  asm volatile("ld.global.cs.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Eight consecutive logits: their raw 16-byte words and the conversion to f32.
template <typename T> struct Vec;
template <> struct Vec<float> {
  uint4 a, b;
  __device__ __forceinline__ void load(const float* p) { a = ld16(p); b = ld16(p + 4); }
  __device__ __forceinline__ uint64_t pair(int i) const {
    const uint4 w = i < 2 ? a : b;
    return i & 1 ? pack2(__uint_as_float(w.z), __uint_as_float(w.w)) : pack2(__uint_as_float(w.x), __uint_as_float(w.y));
  }
  template <int kN> __device__ static float top(const Vec<float> (&r)[kN]) {
    float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      m0 = max3f(m0, __uint_as_float(r[u].a.x), __uint_as_float(r[u].a.y));
      m1 = max3f(m1, __uint_as_float(r[u].a.z), __uint_as_float(r[u].a.w));
      m0 = max3f(m0, __uint_as_float(r[u].b.x), __uint_as_float(r[u].b.y));
      m1 = max3f(m1, __uint_as_float(r[u].b.z), __uint_as_float(r[u].b.w));
    }
    return fmaxf(m0, m1);
  }
  __device__ static float one(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
  }
};
template <> struct Vec<uint16_t> {       // bf16 bit patterns
  uint4 a;
  __device__ __forceinline__ void load(const uint16_t* p) { a = ld16(p); }
  __device__ __forceinline__ uint64_t pair(int i) const {
    const uint32_t w = i == 0 ? a.x : i == 1 ? a.y : i == 2 ? a.z : a.w;
    return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
  }
  template <int kN> __device__ static float top(const Vec<uint16_t> (&r)[kN]) {
    uint32_t m = r[0].a.x;
#pragma unroll
    for (int u = 0; u < kN; ++u) m = max_bf16x2(max_bf16x2(m, max_bf16x2(r[u].a.x, r[u].a.y)), max_bf16x2(r[u].a.z, r[u].a.w));
    return fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u));
  }
  __device__ static float one(const uint16_t* p) {
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return __uint_as_float((uint32_t)v << 16);
  }
};
// The pairs of kLanes neighbouring lanes as one, in all of them: the maximum first, so that every lane has a single exponential.
template <int kLanes>
__device__ __forceinline__ void merge_lanes(Running& r) {
  float top = r.m;
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  float sum = r.s * ex2(r.m - top);
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  r = Running{top, sum};
}
// adds a batch of vectors
template <bool POLY, typename T, int kN>
__device__ __forceinline__ void add_batch(Running& run, const Vec<T> (&r)[kN]) {
  run.raise(Vec<T>::top(r));
  const uint64_t c2 = pack2(kLog2e, kLog2e), nm = pack2(-run.m, -run.m);
  uint64_t acc[2] = {0ull, 0ull};
#pragma unroll
  for (int u = 0; u < kN; ++u)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint64_t x = fma2(r[u].pair(i), c2, nm);
      acc[i & 1] = add2(acc[i & 1], POLY && kN * 4 >= kPolyPairs && (u * 4 + i) % kPolyPairs == 1 ? ex2_pair_fma(x) : ex2_pair_sfu(x));
    }
  float a, b;
  unpack2(add2(acc[0], acc[1]), a, b);
  run.s += a + b;
}
template <typename T> constexpr int kBatch = sizeof(T) == 2 ? 8 : 4;   // 128 bytes per thread in flight

// Rows [0, whole) have a CTA each; every later row is shared by the `parts` CTAs of a cluster
// (parts divides `whole`, so clusters never mix the two), which merge their pairs in the first
// one's shared memory.  A row may start anywhere on the element grid: the values before its first
// and after its last 16-byte boundary (at most fourteen) are read one by one.
template <typename T, bool POLY>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
ppl_nll_kernel(const T* __restrict__ logits, int num_tokens, int vocab, int64_t stride_chunk,
               int64_t stride_token, int whole, int parts, const int32_t* __restrict__ targets,
               float* __restrict__ nll, DeviceStatus* status) {
  __shared__ float sm_m[kThreads / 32], sm_s[kThreads / 32];
  __shared__ float2 sm_part[kMaxParts];
  pdl_launch_dependents();
  const bool split = (int)blockIdx.x >= whole;
  const int part = split ? ((int)blockIdx.x - whole) % parts : 0;
  const int row = split ? whole + ((int)blockIdx.x - whole) / parts : (int)blockIdx.x;
  const int n_parts = split ? parts : 1;
  if (split) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // this CTA has started
  const int chunk = row / num_tokens, t = row % num_tokens;
  const T* x = logits + (int64_t)chunk * stride_chunk + (int64_t)t * stride_token;
  Running r{kNoMax, 0.f};
  // The target is asked for before the row, its logit before the last vectors of it: both at the end, one after the other, and a
  // chain of sixteen merges by one thread, kept a CTA 2 us after its row was read, in waves that all end together.
  const bool writer = part == 0 && threadIdx.x == 0;
  int target = -1;
  const int head = min(vocab, (int)((16u - (unsigned)((uintptr_t)x & 15u)) & 15u) / (int)sizeof(T));
  const T* xv = x + head;
  const int n_vec = (vocab - head) / kVecWidth;
  int i = (int)((int64_t)n_vec * part / n_parts) + threadIdx.x;
  const int i_end = (int)((int64_t)n_vec * (part + 1) / n_parts);
  constexpr int kB = kBatch<T>;
  pdl_wait();
  if (writer) asm volatile("ld.global.s32 %0, [%1];" : "=r"(target) : "l"(targets + t));
  for (; i + (kB - 1) * kThreads < i_end; i += kB * kThreads) {
    Vec<T> raw[kB];
#pragma unroll
    for (int u = 0; u < kB; ++u) raw[u].load(xv + (int64_t)(i + u * kThreads) * kVecWidth);
#pragma unroll
    for (int u = 0; u < kB; u += kGroup) {
      Vec<T> taken[kGroup];
#pragma unroll
      for (int g = 0; g < kGroup; ++g) taken[g] = raw[u + g];
      add_batch<POLY, T, kGroup>(r, taken);
    }
  }
  const bool known = writer && target >= 0 && target < vocab;
  const float at_target = known ? Vec<T>::one(x + target) : 0.0f;
  for (; i < i_end; i += kThreads) {
    Vec<T> raw[1];
    raw[0].load(xv + (int64_t)i * kVecWidth);
    add_batch<POLY, T, 1>(r, raw);
  }
  // the values before the first and after the last whole vector
  if (part == 0) {
    const int tail = head + n_vec * kVecWidth;
    for (int j = threadIdx.x; j < head + vocab - tail; j += kThreads)
      r.merge(Vec<T>::one(x + (j < head ? j : tail + j - head)) * kLog2e, 1.0f);
  }

  merge_lanes<32>(r);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sm_m[warp] = r.m; sm_s[warp] = r.s; }
  __syncthreads();
  Running all{kNoMax, 0.f};
  if (warp == 0) {
    static_assert(kThreads / 32 == 16, "a half warp merges the warps' pairs");
    all = Running{sm_m[lane & 15], sm_s[lane & 15]};
    merge_lanes<16>(all);
  }
  if (split) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // the first CTA has started
    if (threadIdx.x == 0)
      *cg::this_cluster().map_shared_rank(&sm_part[part], 0) = make_float2(all.m, all.s);
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (part != 0) return;
    if (threadIdx.x == 0)
      for (int k = 1; k < parts; ++k) all.merge(sm_part[k].x, sm_part[k].y);
  }
  if (writer) {
    float out = __int_as_float(0x7fc00000);                   // NaN for an invalid token id or a row of masked logits
    if (!known)
      report_error(status, CC_ERR_DEVICE_FLAG, 600);
    else if (all.m > kNoMax)
      out = (all.m + log2f(all.s)) * kLn2 - at_target;
    nll[row] = out;
  }
}

// mean over the query positions, summed in order: one warp per chunk, 32 values per load
__global__ void __launch_bounds__(kMeanThreads)
ppl_mean_kernel(const float* __restrict__ nll, int num_chunks, int num_tokens, float* __restrict__ score) {
  pdl_launch_dependents();
  pdl_wait();
  const int c = blockIdx.x * (kMeanThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= num_chunks) return;
  float acc = 0.f;
  for (int t0 = 0; t0 < num_tokens; t0 += 32) {
    const float v = t0 + lane < num_tokens ? nll[(int64_t)c * num_tokens + t0 + lane] : 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float x = __shfl_sync(0xffffffffu, v, k);
      if (t0 + k < num_tokens) acc = __fadd_rn(acc, x);
    }
  }
  if (lane == 0) score[c] = __fdiv_rn(acc, (float)num_tokens);
}

// rank of every chunk by (score, index); the k best are written in rank order.  A warp ranks one
// chunk against all others.
__global__ void __launch_bounds__(kRankThreads)
select_chunks_kernel(const float* __restrict__ score, int num_chunks, int k, int32_t* __restrict__ chosen) {
  extern __shared__ float key[];
  pdl_launch_dependents();
  pdl_wait();
  for (int i = threadIdx.x; i < num_chunks; i += kRankThreads) {
    const float s = score[i];
    key[i] = s != s ? INFINITY : s;                           // NaN ranks last
  }
  __syncthreads();
  const int i = blockIdx.x * (kRankThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= num_chunks) return;
  const float mine = key[i];
  int rank = 0;
  for (int j = lane; j < num_chunks; j += 32) rank += key[j] < mine || (key[j] == mine && j < i);
  rank = __reduce_add_sync(0xffffffffu, rank);
  if (lane == 0 && rank < k) chosen[rank] = i;
}

}  // namespace

// A row is a few hundred KB, so whole rows quantise badly: the rows that do not fill a last wave of
// `slots` CTAs (all of them, when there are few) are split over clusters as wide as that wave allows, not
// below 8192 values per CTA.  The clusters start at a multiple of their width, so up to seven rows of the
// full waves are split too; no width is taken that adds a wave with them.  8 x 16 rows of 151936 bf16 logits:
// 18.8 -> 14 us with three CTAs per row; splitting beyond one wave, or rows of full waves, is slower
// (cluster scheduling).  Where full waves of 444 were left exactly or nearly, the split used to add a wave:
// 128256 bf16 logits, 444 rows 31.9 -> 24.2 us, 888 rows 47.7 -> 43.9, 497 rows 32.8 -> 32.0.
PplSplit ppl_split(int rows, int vocab, int slots) {
  const int full = rows / slots * slots;
  PplSplit best{rows, 1};
  if (rows == full) return best;
  for (int parts = 2; parts <= kMaxParts && vocab / parts >= 8192; ++parts) {
    const int whole = full - full % parts;
    if ((rows - whole) * parts <= full - whole + slots) best = PplSplit{whole, parts};
  }
  return best;
}

cudaError_t launch_ppl_scores(const Launch& L, const void* logits, bool is_f32, int num_chunks,
                              int num_tokens, int vocab, int64_t stride_chunk, int64_t stride_token,
                              const int32_t* targets, float* nll, float* score) {
  const int rows = num_chunks * num_tokens;
  const PplSplit split = ppl_split(rows, vocab, L.sm_count * kCtasPerSm);
  const int whole = split.whole, parts = split.parts;
  const unsigned grid = (unsigned)(whole + (rows - whole) * parts);
  // The FMA pipe's exponentials (relative error 8e-5) are for bf16 rows on the 16-byte grid alone, where
  // they take 1.6 % off the call (32 x 64 rows of 128256: 94.2 against 95.7 us).  f32 logits leave the
  // special-function unit idle anyway (32 x 32 rows of 128256: 85.1 without, 86.5 us with them), and rows
  // off the grid lose nothing (32 x 64 rows of 50257 bf16 logits: 46.5 / 46.9).
  const bool poly = !is_f32 && (uintptr_t)logits % 16 == 0 && stride_chunk % 8 == 0 && stride_token % 8 == 0;
  const auto bf16_kernel = poly ? ppl_nll_kernel<uint16_t, true> : ppl_nll_kernel<uint16_t, false>;
  const cudaError_t e = is_f32
      ? launch_pdl(ppl_nll_kernel<float, false>, dim3(grid), dim3(kThreads), 0, L.stream, parts, (const float*)logits,
                   num_tokens, vocab, stride_chunk, stride_token, whole, parts, targets, nll, L.status)
      : launch_pdl(bf16_kernel, dim3(grid), dim3(kThreads), 0, L.stream, parts,
                   (const uint16_t*)logits, num_tokens, vocab, stride_chunk, stride_token, whole, parts, targets,
                   nll, L.status);
  if (e != cudaSuccess) return e;
  return launch_pdl(ppl_mean_kernel, dim3((num_chunks + kMeanThreads / 32 - 1) / (kMeanThreads / 32)),
                    dim3(kMeanThreads), 0, L.stream, 1, nll, num_chunks, num_tokens, score);
}

cudaError_t launch_select_chunks(const Launch& L, const float* score, int num_chunks, int k,
                                 int32_t* chosen) {
  return launch_pdl(select_chunks_kernel, dim3((num_chunks + kRankThreads / 32 - 1) / (kRankThreads / 32)),
                    dim3(kRankThreads), (size_t)num_chunks * sizeof(float), L.stream, 1, score, num_chunks, k, chosen);
}

}  // namespace cc

extern "C" void ccx_ppl_split(int rows, int vocab, int slots, int* whole, int* parts) {
  const cc::PplSplit s = cc::ppl_split(rows, vocab, slots);
  *whole = s.whole;
  *parts = s.parts;
}
