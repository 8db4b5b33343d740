// A2 + A3: sliding-window pooling of the scores and fusion with the structural prior.
// Token level: one thread per token; the 2*half neighbours come from L1/L2 (the whole score
// array of a layer is about 1 MB).  Chunk level: one thread per chunk.
// Every floating-point operation is an explicitly rounded f32 operation (no contraction into
// FMA), in a fixed order, so that the result is reproducible bit for bit.
#include "cc_internal.cuh"

namespace cc {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float canonical(float x) { return __fadd_rn(x, 0.0f); }  // -0 -> +0

__global__ void __launch_bounds__(kThreads)
fuse_pool_kernel(const __grid_constant__ BatchTable bt, int pool_kind, int pool_size,
                 float alpha, float beta, const float* __restrict__ scores,
                 const float* __restrict__ prior, float* __restrict__ fused) {
  const int s = blockIdx.z;
  const int h = blockIdx.y;
  const SeqInfo& q = bt.seq[s];
  const float* u = scores + (int64_t)h * bt.n_tot + q.tok_off;
  const float* p = prior + q.tok_off;
  float* f = fused + (int64_t)h * bt.m_tot + q.item_off;

  for (int i = blockIdx.x * kThreads + threadIdx.x; i < q.n_items; i += gridDim.x * kThreads) {
    float val, pr;
    if (bt.chunk > 1) {
      const int lo = i * bt.chunk;
      const int hi = min(q.n, lo + bt.chunk);
      val = u[lo];
      pr = p[lo];
      for (int j = lo + 1; j < hi; ++j) {
        val = __fadd_rn(val, u[j]);
        pr = fmaxf(pr, p[j]);
      }
    } else {
      pr = p[i];
      if (pool_kind == CC_POOL_NONE || pool_size <= 1) {
        val = u[i];
      } else {
        const int half = pool_size / 2;
        if (pool_kind == CC_POOL_MAX) {
          val = u[i];
          for (int j = max(0, i - half); j <= min(q.n - 1, i + half); ++j) val = fmaxf(val, u[j]);
        } else {
          val = 0.0f;
          bool first = true;
          for (int j = i - half; j <= i + half; ++j) {
            const float x = (j >= 0 && j < q.n) ? u[j] : 0.0f;
            val = first ? x : __fadd_rn(val, x);
            first = false;
          }
          val = __fdiv_rn(val, (float)pool_size);
        }
      }
    }
    f[i] = canonical(__fadd_rn(__fmul_rn(alpha, val), __fmul_rn(beta, pr)));
  }
}

// Nearest-to-protected fill (Section 4.4, last sentence of "Token-level protection"): the value of
// a token is minus the distance to the closest protected token (minus n when there is none), the
// same for every head.  One CTA per tile of kNearTile tokens: the protected flags of the tile are
// a bit mask in shared memory (one ballot per 32 tokens), so the closest protected token inside
// the tile is a few bit operations away; the closest ones outside are looked for in both
// directions at once, kNearTile tokens per step, from the tile's edges outwards (protected tokens
// are a few percent of a text, so one step finds them).  Bound by the hkv coalesced rows written;
// 32768 tokens, 8 heads: 4 us (one CTA per sequence with a contiguous segment per thread: 150 us).
constexpr int kNearTile = 1024;
constexpr int kNearWords = kNearTile / 32;

__global__ void __launch_bounds__(kNearTile)
nearest_fill_kernel(const __grid_constant__ BatchTable bt, int hkv, float theta,
                    const float* __restrict__ prior, float* __restrict__ fused) {
  __shared__ unsigned mask[kNearWords];
  __shared__ int s_before, s_after;            // closest protected tokens outside the tile
  pdl_launch_dependents();
  const int s = blockIdx.y;
  const SeqInfo& q = bt.seq[s];
  const int n = q.n, lo = blockIdx.x * kNearTile;
  if (lo >= n) return;
  const float* p = prior + q.tok_off;
  const int t = threadIdx.x, lane = t & 31, word = t >> 5, j = lo + t;
  if (t == 0) { s_before = -1; s_after = 2 * n; }
  pdl_wait();
  // the tile's priors and those of its neighbours, where the search nearly always ends, are asked for together
  const float own = j < n ? p[j] : 0.0f;
  const float left = lo > 0 ? p[j - kNearTile] : 0.0f, right = j + kNearTile < n ? p[j + kNearTile] : 0.0f;
  const unsigned m = __ballot_sync(0xffffffffu, j < n && own >= theta);
  if (lane == 0) mask[word] = m;
  // outside the tile: the last protected token before lo, the first one from lo + kNearTile on
  bool need_b = lo > 0, need_a = lo + kNearTile < n;
  for (int step = 1; need_b || need_a; ++step) {
    __syncthreads();
    const int jb = lo - step * kNearTile + t, ja = lo + step * kNearTile + t;
    if (need_b && (step == 1 ? left : p[jb]) >= theta) atomicMax(&s_before, jb);
    if (need_a && ja < n && (step == 1 ? right : p[ja]) >= theta) atomicMin(&s_after, ja);
    __syncthreads();
    need_b = need_b && s_before < 0 && lo - (step + 1) * kNearTile >= 0;
    need_a = need_a && s_after >= n && lo + (step + 1) * kNearTile < n;
  }
  __syncthreads();
  const unsigned words = __ballot_sync(0xffffffffu, mask[lane] != 0u);   // which words are not empty
  if (j >= n) return;
  int before = s_before, after = s_after;
  const unsigned m_le = m & (0xffffffffu >> (31 - lane)), m_ge = m & (0xffffffffu << lane);
  const unsigned w_lt = words & ((1u << word) - 1u), w_gt = words & ~((2u << word) - 1u);
  if (m_le) before = lo + word * 32 + 31 - __clz(m_le);
  else if (w_lt) { const int w = 31 - __clz(w_lt); before = lo + w * 32 + 31 - __clz(mask[w]); }
  if (m_ge) after = lo + word * 32 + __ffs(m_ge) - 1;
  else if (w_gt) { const int w = __ffs(w_gt) - 1; after = lo + w * 32 + __ffs(mask[w]) - 1; }
  const int d = min(before >= 0 ? j - before : n, after < n ? after - j : n);
  float* f = fused + q.item_off + j;
  for (int h = 0; h < hkv; ++h) f[(int64_t)h * bt.m_tot] = -(float)d;
}

}  // namespace

cudaError_t launch_nearest_fill(const Launch& L, const BatchTable& bt, const Geometry& g,
                                float force_threshold, const float* prior, float* fused) {
  const int tiles = (bt.max_items + kNearTile - 1) / kNearTile;
  return launch_pdl(nearest_fill_kernel, dim3(tiles < 1 ? 1 : tiles, bt.num_seqs), dim3(kNearTile), 0, L.stream, 1,
                    bt, g.hkv, force_threshold, prior, fused);
}

cudaError_t launch_fuse_pool(const Launch& L, const BatchTable& bt, const Geometry& g,
                             int pool_kind, int pool_size, float alpha, float beta,
                             const float* scores, const float* prior, float* fused) {
  int blocks = (bt.max_items + kThreads - 1) / kThreads;
  if (blocks < 1) blocks = 1;
  dim3 grid(blocks, g.hkv, bt.num_seqs);
  fuse_pool_kernel<<<grid, kThreads, 0, L.stream>>>(bt, pool_kind, pool_size, alpha, beta, scores,
                                                    prior, fused);
  return cudaGetLastError();
}

}  // namespace cc
