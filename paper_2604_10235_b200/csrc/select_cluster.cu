// A2 + A3 + A4 on a thread-block cluster: pooling, prior fusion and selection of the retained
// tokens of one (sequence, KV head) by up to eight CTAs that keep their slice of the items in
// shared memory.
//
// Ranking (protected first in sequence order, then larger fused value, then lower index) and the
// output (ascending token indices) are those of select.cu; what differs is where the data
// lives and how the CTAs cooperate:
//   * every item is read from global memory once; its order-preserving integer key and its
//     protected flag stay in shared memory.  A warp owns a run of consecutive items and walks it 32
//     at a time, so accesses are free of bank conflicts and ordered prefixes are ballots;
//   * what the CTAs exchange goes through distributed shared memory.  An exchange costs 1 to 2 us
//     whatever it carries, and at these sizes the kernel's time is mostly a chain of them and of
//     block barriers, so there are three: (1) protected weight and key range, (2) one histogram of
//     1024 bins over the range that is present, (3) the keys of the bin that holds the cut-off,
//     which every CTA then ranks for itself.  A bin usually holds a few dozen keys; one with more
//     than kCand is looked at again (one value? else a finer histogram).  What the ordered emission
//     needs to know about the CTAs before it follows from the same three (histograms and
//     candidates are read per CTA), so no prefix sums are exchanged;
//   * the passes over all items end with two masks per 32 items, from which the indices are written.
//   * with FUSED the kernel starts from the raw scores: it pools them (max / avg, or sums them
//     over a chunk), fuses them with the prior using the same explicitly rounded f32 operations
//     as fuse_pool.cu, and also stores the fused values.
// Measured with its launch, replayed alone (four digit rounds of 8 bits with an exchange each, and a
// contiguous run of items per thread, before): ragged batch of 64 problems, 8 k to 64 k tokens
// 52.6 -> 28.6 us, 256 problems of 2 k with a cap 19.0 -> 12.6, 32768 tokens x 8 heads 17.3 -> 12.6
// (7.4 -> 6.4 when the protected tokens fill the budget), 2048 x 2 9.6 -> 6.9.
// Loops are rolled unless what they hold in registers is the point: behind the score kernel this
// kernel's instructions come from L2, and a CTA of a small problem runs each of them once or twice.
// 75 -> 48 KB of code: whole call on 1691 tokens x 4 heads 22.4 -> 21.3 us, 2048 x 2 20.9 -> 19.9,
// 10007 x 4 with a causal window 41.1 -> 40.5; the widest slices (8192 items per CTA) give back 0.5 us.
#include <cooperative_groups.h>
#include <string.h>

#include <type_traits>

#include "cc_internal.cuh"
#include "select_common.cuh"

namespace cg = cooperative_groups;

namespace cc {

namespace {

constexpr int kBinBits = 10;
constexpr int kBins = 1 << kBinBits;
constexpr int kCand = 512;                // candidates of the cut-off bin that are ranked directly
constexpr int kMaxCluster = 8;
constexpr int kMaxWarps = 32;
constexpr int kStep = 4;                  // items a thread pools per part of the slice
constexpr int kMaxHalf = 32;              // half of the widest pooling window, rounded up
constexpr int kWords = 3;                 // words of an exchange

struct Cand {
  unsigned key, len;
};

struct __align__(16) Shared {
  unsigned hist[2][kBins];                      // alternate between rounds (peers read them)
  Cand own[kCand];                              // this CTA's candidates (peers read them)
  Cand all[kCand];                              // the cluster's, in rank order
  unsigned sub[256];                            // weights of the candidates by their next bits
  unsigned n_own;                               // its length (peers read it)
  unsigned xchg[2][kMaxCluster][kWords];        // [buffer copy][source CTA][word]: written by the peers
  unsigned warp_x[2][kWords][kMaxWarps];        // block reductions, alternating
  unsigned bcast[4];
};

struct ClusterParams {
  int cluster;               // CTAs per (sequence, head)
  int per;                   // steps of 32 items per warp, for the longest sequence
  int hkv;
  float theta;
  // FUSED only
  int pool_kind, pool_size;
  float alpha, beta;
  const float* prior;
  // per layer of the launch
  const float* scores[kMaxLayers];    // FUSED only
  float* fused[kMaxLayers];           // FUSED: written; plain: read
  int32_t* idx[kMaxLayers];
  int32_t* count[kMaxLayers];
};

// CLUSTER: CTAs per (sequence, head).  The loops over them are unrolled, and in code for eight that only looks how many
// there are, the fetch of instructions was most of a small problem's time: alone (no cluster, no exchange) 2048 tokens x 2
// heads 17.7 -> 16.2 us, 1500 x 8 21.0 -> 19.7; in twos and fours 7000 and 10000 tokens x 2, 4, 8 heads -1 to -2 %.  Eight looks
// all the same: with the number known the registers spill and 14000 tokens take 2 % more.
template <int THREADS, int CLUSTER>
struct Ctx {
  static constexpr int kWarps = THREADS / 32, kPeers = CLUSTER;
  Shared* sm;
  int width, rank_;
  __device__ int cluster() const { return CLUSTER == kMaxCluster ? width : CLUSTER; }
  __device__ int rank() const { return CLUSTER == 1 ? 0 : rank_; }
  unsigned n_xchg, n_red, n_hist;   // exchanges, block reductions, histograms so far (select the copy)

  __device__ void sync_all() {
    if (CLUSTER > 1) cg::this_cluster().sync(); else __syncthreads();
  }
  template <class T>
  __device__ const T* peer(const T* p, int r) const {
    if (CLUSTER == 1) return p;
    return cg::this_cluster().map_shared_rank(const_cast<T*>(p), r);
  }
  // Sum of v over the block.  Two copies of the warp totals: a copy is written again only after
  // the barrier of the reduction in between, which every warp reaches after it has read it.
  __device__ unsigned block_sum(unsigned v) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned* w = sm->warp_x[n_red++ & 1u][0];
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) w[warp] = v;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < kWarps ? w[lane] : 0u);
  }
  __device__ void block_sum2(unsigned& a, unsigned& b) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned(*w)[kMaxWarps] = sm->warp_x[n_red++ & 1u];
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    if (lane == 0) { w[0][warp] = a; w[1][warp] = b; }
    __syncthreads();
    a = __reduce_add_sync(0xffffffffu, lane < kWarps ? w[0][lane] : 0u);
    b = __reduce_add_sync(0xffffffffu, lane < kWarps ? w[1][lane] : 0u);
  }
  // Warp totals a, b (the same in all lanes): sums over the warps before this one.
  __device__ void warps_before2(unsigned& a, unsigned& b) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned(*w)[kMaxWarps] = sm->warp_x[n_red++ & 1u];
    if (lane == 0) { w[0][warp] = a; w[1][warp] = b; }
    __syncthreads();
    a = __reduce_add_sync(0xffffffffu, lane < warp ? w[0][lane] : 0u);
    b = __reduce_add_sync(0xffffffffu, lane < warp ? w[1][lane] : 0u);
  }
  // Sum of a, minimum of b, maximum of e over the block.
  __device__ void block_totals(unsigned& a, unsigned& b, unsigned& e) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned(*w)[kMaxWarps] = sm->warp_x[n_red++ & 1u];
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_min_sync(0xffffffffu, b);
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) { w[0][warp] = a; w[1][warp] = b; w[2][warp] = e; }
    __syncthreads();
    const int i = lane < kWarps ? lane : 0;
    a = __reduce_add_sync(0xffffffffu, lane < kWarps ? w[0][i] : 0u);
    b = __reduce_min_sync(0xffffffffu, w[1][i]);
    e = __reduce_max_sync(0xffffffffu, w[2][i]);
  }
  // Exclusive prefix sum over the threads of the block.
  __device__ unsigned block_scan(unsigned v) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    unsigned* w = sm->warp_x[n_red++ & 1u][0];
    if (lane == 31) w[warp] = inc;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < warp ? w[lane] : 0u) + inc - v;
  }
  // Words of every CTA to every CTA: thread r < C stores this CTA's into peer r's shared memory
  // (remote stores need no round trip), the cluster barrier publishes them.  Two buffer copies: a
  // CTA writes copy k & 1 for exchange k only after the barrier of exchange k - 1, which every
  // peer reaches after it has read exchange k - 2.
  __device__ const unsigned (*publish(const unsigned (&w)[kWords]))[kWords] {
    const unsigned bf = n_xchg++ & 1u;
    if ((int)threadIdx.x < cluster()) {
      unsigned* dst = CLUSTER == 1 ? sm->xchg[bf][0] : cg::this_cluster().map_shared_rank(&sm->xchg[bf][rank()][0], (int)threadIdx.x);
#pragma unroll
      for (int i = 0; i < kWords; ++i) dst[i] = w[i];
    }
    sync_all();
    return sm->xchg[bf];
  }
};

// Where the cut-off among a set of items lies.
struct Cut {
  unsigned T;             // items with key > T are above it
  bool whole;             // ... those with key == T too (nothing is tied)
  unsigned above;         // token weight above it
  unsigned above_before;  // ... of that in the CTAs before this one
  unsigned tied_before;   // token weight with key == T in the CTAs before this one
};

// Finds T such that weight(key > T) < R <= weight(key >= T), 1 <= R <= total weight of the
// eligible items, whose keys lie in [kmin, kmax].  get(li, key, len) tells whether the local
// item li is eligible; a warp calls it for its items [lo, hi) 32 at a time.
template <int THREADS, int CLUSTER, class Get>
__device__ Cut find_cut(Ctx<THREADS, CLUSTER>& c, int lo, int hi, unsigned R, unsigned kmin, unsigned kmax, unsigned max_len,
                        bool allow_whole, Get get) {
  constexpr int kPeers = CLUSTER;
  Shared& sm = *c.sm;
  const int lane = threadIdx.x & 31;
  const unsigned range = kmax - kmin;
  Cut cut{kmin, false, 0u, 0u, 0u};
  if (range == 0) {                       // one key value: everything is tied
    unsigned mine = 0;
#pragma unroll 1
    for (int li = lo + lane; li < hi; li += 32) {
      unsigned key, len;
      if (get(li, key, len)) mine += len;
    }
    if (CLUSTER == 1) return cut;
    unsigned w[kWords] = {c.block_sum(mine), 0u, 0u};
    const unsigned(*x)[kWords] = c.publish(w);
#pragma unroll 1
    for (int r = 0; r < c.rank(); ++r) cut.tied_before += x[r][0];
    return cut;
  }
  if (threadIdx.x < 256) sm.sub[threadIdx.x] = 0;     // (published by the barriers below)
  unsigned below = 0;                     // this thread's share of above_before
  const int sh = __clz(range);
  unsigned prefix = 0, remaining = R;     // resolved high bits of the shifted keys; rank inside them
  int shift = 32;                         // ... bits [31, shift)
  bool rank_keys = false;                 // the bin's keys have to be listed and ranked
#pragma unroll 1
  for (;;) {
    const int bits = min(kBinBits, shift), top = shift;
    shift -= bits;
    // two copies: a copy is cleared again only after the barrier of the histogram in between
    unsigned* h = sm.hist[c.n_hist & 1u];
    if (c.n_hist++ > 0) {                 // (the first one is clear from the start)
#pragma unroll 1
      for (int i = threadIdx.x; i < kBins; i += THREADS) h[i] = 0;
      __syncthreads();
    }
#pragma unroll 1
    for (int li = lo + lane; li < hi; li += 32) {
      unsigned key, len;
      if (!get(li, key, len)) continue;
      const unsigned kk = (key - kmin) << sh;
      if (top == 32 || (kk >> top) == (prefix >> top)) atomicAdd(&h[(kk >> shift) & ((1u << bits) - 1u)], len);
    }
    c.sync_all();
    // Thread t < kBins / 4 owns four bins, counted from the top, so a forward scan walks the keys
    // down; a peer's four are one 16-byte load (the exchange is paid per request: 4-byte loads by
    // all threads made this step 4 us long in clusters of eight), and all peers' are requested
    // before the first is used.
    constexpr int kOwn = 4;
    const bool owner = threadIdx.x < kBins / kOwn;
    const int b0 = owner ? kBins - kOwn - (int)threadIdx.x * kOwn : 0;
    unsigned n[kOwn] = {0u, 0u, 0u, 0u}, nb[kOwn] = {0u, 0u, 0u, 0u};   // weight per bin: all CTAs, those before this one
    if (owner) {
      uint4 v[kPeers];
#pragma unroll
      for (int r = 0; r < kPeers; ++r)
        v[r] = r < c.cluster() ? *reinterpret_cast<const uint4*>(c.peer(h + b0, r)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int r = 0; r < kPeers; ++r) {
        n[0] += v[r].x; n[1] += v[r].y; n[2] += v[r].z; n[3] += v[r].w;
        if (r < c.rank()) { nb[0] += v[r].x; nb[1] += v[r].y; nb[2] += v[r].z; nb[3] += v[r].w; }
      }
    }
    unsigned sum = 0;
#pragma unroll
    for (int i = 0; i < kOwn; ++i) sum += n[i];
    unsigned excl = c.block_scan(sum);
#pragma unroll
    for (int i = kOwn - 1; i >= 0; --i) {
      if (owner && excl < remaining && remaining <= excl + n[i]) {
        sm.bcast[0] = (unsigned)(b0 + i);
        sm.bcast[1] = remaining - excl;
        sm.bcast[2] = n[i];
        sm.bcast[3] = nb[i];
      }
      excl += n[i];
    }
    __syncthreads();
    const unsigned bin = sm.bcast[0], in_bin = sm.bcast[2], in_bin_before = sm.bcast[3];
    remaining = sm.bcast[1];
#pragma unroll
    for (int i = 0; i < kOwn; ++i)
      if ((unsigned)(b0 + i) > bin) below += nb[i];
    prefix |= bin << shift;
    cut.T = kmin + (prefix >> sh);
    if (allow_whole && remaining == in_bin) {   // the whole bin is above the cut: nothing is tied
      cut.whole = true;
      cut.above = R;
      cut.above_before = in_bin_before;
      break;
    }
    cut.above = R - remaining;
    if (shift == 0) {                     // every bit resolved: the bin is one key value
      cut.tied_before = in_bin_before;
      break;
    }
    if (in_bin <= (unsigned)(kCand - 1) * max_len) { rank_keys = true; break; }
    // a crowded bin is often a single value (equal distances, clamped scores): look before refining
    unsigned lo_k = 0xffffffffu, hi_k = 0u;
#pragma unroll 1
    for (int li = lo + lane; li < hi; li += 32) {
      unsigned key, len;
      if (!get(li, key, len) || (((key - kmin) << sh) >> shift) != (prefix >> shift)) continue;
      lo_k = min(lo_k, key);
      hi_k = max(hi_k, key);
    }
    unsigned a0 = 0u;
    c.block_totals(a0, lo_k, hi_k);
    if (CLUSTER > 1) {
      const unsigned w[kWords] = {lo_k, hi_k, 0u};
      const unsigned(*x)[kWords] = c.publish(w);
#pragma unroll 1
      for (int r = 0; r < c.cluster(); ++r) {
        lo_k = min(lo_k, x[r][0]);
        hi_k = max(hi_k, x[r][1]);
      }
    }
    if (lo_k == hi_k) {
      cut.T = lo_k;
      cut.tied_before = in_bin_before;
      break;
    }
  }
  unsigned gt_before = below, eq_before = 0;
  if (rank_keys) {
    // Behind this search's histograms all peers have read what an earlier search left in the counter.
    // (A counter per search cleared at the kernel's start, or the clearing right behind the histogram's
    // barrier, cost 0.2-0.3 us on one shape or another.)
    if (threadIdx.x == 0) sm.n_own = 0;
    __syncthreads();
    // the bin's keys, listed per CTA and read by all of them in rank order
#pragma unroll 1
    for (int li = lo + lane; li < hi; li += 32) {
      unsigned key, len;
      if (!get(li, key, len)) continue;
      if ((((key - kmin) << sh) >> shift) == (prefix >> shift)) sm.own[atomicAdd(&sm.n_own, 1u)] = Cand{key, len};
    }
    c.sync_all();
    unsigned first[kPeers + 1];        // places of the CTAs' lists in the common one
    first[0] = 0;
#pragma unroll
    for (int r = 0; r < kPeers; ++r) first[r + 1] = r < c.cluster() ? *c.peer(&sm.n_own, r) : 0u;
    unsigned before = 0;                    // (a sum, not first[rank]: that would put the array into local memory)
#pragma unroll
    for (int r = 0; r < kPeers; ++r) {
      if (r < c.rank()) before += first[r + 1];
      first[r + 1] += first[r];
    }
    const unsigned total = first[kPeers];
    const int sub_bits = min(8, shift), sub_shift = shift - sub_bits;
    auto sub_bin = [&](unsigned key) { return (((key - kmin) << sh) >> sub_shift) & ((1u << sub_bits) - 1u); };
    const bool refine = total > 64;         // narrow a long list down by the next bits before ranking
#pragma unroll 1
    for (unsigned i = threadIdx.x; i < total; i += THREADS) {
      int r = 0;
      unsigned at = i;
#pragma unroll
      for (int k = 1; k < kPeers; ++k)
        if (i >= first[k]) { r = k; at = i - first[k]; }
      const Cand o = c.peer(sm.own, r)[at];
      sm.all[i] = o;
      if (refine) atomicAdd(&sm.sub[sub_bin(o.key)], o.len);
    }
    __syncthreads();
    unsigned sub = 0;
    if (refine) {                           // every warp finds the sub-bin for itself (lane l: bins 255 - 8 l ...)
      unsigned n8[8], sum = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { n8[i] = sm.sub[255 - 8 * lane - i]; sum += n8[i]; }
      unsigned inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      unsigned excl = inc - sum;
      bool found = false;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (excl < remaining && remaining <= excl + n8[i]) { sub = 255 - 8 * lane - i; found = true; }
        excl += n8[i];
      }
      sub = __shfl_sync(0xffffffffu, sub, __ffs(__ballot_sync(0xffffffffu, found)) - 1);
    }
    // a warp ranks one key against all others
#pragma unroll 1
    for (unsigned i = threadIdx.x >> 5; i < total; i += THREADS / 32) {
      const unsigned key = sm.all[i].key;
      if (refine && sub_bin(key) != sub) continue;
      unsigned gt = 0, eq = 0;
#pragma unroll 1
      for (unsigned j = lane; j < total; j += 32) {
        const Cand o = sm.all[j];
        gt += o.key > key ? o.len : 0u;
        eq += o.key == key ? o.len : 0u;
      }
      gt = __reduce_add_sync(0xffffffffu, gt);
      eq = __reduce_add_sync(0xffffffffu, eq);
      if (lane == 0 && gt < remaining && remaining <= gt + eq) { sm.bcast[0] = key; sm.bcast[1] = gt; }
    }
    __syncthreads();
    cut.T = sm.bcast[0];
    cut.above += sm.bcast[1];
#pragma unroll 1
    for (unsigned i = threadIdx.x; i < before; i += THREADS) {
      const Cand o = sm.all[i];
      if (o.key > cut.T) gt_before += o.len;
      if (o.key == cut.T) eq_before += o.len;
    }
  }
  if (CLUSTER > 1) {
    c.block_sum2(gt_before, eq_before);
    cut.above_before += gt_before;
    cut.tied_before += eq_before;
  }
  return cut;
}

// CHUNKED instantiations rank fixed chunks of bt.chunk tokens; the others are compiled for
// token-level items only (bt.chunk == 1), which keeps their code short.  CAPPED ones (any sequence of the launch has a
// cap on its protected tokens, and all CHUNKED ones) hold the search for the cap; without it whole calls on 2000 to 70000
// tokens take 1 to 3 % less.
template <bool FUSED, bool CHUNKED, bool CAPPED, int THREADS, int CLUSTER>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
select_cluster_kernel(const __grid_constant__ BatchTable bt, const __grid_constant__ ClusterParams P) {
  extern __shared__ __align__(16) uint8_t dyn[];
  Shared& sm = *reinterpret_cast<Shared*>(dyn);
  Ctx<THREADS, CLUSTER> c;
  c.sm = &sm;
  c.width = P.cluster;
  c.rank_ = CLUSTER == 1 ? 0 : (int)cg::this_cluster().block_rank();
  c.n_xchg = c.n_red = c.n_hist = 0;

  pdl_launch_dependents();
  if (CLUSTER > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // this CTA has started
  const int h = blockIdx.y, s = blockIdx.z;
  const SeqInfo& q = bt.seq[s];
  const int m = q.n_items, cs = CHUNKED ? bt.chunk : 1;
  const int slice = (m + c.cluster() * THREADS - 1) / (c.cluster() * THREADS) * THREADS;     // items per CTA, a multiple of 32
  const int cta_lo = min(m, c.rank() * slice), cta_items = min(m, cta_lo + slice) - cta_lo;
  unsigned* keys = reinterpret_cast<unsigned*>(dyn + sizeof(Shared));
  uint8_t* flags = reinterpret_cast<uint8_t*>(keys + P.per * THREADS);
  const float* p = P.prior + q.tok_off;
  int32_t* out = P.idx[q.layer] + (int64_t)h * bt.b_tot + q.idx_off;
  const unsigned keep = (unsigned)q.keep;
  const float theta = P.theta;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the run of items of this warp
  const int run = slice / (THREADS / 32);
  const int lo = min(cta_items, warp * run), hi = min(cta_items, lo + run);

  auto item_len = [&](int li) -> unsigned {
    if (cs == 1) return 1u;
    const int i = cta_lo + li;
    return (unsigned)(min(q.n, (i + 1) * cs) - i * cs);
  };
#pragma unroll 1
  for (int i = threadIdx.x; i < kBins; i += THREADS) sm.hist[0][i] = 0;

  // FUSED runs right after the second score pass, which starts only once the caller's inputs are complete and all that was
  // enqueued before the call has ended: what the priors decide, it does before it waits for the scores
  if (!FUSED) pdl_wait();
  // ---- priors: parked in the key slots, with the protected flags, the protected weight and, when there is a cap, the range
  // of the protected items' priors (loads are issued four or eight at a time)
  const bool capped = CAPPED && q.span_cap >= 0;
  unsigned forced_tokens = 0, forced_before = 0;              // before: in the CTAs before this one
  unsigned pri_lo = 0xffffffffu, pri_hi = 0u;
  const bool flags_later = FUSED && !CHUNKED && !capped;      // with the scores, four to a word
  auto park = [&](int li, float pr) {
    const bool forced = pr >= theta;
    keys[li] = __float_as_uint(pr);
    if (flags_later) return;
    flags[li] = forced ? 1 : 0;
    if (!forced) return;
    forced_tokens += item_len(li);
    if (capped) {
      const unsigned pk = mono_key(pr);
      pri_lo = min(pri_lo, pk);
      pri_hi = max(pri_hi, pk);
    }
  };
  auto parked = [&](int li) -> float { return __uint_as_float(keys[li]); };
  if (cs == 1) {
#pragma unroll 1
    for (int t0 = threadIdx.x; t0 < cta_items; t0 += 4 * THREADS) {
      float b[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) b[k] = t0 + k * THREADS < cta_items ? p[cta_lo + t0 + k * THREADS] : 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (t0 + k * THREADS < cta_items) park(t0 + k * THREADS, b[k]);
    }
  } else {
#pragma unroll 1
    for (int li = threadIdx.x; li < cta_items; li += THREADS) {
      const int t0 = (cta_lo + li) * cs, t1 = min(q.n, t0 + cs);
      float pr = -INFINITY;
#pragma unroll 1
      for (int j0 = t0; j0 < t1; j0 += 8) {
        float b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) b[k] = j0 + k < t1 ? p[j0 + k] : -INFINITY;
#pragma unroll
        for (int k = 0; k < 8; ++k) pr = fmaxf(pr, b[k]);
      }
      park(li, pr);
    }
  }
  // Sum (and the sum over the CTAs before this one), minimum and maximum over the cluster (the block reduction's barrier also
  // publishes what was stored to shared memory).
  bool started = CLUSTER == 1;
  auto totals = [&](unsigned& sum, unsigned& before, unsigned& lo0, unsigned& hi0) {
    c.block_totals(sum, lo0, hi0);
    if (CLUSTER == 1) return;
    if (!started) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // so have the others
    started = true;
    const unsigned w[kWords] = {sum, lo0, hi0};
    const unsigned(*x)[kWords] = c.publish(w);
    sum = before = 0;
#pragma unroll 1
    for (int r = 0; r < c.cluster(); ++r) {
      if (r == c.rank()) before = sum;
      sum += x[r][0];
      lo0 = min(lo0, x[r][1]);
      hi0 = max(hi0, x[r][2]);
    }
  };

  // ---- stage 1: cap on the protected items (longest prefix by (prior desc, index asc) within B_span), which hangs on the priors
  // alone and is found before the scores are there; stage 2: cut-off among the unprotected items; one copy of the search.
  // (3 us of search less behind the scores: 32 chunks 243.8 -> 239.7 us, all layers -1 %; 3277 chunks of ten tokens, whose
  // priors had been read with the scores, 56.3 -> 54.0.  Writing the indices as early where protected items fill the budget
  // takes an exchange more in every call: 32768 tokens in clusters of eight +4 %.)
  Cut cut{0u, false, 0u, 0u, 0u};
#pragma unroll 1
  for (int stage = capped ? 1 : 2; stage <= 2; ++stage) {
    const bool first = stage == 1;
    const unsigned cap = (unsigned)q.span_cap;
    unsigned key_lo = pri_lo, key_hi = pri_hi;      // of the items the search is among
    if (first) {
      totals(forced_tokens, forced_before, key_lo, key_hi);
      if (forced_tokens <= cap) continue;
    } else {
      key_lo = 0xffffffffu;
      key_hi = 0u;
      // ---- keys of the CTA's slice (coalesced over the block)
      auto tally = [&](int li, unsigned key) {
        keys[li] = key;
        if (flags[li]) return;
        key_lo = min(key_lo, key);
        key_hi = max(key_hi, key);
      };
      if (FUSED) {
        pdl_wait();                                   // the scores are complete from here on
        const float* u = P.scores[q.layer] + (int64_t)h * bt.n_tot + q.tok_off;
        const int half = (cs == 1 && P.pool_kind != CC_POOL_NONE) ? P.pool_size / 2 : 0;
        auto fuse = [&](float val, float pr) {
          return mono_key(__fadd_rn(__fmul_rn(P.alpha, val), __fmul_rn(P.beta, pr)));
        };
        // Keys and flags of four items in place of their parked priors.  Bound, like the pooling above it, by issue slots (26
        // items a thread: 1.2 us a part of four): bounds as one unsigned compare, two taps per step, and the cap's
        // prior range on its own took the load of a 52437-token sequence by two CTAs from 10.9 to 8.4 us, the call on 2048
        // tokens x 2 heads 18.7 -> 18.2, 10007 x 4 38.9 -> 38.4, 32768 x 8 -0.9 %.  (Walking the slice four items to a lane in the search
        // as well: 65536-token batches -0.5 %, small calls +1 to 2 %.)
        auto store4 = [&](int l4, const float (&v)[4], float4 pr) {
          const uint4 k4 = make_uint4(fuse(v[0], pr.x), fuse(v[1], pr.y), fuse(v[2], pr.z), fuse(v[3], pr.w));
          const int left = cta_items - l4;
          const unsigned key[4] = {k4.x, k4.y, k4.z, k4.w};
          unsigned f = 0;
          if (capped) {
            f = *reinterpret_cast<const unsigned*>(flags + l4);
          } else {
            f = (pr.x >= theta ? 1u : 0u) | (left > 1 && pr.y >= theta ? 1u << 8 : 0u) | (left > 2 && pr.z >= theta ? 1u << 16 : 0u) |
                (left > 3 && pr.w >= theta ? 1u << 24 : 0u);
            forced_tokens += __popc(f);
            *reinterpret_cast<unsigned*>(flags + l4) = f;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const bool counts = j < left && !(f >> (8 * j) & 255u);
            key_lo = min(key_lo, counts ? key[j] : 0xffffffffu);
            key_hi = max(key_hi, counts ? key[j] : 0u);
          }
          *reinterpret_cast<uint4*>(keys + l4) = k4;
        };
        if (cs == 1) {
          // The scores go through two staging buffers of kStep * THREADS items and the pooling halo
          // (zero outside the sequence, which is neutral for the maximum too: scores are not
          // negative); a part is requested while the one before it is pooled.
          float* us = reinterpret_cast<float*>(flags + P.per * THREADS);
          const int part = kStep * THREADS, pitch = part + 2 * kMaxHalf;
          float a[kStep + 1];
          // element e of the slice with its halo is score e - half of the slice; those of [e_lo, e_hi) exist
          const float* uh = u + cta_lo - half;
          const int e_lo = max(0, half - cta_lo);
          const unsigned e_span = (unsigned)max(0, min(cta_items + 2 * half, q.n - cta_lo + half) - e_lo);
          auto request = [&](int c0) {
            const int e = c0 + (int)threadIdx.x;
#pragma unroll
            for (int k = 0; k < kStep; ++k) a[k] = (unsigned)(e + k * THREADS - e_lo) < e_span ? uh[e + k * THREADS] : 0.0f;
            a[kStep] = (int)threadIdx.x < 2 * half && (unsigned)(e + part - e_lo) < e_span ? uh[e + part] : 0.0f;
          };
          if (cta_items > 0) request(0);
#pragma unroll 1
          for (int c0 = 0, buf = 0; c0 < cta_items; c0 += part, buf ^= 1) {
            float* ub = us + buf * pitch;
#pragma unroll
            for (int k = 0; k < kStep; ++k) ub[threadIdx.x + k * THREADS] = a[k];
            if ((int)threadIdx.x < 2 * half) ub[threadIdx.x + part] = a[kStep];
            __syncthreads();
            if (c0 + part < cta_items) request(c0 + part);
            const int l4 = c0 + 4 * (int)threadIdx.x;
            if (l4 < cta_items) {
              const float4 pr = *reinterpret_cast<const float4*>(keys + l4);       // the parked priors
              float v[4];
              // four windows, two taps per step; averages are left-to-right sums, then one division
              const float* w = ub + 4 * threadIdx.x;
              const float4 x = *reinterpret_cast<const float4*>(w);
              float y0 = x.y, y1 = x.z, y2 = x.w;
              v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
              if (P.pool_kind == CC_POOL_MAX) {
#pragma unroll 1
                for (int d = 1; d < 2 * half; d += 2) {
                  const float2 y = *reinterpret_cast<const float2*>(w + d + 3);
                  v[0] = max3(v[0], y0, y1); v[1] = max3(v[1], y1, y2); v[2] = max3(v[2], y2, y.x); v[3] = max3(v[3], y.x, y.y);
                  y0 = y2; y1 = y.x; y2 = y.y;
                }
              } else if (half > 0) {
#pragma unroll 1
                for (int d = 1; d < 2 * half; d += 2) {
                  const float2 y = *reinterpret_cast<const float2*>(w + d + 3);
                  v[0] = __fadd_rn(__fadd_rn(v[0], y0), y1); v[1] = __fadd_rn(__fadd_rn(v[1], y1), y2);
                  v[2] = __fadd_rn(__fadd_rn(v[2], y2), y.x); v[3] = __fadd_rn(__fadd_rn(v[3], y.x), y.y);
                  y0 = y2; y1 = y.x; y2 = y.y;
                }
#pragma unroll 1
                for (int j = 0; j < 4; ++j) {       // (rotates: one copy of the division)
                  const float y = __fdiv_rn(v[0], (float)(2 * half + 1));
                  v[0] = v[1]; v[1] = v[2]; v[2] = v[3]; v[3] = y;
                }
              }
              store4(l4, v, pr);
            }
          }
        } else {
#pragma unroll 1
          for (int li = threadIdx.x; li < cta_items; li += THREADS) {
            // chunk sum in token order; the loads of eight tokens are issued before they are used
            const int t0 = (cta_lo + li) * cs, t1 = min(q.n, t0 + cs);
            float val = 0.0f;
#pragma unroll 1
            for (int j0 = t0; j0 < t1; j0 += 8) {
              float a[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) a[k] = j0 + k < t1 ? u[j0 + k] : 0.0f;
#pragma unroll
              for (int k = 0; k < 8; ++k)
                if (j0 + k < t1) val = (j0 + k == t0) ? a[k] : __fadd_rn(val, a[k]);
            }
            tally(li, fuse(val, parked(li)));
          }
        }
      } else {
        const float* f = P.fused[q.layer] + (int64_t)h * bt.m_tot + q.item_off;
#pragma unroll 1
        for (int l0 = threadIdx.x; l0 < cta_items; l0 += 4 * THREADS) {
          float a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) a[k] = l0 + k * THREADS < cta_items ? f[cta_lo + l0 + k * THREADS] : 0.0f;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (l0 + k * THREADS < cta_items) tally(l0 + k * THREADS, mono_key(a[k]));
        }
      }
      unsigned sum = capped ? 0u : forced_tokens, before = 0u;
      totals(sum, before, key_lo, key_hi);
      if (!capped) { forced_tokens = sum; forced_before = before; }
      if (forced_tokens >= keep) break;       // protected items alone fill the budget: first B in order
    }
    cut = find_cut(c, lo, hi, first ? cap + 1u : keep - forced_tokens, key_lo, key_hi,
                   (unsigned)cs, !first, [&](int li, unsigned& key, unsigned& len) {
                     if ((flags[li] != 0) != first) return false;
                     key = first ? mono_key(parked(li)) : keys[li];
                     len = item_len(li);
                     return true;
                   });
    if (!first) break;
    unsigned ties = 0, none = 0;
#pragma unroll 1
    for (int li = lo + lane; li < hi; li += 32)
      if (flags[li] && mono_key(parked(li)) == cut.T) ties += item_len(li);
    ties = __reduce_add_sync(0xffffffffu, ties);
    c.warps_before2(ties, none);
    unsigned tie_run = cut.tied_before + ties, kept = 0;
#pragma unroll 1
    for (int l0 = lo; l0 < hi; l0 += 32) {
      const int li = l0 + lane;
      const bool forced = li < hi && flags[li];
      const unsigned pk = forced ? mono_key(parked(li)) : 0u, len = forced ? item_len(li) : 0u;
      const unsigned tm = __ballot_sync(0xffffffffu, forced && pk == cut.T);
      const unsigned before = tie_run + __popc(tm & ((1u << lane) - 1u)) * (unsigned)cs;
      tie_run += __popc(tm) * (unsigned)cs;
      if (!forced) continue;
      if (pk > cut.T || (pk == cut.T && cut.above + before + len <= cap)) kept += len;
      else flags[li] = 0;
    }
    if (cs == 1) {                 // items of one token fill the cap exactly
      forced_tokens = cap;
      forced_before = cut.above_before + min(cut.tied_before, cap - cut.above);
    } else {
      forced_tokens = c.block_sum(kept);
      if (CLUSTER > 1) {
        const unsigned w[kWords] = {forced_tokens, 0u, 0u};
        const unsigned(*x)[kWords] = c.publish(w);
        forced_tokens = forced_before = 0;
#pragma unroll 1
        for (int r = 0; r < c.cluster(); ++r) {
          if (r == c.rank()) forced_before = forced_tokens;
          forced_tokens += x[r][0];
        }
      }
    }
    __syncthreads();               // the load replaces parked priors and reads flags of other warps' items
  }
  const bool ties_are_forced = forced_tokens >= keep;
  if (ties_are_forced) cut = Cut{0u, false, 0u, 0u, 0u};
  const unsigned tie_budget = ties_are_forced ? keep : keep - forced_tokens - cut.above;
  // last read of a peer's shared memory is done: announce it now, wait for the peers at the
  // very end, and write the indices in between
  // (relaxed: nothing is published by it, so it need not wait for stores in flight)
  if (CLUSTER > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

  // ordered emission.  Items kept for sure (def) and the tied ones in sequence order,
  // until the budget is full
  auto classify = [&](int li, bool& def, bool& tie) {
    def = tie = false;
    if (li >= hi) return;
    if (flags[li]) {
      def = !ties_are_forced;
      tie = ties_are_forced;
    } else if (!ties_are_forced) {
      const unsigned key = keys[li];
      def = key > cut.T || (cut.whole && key == cut.T);
      tie = !cut.whole && key == cut.T;
    }
  };
  // Step k of a warp's run (at most 32 steps) leaves two masks of its 32 items in lane k, and the
  // indices are written from the masks: the passes over all items end here.  The fused
  // values are stored on the way, from their keys: earlier, the stores in flight would have to
  // land before every exchange of the CTAs.
  float* fo = FUSED ? P.fused[q.layer] + (int64_t)h * bt.m_tot + q.item_off + cta_lo : nullptr;
  unsigned defs = 0, ties = 0;
#pragma unroll 2
  for (int k = 0; k < run / 32; ++k) {
    const int li = lo + k * 32 + lane;
    bool def, tie;
    classify(li, def, tie);
    if (FUSED && li < hi) fo[li] = mono_value(keys[li]);
    const unsigned dm = __ballot_sync(0xffffffffu, def), tm = __ballot_sync(0xffffffffu, tie);
    if (lane == k) { defs = dm; ties = tm; }
  }
  // tokens of this lane's step and of the steps and warps before it
  const int base = lo + lane * 32, last = m - 1 - cta_lo - base;         // bit of the sequence's last item
  const unsigned cut_short = CHUNKED && last >= 0 && last < 32 ? (unsigned)(cs - (q.n - (m - 1) * cs)) << 1 : 0u;
  auto tokens = [&](unsigned mask) {
    unsigned n = (unsigned)__popc(mask) * (unsigned)cs;
    if (CHUNKED && cut_short && (mask >> last & 1u)) n -= cut_short >> 1;
    return n;
  };
  const unsigned def_own = tokens(defs), tie_own = tokens(ties);
  unsigned def_run = def_own, tie_run = tie_own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned a = __shfl_up_sync(0xffffffffu, def_run, o), b = __shfl_up_sync(0xffffffffu, tie_run, o);
    if (lane >= o) { def_run += a; tie_run += b; }
  }
  unsigned def_warps = __shfl_sync(0xffffffffu, def_run, 31), tie_warps = __shfl_sync(0xffffffffu, tie_run, 31);
  c.warps_before2(def_warps, tie_warps);
  def_run += def_warps - def_own + (ties_are_forced ? 0u : forced_before) + cut.above_before;
  tie_run += tie_warps - tie_own + (ties_are_forced ? forced_before : cut.tied_before);
  auto emit = [&](int li, bool tie, unsigned def_before, unsigned tie_before) {
    const unsigned len = item_len(li), pos = def_before + min(tie_before, tie_budget);
    const unsigned take = !tie ? len : (tie_before < tie_budget ? min(len, tie_budget - tie_before) : 0u);
    const int tok0 = (cta_lo + li) * cs;
#pragma unroll 1
    for (unsigned k = 0; k < take; ++k)
      if (pos + k < keep) out[pos + k] = tok0 + (int)k;
    return len;
  };
  if (run / 32 > 10) {           // a step per lane
#pragma unroll 1
    for (unsigned left = defs | ties; left; left &= left - 1u) {
      const int bit = __ffs(left) - 1;
      const bool tie = ties >> bit & 1u;
      const unsigned len = emit(base + bit, tie, def_run, tie_run);
      if (tie) tie_run += len; else def_run += len;
    }
  } else {                       // few steps: one after the other, an item per lane
    const unsigned lt = (1u << lane) - 1u;
    for (int k = 0; k < run / 32; ++k) {
      const unsigned dm = __shfl_sync(0xffffffffu, defs, k), tm = __shfl_sync(0xffffffffu, ties, k);
      const unsigned db = __shfl_sync(0xffffffffu, def_run, k) + __popc(dm & lt) * (unsigned)cs;
      const unsigned tb = __shfl_sync(0xffffffffu, tie_run, k) + __popc(tm & lt) * (unsigned)cs;
      if ((dm | tm) >> lane & 1u) emit(lo + k * 32 + lane, tm >> lane & 1u, db, tb);
    }
  }
  for (int i = (int)keep + c.rank() * THREADS + threadIdx.x; i < q.budget; i += c.cluster() * THREADS)
    out[i] = -1;
  if (c.rank() == 0 && threadIdx.x == 0) P.count[q.layer][q.src * P.hkv + h] = (int)keep;
  // no CTA may leave while a peer can still read its shared memory
  if (CLUSTER > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

size_t cluster_smem_bytes(int slots, int threads, bool staging) {
  size_t b = sizeof(Shared) + (size_t)slots * 5;                   // keys, flags
  if (staging) b += 2 * (size_t)(kStep * threads + 2 * kMaxHalf) * sizeof(float);
  return (b + 15) / 16 * 16;
}

template <bool FUSED, bool CHUNKED, bool CAPPED, int THREADS, int CLUSTER>
cudaError_t launch_one(const Launch& L, const BatchTable& bt, const Geometry& g, const ClusterParams& P, size_t smem) {
  auto kern = select_cluster_kernel<FUSED, CHUNKED, CAPPED, THREADS, CLUSTER>;
  const cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(CLUSTER, g.hkv, bt.num_seqs), dim3(THREADS), smem, L.stream, CLUSTER, bt, P);
}
// Shapes there is code for: those that are the cheapest (launch_cost) for some batch on 148 SMs.  Of the ones with 512 threads
// these are a CTA alone, for short sequences, and clusters of four and eight for chunks; the others lost to 1024 threads or to
// another width on each of 400000 batches (1 to 10^6 items, 1 to 128 sequences, 1 to 32 heads, chunks of 1 to 64 tokens).
constexpr bool has_shape(bool chunked, int cluster, int threads) {
  return threads == 1024 || cluster == 1 || (chunked && cluster >= 4);
}
template <bool FUSED, bool CHUNKED, bool CAPPED, int CLUSTER>
cudaError_t launch_width(const Launch& L, const BatchTable& bt, const Geometry& g, const ClusterParams& P, int threads, size_t smem) {
  if (threads == 1024) return launch_one<FUSED, CHUNKED, CAPPED, 1024, CLUSTER>(L, bt, g, P, smem);
  if constexpr (has_shape(CHUNKED, CLUSTER, 512)) return launch_one<FUSED, CHUNKED, CAPPED, 512, CLUSTER>(L, bt, g, P, smem);
  return cudaErrorInvalidConfiguration;
}
template <bool FUSED, bool CHUNKED, bool CAPPED>
cudaError_t launch_shape(const Launch& L, const BatchTable& bt, const Geometry& g, const ClusterParams& P, SelectShape sh,
                         size_t smem) {
  switch (sh.cluster) {
    case 1: return launch_width<FUSED, CHUNKED, CAPPED, 1>(L, bt, g, P, sh.threads, smem);
    case 2: return launch_width<FUSED, CHUNKED, CAPPED, 2>(L, bt, g, P, sh.threads, smem);
    case 4: return launch_width<FUSED, CHUNKED, CAPPED, 4>(L, bt, g, P, sh.threads, smem);
    default: return launch_width<FUSED, CHUNKED, CAPPED, 8>(L, bt, g, P, sh.threads, smem);
  }
}

// Two CTAs of 512 threads share an SM when their shared memory (and 1 KB that each is charged besides)
// fits its 228 KB.
constexpr size_t kPairSmem = (228 * 1024 - 2 * 1024) / 2;

int steps_per_warp(int max_items, int cluster, int threads) {
  return max_items > 0 ? (max_items + cluster * threads - 1) / (cluster * threads) : 1;
}

// Time of a launch with clusters of 1 << lc CTAs of `threads` threads, in us, from launches of one wave
// on a B200 (n = 2048 .. 131072 items, 2 .. 256 problems): a constant that grows with what the
// exchanges of wider clusters cost, something for the barriers of 1024 threads (less than in replays
// of this kernel alone: behind other kernels its code is cold, which more warps hide better), and
// 0.48 (0.6) us per item of a thread of 512 (1024).  A chunk's tokens count a fifth of an item each.
// A CTA of 1024 threads fills an SM, CTAs of 512 share it in pairs; a cluster sits inside one GPC, so
// fewer CTAs run at a time in wide ones.  (One CTA: 6.1 until it had its own code; with 4.8 3500 tokens x 2, 4, 8 heads -4 %,
// three sequences of up to 3000 -7 %; 5.2: 5000 tokens +1 %, 4.2: 7000 tokens +3 to 6 %.)
double launch_cost(const BatchTable& bt, int hkv, const SelectRoom& room, bool staging, int lc, int threads) {
  static const double base[4] = {4.8, 7.7, 7.8, 8.6};
  const int c = 1 << lc;
  const double per_thread = (bt.max_items + (bt.chunk > 1 ? 0.2 * bt.chunk * bt.max_items : 0.0)) / (double)(c * threads);
  const size_t smem = cluster_smem_bytes(steps_per_warp(bt.max_items, c, threads) * threads, threads, staging);
  const int ctas = bt.num_seqs * hkv * c, fit = threads == 512 && smem <= kPairSmem ? room.two[lc] : room.one[lc];
  const int waves = (ctas + fit - 1) / fit;
  const double slope = threads == 1024 ? 0.6 : (ctas > room.one[lc] ? 0.96 : 0.48);
  return waves * (base[lc] + (threads == 512 ? 0.0 : bt.chunk > 1 ? 1.0 : lc == 0 ? 0.8 : 0.3) + slope * per_thread);
}

}  // namespace

// CTAs that run at a time, in clusters of 1, 2, 4, 8: how many SMs the GPCs of a part have is not the same
// on all parts, so the runtime is asked, once per context.  (148, 148, 132, 120 on the part at hand; 296, 296,
// 284, 264 in pairs.)
cudaError_t query_select_room(SelectRoom* room) {
  auto one = select_cluster_kernel<true, false, true, 1024, 8>;
  auto two = select_cluster_kernel<true, true, true, 512, 8>;
  cudaError_t e = allow_smem(one);
  if (e == cudaSuccess) e = allow_smem(two);
  for (int lc = 0; lc <= 3 && e == cudaSuccess; ++lc) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1u << lc;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << lc);
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = kSmemPerCta;
    e = cudaOccupancyMaxActiveClusters(&room->one[lc], one, &cfg);
    if (e != cudaSuccess) break;
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = kPairSmem;
    e = cudaOccupancyMaxActiveClusters(&room->two[lc], two, &cfg);
    room->one[lc] <<= lc;
    room->two[lc] <<= lc;
  }
  return e;
}

// The cheapest shape; cluster 0 when a sequence has more items than the widest cluster holds.
SelectShape select_shape(const BatchTable& bt, int hkv, const SelectRoom& room, bool fused_input) {
  if (bt.max_items <= 0) return SelectShape{1, 512};
  SelectShape best{0, 0};
  double best_us = 1e30;
  for (int lc = 0; lc <= 3; ++lc)
    for (int threads = 512; threads <= 1024; threads += 512) {
      if (!has_shape(bt.chunk > 1, 1 << lc, threads) || room.one[lc] <= 0 || room.two[lc] <= 0) continue;
      if (steps_per_warp(bt.max_items, 1 << lc, threads) > 32) continue;   // a warp's run has at most 32 steps
      const double us = launch_cost(bt, hkv, room, fused_input && bt.chunk == 1, lc, threads);
      if (us < best_us) { best_us = us; best = SelectShape{1 << lc, threads}; }
    }
  return best;
}

cudaError_t launch_select_cluster(const Launch& L, const BatchTable& bt, const Geometry& g,
                                  float force_threshold, bool fused_input, int pool_kind,
                                  int pool_size, float alpha, float beta, const LayerPtrs& lp,
                                  const float* prior, SelectShape sh) {
  ClusterParams P;
  P.cluster = sh.cluster;
  P.per = steps_per_warp(bt.max_items, sh.cluster, sh.threads);
  P.hkv = g.hkv;
  P.theta = force_threshold;
  P.pool_kind = pool_kind;
  P.pool_size = pool_kind == CC_POOL_NONE ? 1 : pool_size;
  P.alpha = alpha;
  P.beta = beta;
  P.prior = prior;
  for (int l = 0; l < lp.n; ++l) {
    P.scores[l] = lp.scores[l];
    P.fused[l] = lp.fused[l];
    P.idx[l] = lp.idx[l];
    P.count[l] = lp.count[l];
  }
  const size_t smem = cluster_smem_bytes(P.per * sh.threads, sh.threads, fused_input && bt.chunk == 1);
  bool capped = false;
  for (int i = 0; i < bt.num_seqs; ++i) capped |= bt.seq[i].span_cap >= 0;
  if (fused_input)
    return bt.chunk > 1 ? launch_shape<true, true, true>(L, bt, g, P, sh, smem)
           : capped     ? launch_shape<true, false, true>(L, bt, g, P, sh, smem)
                        : launch_shape<true, false, false>(L, bt, g, P, sh, smem);
  return bt.chunk > 1 ? launch_shape<false, true, true>(L, bt, g, P, sh, smem)
         : capped     ? launch_shape<false, false, true>(L, bt, g, P, sh, smem)
                      : launch_shape<false, false, false>(L, bt, g, P, sh, smem);
}

}  // namespace cc

extern "C" void ccx_select_shape(int max_items, int num_seqs, int hkv, int chunk, int fused_input, const int* one,
                                 const int* two, int* cluster, int* threads) {
  static thread_local cc::BatchTable bt;
  bt.max_items = max_items;
  bt.num_seqs = num_seqs;
  bt.chunk = chunk;
  cc::SelectRoom room;
  for (int i = 0; i < 4; ++i) { room.one[i] = one[i]; room.two[i] = two[i]; }
  const cc::SelectShape sh = cc::select_shape(bt, hkv, room, fused_input != 0);
  *cluster = sh.cluster;
  *threads = sh.threads;
}
extern "C" int ccx_select_has_shape(int chunk, int cluster, int threads) {
  return cc::has_shape(chunk > 1, cluster, threads);
}
