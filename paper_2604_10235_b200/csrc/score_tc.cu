// A1, tensor-core mode (CC_MODE_BF16): window attention scores on sm_100a.
//
// u_h(j) = sum_r exp(s_rj - L_r) with s = q_r . k_j / sqrt(d) and L_r = log sum_j exp(s_rj),
// where r runs over the w * G query rows that share KV head h.  L_r needs every key before
// any column can be reduced, so the keys are streamed twice with the same persistent kernel:
//
//   pass 1  S = Q K^T with query rows on the MMA M axis: one TMEM lane, hence one thread, per
//           query row, so the running maximum and sum of exp need no cross-thread traffic.
//           Each CTA covers a contiguous span of key tiles and writes one (max, sum) pair per
//           row; the spans of a (sequence, head) are merged in pass 2.
//   pass 2  S^T = K Q^T with keys on the M axis: one thread per key, the query rows along the
//           TMEM columns, so u(j) is a plain in-thread sum and is stored coalesced.
//
// Pipeline per CTA (one CTA per SM, 608 threads): warp 0 issues TMA loads (K tiles of 128 keys
// through a ring of shared-memory stages, Q once per (sequence, head)), two warps issue
// tcgen05.mma into four TMEM accumulator buffers, sixteen warps drain the accumulators with
// tcgen05.ld and do the exp / reduction work while later tiles are being multiplied.
// All operands sit in shared memory in the 128-byte-swizzled K-major layout that both TMA
// and the MMA descriptors understand; Q and K simply swap the A / B roles between passes.
//
// TMEM holds four accumulator buffers of 128 columns; work item i (one 128 x 128 block of S or
// S^T) lands in buffer i mod 4.  The sixteen epilogue warps form four sets of four (one warp
// per TMEM lane quadrant); set k drains buffer k, so every scheduler hosts one warp of each set
// and the sets run staggered: while one set waits for its buffer to be refilled, the other
// three keep the special-function unit busy.  The exponentials are the bottleneck of both
// passes (16 per clock on the special-function unit against 8192 tensor flops per clock), and
// what counts is that the unit never idles: a warp reads 32 columns at a time, so it needs few
// registers and four warps fit per scheduler; scaling and accumulation use packed f32x2
// instructions; one pair of exponentials in three is evaluated on the FMA pipe instead
// (round to nearest integer, degree-3 polynomial for the fraction, exponent patched in by
// integer arithmetic; relative error 8e-5).
//
// Every wait on an mbarrier is bounded: when the bound is hit the kernel records
// CC_ERR_TIMEOUT, every role leaves its loop, TMEM is released and the kernel returns.
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "cc_internal.cuh"
#include "exp2_poly.cuh"

namespace cc {

namespace {

constexpr int kIssuers = 2;                               // MMA issuers: items go to them in pairs, one per epilogue set and turn
constexpr int kEpiWarps = 16;
constexpr int kThreads = (1 + kIssuers + kEpiWarps) * 32; // TMA, the MMA issuers, 16 epilogue warps
constexpr int kMmaWarpB = 2 + kEpiWarps;                  // second MMA issuer (the last warp)
static_assert(kThreads / 32 == kMmaWarpB + 1, "warps 0, 1, the epilogue warps, the second issuer");
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kMaxStages = 6;
constexpr uint32_t kPanelBytes = kTileKeys * 128;        // one 64-channel half of a K tile
constexpr uint32_t kStageBytes = 2 * kPanelBytes;        // 32 KB
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kBufCols = 128;                        // accumulator buffer stride
constexpr int kBufs = 4;                                  // accumulator buffers in TMEM
constexpr int kSets = 4;                                  // epilogue warp sets, one per buffer
constexpr uint32_t kSmemLimit = 232448;                   // 227 KB
constexpr float kLn2 = 0.6931471805599453f;

struct TcParams {
  int grid;            // CTAs (same for both passes)
  int total_tiles;     // H_kv * sum of tiles over the sequences
  int change;          // weight of the start of a (sequence, head) when the spans are cut
  long long weight;    // of all tiles and starts
  int halves;          // units of work per tile: 1, or 2 (its row blocks in two halves); HALVES of the kernel
  int rows;            // w * G
  int rows_pad;        // G * w_pad, a multiple of 16
  int w_pad;
  int n_stages;
  int n_sub;           // pass 1: 128-row blocks; pass 2: column chunks
  int sub_cols;        // pass 2: rows per column chunk (multiple of 16, <= 128)
  float2* part;        // [(grid + problems)][rows_pad] (max, sum) in the log2 domain
  float* lse;
  int64_t pool_rows;
  // K tile in shared memory.  Contiguous cache: two panels of 64 channels, each 128 rows of 128
  // bytes (8-row groups 1024 bytes apart, second panel 16 KB on).  Paged cache: one copy per page
  // lays the rows out in 8-token groups of 2 KB, first panel then second (8-row groups of a panel
  // 2048 bytes apart, second panel 1 KB on), whatever the page size.
  uint32_t k_sbo16;      // stride between 8-row groups of a panel, in 16-byte units
  uint32_t k_panel16;    // offset of the second panel, in 16-byte units
};

// Tensor maps and score arrays of the layers of a launch.
template <int LAYERS>
struct TcLayers {
  CUtensorMap q[LAYERS], k[LAYERS];
  float* scores[LAYERS];
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One probe of the barrier phase; the hardware may park the thread for up to the given number
// of nanoseconds while the phase is incomplete, so a waiting warp does not take issue slots
// from the warps that have work.
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
  return ok;
}
// Up to 64 probes in a short loop (a suspended thread is woken by every arrival in the CTA,
// whatever the barrier, so waiting threads go round often); whether the phase completed.
__device__ __forceinline__ bool mbar_spin(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 n;\n\tmov.u32 n, 64;\n"
      "W%=:\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "@p bra D%=;\n\tsub.u32 n, n, 1;\n\tsetp.ne.u32 q, n, 0;\n\t@q bra W%=;\n"
      "D%=:\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
  return ok != 0;
}
// This thread's stores to shared memory before, the tensor core's reads after.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// K tile copy with an L2 eviction-priority hint: pass 1 asks L2 to keep the tile (pass 2 reads
// it again), pass 2 marks it as the first to go.
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                 int c0, int c1, int c2, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}
// One page of a paged cache: box (64 channels, 8 tokens, 2 panels, page_size / 8 groups, 1 head).
__device__ __forceinline__ void tma_load_5d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                 int c3, int c4, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %3, %3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(c3), "r"(c4), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
               ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}
// One lane of the warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
  uint32_t yes;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(yes));
  return yes != 0;
}
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]),
        "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
        "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void epi_barrier() {      // the sixteen epilogue warps only
  asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max32(const uint32_t (&v)[32]) {
  float m0 = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
  float m1 = max3(__uint_as_float(v[3]), __uint_as_float(v[4]), __uint_as_float(v[5]));
#pragma unroll
  for (int i = 6; i < 30; i += 4) {
    m0 = max3(m0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
    m1 = max3(m1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
  }
  return max3(max3(m0, m1, __uint_as_float(v[30])), __uint_as_float(v[31]), __uint_as_float(v[31]));
}

// Instruction descriptor: bf16 x bf16 -> f32, both operands K-major.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t m, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

// Operands of the step of 16 channels that adds -L_r: ones from the keys' side; the rows' side is 16 bytes a row, the second 8
// channels of a group of rows lie on the next group's first and meet zeros.
__device__ __forceinline__ uint64_t ones_desc(const void* ones) {
  return (uint64_t)(((smem_u32(ones) & 0x3FFFFu) >> 4) | (8u << 16)) | ((uint64_t)(16u | (1u << 14)) << 32);
}
__device__ __forceinline__ uint64_t stat_desc(const void* rows) {
  return (uint64_t)(((smem_u32(rows) & 0x3FFFFu) >> 4) | (8u << 16)) | ((uint64_t)(8u | (1u << 14)) << 32);
}

// ------------------------------------------------------------------ shared state
struct Barriers {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t q_full, q_empty, l_full;
  uint64_t acc_full[kBufs], acc_empty[kBufs];
  uint64_t late_full[kBufs];         // ADDED: -L_r has been added to the first item of the set in the (sequence, head)
  uint64_t u_full[8][4];             // pass 2: the other sets' partial sums of (slot, quadrant)
  uint64_t edge_full[2][4];          // ... of a first / last tile of which the CTA has one half
};

struct Misc {                        // behind the ring of K tiles in dynamic shared memory
  union {
    float2 xchg[kSets][kMaxRows];    // (max, sum) hand-over: pass 1 per set, pass 2 while merging (the first of them)
    struct {
      float u_part[8][kSets - 1][kTileKeys];   // pass 2: partial column sums, slot = tile & 7
      uint4 ones[2 * kTileKeys];     // pass 2: the other side of the operand with -L_r: 128 keys x 16 channels, (1, 1, 1, 0, ...)
    };
  };
  float edge_part[2][kTileKeys];     // pass 2: partial column sums of cut tiles
  Barriers bar;
  long long span[2];                 // first unit of the CTA, first unit behind it
  uint32_t tmem_base;
  volatile int abort_flag;
};
static_assert(sizeof(Misc) % 16 == 0, "the operand behind Misc starts on 16 bytes");

struct Pipe {
  Misc* misc;
  DeviceStatus* status;
};

// Bounded wait; false (and the abort flag set) when the bound is hit or another role gave up.
// A healthy wait lasts microseconds; the bound is 50 ms of wall-clock time (the global timer is
// read only after the first probes have failed, and then once every eight probes).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Every lane of the warp waits; the answer is the same in all of them.
__device__ __forceinline__ bool warp_wait(const Pipe& p, uint64_t* bar, uint32_t parity, int where) {
  const uint32_t b = smem_u32(bar);
  if (__all_sync(0xffffffffu, mbar_try_wait(b, parity))) return true;
  unsigned long long t0 = 0;
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_spin(b, parity))) return true;
    if (__any_sync(0xffffffffu, p.misc->abort_flag)) return false;
    const unsigned long long now = global_ns();
    if (t0 == 0) t0 = now;
    if (__any_sync(0xffffffffu, now - t0 > 50ull * 1000 * 1000)) break;
  }
  p.misc->abort_flag = 1;
  if ((threadIdx.x & 31) == 0) report_error(p.status, CC_ERR_TIMEOUT, where);
  __syncwarp();
  return false;
}

// ------------------------------------------------------------------ the four drains
// One accumulator buffer through a warp, 32 columns at a time.  The common forms and the masked ones
// are loops of their own, so that the common ones hold no range tests and no moves of values that
// only the others overwrite.  Bound by the exponentials and the issue slots around them: the arithmetic and the reads alone reach 20.1
// per clock per SM.
__device__ __forceinline__ void hand_back(uint32_t empty_bar, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(empty_bar);
}

// pass 1, all 128 keys count.  The reference of the exponentials only has to be near the row
// maximum, not equal to it: it is replaced when a value lies more than 2^64 above it.  It is an integer, for the sake of
// the polynomial's arguments.  Only the first chunk of a row and the last of an item look at their maximum beforehand, a serial stretch
// of 16 instructions, a vote and a branch before the first exponential.  The sums of the others, which grow beyond 2^70 or are no numbers
// where a value is out of the arithmetic's range, and the ranges of the reference and of the last chunk are looked at before the
// buffer goes back; when one is not as it should be, nothing has been changed and the answer is false: the caller goes through
// the item again, chunk by chunk.  HALF: only the lanes in `real` decide; the others
// multiply whatever lies behind the rows of Q, keys among it, whose products with keys are large where a channel of all keys is
// (300 in two channels, 65536 tokens: 8 heads of 48 rows 49.7 -> 46.7 us, causal 59 -> 50, 4 of 448 rows causal 80 -> 74; without
// such channels 48 rows +1 us).
constexpr float kRedo = 1.1805916e21f;     // 2^70
constexpr float kMaxProduct = 1.0995116e12f;     // 2^40
template <bool HALF>
__device__ __forceinline__ bool drain_keys(uint32_t addr, uint32_t empty_bar, int lane, unsigned real, float& m_run, float& l_run) {
  uint64_t acc[2] = {0ull, 0ull};
  float m = m_run, l = l_run;
  PolyRef r = poly_ref(m);
  bool look = __any_sync(0xffffffffu, m == -INFINITY);
#pragma unroll 1
  for (int cc0 = 0; cc0 < kTileKeys; cc0 += 32) {
    uint32_t v[32];
    tmem_ld32(addr + (uint32_t)cc0, v);
    tmem_wait_ld();
    if (look) {
      const float mx = max32(v) * kScale;
      if (cc0 + 32 == kTileKeys) {
        const bool fine = acc_total(acc) < kRedo && fmaxf(fabsf(m), mx) < kMaxRef && poly_reach(v) < kMaxProduct;
        if (HALF) {
          if (__ballot_sync(0xffffffffu, !fine) & real) return false;
        } else if (!__all_sync(0xffffffffu, fine)) {
          return false;
        }
        hand_back(empty_bar, lane);
      }
      if (m == -INFINITY || mx > m + 64.0f) {
        const float ref = rintf(mx);
        if (m > -INFINITY) l = (l + acc_total(acc)) * ex2(m - ref);
        acc[0] = acc[1] = 0ull;
        m = ref;
        r = poly_ref(m);
      }
      __syncwarp();
    }
    look = cc0 + 64 == kTileKeys;
    exp_accumulate(v, m, r, acc);
  }
  m_run = m;
  l_run = l + acc_total(acc);
  return true;
}

// Stands for a product that does not count: minus infinity, since a row's own logits may lie anywhere.
constexpr uint32_t kMasked = 0xff800000u;

// pass 1, keys from valid_r on (a bound of the thread's own) do not count (returns the row's new reference and sum); logits of any
// size.  Of chunks that no row of the warp attends to all but the read is skipped, and in those that all do nothing is masked: with
// a causal window most are one or the other, and the CTA with the last tiles of a sequence is what a short call waits for
// (10007 tokens x 4 heads: 7 us of work there, 4.5 to 5.5 elsewhere; score stage 24.1 -> 22.8 us).
__device__ __forceinline__ float2 drain_keys_masked(uint32_t addr, uint32_t empty_bar, int lane, int valid_r, float m_run, float l_run) {
  uint64_t acc[2] = {0ull, 0ull};
#pragma unroll 1
  for (int cc0 = 0; cc0 < kTileKeys; cc0 += 32) {
    uint32_t v[32];
    __syncwarp();                       // the rows of a warp skip different chunks
    tmem_ld32(addr + (uint32_t)cc0, v);
    tmem_wait_ld();
    if (cc0 + 32 == kTileKeys) hand_back(empty_bar, lane);
    const bool whole = __all_sync(0xffffffffu, cc0 + 32 <= valid_r);
    if (cc0 >= valid_r) continue;
    if (!whole) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (cc0 + i >= valid_r) v[i] = kMasked;
    }
    const float mx = max32(v) * kScale;
    if (m_run == -INFINITY || mx > m_run + 64.0f) {
      const float ref = rintf(mx);
      if (m_run > -INFINITY) l_run = (l_run + acc_total(acc)) * ex2(m_run - ref);
      acc[0] = acc[1] = 0ull;
      m_run = ref;
    }
    exp_accumulate_any(v, -m_run, acc);
  }
  return make_float2(m_run, l_run + acc_total(acc));
}

// pass 2: nc columns (a multiple of 16).  ADDED: the products come with -L_r; otherwise nl is the shared-space address of
// that of the first column
template <bool ADDED>
__device__ __forceinline__ float drain_rows(uint32_t addr, uint32_t empty_bar, int lane, uint32_t nl, int nc) {
  uint64_t acc[2] = {0ull, 0ull};
#pragma unroll 1
  for (int cc0 = 0; cc0 + 32 <= nc; cc0 += 32) {
    uint32_t v[32];
    tmem_ld32(addr + (uint32_t)cc0, v);               // stays inside the 128-column buffer
    tmem_wait_ld();
    if (cc0 + 32 == nc) hand_back(empty_bar, lane);
    if (ADDED) exp_accumulate_below<32>(v, acc);
    else exp_accumulate_columns<32>(v, nl + 4u * (uint32_t)cc0, acc);
  }
  if (nc & 16) {
    uint32_t v[32];
    tmem_ld32(addr + (uint32_t)(nc - 16), v);
    tmem_wait_ld();
    hand_back(empty_bar, lane);
    if (ADDED) exp_accumulate_below<16>(v, acc);
    else exp_accumulate_columns<16>(v, nl + 4u * (uint32_t)(nc - 16), acc);
  }
  return acc_total(acc);
}

// pass 2, columns before first_col (a bound of the thread's own) do not count, and nothing does for a thread without a key
// (returns the sum).  Skips and masks as above.
template <bool ADDED>
__device__ __forceinline__ float drain_rows_masked(uint32_t addr, uint32_t empty_bar, int lane, uint32_t nl, int nc, int first_col,
                                                   bool key) {
  uint64_t acc[2] = {0ull, 0ull};
#pragma unroll 1
  for (int cc0 = 0; cc0 < nc; cc0 += 32) {
    uint32_t v[32];
    __syncwarp();
    tmem_ld32(addr + (uint32_t)cc0, v);
    tmem_wait_ld();
    if (cc0 + 32 >= nc) hand_back(empty_bar, lane);
    if (!__any_sync(0xffffffffu, key && cc0 + 32 > first_col)) continue;
    if (!__all_sync(0xffffffffu, !key || cc0 >= first_col)) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (cc0 + i < first_col) v[i] = kMasked;
    }
    if (ADDED) {
      if (cc0 + 32 <= nc) exp_accumulate_below<32>(v, acc);
      else                exp_accumulate_below<16>(v, acc);
    } else {
      if (cc0 + 32 <= nc) exp_accumulate_columns<32>(v, nl + 4u * (uint32_t)cc0, acc);
      else                exp_accumulate_columns<16>(v, nl + 4u * (uint32_t)cc0, acc);
    }
  }
  return acc_total(acc);
}

// Walks the tiles of a CTA's span in (sequence, head, tile) order.
struct TileCursor {
  int s, h, local, n_tiles;
  __device__ void locate(const BatchTable& bt, int hkv, int t) {
    for (s = 0; s < bt.num_seqs; ++s) {
      const int lo = hkv * bt.seq[s].tile_off, cnt = hkv * bt.seq[s].n_tiles;
      if (t < lo + cnt) {
        n_tiles = bt.seq[s].n_tiles;
        h = (t - lo) / n_tiles;
        local = (t - lo) % n_tiles;
        return;
      }
    }
    s = bt.num_seqs - 1; h = 0; local = 0; n_tiles = 1;   // not reached for t < total_tiles
  }
  __device__ void advance(const BatchTable& bt, int hkv) {
    if (++local < n_tiles) return;
    local = 0;
    if (++h < hkv) return;
    h = 0;
    do { ++s; } while (s < bt.num_seqs && bt.seq[s].n_tiles == 0);
    n_tiles = s < bt.num_seqs ? bt.seq[s].n_tiles : 1;
  }
  __device__ int problem(int hkv) const { return s * hkv + h; }
};

// The CTAs' spans are runs of units (tiles, or halves of tiles) of equal weight.  A tile weighs 4, and
// the start of a (sequence, head) weighs P.change besides: a CTA that goes from one to the next
// replaces Q, drains its pipeline and hands row statistics over.  The first unit of CTA b is the
// one at weight b * P.weight / grid.
constexpr int kTileWeight = 4;

// a / b in 32 bits where they fit, which is always but for batches of millions of tiles: the 64-bit division is a call of some
// hundred instructions, run once per CTA from a cold instruction cache.
__device__ __forceinline__ long long quotient(long long a, long long b) {
  if (((a | b) >> 32) == 0) return (unsigned)a / (unsigned)b;
  return a / b;
}
// The unit at weight w, counted over all (sequence, head)s.
template <int HALVES>
__device__ long long unit_at(const BatchTable& bt, int hkv, const TcParams& P, long long w) {
  long long unit = 0;
#pragma unroll 1
  for (int s = 0; s < bt.num_seqs; ++s) {
    const int n_tiles = bt.seq[s].n_tiles;
    if (n_tiles == 0) continue;
    const unsigned per = (unsigned)(n_tiles * kTileWeight + P.change);       // weight of one head
    if (w < (long long)per * hkv) {
      const unsigned h = (unsigned)w / per;
      const int in = (int)((unsigned)w - h * per) - P.change;
      return unit + ((long long)h * n_tiles) * HALVES + max(in, 0) / (kTileWeight / HALVES);
    }
    w -= (long long)per * hkv;
    unit += (long long)n_tiles * HALVES * hkv;
  }
  return unit;
}
// CTA that has unit `local` of head h of sequence s.
template <int HALVES>
__device__ __forceinline__ int cta_of_unit(const BatchTable& bt, int hkv, const TcParams& P, int s, int h, int local) {
  long long w = 0;
#pragma unroll 1
  for (int i = 0; i < s; ++i)
    if (bt.seq[i].n_tiles) w += (long long)(bt.seq[i].n_tiles * kTileWeight + P.change) * hkv;
  w += (long long)(bt.seq[s].n_tiles * kTileWeight + P.change) * h + P.change + (long long)(local + 1) * (kTileWeight / HALVES);
  return (int)quotient(w * P.grid - 1, P.weight);      // w: the weight behind the unit
}

// A value that is the same in all lanes, in a form in which the compiler knows it: loop bounds and
// addresses derived from it then live in uniform registers.  (With the span's bounds not known to be
// uniform the ragged batch took 363 instead of 354 us.)
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// ------------------------------------------------------------------ the kernel
// CAUSAL instantiations carry the masked copies of the epilogue loops; the others have none of that code.  PAD (pass 1): 1 ones
// skip the items of warps whose 32 rows all lie behind the last one, one item in four on two of the four schedulers for 448
// rows: 65536 tokens x 4 heads of 448 rows 92.8 -> 91.9 us, 30000 x 8 of 400 rows 82.2 -> 81.0; with the test in all instantiations
// the others were 0.2-0.5 % slower.  2 ones know of warps with rows in half of their lanes besides (448 rows +1.5 % with that test).
// ADDED ones (pass 2) have -L_r added by the product, a ninth step of 16 channels (ones x three
// bf16 that sum to it), instead of reading it from shared memory for every column: eight loads fewer per chunk (figures: kAddedItems).
template <int PASS, bool CAUSAL, int LAYERS, int HALVES, int PAD, bool ADDED>
__global__ void __launch_bounds__(kThreads, 1)
score_tc_kernel(const __grid_constant__ BatchTable bt, const __grid_constant__ Geometry g,
                const __grid_constant__ TcParams P, const __grid_constant__ TcLayers<LAYERS> M,
                DeviceStatus* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t q_bytes = (uint32_t)P.rows_pad * 256u;
  const uint32_t q_panel = (uint32_t)P.rows_pad * 128u;
  uint8_t* q_smem = smem;
  uint8_t* k_smem = smem + q_bytes;
  Misc* misc = reinterpret_cast<Misc*>(k_smem + (size_t)P.n_stages * kStageBytes);
  // pass 2: -L_r, as an operand (ADDED; rows_pad + 8 rows) or in the log2 domain (-1e4 for padded rows)
  uint4* l_smem = reinterpret_cast<uint4*>(misc + 1);
  float* neg_lc = reinterpret_cast<float*>(misc + 1);
  Pipe pipe{misc, status};

  // the warp index as a value the compiler knows to be the same in all lanes: the MMA issuer's
  // descriptors then live in uniform registers
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 32) {
    // fetch the two TMA descriptors (kernel parameters) while the barriers are being set up
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&M.q[0])) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&M.k[0])) : "memory");
  }
  if (warp == 0) {               // one or two of each kind per lane: 64 in a row by one thread took 0.2 us
    if (lane < kMaxStages) {
      mbar_init(smem_u32(&misc->bar.full[lane]), 1);
      mbar_init(smem_u32(&misc->bar.empty[lane]), kIssuers);   // one arrival per MMA issuer
    }
    if (lane < kBufs) {
      mbar_init(smem_u32(&misc->bar.acc_full[lane]), 1);
      mbar_init(smem_u32(&misc->bar.acc_empty[lane]), 4);       // the four warps of a set
      mbar_init(smem_u32(&misc->bar.late_full[lane]), 1);
    }
    // one arrival per set that hands its partial sums over
    mbar_init(smem_u32(&misc->bar.u_full[lane >> 2][lane & 3]), P.n_sub > 1 ? P.n_sub - 1 : 1);
    if (lane < 8) mbar_init(smem_u32(&misc->bar.edge_full[lane >> 2][lane & 3]), 1);
    if (lane == 0) {
      mbar_init(smem_u32(&misc->bar.q_full), 1);
      mbar_init(smem_u32(&misc->bar.q_empty), kIssuers);
      mbar_init(smem_u32(&misc->bar.l_full), 1);
      misc->abort_flag = 0;
    }
    fence_barrier_init();
  }
  if (warp >= 2 && warp < 4 && lane == 0)      // the ends of the span, computed once (it is a slow piece of code)
    misc->span[warp - 2] = unit_at<HALVES>(bt, g.hkv, P, quotient((blockIdx.x + warp - 2) * P.weight, P.grid));
  if (warp == 1) {
    tmem_alloc(smem_u32(&misc->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  if (ADDED && threadIdx.x >= 128 && threadIdx.x < 128 + 2 * kTileKeys) {
    const int i = threadIdx.x - 128;       // 8-row groups of 256 bytes: channels 0-7 of the rows, channels 8-15
    misc->ones[i] = (i & 8) ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);
    if (i < 8) l_smem[P.rows_pad + i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
  }
  if (PASS == 2) pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, misc->tmem_base, 0);
  // Tiles [t_begin, t_end) of the span; of the first one only the row blocks from sub_begin on, of
  // the last one only those before sub_end (a tile cut at its middle belongs to two CTAs, which add
  // their column sums to zeroed scores: two addends, so their order does not matter).
  const long long u_begin = misc->span[0], u_end = misc->span[1];
  const int t_begin = uniform((int)(u_begin / HALVES)), t_end = uniform((int)((u_end + HALVES - 1) / HALVES));
  const int sub_begin = HALVES > 1 ? uniform(u_begin % HALVES ? P.n_sub / 2 : 0) : 0;
  const int sub_end = HALVES > 1 ? uniform(u_end % HALVES ? P.n_sub / 2 : P.n_sub) : P.n_sub;
  // Pass 1 reads Q and K, which the launch before it in the stream may have produced: every
  // thread waits for that launch, and only then lets pass 2 be scheduled, so that whatever runs
  // after pass 1 has begun finds the caller's inputs complete.  The launch before pass 2 is
  // pass 1, which only produces the row statistics: the TMA and MMA roles of pass 2 start at
  // once (their first K tiles and products overlap the tail of pass 1) and only the epilogue
  // warps, which read the statistics and write the scores, wait.
  auto pass1_wait = [] {
    if (PASS == 1) {
      pdl_wait();
      pdl_launch_dependents();
    }
  };

  if (warp == 0) {
    // ================================================================ TMA producer
    // The whole warp walks the tile list; one lane issues the copies.  With a paged cache every
    // lane reads and checks the id of one page of the tile (before the wait for the stage, so the
    // load is covered): the page-table look-ups of a tile are one parallel load, not a chain.
    {
      TileCursor cur;
      cur.locate(bt, g.hkv, t_begin);
      pass1_wait();
      const bool elected = elect_one();
      int stage = 0, cur_problem = -1;
      uint32_t phase = 0, qe_phase = 0;
      const int ps = bt.page_size;
      uint64_t k_policy;
      if (PASS == 1) asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(k_policy));
      else           asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(k_policy));
      for (int t = t_begin; t < t_end; ++t, cur.advance(bt, g.hkv)) {
        const SeqInfo& sq = bt.seq[cur.s];
        const int layer = LAYERS > 1 ? sq.layer : 0;
        const CUtensorMap* q_map = &M.q[layer];
        const CUtensorMap* k_map = &M.k[layer];
        if (cur.problem(g.hkv) != cur_problem) {
          if (cur_problem >= 0) {
            if (!warp_wait(pipe, &misc->bar.q_empty, qe_phase, 10)) break;
            qe_phase ^= 1;
          }
          cur_problem = cur.problem(g.hkv);
          if (elected) {
            const uint32_t qb = smem_u32(&misc->bar.q_full);
            mbar_expect_tx(qb, q_bytes);
            tma_load_4d(smem_u32(q_smem), q_map, qb, 0, cur.h * g.group, 0, sq.src);
            tma_load_4d(smem_u32(q_smem) + q_panel, q_map, qb, 64, cur.h * g.group, 0, sq.src);
          }
        }
        const int key0 = cur.local * kTileKeys;
        int page_id = -1;
        bool mine = false;               // this lane owns a page of the tile
        if (ps > 0) {
          const int valid = min(kTileKeys, sq.n - key0);
          mine = lane < (valid + ps - 1) / ps;
          if (mine) page_id = g.page_table[(int64_t)sq.src * g.page_table_stride + key0 / ps + lane];
        }
        if (!warp_wait(pipe, &misc->bar.empty[stage], phase ^ 1, 11)) break;
        const uint32_t fb = smem_u32(&misc->bar.full[stage]);
        const uint32_t dst = smem_u32(k_smem) + (uint32_t)stage * kStageBytes;
        if (ps == 0) {
          if (elected) {
            mbar_expect_tx(fb, kStageBytes);
            tma_load_3d_hint(dst, k_map, fb, 0, cur.h, sq.tok_off + key0, k_policy);
            tma_load_3d_hint(dst + kPanelBytes, k_map, fb, 64, cur.h, sq.tok_off + key0, k_policy);
          }
        } else {
          const bool good = mine && page_id >= 0 && ((int64_t)page_id + 1) * ps <= P.pool_rows;
          if (mine && !good) report_error(status, CC_ERR_DEVICE_FLAG, 12);
          const unsigned good_mask = __ballot_sync(0xffffffffu, good);
          // the stage completes when the bytes of the good pages have landed; one lane issues the
          // copies, so that their operands are uniform
          if (elected) mbar_expect_tx(fb, (uint32_t)__popc(good_mask) * (uint32_t)ps * 256u);
          for (unsigned left = good_mask; left; left &= left - 1) {
            const int p = __ffs(left) - 1;
            const int id = __shfl_sync(0xffffffffu, page_id, p);
            if (elected)       // the page's rows, both panels, in one copy
              tma_load_5d_hint(dst + (uint32_t)p * (uint32_t)ps * 256u, k_map, fb, id * (ps >> 3), cur.h, k_policy);
          }
        }
        if (++stage == P.n_stages) { stage = 0; phase ^= 1; }
      }
    }
  } else if (warp == 1 || warp == kMmaWarpB) {
    // ================================================================ MMA issuers
    // The whole warp walks the items and waits; one elected lane issues the multiplications.  With
    // all of it inside `if (lane == 0)` the compiler cannot know that the operands of tcgen05.mma
    // (uniform registers) are the same in all lanes and wraps each one in a loop over the lanes:
    // that was 30 of the 227 instructions the SM issued per 32-column chunk of a warp, and as long
    // a serial stream between a buffer's return and its refill (llama3_8b shape, both passes:
    // 52.1 -> 49.4 us together with the waits and the single issuing lane of the K copies).
    // Two issuers still refill a little sooner than one (chunk batch 190 against 194 us); items go
    // to them in pairs (0, 1 -> first; 2, 3 -> second; ...); both wait for every K tile and both
    // hand it back.  Descriptors are formed by adding small constants to a base word, and the tile
    // bookkeeping is a countdown instead of a cursor walk.
    const int my_half = warp == 1 ? 0 : 1;
    {
      TileCursor cur;
      cur.locate(bt, g.hkv, t_begin);
      pass1_wait();
      int left = cur.n_tiles - cur.local;          // tiles of the current (sequence, head) still to do
      int stage = 0;
      uint32_t phase = 0, qf_phase = 0, item = 0;
      bool need_q = true;
      // descriptor words: low = start address >> 4 | LBO field, high = SBO 1024 B, version 1,
      // 128-byte swizzle
      const uint32_t q_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
      const uint32_t k_hi = P.k_sbo16 | (1u << 14) | (2u << 29);
      const uint32_t a_hi = PASS == 1 ? q_hi : k_hi, b_hi = PASS == 1 ? k_hi : q_hi;
      const uint32_t q_lo0 = ((smem_u32(q_smem) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t k_lo0 = ((smem_u32(k_smem) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t q_panel16 = q_panel >> 4;
      const uint32_t q_step16 = PASS == 1 ? (128u * 128u) >> 4 : ((uint32_t)P.sub_cols * 128u) >> 4;
      const uint32_t idesc_full =
          PASS == 1 ? instr_desc(128, kTileKeys) : instr_desc(128, (uint32_t)P.sub_cols);
      const uint32_t idesc_last =
          PASS == 1 ? idesc_full
                    : instr_desc(128, (uint32_t)(P.rows_pad - (P.n_sub - 1) * P.sub_cols));
      const uint32_t empty0 = smem_u32(&misc->bar.empty[0]);
      const uint32_t accf0 = smem_u32(&misc->bar.acc_full[0]);
      // pass 2: one more step adds -L_r, but for the first two of an issuer's items of a (sequence, head), the first of each set:
      // L_r may not be known yet, and the set takes that step itself
      const uint64_t ones = ones_desc(misc->ones), stat = stat_desc(l_smem);
      uint32_t l_phase = 0, n_own = 0;
      bool l_known = false;
      const bool elected = elect_one();
      bool ok = true;
      for (int t = t_begin; t < t_end && ok; ++t) {
        if (need_q) {
          if (!warp_wait(pipe, &misc->bar.q_full, qf_phase, 20)) break;
          qf_phase ^= 1;
          need_q = false;
        }
        if (!warp_wait(pipe, &misc->bar.full[stage], phase, 21)) break;
        tc_fence_after();
        const uint32_t k_lo = k_lo0 + (uint32_t)stage * (kStageBytes >> 4);
#pragma unroll 1
        for (int sub = t == t_begin ? sub_begin : 0; sub < (t == t_end - 1 ? sub_end : P.n_sub); ++sub, ++item) {
          if ((int)((item >> 1) & 1u) != my_half) continue;
          const uint32_t buf = item & (kBufs - 1);
          const uint32_t par = ((item >> 2) & 1u) ^ 1u;
          if (!warp_wait(pipe, &misc->bar.acc_empty[buf], par, 22)) {
            ok = false;
            break;
          }
          if (ADDED && n_own++ == 2) {
            if (!warp_wait(pipe, &misc->bar.l_full, l_phase, 23)) {
              ok = false;
              break;
            }
            l_known = true;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + buf * kBufCols;
          const uint32_t idesc = sub == P.n_sub - 1 ? idesc_last : idesc_full;
          const uint32_t q_lo = q_lo0 + (uint32_t)sub * q_step16;
          if (elected) {
#pragma unroll
            for (int ks = 0; ks < kHeadDim / 16; ++ks) {
              const uint32_t ql = q_lo + (ks >= 4 ? q_panel16 : 0u) + (uint32_t)(ks & 3) * 2u;
              const uint32_t kl = k_lo + (ks >= 4 ? P.k_panel16 : 0u) + (uint32_t)(ks & 3) * 2u;
              const uint64_t al = PASS == 1 ? ql : kl, bl = PASS == 1 ? kl : ql;
              umma(d_tmem, al | ((uint64_t)a_hi << 32), bl | ((uint64_t)b_hi << 32), idesc, ks > 0);
            }
            if (ADDED && l_known)
              umma(d_tmem, ones, stat + (uint64_t)((uint32_t)sub * (uint32_t)P.sub_cols), idesc, true);
            umma_commit(accf0 + 8u * buf);
          }
        }
        if (!ok) break;
        if (elected) umma_commit(empty0 + 8u * (uint32_t)stage);
        if (++stage == P.n_stages) { stage = 0; phase ^= 1; }
        if (--left == 0 && t + 1 < t_end) {
          l_known = false;
          n_own = 0;
          l_phase ^= 1;      // (without a third item there is no wait; with one the next L_r waits for that item)
          // the next tile belongs to another (sequence, head): Q may be replaced once the
          // multiplications issued so far have read it
          if (elected) umma_commit(smem_u32(&misc->bar.q_empty));
          cur.local = cur.n_tiles - 1;
          cur.advance(bt, g.hkv);
          left = cur.n_tiles;
          need_q = true;
        }
      }
    }
  } else if (warp >= 2 && warp < 2 + kEpiWarps) {
    // ================================================================ epilogue warps
    const int ew = warp - 2;                 // 0..15
    const int quad = warp & 3;               // TMEM lane quadrant this warp may read
    const int set = ew >> 2;                 // consecutive warps cover the four quadrants
    const int row_in_tile = quad * 32 + lane;
    const int etid = ew * 32 + lane;         // 0..511, unique per epilogue thread
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    TileCursor cur;
    cur.locate(bt, g.hkv, t_begin);
    pass1_wait();
    int cur_problem = -1;
    bool dead = false;      // after a failed wait: keep the loop structure (and its barriers), skip the work
    float run_m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    float run_l[4] = {0.f, 0.f, 0.f, 0.f};

    // pass 1: merge the four sets' (max, sum) of every row and write the span's partial
    auto flush_partial = [&](int problem) {
#pragma unroll
      for (int rb = 0; rb < 4; ++rb) {
        if (rb >= P.n_sub) break;
        // a set whose row block never changes keeps its state in slot 0
        const int own = P.n_sub == 3 ? rb : (rb == (sub_begin + set) % P.n_sub ? 0 : -1);
        float2 st = make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) if (k == own) st = make_float2(run_m[k], run_l[k]);
        misc->xchg[set][rb * 128 + row_in_tile] = st;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) { run_m[k] = -INFINITY; run_l[k] = 0.f; }
      epi_barrier();
      for (int row = etid; row < P.rows_pad; row += kEpiThreads) {
        float m = -INFINITY;
#pragma unroll
        for (int k = 0; k < kSets; ++k) m = fmaxf(m, misc->xchg[k][row].x);
        float l = 0.f;
#pragma unroll
        for (int k = 0; k < kSets; ++k) {
          const float2 o = misc->xchg[k][row];
          if (o.y > 0.f) l += o.y * ex2(o.x - m);
        }
        P.part[(int64_t)(blockIdx.x + problem) * P.rows_pad + row] = make_float2(m, l);
      }
      epi_barrier();
    };

    // pass 2: merge the spans' (max, sum) of a (sequence, head) into -L_r.  b0, b1: the first and the last CTA
    // that have tiles of it; write_lse: this CTA has its first.  A thread takes two neighbouring rows, one 16-byte load
    // a span; the threads that share a pair of rows take every ways-th span, issue up to kPartLoads loads before they use the
    // first, and meet through shared memory.  Bound by that latency and by the fetch of its instructions, on the path between
    // the passes: with a row per thread, rounds of eight loads, a chain of exponentials and the spans looked up on the
    // way it took 2.5 us on 2048 tokens x 2 heads, 3.1 on 32768 x 8, 4.5 on 10007 x 4 of 448 rows (37 spans), now
    // 2.1, 2.2 and 3.0; whole calls -2 to -4 %.  (Eight loads: 10007 x 4 +1 %; four: +1 % there, 2048 x 2 level.  A first round on
    // whatever the buffer holds while pass 1 ends, to have the code at hand: 1.65 us, but late where pass 2 starts late, 10007 x 4 +7 %.)
    auto merge_lse = [&](int b0, int b1, bool write_lse) {
      constexpr int kPartLoads = 10;
      const int problem = cur.problem(g.hkv);
      const int pairs = P.rows_pad / 2, ways = min(16, kEpiThreads / pairs);
      const int way = etid / pairs, pair = etid - way * pairs;
      float2* fold = &misc->xchg[0][0];          // [ways][rows_pad]; no tile is in flight here, the union is free
      float m0 = -INFINITY, l0 = 0.f, m1 = -INFINITY, l1 = 0.f;
      if (way < ways) {
        const float4* part = reinterpret_cast<const float4*>(P.part + (int64_t)(b0 + way + problem) * P.rows_pad) + pair;
        const int64_t pitch = (int64_t)ways * pairs;
#pragma unroll 1
        for (int b = b0 + way; b <= b1; b += kPartLoads * ways) {
          float4 o[kPartLoads];
#pragma unroll
          for (int k = 0; k < kPartLoads; ++k) {
            o[k] = b + k * ways <= b1 ? __ldcg(part) : make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
            part += pitch;
          }
          float n0 = m0, n1 = m1;
#pragma unroll
          for (int k = 0; k < kPartLoads; ++k) { n0 = fmaxf(n0, o[k].x); n1 = fmaxf(n1, o[k].z); }
          // (a row without a key in any of the spans so far: m - n is a difference of infinities)
          l0 = l0 > 0.f ? l0 * ex2(m0 - n0) : 0.f;
          l1 = l1 > 0.f ? l1 * ex2(m1 - n1) : 0.f;
#pragma unroll
          for (int k = 0; k < kPartLoads; ++k) {
            l0 += o[k].y > 0.f ? o[k].y * ex2(o[k].x - n0) : 0.f;
            l1 += o[k].w > 0.f ? o[k].w * ex2(o[k].z - n1) : 0.f;
          }
          m0 = n0;
          m1 = n1;
        }
      }
      epi_barrier();                             // all sets are done with the (sequence, head) before
      if (way < ways) *reinterpret_cast<float4*>(&fold[way * P.rows_pad + 2 * pair]) = make_float4(m0, l0, m1, l1);
      epi_barrier();
      const int row = etid;
      if (row < P.rows_pad) {
        float m = -INFINITY, l = 0.f;
        for (int k = 0; k < ways; ++k) m = fmaxf(m, fold[k * P.rows_pad + row].x);
        for (int k = 0; k < ways; ++k) {
          const float2 o = fold[k * P.rows_pad + row];
          l += o.y > 0.f ? o.y * ex2(o.x - m) : 0.f;
        }
        const float lc = m + log2f(l);
        const bool real = row < P.rows;          // row = t * G + g
        if (!ADDED) {
          neg_lc[row] = real ? -lc : -1.0e4f;
        } else {
          // in units of the products, as three bf16 that add up to it (padded rows: far below everything)
          const float nl = real ? -lc * (1.0f / kScale) : -8.0e4f;
          const float rest = real ? fmaf(nl, kScale, lc) * (-1.0f / kScale) : 0.0f;       // rounding of the division
          const __nv_bfloat16 x0 = __float2bfloat16_rn(nl), x1 = __float2bfloat16_rn(nl - __bfloat162float(x0));
          const __nv_bfloat16 x2 = __float2bfloat16_rn(nl - __bfloat162float(x0) - __bfloat162float(x1) + rest);
          l_smem[row] = make_uint4((uint32_t)__bfloat16_as_ushort(x0) | (uint32_t)__bfloat16_as_ushort(x1) << 16,
                                   (uint32_t)__bfloat16_as_ushort(x2), 0u, 0u);
          fence_proxy_async();
        }
        if (real && P.lse != nullptr && write_lse) {
          const int gq = row % g.group, tq = row / g.group;
          P.lse[((int64_t)cur.s * g.hq + cur.h * g.group + gq) * g.window + tq] = lc * kLn2;
        }
      }
      epi_barrier();
      if (ADDED && etid == 0) mbar_arrive(smem_u32(&misc->bar.l_full));
    };

    // A set works on every fourth item of the span, item = (tile - t_begin) * n_sub + sub, and
    // steps from one of its items to the next by a precomputed (tiles, subs) stride; the
    // cursor is walked only where the (sequence, head) changes.  Buffer = set, and the phase
    // of its barrier flips with every item.
    const int n_sub = P.n_sub;
    const int dt = kSets / n_sub, ds = kSets % n_sub;
    const bool rotating = ds != 0;          // the set's row block changes from item to item
    int sub = (sub_begin + set) % n_sub, t = t_begin + (sub_begin + set) / n_sub;
    const int set_end = t_end - (sub >= sub_end ? 1 : 0);     // (a cut tile: sub is the same in all items of a set)
    // cut tiles of the span; the others use the eight slots of u_part in turn, from t_slot on
    const int cut_first = sub_begin > 0 ? t_begin : -1, cut_last = sub_end < n_sub ? t_end - 1 : -1;
    const int t_slot = t_begin + (sub_begin > 0 ? 1 : 0);
    const int idle_from = (max(P.rows_pad - quad * 32, 0) + 127) / 128;   // row blocks from here on have no row of this warp
    // lanes of a warp that have a row in the last block of rows (a multiple of 16 in all), if any do
    const unsigned last_rows = P.rows_pad - (n_sub - 1) * 128 - quad * 32 >= 32 ? ~0u : 0xffffu;
    uint32_t par = 0;
    bool first_item = true;     // ADDED: of the set in the (sequence, head); these come without -L_r
    uint32_t late_par = 0;
    int prob_end = t_begin, first_tile = 0, n_cur = 0;
    float* out = nullptr;
    const uint32_t full_bar = smem_u32(&misc->bar.acc_full[set]);
    const uint32_t empty_bar = smem_u32(&misc->bar.acc_empty[set]);
    const uint32_t acc_addr = lane_addr + (uint32_t)set * kBufCols;
    // CTA with the first unit of the span's first (sequence, head), CTA with the last one of its last
    int b_first = 0, b_last = 0;
    if (PASS == 2) {
      if (t_begin < t_end) {
        TileCursor last;
        last.locate(bt, g.hkv, t_end - 1);
        b_first = cta_of_unit<HALVES>(bt, g.hkv, P, cur.s, cur.h, 0);
        b_last = cta_of_unit<HALVES>(bt, g.hkv, P, last.s, last.h, last.n_tiles * HALVES - 1);
      }
      pdl_wait();
    }
    if (HALVES > 1 && PASS == 1 && sub_end < n_sub && etid < kTileKeys) {
      // pass 2 adds to the scores of the tile this span shares with the next one
      TileCursor last;
      last.locate(bt, g.hkv, t_end - 1);
      const SeqInfo& sq = bt.seq[last.s];
      const int key = last.local * kTileKeys + etid;
      if (key < sq.n) M.scores[LAYERS > 1 ? sq.layer : 0][(int64_t)last.h * bt.n_tot + sq.tok_off + key] = 0.f;
    }
    for (;;) {
      if (t >= min(prob_end, set_end)) {
        bool done = false;
        do {
          if (PASS == 1 && cur_problem >= 0) flush_partial(cur_problem);
          if (prob_end >= t_end) { done = true; break; }
          if (cur_problem >= 0) {
            cur.local = cur.n_tiles - 1;
            cur.advance(bt, g.hkv);
          }
          const SeqInfo& sq = bt.seq[cur.s];
          first_tile = g.hkv * sq.tile_off + cur.h * sq.n_tiles;
          if (PASS == 2) {
            // (sequence, head)s that begin or end in this span: this CTA is their first or last
            const bool begins = first_tile * HALVES >= u_begin, ends = (first_tile + sq.n_tiles) * HALVES <= u_end;
            merge_lse(begins ? (int)blockIdx.x : b_first, ends ? (int)blockIdx.x : b_last, begins);
          }
          first_item = true;
          cur_problem = cur.problem(g.hkv);
          prob_end = min(t_end, first_tile + sq.n_tiles);
          n_cur = sq.n;
          out = M.scores[LAYERS > 1 ? sq.layer : 0] + (int64_t)cur.h * bt.n_tot + sq.tok_off;
        } while (t >= min(prob_end, set_end));
        if (done) break;
      }
      const int key0 = (t - first_tile) * kTileKeys;
      const int valid = min(kTileKeys, n_cur - key0);
      if (!dead) {
        dead = !warp_wait(pipe, &misc->bar.acc_full[set], par, 30);
      }
      par ^= 1u;
      if (ADDED && first_item) {
        // The step that the issuer could not take, so that all items are rounded alike and equal keys have equal scores.  (With the
        // offset added to the product when it is read, keys of these items differed from their equals in the last places;
        // the calls take 0 to 0.4 % more, 32768 tokens x 8 heads 55.8 -> 56.0 us.)
        if (!dead) {
          tc_fence_after();
          if ((ew & 3) == 0 && elect_one()) {
            const int c0 = sub * P.sub_cols;
            umma(tmem_base + (uint32_t)set * kBufCols, ones_desc(misc->ones), stat_desc(l_smem) + (uint64_t)(uint32_t)c0,
                 instr_desc(128, (uint32_t)min(P.sub_cols, P.rows_pad - c0)), true);
            umma_commit(smem_u32(&misc->bar.late_full[set]));
          }
          __syncwarp();
          dead = !warp_wait(pipe, &misc->bar.late_full[set], late_par, 35);
        }
        late_par ^= 1u;
        first_item = false;
      }
      float u_acc = 0.f;
      if (!dead) {
        tc_fence_after();
        const bool edge = PASS == 1 ? valid < kTileKeys || (CAUSAL && key0 + kTileKeys > n_cur - g.window + 1)
                                    : CAUSAL && key0 + kTileKeys > n_cur - g.window + 1;
        if (PAD && sub >= idle_from) {
          hand_back(empty_bar, lane);
        } else if (PASS == 1) {
          // thread = query row (sub * 128 + row_in_tile); columns = the 128 keys of the tile
          float m_run = run_m[0], l_run = run_l[0];
          if (rotating) {
#pragma unroll
            for (int rb = 1; rb < 4; ++rb) if (rb == sub) { m_run = run_m[rb]; l_run = run_l[rb]; }
          }
          if (edge || !drain_keys<PAD == 2>(acc_addr, empty_bar, lane, sub == n_sub - 1 ? last_rows : ~0u, m_run, l_run)) {
            // keys of the tile this row attends to: the valid ones, or (causal window) those up to the
            // row's own position n - w + t
            int valid_r = valid;
            if (CAUSAL) {
              const int t_row = (sub * 128 + row_in_tile) / g.group;
              if (t_row < g.window) valid_r = min(valid, n_cur - g.window + t_row + 1 - key0);
            }
            const float2 st = drain_keys_masked(acc_addr, empty_bar, lane, valid_r, m_run, l_run);
            m_run = st.x;
            l_run = st.y;
          }
          if (rotating) {
#pragma unroll
            for (int rb = 0; rb < 4; ++rb) if (rb == sub) { run_m[rb] = m_run; run_l[rb] = l_run; }
          } else {
            run_m[0] = m_run;
            run_l[0] = l_run;
          }
        } else {
          // thread = key (key0 + row_in_tile); columns = the query rows of this chunk
          const int c0 = sub * P.sub_cols;
          const int nc = min(P.sub_cols, P.rows_pad - c0);        // multiple of 16
          // causal window: key j is seen by the rows t >= j - (n - w), i.e. by the columns from
          // G * (j - n + w) on; the columns before it contribute nothing
          if (edge)
            u_acc = drain_rows_masked<ADDED>(acc_addr, empty_bar, lane, smem_u32(neg_lc + c0), nc,
                                             g.group * (key0 + row_in_tile - n_cur + g.window) - c0, row_in_tile < valid);
          else
            u_acc = drain_rows<ADDED>(acc_addr, empty_bar, lane, smem_u32(neg_lc + c0), nc);
        }
      }
      if (PASS == 2) {
        if (n_sub > 1) {
          // The sets that hold partial sums of the tile (one per item) meet through shared
          // memory: the set that drained the tile's last item adds the others' sums and stores;
          // n_sub - 1 arrivals complete a (slot, quadrant).  Eight slots: a slot is written
          // again only after the accumulator hand-shake has forced the reader past the tile it
          // belongs to.
          if (HALVES > 1 && (t == cut_first || t == cut_last)) {
            // half of a tile: one other set at most has a part of it
            const int e = t == cut_first ? 0 : 1;
            const bool finish = sub == (e == 0 ? n_sub : sub_end) - 1;
            if (!finish) {
              misc->edge_part[e][row_in_tile] = u_acc;
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&misc->bar.edge_full[e][quad]));
            } else {
              if (n_sub == 4 && !dead) dead = !warp_wait(pipe, &misc->bar.edge_full[e][quad], 0u, 34);
              if (!dead && row_in_tile < valid)
                atomicAdd(out + key0 + row_in_tile, n_sub == 4 ? u_acc + misc->edge_part[e][row_in_tile] : u_acc);
            }
          } else {
            const int slot = (t - t_slot) & 7;
            if (sub != n_sub - 1) {
              misc->u_part[slot][sub][row_in_tile] = u_acc;
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&misc->bar.u_full[slot][quad]));
            } else {
              if (!dead) dead = !warp_wait(pipe, &misc->bar.u_full[slot][quad], (uint32_t)((t - t_slot) >> 3) & 1u, 31);
              if (!dead && row_in_tile < valid) {
                float u = u_acc;
                for (int k = 0; k < n_sub - 1; ++k) u += misc->u_part[slot][k][row_in_tile];
                out[key0 + row_in_tile] = u;
              }
            }
          }
        } else if (!dead && row_in_tile < valid) {
          out[key0 + row_in_tile] = u_acc;
        }
      }
      sub += ds;
      t += dt;
      if (sub >= n_sub) { sub -= n_sub; ++t; }
    }
  }

  // ---------------------------------------------------------------- teardown
  if (misc->abort_flag) {
    // give copies still in flight time to land before shared memory is released
#pragma unroll 1
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Items of a CTA from which on pass 2 lets the products add -L_r (ADDED).  The first item of each set gets it late, and the
// operand has to be prepared: 20480 tokens x 8 heads of 256 rows (17 items) -0.8 %, 65536 x 4 of 448 -1.3 %, 131072 x 8 -2.0 %,
// 32 x 2200 x 8 of 512 -2.0 %; level at 7 to 14 items, +0.9 % on 131072 x 2 of 128 rows (14 items) and 12 x 300 x 8 of 512.
// Spans with cut tiles have few items.
constexpr int kAddedItems = 16;

// Shared memory of a launch: Q, a ring of as many K tiles as there is room for, Misc, and in pass 2 the row statistics.  Each
// launch has the ring that its own needs leave: 5 tiles at 176 rows, 4 at 304 (320 in pass 1), 3 at 432 (448 in pass 1).
struct Ring {
  int stages;
  size_t smem_bytes;
};
Ring ring_of(int rows_pad, size_t l_bytes) {
  const size_t fixed = 1024 + (size_t)rows_pad * 256 + sizeof(Misc) + l_bytes;
  const int stages = fixed < kSmemLimit ? (int)((kSmemLimit - fixed) / kStageBytes) : 0;
  const int n = stages < kMaxStages ? stages : kMaxStages;
  return Ring{n, fixed + (size_t)n * kStageBytes};
}
Ring ring_pass1(int rows_pad) { return ring_of(rows_pad, 0); }
Ring ring_pass2(int rows_pad, bool added) { return ring_of(rows_pad, added ? (size_t)(rows_pad + 8) * 16 : (size_t)rows_pad * 4); }
// Whether pass 2 lets the products add -L_r (ADDED): with items enough (kAddedItems), and not where the operand costs the ring a tile
// (64, 304, 432 rows): 131072 tokens x 8 heads of 64 rows 86.6 with it and 84.9 us without, 65536 x 8 of 304 rows 102.6 and 102.0,
// of 432 130.3 and 129.7.
bool adds_statistic(int rows_pad, int items, int grid) {
  return items >= kAddedItems * grid && ring_pass2(rows_pad, true).stages == ring_pass2(rows_pad, false).stages;
}

struct TcPlan {
  TcParams P;
  bool ok;
};

TcPlan make_plan(const BatchTable& bt, const Geometry& g, int sm_count, int layers) {
  TcPlan pl;
  TcParams& P = pl.P;
  memset(&pl, 0, sizeof(pl));
  P.total_tiles = g.hkv * bt.tiles_per_head;
  P.rows = g.rows;
  // pad the window so that the padded row count is a multiple of 16 (UMMA N granularity)
  int w_pad = g.window;
  while ((g.group * w_pad) % 16 != 0) ++w_pad;
  P.w_pad = w_pad;
  P.rows_pad = g.group * w_pad;
  P.n_sub = (P.rows_pad + 127) / 128;
  // Whole tiles, or half ones where the CTA with the most whole tiles, ceil(tiles / SMs) of them,
  // has a tenth more than that in halves (10007 tokens x 4 heads: 3 where the average is 2.1, 2.5 in
  // halves).  Not below two tiles per SM: half of a lone tile occupies half of the epilogue sets,
  // and the cut tiles' keys are loaded twice (2546 tokens x 8 heads: 20.2 -> 21.7 us with halves).
  const int whole = (P.total_tiles + sm_count - 1) / sm_count, half = (2 * P.total_tiles + sm_count - 1) / sm_count;
  P.halves = layers == 1 && P.n_sub % 2 == 0 && P.total_tiles > 2 * sm_count && half * 1.1 < 2 * whole ? 2 : 1;
  int starts = 0;
  for (int s = 0; s < bt.num_seqs; ++s) starts += bt.seq[s].n_tiles > 0;
  // A start weighs as much as 2000 / rows quarters of a tile (2 tiles at 256 rows, 1 at 512; spans
  // that straddle one are that late in pass 2): llama3_8b shape 49.0 -> 47.3 us, 32 chunks 188 -> 178.  Against 2500 / rows
  // 32 chunks -1.2 to -1.6 %, batches of 32 and 16 sequences -1.5 and -1.9 %, the others level; 1500 and 1000: +1 to 3 % on batches
  // of 448 rows.  With few tiles per CTA whole tiles are too coarse to pay it back.
  P.change = P.total_tiles >= 4 * sm_count ? (2000 + P.rows_pad / 2) / P.rows_pad : 0;
  P.weight = (long long)P.total_tiles * 4 + (long long)starts * g.hkv * P.change;
  const int units = P.total_tiles * P.halves;
  P.grid = units < sm_count ? units : sm_count;
  if (P.grid < 1) P.grid = 1;
  pl.ok = P.rows_pad <= kMaxRows && w_pad <= 256 && g.group <= 256;
  if (ring_pass2(P.rows_pad, false).stages < 2) pl.ok = false;
  return pl;
}

}  // namespace

size_t score_tc_ws_bytes(const BatchTable& bt, const Geometry& g, int sm_count) {
  TcPlan pl = make_plan(bt, g, sm_count, bt.num_seqs ? bt.seq[bt.num_seqs - 1].layer + 1 : 1);
  const size_t entries = (size_t)pl.P.grid + (size_t)bt.num_seqs * g.hkv;
  return (entries * pl.P.rows_pad * sizeof(float2) + 255) / 256 * 256;
}

namespace {

// The tensor maps of one layer.
CUresult encode_maps(EncodeTiledFn encode, const BatchTable& bt, const Geometry& g, const TcParams& P, int num_seqs,
                     const void* q, const void* k, CUtensorMap* q_map, CUtensorMap* k_map) {
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  {
    const cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.hq, (cuuint64_t)g.window, (cuuint64_t)num_seqs};
    int64_t seq_stride = g.q_stride_seq;
    if (num_seqs == 1 || seq_stride <= 0) seq_stride = g.q_stride_row * g.window;
    const cuuint64_t strides[3] = {(cuuint64_t)g.q_stride_head * 2, (cuuint64_t)g.q_stride_row * 2,
                                   (cuuint64_t)seq_stride * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)g.group, (cuuint32_t)P.w_pad, 1};
    const CUresult r = encode(q_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return r;
  }
  if (bt.page_size > 0) {
    // A page (page_size tokens, a multiple of 8, starting at a multiple of 8 rows) as one box: 64
    // channels x 8 tokens x 2 panels x page_size / 8 groups of one head.  In shared memory that is
    // page_size / 8 blocks of 2 KB, each the eight rows of the first panel followed by the eight
    // rows of the second: two copies per page become one (a 16-token page: 4 KB per copy).
    const cuuint64_t dims[5] = {64, 8, 2, (cuuint64_t)(P.pool_rows / 8), (cuuint64_t)g.hkv};
    const cuuint64_t strides[4] = {(cuuint64_t)g.kv_stride_tok * 2, 128, (cuuint64_t)g.kv_stride_tok * 16,
                                   (cuuint64_t)g.kv_stride_head * 2};
    const cuuint32_t box[5] = {64, 8, 2, (cuuint32_t)(bt.page_size / 8), 1};
    return encode(k_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(k), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.hkv, (cuuint64_t)P.pool_rows};
  const cuuint64_t strides[2] = {(cuuint64_t)g.kv_stride_head * 2, (cuuint64_t)g.kv_stride_tok * 2};
  const cuuint32_t box[3] = {64, 1, (cuuint32_t)kTileKeys};
  return encode(k_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(k), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int LAYERS, int HALVES>
cudaError_t launch_passes(const Launch& L, const BatchTable& bt, const Geometry& g, const LayerPtrs& lp,
                          const TcPlan& pl, EncodeTiledFn encode, int* drv_err) {
  TcParams P = pl.P;
  TcLayers<LAYERS> M;
  for (int l = 0; l < lp.n; ++l) {
    const CUresult r = encode_maps(encode, bt, g, P, bt.num_seqs / lp.n, lp.q[l], lp.k[l], &M.q[l], &M.k[l]);
    if (r != CUDA_SUCCESS) { *drv_err = (int)r; return cudaErrorUnknown; }
    M.scores[l] = lp.scores[l];
  }
  // PAD: the last block of rows is not full; a warp has rows in half of its lanes, or some warps have none (causal calls gain nothing
  // from a form of their own for that: 10007 tokens x 4 heads of 448 rows level)
  const int pad = P.rows_pad % 32 != 0 ? 2 : P.rows_pad % 128 != 0 ? 1 : 0;
  auto pass1 = g.causal ? (pad ? score_tc_kernel<1, true, LAYERS, HALVES, 2, false> : score_tc_kernel<1, true, LAYERS, HALVES, 0, false>)
               : pad == 2 ? score_tc_kernel<1, false, LAYERS, HALVES, 2, false>
               : pad == 1 ? score_tc_kernel<1, false, LAYERS, HALVES, 1, false>
                          : score_tc_kernel<1, false, LAYERS, HALVES, 0, false>;
  auto pass2 = g.causal ? score_tc_kernel<2, true, LAYERS, HALVES, 0, false> : score_tc_kernel<2, false, LAYERS, HALVES, 0, false>;
  const bool added = HALVES == 1 && adds_statistic(P.rows_pad, P.total_tiles * P.n_sub, P.grid);
  if (added)
    pass2 = g.causal ? score_tc_kernel<2, true, LAYERS, HALVES, 0, HALVES == 1>
                     : score_tc_kernel<2, false, LAYERS, HALVES, 0, HALVES == 1>;
  cudaError_t e = allow_smem(pass1);
  if (e == cudaSuccess) e = allow_smem(pass2);
  if (e != cudaSuccess) return e;

  P.n_sub = (P.rows_pad + 127) / 128;
  P.sub_cols = 0;
  const Ring ring1 = ring_pass1(P.rows_pad), ring2 = ring_pass2(P.rows_pad, added);
  P.n_stages = ring1.stages;
  e = launch_pdl(pass1, dim3(P.grid), dim3(kThreads), ring1.smem_bytes, L.stream, 1, bt, g, P, M, L.status);
  if (e != cudaSuccess) return e;
  P.sub_cols = ((P.rows_pad + P.n_sub - 1) / P.n_sub + 15) / 16 * 16;
  P.n_stages = ring2.stages;
  return launch_pdl(pass2, dim3(P.grid), dim3(kThreads), ring2.smem_bytes, L.stream, 1, bt, g, P, M, L.status);
}

}  // namespace

cudaError_t launch_score_tc(const Launch& L, const BatchTable& bt, const Geometry& g, const LayerPtrs& lp,
                            float* lse, void* ws, void* encode_fn, int64_t pool_rows, int* drv_err) {
  *drv_err = 0;
  TcPlan pl = make_plan(bt, g, L.sm_count, lp.n);
  if (!pl.ok) return cudaErrorInvalidConfiguration;
  pl.P.part = (float2*)ws;
  pl.P.lse = lse;
  pl.P.pool_rows = bt.page_size > 0 ? pool_rows : (int64_t)bt.n_tot;
  // 8-row groups and panels of a K tile in shared memory (see TcParams)
  pl.P.k_sbo16 = (bt.page_size > 0 ? 2048u : 1024u) >> 4;
  pl.P.k_panel16 = (bt.page_size > 0 ? 1024u : kPanelBytes) >> 4;
  EncodeTiledFn encode = (EncodeTiledFn)encode_fn;
  if (lp.n > 1) return launch_passes<kMaxLayers, 1>(L, bt, g, lp, pl, encode, drv_err);
  return pl.P.halves == 2 ? launch_passes<1, 2>(L, bt, g, lp, pl, encode, drv_err)
                          : launch_passes<1, 1>(L, bt, g, lp, pl, encode, drv_err);
}

}  // namespace cc

extern "C" void ccx_score_ring(int rows_pad, int items, int grid, int* pass1, int* pass2, int* added, size_t* smem_bytes) {
  *added = cc::adds_statistic(rows_pad, items, grid);
  const cc::Ring one = cc::ring_pass1(rows_pad), two = cc::ring_pass2(rows_pad, *added != 0);
  *pass1 = one.stages;
  *pass2 = two.stages;
  *smem_bytes = one.smem_bytes > two.smem_bytes ? one.smem_bytes : two.smem_bytes;
}
