// Causal append-chunk attention on the 5th-generation tensor cores
// (tcgen05 + TMEM), for rows that append a tool-observation chunk (L > 1).
//
// One CTA per SM, persistent, 12 warps. A work item is 256 query rows of one
// append row and kv head: (256 / g) consecutive tokens x the g query heads of
// that kv head, held as two 128-row tiles A and B (TMEM lanes = rows). Both
// tiles read the same K/V stream, so each K/V block in shared memory feeds
// four MMA chains (S_A, S_B, O_A, O_B), and the K/V bytes per flop are half
// those of a one-tile CTA.
//   warps 0-3  softmax of tile A, warps 4-7 softmax of tile B: thread t owns
//              row t & 127 of its tile. Per 128-key block it reads the 128
//              scores from TMEM in two chunks of 64, exponentiates them
//              against the row's reference (the max of the row's first chunk,
//              raised when a later chunk's max exceeds it by more than 2^8),
//              adds up the row sum and writes P (bf16) to the tile's TMEM P
//              buffer. The S buffer is released as soon as both chunks have
//              been loaded.
//              Epilogue: O / l and the log-sum-exp to global (or page-locked
//              host) memory, each row as four 32-byte stores, whole sectors;
//   warps 8, 11  TMA producers: warp 8 the item queue, both query tiles (one
//              3-D box of (256 / g) tokens x g heads x 64 dims) and K, warp 11
//              V, in blocks of 8 pages = 128 keys (16 KiB) through two rings of
//              their own: a K block is released as soon as S_A and S_B have
//              read it, a V block only after both PVs, so K runs a block ahead
//              of V. A warp issues a 2 KiB box every 100-130 cycles (measured),
//              so the 16 boxes of a block need two warps;
//   warps 9, 10  MMA issuers of tile A and tile B: S_X(b) = Q_X K_b^T (M 128,
//              N 128, K 64, both operands K-major from shared memory), then
//              O_X += P_X(b - 1) V_(b-1) (M 128, N 64, K 128; P from TMEM,
//              V MN-major from shared memory).
// TMEM (512 columns): S_A, S_B (128 each), O_A, O_B, P_A, P_B (64 each).
//
// What bounds it: instruction fetch and the issuers' latency, not the tensor
// pipe (46 % active) or the exponentials (47 % of the MUFU's rate). An SM
// sub-partition runs at full rate from about 6 KiB of loop code (a 172-instruction
// chunk body copied 1 / 3 / 6 times in straight line: 389 / 510 / 632 cycles per
// chunk), and code run once costs about 5 cycles per instruction. So the code is kept small: one
// rolled chunk body for every block, masks and maxima in a short loop over
// TMEM that is called for an item's first and edge blocks only, the rare search
// for a higher reference out of line, and the warp index broadcast so that what depends on it stays in
// the uniform datapath. (Masks applied to the scores in registers also made the
// compiler copy all 64 of them on the unmasked path.) Against the unrolled form
// (73 KB of code, now 45): 256-row mixed batch 5300 -> 4588 us beside the
// decode kernel, prefill of 8 prompts (35681 tokens, 1.61 TFLOP) 1677 -> 1470 us
// = 1.09 PFLOP/s, window layer of 384 rows 250 -> 236 us (188 with the short form). Measured slower:
// four issuers (1737 us for the prefill), 16 softmax warps on key halves (1528),
// 32-key chunks (1838), per-MMA elect (1556), waits in a called function (1535).
//
// Ordering (all mbarriers, all waits bounded; X = tile A or B, phase = the
// CTA's running block count, so no waiter can fall two phases behind):
//   k_full/k_empty     K ring; a stage is released by the commits after S_A, S_B
//   v_full/v_empty     V ring; a stage is released by the commits after PV_A, PV_B
//   s_full[X]          S_X(b) complete (commit after its 4 MMAs)
//   s_free[X]          S_X(b) loaded into registers (4 warps arrive)
//   p_full[X]          P_X(b) stored and O_X rescaled (4 warps arrive)
//   o_ready[X]         PV_X(b) complete; also guards the single P buffer
//   o_free[X]          epilogue has read O_X (next item may overwrite it)
//   q_full/q_empty     query tiles loaded / last QK^T of the item done
//   item_full/empty[2] two-slot queue of work items from the K producer
//
// A wait that runs out sets an abort flag in shared memory that every other
// role's waits poll, so the whole CTA leaves within microseconds; before TMEM
// is freed the issuers wait for their MMAs and the producers for their copies
// still in flight. append_tc_kernel<true, false> is the self-test form of the same
// kernel (mcpu_selftest_append_abort): one chosen role stops at the second
// key block of its first item and waits on a barrier nothing completes (for
// half the wait limit), and each warp reports when it left (the two producers
// under one entry).
#include "tcgen05.cuh"

namespace mcpu {

constexpr int kTcRows = 128;                          // rows per tile (TMEM lanes)
constexpr int kTcKeys = 128;                          // keys per block
// Ring depths and registers leave room on every SM for one CTA of the
// memory-bound decode kernel (side stream): 145 KiB of shared memory here, and 3
// warps x 136 registers on each SM sub-partition of 512, which leaves 104 for the
// decode kernel's warp (96). The kernel takes 134; a test holds both to that sum.
// Its own cap is 144 all the same: capped at 136 the compiler takes 128 and a
// slower schedule (prefill of 8 prompts 1508 -> 1767 us). With no room for the
// decode CTA its work follows the append kernel's: a form of this kernel that took
// 144 registers lost 1700 us of the mixed batch's 4923 and 350 of the prefill's 1508.
constexpr int kTcKStages = 4, kTcVStages = 3;
constexpr int kTcQBytes = kAppendTcRows * kRowBytes;  // both tiles: 32 KiB
constexpr int kTcTileQBytes = kTcRows * kRowBytes;    // 16 KiB
constexpr int kTcKvBytes = kTcKeys * kRowBytes;       // one K or V block: 16 KiB
constexpr int kTcSoftmaxWarps = 8;
constexpr int kTcKWarp = 8, kTcIssuerA = 9, kTcIssuerB = 10, kTcVWarp = 11;
constexpr int kTcThreads = 384;
constexpr uint32_t kTmemCols = 512;
// TMEM columns of tile x (0 = A, 1 = B)
__device__ __forceinline__ uint32_t col_s(int x) { return x ? 128u : 0u; }
__device__ __forceinline__ uint32_t col_o(int x) { return x ? 320u : 256u; }
__device__ __forceinline__ uint32_t col_p(int x) { return x ? 448u : 384u; }
// A row's reference is raised when a chunk's max exceeds it by more than
// kRescaleThreshold (log2 units). A chunk whose sum is below 2^kRescaleThreshold
// holds no such score, so only other chunks are searched for their max. The weights
// that dominate a row then stand close to its reference, where a bf16 weight of
// exactly 1 rounds nothing away: with a threshold of 2^16 the errors of full-context
// rows grew by 8-12 % for scores of 4 and 16 times unit variance.
constexpr float kRescaleThreshold = 8.f;
constexpr float kSearchAt = 256.f;

static_assert(kAppendTcRows == 2 * kTcRows, "an item is two tiles");

// The form for sliding windows of at most kShortWindow keys (kShort), whose items
// are a few blocks long: an item's last block is half a block when its keys fit,
// with half the copies, MMAs and exponentials. A window of 128 keys is then 1.5
// blocks for most items instead of 2: a window layer of 384 rows 267 -> 239 us,
// 23 thousand tokens with windows of 16 / 256 / 512 / 1000 keys 157 / 254 / 333 /
// 537 -> 130 / 232 / 311 / 525 us, and 654 -> 654 at 2000. In the general form the
// same code made full-context layers 1.5-2 % slower.
constexpr int kShortWindow = 1024;
template <bool kShort>
__device__ __forceinline__ bool half_block(const AppendItem& a, int kb0, int b) {
  return kShort && a.key_end - (kb0 + b * kTcKeys) <= kTcKeys / 2;
}

struct TcSmem {  // barriers and small state, after the tiles
  uint64_t q_full, q_empty;
  uint64_t k_full[kTcKStages], k_empty[kTcKStages], v_full[kTcVStages], v_empty[kTcVStages];
  uint64_t s_full[2], s_free[2], p_full[2], o_ready[2], o_free[2];
  uint64_t item_full[2], item_empty[2];
  uint64_t drain[2];  // each issuer's last MMAs complete (before TMEM is freed)
  uint64_t never;     // self-test form only: a barrier nothing completes
  AppendItem items[2];
  int32_t item_idx[2];
  uint32_t tmem_base;
  int32_t abort_flag;  // 1: a wait ran out; 2: the self-test's stalled role gave up
  uint64_t t_start;    // self-test form only: %globaltimer at kernel start
};

size_t append_tc_smem_bytes() {
  return 1024 + kTcQBytes + (size_t)(kTcKStages + kTcVStages) * kTcKvBytes + sizeof(TcSmem);
}

namespace {

__device__ __forceinline__ uint32_t elect_lane() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}" : "=r"(r));
  return r;
}

// tma_load_2d executed by a whole warp in step with warp-uniform operands; one
// elected lane issues.
__device__ __forceinline__ void tma_load_2d_e(uint32_t dst, const CUtensorMap* map, int32_t x, int32_t y, uint32_t bar,
                                              uint64_t policy) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;\n\t}" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}

// Bounded wait that also gives up when another role has aborted. The polls
// sleep (the producers and the MMA issuers wait most of the time and share
// sub-partitions with the softmax warps) and are out of line, to keep the
// loops of these roles short. Used by the producers and issuers.
__device__ __noinline__ bool wait_bar_slow(uint32_t bar, uint32_t parity, volatile int32_t* abort_flag) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait_sleep(bar, parity, 10000)) {
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > kWaitTimeoutNs) {
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int32_t* abort_flag) {
  return mbar_try_wait(bar, parity) || wait_bar_slow(bar, parity, abort_flag);
}

// The softmax warps' bounded wait: the same, with plain polls (no
// suspend-time hint). The softmax is the critical path and rarely waits
// long; a sleeping poll there made the mixed batch's step ~0.65 % slower.
__device__ __forceinline__ bool wait_bar_poll(uint32_t bar, uint32_t parity, volatile int32_t* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > kWaitTimeoutNs) {
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// A block with keys some row does not see, or without a reference yet: writes
// -inf over the scores in TMEM (columns cS ..) of keys outside [lo, pos] and
// returns the largest visible score (raw) of the first 64 keys, or, if the row
// sees none of them, of the others. A short loop, called once or
// twice per item: the code that turns scores into probabilities stays the same
// for every block, and small.
__device__ __noinline__ float mask_block(uint32_t cS, int kb, int pos, int lo) {
  float m0 = -INFINITY, m1 = -INFINITY, first = -INFINITY;
  const unsigned span = (unsigned)(pos - lo);
#pragma unroll 1
  for (int c = 0; c < kTcKeys / 32; ++c) {
    if (c == 2) first = fmaxf(m0, m1);
    uint32_t v[32];
    tmem_ld32(cS + 32 * c, v);
    tmem_ld_wait();
    const int r = kb + 32 * c - lo;
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if ((unsigned)(r + e) > span) v[e] = 0xff800000u;
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      m0 = fmax3(m0, __uint_as_float(v[e]), __uint_as_float(v[e + 1]));
      m1 = fmax3(m1, __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
    }
    tmem_st32(cS + 32 * c, v);
  }
  tmem_st_wait();
  return first > -INFINITY ? first : fmaxf(m0, m1);
}

// The same for the short form, whose items are mostly such blocks. The warp's rows
// are a few neighbouring tokens, so most chunks of 32 keys are seen by all of them
// or by none: only the others need the compares, which the ALU pipe issues at half
// rate (460 cycles a chunk; a load and the maxima 150). The max is taken if
// want_max. A window layer of 384 rows: 238 -> 225.5 us. In the general form, where
// it runs once or twice in an item of many blocks, it made a rollout step 1 % slower.
__device__ __noinline__ float mask_block_short(uint32_t cS, int n, int kb, int pos, int lo, bool want_max) {
  float m0 = -INFINITY, m1 = -INFINITY, first = -INFINITY;
  const unsigned span = (unsigned)(pos - lo);
  // keys that every row sees, and that some row sees
  const int all_lo = __reduce_max_sync(0xffffffffu, lo), all_hi = __reduce_min_sync(0xffffffffu, pos);
  const int any_lo = __reduce_min_sync(0xffffffffu, lo), any_hi = __reduce_max_sync(0xffffffffu, pos);
#pragma unroll 1
  for (int c = 0; c < n; ++c) {
    if (c == 2) first = fmaxf(m0, m1);
    uint32_t v[32];
    const int k0 = kb + 32 * c;
    const bool whole = k0 >= all_lo && k0 + 31 <= all_hi;
    if (whole && !want_max) continue;
    if (k0 > any_hi || k0 + 31 < any_lo) {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = 0xff800000u;
      tmem_st32(cS + 32 * c, v);
      continue;
    }
    tmem_ld32(cS + 32 * c, v);
    tmem_ld_wait();
    if (!whole) {
      const int r = k0 - lo;
#pragma unroll
      for (int e = 0; e < 32; ++e)
        if ((unsigned)(r + e) > span) v[e] = 0xff800000u;
      tmem_st32(cS + 32 * c, v);
    }
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      m0 = fmax3(m0, __uint_as_float(v[e]), __uint_as_float(v[e + 1]));
      m1 = fmax3(m1, __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
    }
  }
  tmem_st_wait();
  return first > -INFINITY ? first : fmaxf(m0, m1);
}

// p = 2^(s * scale_log2 - m) for the 64 scores, packed to bf16 pairs; returns
// the fp32 sum of the 64 values.
__device__ __forceinline__ float chunk_exp(const uint32_t (&sv)[2][32], float scale_log2, float neg_mu,
                                           uint32_t (&pk)[32]) {
  const uint64_t sl2x2 = pack_f32x2(scale_log2, scale_log2);
  const uint64_t nmux2 = pack_f32x2(neg_mu, neg_mu);
  uint64_t lsum[2] = {0, 0};
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
      const uint64_t x = fma2((uint64_t)sv[c][e] | ((uint64_t)sv[c][e + 1] << 32), sl2x2, nmux2);
      const float p0 = ex2_approx(lo_f32(x));
      const float p1 = ex2_approx(hi_f32(x));
      lsum[(e >> 1) & 1] = add2(lsum[(e >> 1) & 1], pack_f32x2(p0, p1));
      pk[c * 16 + e / 2] = pack_bf16x2(p0, p1);
    }
  const uint64_t ls = add2(lsum[0], lsum[1]);
  return lo_f32(ls) + hi_f32(ls);
}

__device__ __forceinline__ void st_shared_zero16(uint32_t addr) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
}
// 16 bytes of local memory (a: address in the local window)
__device__ __forceinline__ void st_local_v4(uint32_t a, const uint32_t* w) {
  asm volatile("st.local.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
               : "memory");
}
__device__ __forceinline__ void ld_local_v4(uint32_t a, uint32_t* w) {
  asm volatile("ld.local.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
               : "r"(a));
}
// one 32-byte store (p 32-byte aligned)
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]),
               "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}

// Self-test form only: the stalled role waits on a barrier nothing completes
// for half the library's wait limit, without polling the abort flag; then it
// raises the flag with its own mark (2) unless another role already did. The
// other roles, which began waiting at about the same time with the full
// limit, must leave on seeing the flag; one that ran out of its own wait
// instead would overwrite the mark with 1, and leave a half limit later.
constexpr uint64_t kSelftestStallNs = kWaitTimeoutNs / 2;
__device__ __forceinline__ void selftest_stall(uint32_t never_bar, int32_t* abort_flag) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait_sleep(never_bar, 0, 10000)) {
    if (global_timer_ns() - t0 > kSelftestStallNs) break;
  }
  atomicCAS(abort_flag, 0, 2);
}

__device__ __forceinline__ float chunk_max(const uint32_t (&sv)[2][32]) {
  float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      m0 = fmax3(m0, __uint_as_float(sv[c][e]), __uint_as_float(sv[c][e + 1]));
      m1 = fmax3(m1, __uint_as_float(sv[c][e + 2]), __uint_as_float(sv[c][e + 3]));
    }
  return fmaxf(m0, m1);
}

// A chunk whose probabilities sum to kSearchAt or more (or overflow, or are NaN)
// in some row of the warp: searched for its max, and where that exceeds the row's
// reference by more than the threshold, the reference is raised to it. Writes the
// chunk's P to columns cP, and rescales the block's first chunk of P (columns cP0)
// if it is not this one. Called, not inlined: with this code in the chunk loop the
// prefill of 8 prompts takes 1764 us instead of 1508. The scores are read from
// columns cS, or, if S has been released, from local memory (`scores`). With scores
// of 4 / 16 times unit variance, where most chunks of a warp raise some row, that
// prefill takes 2347 / 2986 us; with all scores through local memory 2525 / 3471,
// with S released only after the search 2181 / 2568 but 1801 at unit variance. The
// short form's items are a few blocks long, and its code the better for being
// shorter: always through local memory, by plain accesses (a window layer of 384
// rows 209.6 -> 207.0 us; in the general form plain ones made the prefill 1508 -> 1534).
struct SearchedChunk {
  float m_ref, sum, alpha;  // alpha: factor of what was summed under the old reference
};
template <bool kShort, typename Scores>  // uint4*, or an address in the local window
__device__ __noinline__ SearchedChunk search_chunk(uint32_t cS, bool released, Scores scores, float scale_log2,
                                                   float m_ref, float sum, uint32_t cP, uint32_t cP0) {
  SearchedChunk r = {m_ref, sum, 1.f};
  uint32_t sv[2][32], pk[32];
  if (!kShort && !released) {
    tmem_ld32(cS, sv[0]);
    tmem_ld32(cS + 32, sv[1]);
    tmem_ld_wait();
  } else {
#pragma unroll
    for (int e = 0; e < 64; e += 4) {
      if constexpr (kShort) {
        const uint4 v = scores[e / 4];
        uint32_t* at = &sv[e >> 5][e & 31];
        at[0] = v.x, at[1] = v.y, at[2] = v.z, at[3] = v.w;
      } else {
        ld_local_v4(scores + 4 * e, &sv[e >> 5][e & 31]);
      }
    }
  }
  const float mx = chunk_max(sv) * scale_log2;
  if (!(sum < kSearchAt) && mx > m_ref + kRescaleThreshold) {
    r.alpha = ex2_approx(m_ref - mx);
    r.m_ref = mx;
  }
  __syncwarp();
  r.sum = chunk_exp(sv, scale_log2, r.m_ref == -INFINITY ? 0.f : -r.m_ref, pk);
  tmem_st32(cP, pk);
  if (cP != cP0 && __any_sync(0xffffffffu, r.alpha != 1.f)) {
    tmem_st_wait();
    tmem_ld32(cP0, pk);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pk[e]));
      pk[e] = pack_bf16x2(f.x * r.alpha, f.y * r.alpha);
    }
    tmem_st32(cP0, pk);
  }
  return r;
}
// O (64 columns) times alpha. Whole warp.
__device__ __noinline__ void rescale_o(uint32_t cO, float alpha) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    uint32_t v[32];
    tmem_ld32(cO + 32 * h, v);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * alpha);
    tmem_st32(cO + 32 * h, v);
  }
}

}  // namespace

// kShort: for sliding windows of at most kShortWindow keys (see half_block)
template <bool kSelfTest, bool kShort>
__global__ void __maxnreg__(144)
    append_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                     const __grid_constant__ CUtensorMap qmap, const AttnParams p) {
  // launched programmatically (a call that may have decode rows only): wait for
  // the planner's records, then let the decode kernel be launched (it waits for
  // this grid). Without the condition the kernel's main loop ran 1.5 % slower in
  // every other call.
  if (p.chained) {
    grid_dep_wait();
    grid_dep_launch();
  }
  // nothing to do (no append rows this call): leave before TMEM and barriers
  if (header(p)->n_append == 0) return;
  extern __shared__ uint8_t smem_raw[];
  // broadcast from lane 0: what depends on the warp index alone stays in the uniform datapath
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t sQ = base;
  const uint32_t sK = base + kTcQBytes;
  const uint32_t sV = sK + kTcKStages * kTcKvBytes;
  TcSmem& st = *reinterpret_cast<TcSmem*>(smem_raw + (base - raw) + kTcQBytes +
                                          (kTcKStages + kTcVStages) * kTcKvBytes);
  volatile int32_t* abort_flag = &st.abort_flag;
  // shared-memory addresses of the barriers: one base register and an offset
  const uint32_t st_addr = sV + kTcVStages * kTcKvBytes;
  auto bar = [&](const uint64_t& b) {
    return st_addr + (uint32_t)(reinterpret_cast<const uint8_t*>(&b) - reinterpret_cast<const uint8_t*>(&st));
  };

  if (threadIdx.x == 0) {
    mbar_init(bar(st.q_full), 1);
    mbar_init(bar(st.q_empty), 2);  // one commit per tile issuer
    for (int s = 0; s < kTcKStages; ++s) {
      mbar_init(bar(st.k_full[s]), 1);
      mbar_init(bar(st.k_empty[s]), 2);
    }
    for (int s = 0; s < kTcVStages; ++s) {
      mbar_init(bar(st.v_full[s]), 1);
      mbar_init(bar(st.v_empty[s]), 2);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar(st.s_full[x]), 1);
      mbar_init(bar(st.s_free[x]), 4);
      mbar_init(bar(st.p_full[x]), 4);
      mbar_init(bar(st.o_ready[x]), 1);
      mbar_init(bar(st.o_free[x]), 4);
      mbar_init(bar(st.item_full[x]), 1);
      mbar_init(bar(st.item_empty[x]), kTcSoftmaxWarps + 3);  // softmax warps, both issuers, V producer
      mbar_init(bar(st.drain[x]), 1);
    }
    mbar_init(bar(st.never), 1);
    st.abort_flag = 0;
    if (kSelfTest) st.t_start = global_timer_ns();
    fence_barrier_init();
  }
  if (warp == kTcIssuerA) {
    tmem_alloc(smem_addr(&st.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = st.tmem_base;

  PlanHeader* hdr = header(p);
  const int Hkv = p.num_kv_heads, Hq = p.num_q_heads, g = p.group;
  const int n_items = hdr->n_append * Hkv;
  const AppendItem* items = reinterpret_cast<const AppendItem*>(p.ws + p.lay.append_items);

  if (warp == kTcKWarp || warp == kTcVWarp) {
    // ----------------------------------------------------------- producers
    // Two warps, one for K (and the item queue and the query tiles) and one
    // for V. The whole warp runs this loop: lane i keeps the page id of page
    // (chunk + i) for the current and the next 32-page chunk, so the block
    // table is read ahead with coalesced loads; an elected lane issues the copies.
    const bool is_k = warp == kTcKWarp;
    const CUtensorMap* map = is_k ? &kmap : &vmap;
    if (lane == 0) {
      prefetch_tensormap(map);
      if (is_k) prefetch_tensormap(&qmap);
    }
    const uint64_t pol = policy_evict_last();
    const int nst = is_k ? kTcKStages : kTcVStages;
    const uint32_t ring = is_k ? sK : sV;
    const uint32_t full0 = is_k ? bar(st.k_full[0]) : bar(st.v_full[0]);
    const uint32_t empty0 = is_k ? bar(st.k_empty[0]) : bar(st.v_empty[0]);
    uint32_t issued = 0, q_issued = 0;  // copies issued so far: blocks, query tiles
    int s = 0;                          // ring stage and phase of the next block
    uint32_t round = 0;
    for (int i = 0;; ++i) {
      const int slot = i & 1;
      AppendItem a;
      int idx = 0;
      if (is_k) {
        if (i >= 2 && !__all_sync(0xffffffffu, wait_bar(bar(st.item_empty[slot]), ((i >> 1) - 1) & 1, abort_flag)))
          break;
        if (lane == 0) idx = atomicAdd(&hdr->append_ticket, 1);
        idx = __shfl_sync(0xffffffffu, idx, 0);
        if (idx < n_items) a = items[idx / Hkv];
        if (lane == 0) {
          st.item_idx[slot] = idx;
          st.items[slot] = a;
          mbar_arrive(bar(st.item_full[slot]));
        }
      } else {
        if (!__all_sync(0xffffffffu, wait_bar(bar(st.item_full[slot]), (i >> 1) & 1, abort_flag))) break;
        idx = st.item_idx[slot];
        a = st.items[slot];
      }
      if (idx >= n_items) break;
      const int kvh = idx % Hkv;
      const int* bt_row = p.block_table + (size_t)a.row * p.max_pages;
      const int pg0 = a.key_begin / kPage;
      const int kb0 = pg0 * kPage;
      const int nb = (a.key_end - kb0 + kTcKeys - 1) / kTcKeys;
      const int page_end = (a.key_end + kPage - 1) / kPage;
      auto load_chunk = [&](int c) -> int {  // pool row of page pg0 + 32c + lane
        const int lp = pg0 + 32 * c + lane;
        int v = -1;
        if (lp < page_end) {
          v = __ldg(bt_row + lp);
          if (v < 0 || v >= p.num_pages) {
            raise_status(p, kStatusBadPage);
            v = -1;
          }
        }
        return v < 0 ? p.oob_row : (v * Hkv + kvh) * kPage;
      };
      int y_cur = load_chunk(0), y_next = load_chunk(1);
      if (is_k) {
        if (i >= 1 && !__all_sync(0xffffffffu, wait_bar(bar(st.q_empty), (i - 1) & 1, abort_flag))) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(bar(st.q_full), kTcQBytes);
          tma_load_3d(sQ, &qmap, 0, kvh * g, a.token_begin, bar(st.q_full));
        }
        q_issued = i + 1;
      }
      bool ok = true;
      constexpr int kPagesPerBlock = kTcKeys / kPage;  // 8: four blocks per 32-page chunk
      for (int b = 0; b < nb; ++b) {
        if (kSelfTest && is_k && p.selftest_stall == 1 && i == 0 && b == 1) {
          if (lane == 0) selftest_stall(bar(st.never), &st.abort_flag);
          __syncwarp();
          ok = false;
          break;
        }
        if (b > 0 && (b * kPagesPerBlock) % 32 == 0) {
          y_cur = y_next;
          y_next = load_chunk(b * kPagesPerBlock / 32 + 1);
        }
        const int lane0 = (b * kPagesPerBlock) % 32;
        if (round > 0 && !__all_sync(0xffffffffu, wait_bar(empty0 + 8 * s, (round - 1) & 1, abort_flag))) {
          ok = false;
          break;
        }
        const uint32_t dst = ring + s * kTcKvBytes, fb = full0 + 8 * s;
        const int n_pages = half_block<kShort>(a, kb0, b) ? kPagesPerBlock / 2 : kPagesPerBlock;
        if (lane == 0) mbar_arrive_expect_tx(fb, n_pages * kTileBytes);
        __syncwarp();
#pragma unroll 1
        for (int j = 0; j < n_pages; ++j)
          tma_load_2d_e(dst + j * kTileBytes, map, 0, __shfl_sync(0xffffffffu, y_cur, lane0 + j), fb, pol);
        ++issued;
        if (++s == nst) {
          s = 0;
          ++round;
        }
      }
      if (!ok) break;
      if (!is_k && lane == 0) mbar_arrive(bar(st.item_empty[slot]));
    }
    // After an abort, copies may still be in flight into the ring: wait
    // (bounded) for the last ones issued. Each such copy is the latest of its
    // stage, so its full barrier's phase parity identifies it. A finished
    // kernel has none in flight.
    if (*abort_flag && lane == 0) {
      for (uint32_t it = issued > (uint32_t)nst ? issued - nst : 0; it < issued; ++it)
        mbar_wait(full0 + 8 * (it % nst), (it / nst) & 1);
      if (q_issued > 0) mbar_wait(bar(st.q_full), (q_issued - 1) & 1);
    }
  } else if (warp == kTcIssuerA || warp == kTcIssuerB) {
    // ---------------------------------------------------------- MMA issuers
    // One issuing warp per tile (warp 9: tile A, warp 10: tile B), each in
    // its tile's own order S(b), PV(b - 1), so that neither tile's MMAs wait
    // behind the other tile's softmax. The whole warp runs the loop, the
    // operands are warp-uniform, and one elected lane issues a block's S or PV
    // MMAs and their commits in one branch: 2 instructions per MMA, where an
    // elect per MMA took about 20 and made the prefill of 8 prompts 5 % slower
    // (1475 -> 1556 us; the issuers' loop is on the critical path). Their MMAs
    // touch disjoint TMEM and are ordered only through the mbarriers; a K or V
    // stage and the query tiles are released by two commits, one per tile. The
    // loops are lean: descriptors are computed once and stepped by constants
    // (the start-address field counts 16-byte units and cannot overflow:
    // shared memory ends below 256 KiB).
    {
      constexpr uint32_t idS = idesc_bf16(kTcRows, kTcKeys, false, false);
      constexpr uint32_t idSHalf = idesc_bf16(kTcRows, kTcKeys / 2, false, false);
      constexpr uint32_t idO = idesc_bf16(kTcRows, kHeadDim, false, true);
      constexpr uint64_t kStageStep = kTcKvBytes / 16, kVStep = 16 * kRowBytes / 16;
      const uint64_t kdesc0 = smem_desc_sw128(sK, 16, 1024);
      const uint64_t vdesc0 = smem_desc_sw128(sV, 1024, 1024);
      // issuer x drives tile x: S_x(b) as soon as K(b) and its S buffer are
      // free, then O_x += P_x(b - 1) V(b - 1) once that P is ready; the two
      // tiles never wait on each other's softmax
      const int x = warp == kTcIssuerA ? 0 : 1;
      const uint32_t scol = tmem + col_s(x), pcol = tmem + col_p(x), ocol = tmem + col_o(x);
      const uint64_t qd = smem_desc_sw128(sQ + x * kTcTileQBytes, 16, 1024);
      uint32_t blk = 0;
      bool ok = true;
      for (int i = 0; ok; ++i) {
        const int slot = i & 1;
        if (!wait_bar(bar(st.item_full[slot]), (i >> 1) & 1, abort_flag)) break;
        const int idx = st.item_idx[slot];
        const AppendItem a = st.items[slot];
        if (idx >= n_items) break;
        const int kb0 = (a.key_begin / kPage) * kPage;
        const int nb = __shfl_sync(0xffffffffu, (a.key_end - kb0 + kTcKeys - 1) / kTcKeys, 0);  // uniform
        const bool last_half = kShort && __shfl_sync(0xffffffffu, (int)half_block<kShort>(a, kb0, nb - 1), 0);
        if (!wait_bar(bar(st.q_full), i & 1, abort_flag)) break;
        for (int b = 0; b <= nb && ok; ++b) {
          if (kSelfTest && p.selftest_stall == 2 && x == 0 && i == 0 && b == 1) {
            selftest_stall(bar(st.never), &st.abort_flag);
            ok = false;
            break;
          }
          if (b < nb) {  // S_x(b)
            const uint32_t bk = blk + b;
            const int s = bk % kTcKStages;
            // S buffer x was last loaded by the softmax of block bk - 1
            if (!wait_bar(bar(st.k_full[s]), (bk / kTcKStages) & 1, abort_flag) ||
                (bk >= 1 && !wait_bar(bar(st.s_free[x]), (bk - 1) & 1, abort_flag))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t kd = kdesc0 + s * kStageStep;
            const uint32_t id = last_half && b == nb - 1 ? idSHalf : idS;
            if (elect_lane()) {
              tc_mma_ss(scol, qd, kd, id, 0u);
#pragma unroll
              for (int kk = 1; kk < kHeadDim / 16; ++kk)
                tc_mma_ss(scol, qd + (uint64_t)(kk * 2), kd + (uint64_t)(kk * 2), id, 1u);
              tc_commit(bar(st.s_full[x]));
              tc_commit(bar(st.k_empty[s]));              // released when both tiles have read it
              if (b == nb - 1) tc_commit(bar(st.q_empty));  // likewise
            }
            __syncwarp();
          }
          if (b >= 1) {  // O_x += P_x(b - 1) V(b - 1)
            const uint32_t bv = blk + b - 1;
            const int sv = bv % kTcVStages;
            if (!wait_bar(bar(st.v_full[sv]), (bv / kTcVStages) & 1, abort_flag) ||
                !wait_bar(bar(st.p_full[x]), bv & 1, abort_flag) ||
                (b == 1 && i >= 1 && !wait_bar(bar(st.o_free[x]), (i - 1) & 1, abort_flag))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t vd = vdesc0 + sv * kStageStep;
            const bool half = last_half && b == nb;
            if (elect_lane()) {
              tc_mma_ts(ocol, pcol, vd, idO, b > 1 ? 1u : 0u);
#pragma unroll
              for (int kk = 1; kk < kTcKeys / 32; ++kk) tc_mma_ts(ocol, pcol + kk * 8, vd + kk * kVStep, idO, 1u);
              if (!half)
#pragma unroll
                for (int kk = kTcKeys / 32; kk < kTcKeys / 16; ++kk)
                  tc_mma_ts(ocol, pcol + kk * 8, vd + kk * kVStep, idO, 1u);
              tc_commit(bar(st.o_ready[x]));
              tc_commit(bar(st.v_empty[sv]));  // released when both tiles have read it
            }
            __syncwarp();
          }
        }
        if (!ok) break;
        blk += nb;
        if (lane == 0) mbar_arrive(bar(st.item_empty[slot]));
      }
      // wait for this thread's MMAs still in flight (only after an abort can
      // any be), so that TMEM is not freed under them
      if (elect_lane()) tc_commit(bar(st.drain[x]));
      __syncwarp();
      mbar_wait(bar(st.drain[x]), 0);
    }
  } else {
    // ------------------------------------------------------------- softmax
    const int x = warp >> 2;                      // tile A (0) or B (1)
    const int row = threadIdx.x & (kTcRows - 1);  // TMEM lane
    const int wq = warp & 3;
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    const uint32_t cS = tmem + lane_off + col_s(x), cP = tmem + lane_off + col_p(x), cO = tmem + lane_off + col_o(x);
    const int tile_tok = kTcRows / g;
    uint32_t blk = 0;
    bool ok = true;
    for (int i = 0; ok; ++i) {
      const int slot = i & 1;
      ok = __all_sync(0xffffffffu, wait_bar_poll(bar(st.item_full[slot]), (i >> 1) & 1, abort_flag));
      if (!ok) break;
      const int idx = st.item_idx[slot];
      const AppendItem a = st.items[slot];
      if (idx >= n_items) break;
      const int kvh = idx % Hkv;
      const int tok = x * tile_tok + row / g, head = row % g;
      const bool valid = tok < a.n_tok;
      const int last_tok = max(a.n_tok - 1, 0);
      const int pos = a.pos_begin + min(tok, last_tok);
      const int lo = p.window > 0 ? pos - p.window + 1 : 0;
      const int kb0 = (a.key_begin / kPage) * kPage;
      const int nb = (a.key_end - kb0 + kTcKeys - 1) / kTcKeys;
      // warp-uniform position range of this warp's rows, for mask skipping
      const int wp_min = a.pos_begin + min(x * tile_tok + (wq * 32) / g, last_tok);
      const int wp_max = a.pos_begin + min(x * tile_tok + (wq * 32 + 31) / g, last_tok);
      float m_ref = -INFINITY, l = 0.f;
      for (int b = 0; b < nb; ++b, ++blk) {
        if (kSelfTest && p.selftest_stall == 0 && x == 0 && i == 0 && b == 1) {
          if (lane == 0) selftest_stall(bar(st.never), &st.abort_flag);
          __syncwarp();
          ok = false;
          break;
        }
        ok = __all_sync(0xffffffffu, wait_bar_poll(bar(st.s_full[x]), blk & 1, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const int kb = kb0 + b * kTcKeys;
        const int nc = half_block<kShort>(a, kb0, b) ? 1 : 2;  // chunks of 64 keys
        // an item's first block, blocks that some row does not see whole
        if (kShort) {
          const bool want_max = __any_sync(0xffffffffu, m_ref == -INFINITY);
          if (want_max || kb + kTcKeys - 1 > wp_min || kb <= wp_max - p.window) {
            const float mx = mask_block_short(cS, 2 * nc, kb, pos, lo, want_max) * p.scale_log2;
            if (m_ref == -INFINITY) m_ref = mx;
          }
        } else if (b == 0 || kb + kTcKeys - 1 > wp_min || (p.window > 0 && kb <= wp_max - p.window) ||
                   __any_sync(0xffffffffu, m_ref == -INFINITY)) {
          const float mx = mask_block(cS, kb, pos, lo) * p.scale_log2;
          if (m_ref == -INFINITY) m_ref = mx;
        }
        float lb = 0.f, alpha = 1.f;  // the block's sum; factor of what came before it
        bool searched = false;
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {  // keys kb + 64c .. kb + 64c + 63
          uint32_t sv[2][32], pk[32];
          tmem_ld32(cS + 64 * c, sv[0]);
          tmem_ld32(cS + 64 * c + 32, sv[1]);
          tmem_ld_wait();
          if (c == nc - 1) {  // S_X is in registers
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(st.s_free[x]));
          }
          const float lc = chunk_exp(sv, p.scale_log2, m_ref == -INFINITY ? 0.f : -m_ref, pk);
          // the single P buffer was last read by PV_X(blk - 1)
          if (c == 0 && blk >= 1) {
            ok = __all_sync(0xffffffffu, wait_bar_poll(bar(st.o_ready[x]), (blk - 1) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
          }
          if (__any_sync(0xffffffffu, !(lc < kSearchAt))) {  // also for inf / NaN
            uint4 copy[16];
            SearchedChunk r;
            if constexpr (kShort) {
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const uint32_t* v = &sv[e >> 3][4 * (e & 7)];
                copy[e] = make_uint4(v[0], v[1], v[2], v[3]);
              }
              r = search_chunk<true, const uint4*>(cS + 64 * c, true, copy, p.scale_log2, m_ref, lc, cP + 32 * c, cP);
            } else {
              const uint32_t scores = (uint32_t)__cvta_generic_to_local(copy);
              if (c == nc - 1) {
#pragma unroll
                for (int e = 0; e < 64; e += 4) st_local_v4(scores + 4 * e, &sv[e >> 5][e & 31]);
              }
              r = search_chunk<false, uint32_t>(cS + 64 * c, c == nc - 1, scores, p.scale_log2, m_ref, lc, cP + 32 * c,
                                                cP);
            }
            m_ref = r.m_ref;
            alpha *= r.alpha;
            searched = true;
            lb = __fmul_rn(lb, r.alpha);  // no fused multiply-add with the sum
            lb += r.sum;
          } else {
            lb += lc;
            tmem_st32(cP + 32 * c, pk);
          }
        }
        if (!ok) break;
        l = fmaf(l, alpha, lb);
        // O_X may only be rescaled once PV_X(blk - 1) has completed (waited above)
        if (b > 0 && searched && __any_sync(0xffffffffu, alpha != 1.f)) rescale_o(cO, alpha);
        // V rows of slots no query of the item sees (before key_begin on the
        // partial first page of a window, from key_end on the partial last
        // page) were perhaps never written and may hold NaN, which a zero
        // weight does not cancel (0 x NaN = NaN). Once the block's V stage
        // has landed they are zeroed in shared memory (at most 15 rows each;
        // whole pages past the row's end arrive as zeros already), then
        // handed to the async proxy before this tile's PV may read them. Both
        // tiles' warps write the same zeros, each before its own p_full.
        const bool lo_edge = b == 0 && kb0 < a.key_begin;
        const bool hi_edge = b == nb - 1 && (a.key_end & (kPage - 1)) != 0;
        if (lo_edge || hi_edge) {
          const uint32_t sv_i = blk % kTcVStages;
          ok = __all_sync(0xffffffffu, wait_bar_poll(bar(st.v_full[sv_i]), (blk / kTcVStages) & 1, abort_flag));
          if (!ok) break;
          const uint32_t vst = sV + sv_i * kTcKvBytes;
          const int zr = row >> 3, zc = row & 7;  // key row (0..15) and 16-byte chunk of this thread
          if (lo_edge && zr < a.key_begin - kb0) st_shared_zero16(vst + zr * kRowBytes + zc * 16);
          if (hi_edge) {
            const int r0 = a.key_end - kb;  // first row past the row's end, inside this block
            if (zr < kPage - (r0 & (kPage - 1))) st_shared_zero16(vst + (r0 + zr) * kRowBytes + zc * 16);
          }
          fence_proxy_async();
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(st.p_full[x]));
      }
      if (!ok) break;
      // epilogue: the last PV_X of the item
      if (nb > 0) {
        ok = __all_sync(0xffffffffu, wait_bar_poll(bar(st.o_ready[x]), (blk - 1) & 1, abort_flag));
        if (!ok) break;
      }
      tc_fence_after();
      float inv = l > 0.f ? 1.f / l : 0.f;
      float lse2 = l > 0.f ? m_ref + __log2f(l) : -INFINITY;
      if (p.sinks != nullptr) inv = finish_with_sink(m_ref, l, sink_log2(p, kvh * g + head), &lse2);
      const size_t orow = (size_t)(a.token_begin + tok) * Hq + kvh * g + head;
      uint8_t* dst = reinterpret_cast<uint8_t*>(p.out + orow * kHeadDim);
      uint32_t ov[2][32];
      tmem_ld32(cO, ov[0]);
      tmem_ld32(cO + 32, ov[1]);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar(st.o_free[x]));
        mbar_arrive(bar(st.item_empty[slot]));
      }
      if (valid) {
        // O / l as bf16 words (dims 2j, 2j + 1), in whole 32-byte sectors: a
        // store of the warp touches 32 rows, and halves of sectors cost twice
        // the stores (a window layer of 384 rows 225.5 -> 211 us) and, in host
        // memory, far more
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint32_t w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            w[j] = pack_bf16x2(__uint_as_float(ov[h >> 1][16 * (h & 1) + 2 * j]) * inv,
                               __uint_as_float(ov[h >> 1][16 * (h & 1) + 2 * j + 1]) * inv);
          if ((reinterpret_cast<uintptr_t>(p.out) & 31) == 0) {
            st_global_v8(dst + 32 * h, w);
          } else {
            reinterpret_cast<uint4*>(dst)[2 * h] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4*>(dst)[2 * h + 1] = make_uint4(w[4], w[5], w[6], w[7]);
          }
        }
        p.lse[orow] = lse2 * 0.69314718055994531f;
      }
    }
  }

  // every role ends here; a timed-out role has set the abort flag
  __syncwarp();
  if (kSelfTest && lane == 0 && blockIdx.x == 0)  // the later of the two producers under one entry
    atomicMax(reinterpret_cast<unsigned long long*>(p.selftest_report + 1 + (warp == kTcVWarp ? kTcKWarp : warp)),
              (unsigned long long)(global_timer_ns() - st.t_start));
  if (threadIdx.x == 0 && *abort_flag) raise_status(p, kStatusTimeout);
  tc_fence_before();
  __syncthreads();
  if (warp == kTcIssuerA) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
    if (kSelfTest && lane == 0 && blockIdx.x == 0) {
      p.selftest_report[0] = *abort_flag;
      p.selftest_report[12] = (int64_t)kSelftestStallNs;
      p.selftest_report[13] = (int64_t)kWaitTimeoutNs;
      p.selftest_report[14] = 1;  // TMEM freed
    }
  }
}

// programmatic: launched with programmatic stream serialization after the planner.
cudaError_t launch_append_tc(const CUtensorMap& kmap, const CUtensorMap& vmap, const CUtensorMap& qmap,
                             const AttnParams& p, int grid, cudaStream_t stream, bool programmatic) {
  LaunchCfg lc(dim3(grid), dim3(kTcThreads), append_tc_smem_bytes(), stream, programmatic);
  const bool is_short = p.window > 0 && p.window <= kShortWindow;
  return cudaLaunchKernelEx(&lc.cfg, is_short ? append_tc_kernel<false, true> : append_tc_kernel<false, false>, kmap,
                            vmap, qmap, p);
}

// The self-test form: one CTA, p.selftest_stall names the stalled role and
// p.selftest_report receives the abort flag and each warp's exit time.
cudaError_t launch_append_tc_selftest(const CUtensorMap& kmap, const CUtensorMap& vmap, const CUtensorMap& qmap,
                                      const AttnParams& p, cudaStream_t stream) {
  append_tc_kernel<true, false><<<1, kTcThreads, append_tc_smem_bytes(), stream>>>(kmap, vmap, qmap, p);
  return cudaGetLastError();
}

cudaError_t prepare_append_tc_kernel(int* blocks_per_sm) {
  for (auto fn : {append_tc_kernel<false, false>, append_tc_kernel<false, true>, append_tc_kernel<true, false>}) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)append_tc_smem_bytes());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, append_tc_kernel<false, false>, kTcThreads,
                                                       append_tc_smem_bytes());
}

}  // namespace mcpu
