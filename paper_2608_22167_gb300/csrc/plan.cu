// Work planner: one CTA reads seq_lens / query_start_loc / block_table on the
// device and writes the work lists of the attention kernels into the
// workspace, so a forward call needs no host round trip and can be captured
// in a CUDA graph.
//
// It decides, per row: decode (L = 1), append (L > 1) or nothing; for decode
// rows, the KV split length and the partial-result slots merged later by
// log-sum-exp; for runs of adjacent rows whose block tables begin with the
// same physical pages (the G samples of a GRPO task sharing their prompt,
// paper §4), the shared prefix that one cascade pass reads once for the
// whole group; for append rows, the query tiles of the chunk kernel.
//
// One thread owns a row (two above 1024 rows) and keeps its quantities in
// registers; one fused prefix sum turns the counts into record offsets. The
// owner writes a row's first record; further records of split rows are written
// by eight lanes per row.
//
// What bounds it: the latency of one CTA, i.e. barriers, dependent loads and
// instruction fetch (code that runs once costs about 5 cycles per
// instruction). So no loop is unrolled, nothing is scanned twice, and what a
// call does not need (groups, append rows, split rows) is branched over as a
// whole. Measured against ten scans over shared memory with a binary search per
// record (67 KB of code, now 22): 64 decode rows 9.6 -> 4.9 us, 384 rows of a
// window layer 13.5 -> 7.7, 512 long rows 18.3 -> 13.1, 256 mixed rows 14.8 -> 10.2.
#include "common.cuh"

namespace mcpu {

// Row flags
constexpr int kFlagDirect = 1;    // decode row with one part: writes out/lse itself
constexpr int kFlagSubFirst = 2;  // first member of its cascade subgroup

struct PlanSmem {
  int S[kMaxSeqs];           // seq_len, -1 if the row is invalid
  int L[kMaxSeqs];           // query tokens (0 if the row is invalid)
  int Q0[kMaxSeqs];          // first query token
  int own_pb[kMaxSeqs];      // first page of the row's own decode range
  int n_own[kMaxSeqs];       // decode records
  int item_off[kMaxSeqs];    // first decode record
  int slot0[kMaxSeqs];       // partial slot of the row's first own split
  int sg_off[kMaxSeqs];      // first cascade record (subgroup-first rows)
  int gs[kMaxSeqs];          // first row of the row's run (group)
  int mrank[kMaxSeqs];       // members in the rows before
  int grp_pages[kMaxSeqs];   // per group, at its first row: shared full pages
  int grp_ndec[kMaxSeqs];    // per group, at its first row: decode rows
  int app_row[kMaxSeqs];     // append rows, longest first
  int app_off[kMaxSeqs];     // first append record of the row of that rank
  int warp_max[32];          // warp totals of the scans
  int warp_sum[6][32];
  int total_wm, total_wlb;
  int cascade_pages;         // pages of all cascade items of kCascadeVectors vectors
};

namespace {

__device__ __forceinline__ int cdiv(int a, int b) { return (a + b - 1) / b; }

// Inclusive sum over the warp's lanes.
__device__ __forceinline__ int warp_scan(int x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Exclusive prefix sum over the CTA, one value per thread; `part` holds the
// warps' totals and is used by this scan alone (one barrier).
template <int NT>
__device__ __forceinline__ int cta_scan(int v, int* total, int* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = warp_scan(v);
  if (lane == 31) part[warp] = x;
  __syncthreads();
  const int t = lane < NT / 32 ? part[lane] : 0;
  *total = (int)__reduce_add_sync(0xffffffffu, (unsigned)t);
  return (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? t : 0)) + x - v;
}

}  // namespace

// Number of leading block-table entries that rows r - 1 and r share, over the
// pages full in both (lengths outside the table count as none); one warp, the
// result in every lane. A step compares 32 * PER entries: PER loads of each row
// per lane in flight, one ballot per 32. FIRST: the first step's PER, fewer
// where the code is cold and most rows differ at once.
template <int PER>
__device__ __forceinline__ bool shared_step(const int* ba, const int* bb, int base, int lim, int& n) {
  const int lane = threadIdx.x & 31;
  int va[PER], vb[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = base + 32 * j + lane;
    va[j] = i < lim ? __ldg(ba + i) : 0;
    vb[j] = i < lim ? __ldg(bb + i) : 1;
  }
  bool stop = false;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const unsigned m = __ballot_sync(0xffffffffu, va[j] == vb[j]);
    if (!stop) {
      if (m == 0xffffffffu) {
        n += 32;
      } else {
        n += __ffs(~m) - 1;
        stop = true;
      }
    }
  }
  return stop;
}

template <int FIRST>
__device__ __forceinline__ int shared_entries(const AttnParams& p, int r) {
  constexpr int kPer = 16;
  const int cap = p.max_pages * kPage;
  const int sa = __ldg(p.seq_lens + r - 1), sb = __ldg(p.seq_lens + r);
  const int lim = (sa < 0 || sb < 0 || sa > cap || sb > cap) ? 0 : min(sa, sb) / kPage;
  const int* ba = p.block_table + (size_t)(r - 1) * p.max_pages;
  const int* bb = p.block_table + (size_t)r * p.max_pages;
  int n = 0, base = 0;
  bool stop = lim == 0;
  if (FIRST < kPer && !stop) {
    stop = shared_step<FIRST>(ba, bb, 0, lim, n);
    base = 32 * FIRST;
  }
#pragma unroll 1
  for (; !stop && base < lim; base += 32 * kPer) stop = shared_step<kPer>(ba, bb, base, lim, n);
  return min(n, lim);
}

// Batches of at most this many rows (one per warp of the smallest form) are
// scanned by the planner itself, a warp per row beside phase 1: one launch fewer
// (1 / 8 short rows 18.5 / 20.5 -> 16.5 / 19.4 us as a graph, 5 rows of 20-65 thousand
// keys 85.1 -> 84.1; eager calls 1-3 us). With more rows the scan is a kernel of its
// own, a warp per row across the GPU.
constexpr int kScanInPlanner = 8;

// lcp[r] of every row r > 0, lcp[0] = 0.
constexpr int kLcpWarps = 8;

__global__ void __launch_bounds__(kLcpWarps * 32) lcp_kernel(const AttnParams p) {
  grid_dep_launch();  // the planner may start its first phase meanwhile
  const int r = blockIdx.x * kLcpWarps + (threadIdx.x >> 5);
  int* lcp = reinterpret_cast<int*>(p.ws + p.lay.lcp);
  if (r >= p.num_seqs) return;
  const int n = r > 0 ? shared_entries<16>(p, r) : 0;
  if ((threadIdx.x & 31) == 0) lcp[r] = n;
}

template <int NT, int R>
__global__ void __launch_bounds__(NT, 1) plan_kernel(AttnParams p) {
  extern __shared__ __align__(16) uint8_t plan_smem_raw[];
  PlanSmem& sm = *reinterpret_cast<PlanSmem*>(plan_smem_raw);
  PlanHeader* hdr = header(p);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int B = p.num_seqs;
  int sub_cap = kCascadeVectors / p.group;  // rows per cascade item
  auto publish = [&](int n_decode, int n_cascade, int n_append, int n_merge, int n_parts) {
    hdr->n_decode = n_decode;
    hdr->n_cascade = n_cascade;
    hdr->n_append = n_append;
    hdr->n_merge = n_merge;
    hdr->n_parts = n_parts;
    hdr->cascade_wide = sub_cap > kCascadeVectors / p.group;
    hdr->append_ticket = hdr->decode_ticket = hdr->cascade_ticket = 0;
  };

  if (p.chained) grid_dep_launch();  // the next kernel may be launched meanwhile (it waits for this grid)

  // ---- phase 1: per-row kind (0 none / invalid, 1 decode, 2 append) and lengths
  int S[R], L[R], Q0[R], kind[R];
  int status = 0, bad_global = 0;
  if (tid == 0) sm.total_wm = sm.total_wlb = sm.cascade_pages = 0;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = tid * R + i;
    S[i] = -1, L[i] = 0, Q0[i] = 0, kind[i] = 0;
    if (r < B) {
      const int q0 = p.qsl[r], q1 = p.qsl[r + 1], s = p.seq_lens[r];
      if ((r == 0 && q0 != 0) || (r == B - 1 && q1 != p.total_q)) bad_global = 1;
      const int len = q1 - q0;
      // a row's tokens lie in [0, total_q): every kernel after this one trusts its record's token
      const bool bad = q0 < 0 || q1 > p.total_q || len < 0 || s < len || s > p.max_pages * kPage;
      // decode-only calls (fp8 pools) report and skip append rows
      const bool skip = !bad && p.decode_only && len > 1;
      if (bad) status |= kStatusBadLengths;
      if (skip) status |= kStatusUnsupportedRow;
      Q0[i] = q0;
      if (!bad && !skip) S[i] = s, L[i] = len, kind[i] = min(len, 2);
      sm.S[r] = S[i];
      sm.grp_pages[r] = 0x7fffffff;
      sm.grp_ndec[r] = 0;
    }
  }
  if (NT == 256 && B <= kScanInPlanner && p.cascade_enabled && p.window <= 0 && warp < B) {
    const int n = warp > 0 ? shared_entries<1>(p, warp) : 0;
    if (lane == 0) reinterpret_cast<int*>(p.ws + p.lay.lcp)[warp] = n;  // read after the barrier
  }
  if (__syncthreads_or(bad_global)) {
    grid_dep_wait();  // nothing of this call ends before the prefix scan
    if (tid == 0) {
      atomicOr(&hdr->status, kStatusBadLengths);
      publish(0, 0, 0, 0, 0);
    }
    return;
  }
  if (status) atomicOr(&hdr->status, status);

  // ---- phase 2: shared-prefix groups (full-context calls only)
  // lcp[r] = leading physical pages row r shares with row r - 1 (full pages
  // of both), scanned in phase 1 (few rows) or beforehand by lcp_kernel across
  // the whole GPU. The planner may have been launched while that scan ran (phase 1 reads only
  // the caller's arrays): wait for it here.
  grid_dep_wait();
  int gp[R], flags[R], pb[R], sub_idx[R], sub_n[R];  // shared pages (members); first own page; subgroup
#pragma unroll
  for (int i = 0; i < R; ++i) gp[i] = 0, flags[i] = 0, pb[i] = 0, sub_idx[i] = -1, sub_n[i] = 0;
  if (p.cascade_enabled && p.window <= 0) {
    const int* lcp_ws = reinterpret_cast<const int*>(p.ws + p.lay.lcp);
    int lcp[R], gs[R], run = -1;  // a run's first row has lcp = 0 here
    bool any = false;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = tid * R + i;
      const int sa = r > 0 && r < B ? sm.S[r - 1] : -1;
      lcp[i] = (sa < 0 || S[i] < 0) ? 0 : min(lcp_ws[r], min(sa, S[i]) / kPage);
      if (lcp[i] < kMinSharedPages) lcp[i] = 0;
      any |= lcp[i] > 0;
      if (r < B && lcp[i] == 0) run = r;
      gs[i] = run;
    }
    if (__syncthreads_or(any)) {
      // first row of each row's run: the last run start at or before it
      int x = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = max(x, y);
      }
      int before = __shfl_up_sync(0xffffffffu, x, 1);
      if (lane == 0) before = -1;
      if (lane == 31) sm.warp_max[warp] = x;
      __syncthreads();
      before = max(before, __reduce_max_sync(0xffffffffu, lane < warp ? sm.warp_max[lane] : -1));
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = tid * R + i;
        if (r >= B) continue;
        if (gs[i] < 0) gs[i] = before;
        sm.gs[r] = gs[i];
        if (lcp[i] > 0) atomicMin(&sm.grp_pages[gs[i]], lcp[i]);
        if (kind[i] == 1) {
          atomicMin(&sm.grp_pages[gs[i]], S[i] / kPage);
          atomicAdd(&sm.grp_ndec[gs[i]], 1);
        }
      }
      __syncthreads();
      // members: decode rows of a group with >= 2 decode rows and a long enough prefix
      int m[R], n_m = 0, tot;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        m[i] = kind[i] == 1 && sm.grp_ndec[gs[i]] >= 2 && sm.grp_pages[gs[i]] >= kMinSharedPages;
        n_m += m[i];
      }
      int rank = cta_scan<NT>(n_m, &tot, sm.warp_sum[0]);
      int mr[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = tid * R + i;
        mr[i] = rank;
        if (r < B) sm.mrank[r] = rank;
        rank += m[i];
        if (r < B && gs[i] == r && sm.grp_ndec[r] >= 2 && sm.grp_pages[r] >= kMinSharedPages)
          atomicAdd(&sm.cascade_pages, sm.grp_pages[r] * cdiv(sm.grp_ndec[r], sub_cap));
      }
      __syncthreads();
      if (p.wide_cascade && (long long)sm.cascade_pages * p.num_kv_heads > (long long)kWidePages * p.total_warps_hint)
        sub_cap *= 2;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        if (!m[i]) continue;
        const int nd = sm.grp_ndec[gs[i]], base = sm.mrank[gs[i]], idx = mr[i] - base;
        gp[i] = pb[i] = sm.grp_pages[gs[i]];
        const int nsub = cdiv(nd, sub_cap), sub = idx * nsub / nd;
        const int first = cdiv(sub * nd, nsub);
        sub_idx[i] = base + first;
        sub_n[i] = cdiv((sub + 1) * nd, nsub) - first;
        if (idx == first) flags[i] |= kFlagSubFirst;
      }
    }
  }

  // ---- phase 3: split length
  int w_m = 0, w_lb = 0;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    if (kind[i] != 1) continue;
    if (gp[i] == 0) pb[i] = p.window > 0 ? max(0, S[i] - p.window) / kPage : 0;
    const int own = cdiv(S[i], kPage) - pb[i];
    w_m += own + gp[i];
    w_lb += own + ((flags[i] & kFlagSubFirst) ? gp[i] : 0);
  }
  w_m = (int)__reduce_add_sync(0xffffffffu, (unsigned)w_m);
  w_lb = (int)__reduce_add_sync(0xffffffffu, (unsigned)w_lb);
  if (lane == 0) {
    atomicAdd(&sm.total_wm, w_m);
    atomicAdd(&sm.total_wlb, w_lb);
  }
  __syncthreads();
  const int c_bound = max(1, cdiv(sm.total_wm, kSplitBudget));
  int C;
  if (p.forced_split_pages > 0) {
    C = max(p.forced_split_pages, c_bound);
  } else {
    // W = (page, kv head) blocks per decode warp. A split of C pages costs a
    // fixed overhead of about 12 pages' time (query setup, ring ramp, the
    // partial's write and merge) and leaves a tail of about C / 2 pages at the
    // end, so the time per warp ~ W + 12 W / C + C / 2 is least at
    // C = sqrt(24 W) (measured optimum 64 pages at W = 162 and 384-512 at
    // W = 4441 for bf16 pages, 48 at W = 121 and 256 at W = 3330 for fp8).
    const float w = (float)sm.total_wlb * (float)p.num_kv_heads / (float)max(p.total_warps_hint, 1);
    C = max(kMinSplitPages, max((int)(sqrtf(24.f * w) + 0.5f), c_bound));
    if (rows_unsplit(p)) C = max(C, p.window / kPage + 2);  // the most pages that a window touches
  }

  // ---- phase 4: per-row counts -> offsets, all in one scan
  int n_own[R], n_cs[R], parts[R];
  int c_parts = 0, c_items = 0, c_sg = 0, c_rows = 0, c_tiles = 0;  // c_rows: merge rows + append rows << 16
#pragma unroll
  for (int i = 0; i < R; ++i) {
    n_own[i] = n_cs[i] = parts[i] = 0;
    if (kind[i] == 1) {
      n_own[i] = cdiv(cdiv(S[i], kPage) - pb[i], C);
      if (gp[i] > 0) n_cs[i] = cdiv(gp[i], C);
      parts[i] = n_own[i] + n_cs[i];
      if (gp[i] == 0 && parts[i] == 1) {
        flags[i] |= kFlagDirect;
        parts[i] = 0;
      }
      c_parts += parts[i];
      c_items += n_own[i];
      if (flags[i] & kFlagSubFirst) c_sg += n_cs[i];
      c_rows += (flags[i] & kFlagDirect) ? 0 : 1;
    } else if (kind[i] == 2) {
      c_rows += 1 << 16;
      c_tiles += cdiv(L[i], p.append_tile_tok);
    }
  }
  int o_parts = warp_scan(c_parts), o_items = warp_scan(c_items), o_sg = warp_scan(c_sg), o_rows = warp_scan(c_rows);
  const int t_tiles = (int)__reduce_add_sync(0xffffffffu, (unsigned)c_tiles);
  if (lane == 31) {
    sm.warp_sum[1][warp] = o_parts;
    sm.warp_sum[2][warp] = o_items;
    sm.warp_sum[3][warp] = o_sg;
    sm.warp_sum[4][warp] = o_rows;
    sm.warp_sum[5][warp] = t_tiles;
  }
  __syncthreads();
  int tot[6];
  {
    int before[6];
#pragma unroll
    for (int k = 1; k < 6; ++k) {
      const int t = lane < NT / 32 ? sm.warp_sum[k][lane] : 0;
      tot[k] = (int)__reduce_add_sync(0xffffffffu, (unsigned)t);
      before[k] = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? t : 0));
    }
    o_parts += before[1] - c_parts;
    o_items += before[2] - c_items;
    o_sg += before[3] - c_sg;
    o_rows += before[4] - c_rows;
  }
  const int tot_parts = tot[1], tot_items = tot[2], tot_cascade = tot[3], n_merge = tot[4] & 0xffff, n_app = tot[4] >> 16,
            tot_tiles = tot[5];
  if (tot_items > p.lay.max_decode || tot_cascade > p.lay.max_cascade || tot_tiles > p.lay.max_append ||
      tot_parts > p.lay.max_parts) {
    if (tid == 0) {
      atomicOr(&hdr->status, kStatusPlanOverflow);
      publish(0, 0, 0, 0, 0);
    }
    return;
  }

  // ---- phase 5: per-row records, and each row's first decode record
  DecodeItem* ditems = reinterpret_cast<DecodeItem*>(p.ws + p.lay.decode_items);
  MergeRow* mrows = reinterpret_cast<MergeRow*>(p.ws + p.lay.merge_rows);
  CascadeMember* members = reinterpret_cast<CascadeMember*>(p.ws + p.lay.members);
  int more = 0;  // some row has a second decode record
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = tid * R + i;
    if (r >= B) continue;
    sm.n_own[r] = n_own[i];
    if (kind[i] == 1) {
      const bool direct = flags[i] & kFlagDirect;
      if (!direct) {
        mrows[o_rows & 0xffff] = MergeRow{Q0[i], parts[i], o_parts, 0};
        ++o_rows;
      }
      if (gp[i] > 0) members[sm.mrank[r]] = CascadeMember{r, Q0[i], o_parts, 0};
      const int slot0 = direct ? -1 : o_parts + n_cs[i];
      if (n_own[i] > 0)
        ditems[o_items] = DecodeItem{r, Q0[i], S[i], p.window > 0 ? max(0, S[i] - p.window) : 0,
                                     pb[i], min(cdiv(S[i], kPage), pb[i] + C), slot0, 0};
      if (n_own[i] > 1) {
        more = 1;
        sm.Q0[r] = Q0[i], sm.own_pb[r] = pb[i], sm.item_off[r] = o_items, sm.slot0[r] = slot0;
      }
      o_parts += parts[i];
      o_items += n_own[i];
    } else if (kind[i] == 2) {
      sm.app_row[o_rows >> 16] = r;
      sm.L[r] = L[i], sm.Q0[r] = Q0[i];
      o_rows += 1 << 16;
    }
    if (tot_cascade > 0) {
      sm.sg_off[r] = o_sg;
      if (flags[i] & kFlagSubFirst) o_sg += n_cs[i];
    }
  }
  if (__syncthreads_or(more)) {
    // further decode records of split rows: eight lanes per row
#pragma unroll 1
    for (int r = tid >> 3; r < B; r += NT / 8) {
      const int n = sm.n_own[r];
#pragma unroll 1
      for (int k = 1 + (tid & 7); k < n; k += 8) {
        const int s = sm.S[r], b = sm.own_pb[r] + k * C;
        ditems[sm.item_off[r] + k] = DecodeItem{r, sm.Q0[r], s, p.window > 0 ? max(0, s - p.window) : 0,
                                                b, min(cdiv(s, kPage), b + C), sm.slot0[r] + k, 0};
      }
    }
  }
  if (tot_cascade > 0) {
    // Cascade records of one group go split-major: (split k, subgroup s) at
    // the group's base + k * nsub + s, so the subgroups of a group (8 rows at
    // g = 8: four of 2) read the same pages within a few tickets of each other
    // and the later reads of a page are L2 hits, not further HBM reads.
    CascadeItem* citems = reinterpret_cast<CascadeItem*>(p.ws + p.lay.cascade_items);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (!(flags[i] & kFlagSubFirst)) continue;
      const int r = tid * R + i, g0 = sm.gs[r], n = n_cs[i];
      const int nd = sm.grp_ndec[g0], nsub = cdiv(nd, sub_cap);
      const int sub = (sm.mrank[r] - sm.mrank[g0]) * nsub / nd;
      const int dst = sm.sg_off[r] - sub * n + sub;
#pragma unroll 1
      for (int k = 0; k < n; ++k)
        citems[dst + k * nsub] = CascadeItem{sub_idx[i], sub_n[i], k * C, min(gp[i], (k + 1) * C), k, r, 0, 0};
    }
  }

  // ---- append rows, longest first: the persistent append kernel takes its
  // items in record order, so it starts with the rows that have the most
  // keys (the longest items) and ends on short ones, which shortens its tail
  // (a list-scheduling model of the 256-row mixed batch: 2.0 % -> 0.6 % idle
  // at the end). Ties keep row order; above kMaxRanked rows the ranking's
  // n^2 comparisons are skipped and row order stays.
  if (n_app > 0) {
    const int tile_tok = p.append_tile_tok;
    AppendItem* aitems = reinterpret_cast<AppendItem*>(p.ws + p.lay.append_items);
    constexpr int kMaxRanked = 512;
    if (n_app <= kMaxRanked) {
#pragma unroll 1
      for (int i = tid; i < n_app; i += NT) {
        const int r = sm.app_row[i], Sr = sm.S[r];
        int rank = 0;
#pragma unroll 4
        for (int j = 0; j < n_app; ++j) {
          const int q = sm.app_row[j], Sq = sm.S[q];
          rank += (Sq > Sr || (Sq == Sr && q < r)) ? 1 : 0;
        }
        sm.app_off[rank] = r;  // app_off as scratch: row of each rank
      }
      __syncthreads();
#pragma unroll 1
      for (int i = tid; i < n_app; i += NT) sm.app_row[i] = sm.app_off[i];
      __syncthreads();
    }
    // offsets of the ranked rows' tiles: ranks tid * R .. + R - 1
    int t[R], sum = 0, total;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int k = tid * R + i;
      t[i] = k < n_app ? cdiv(sm.L[sm.app_row[k]], tile_tok) : 0;
      sum += t[i];
    }
    int off = cta_scan<NT>(sum, &total, sm.warp_max);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int k = tid * R + i;
      if (k < n_app) sm.app_off[k] = off;
      off += t[i];
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < tot_tiles; e += NT) {
      int lo = 0, hi = n_app;  // the row whose tiles hold record e: app_off[lo] <= e < app_off[hi]
#pragma unroll 1
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sm.app_off[mid] <= e) lo = mid; else hi = mid;
      }
      const int r = sm.app_row[lo], s = sm.S[r], len = sm.L[r];
      const int k = cdiv(len, tile_tok) - 1 - (e - sm.app_off[lo]);  // a row's last (longest) tile first
      AppendItem a;
      a.row = r;
      a.token_begin = sm.Q0[r] + k * tile_tok;
      a.n_tok = min(tile_tok, len - k * tile_tok);
      a.seq_len = s;
      a.pos_begin = s - len + k * tile_tok;
      a.key_begin = p.window > 0 ? max(0, a.pos_begin - p.window + 1) : 0;
      a.key_end = a.pos_begin + a.n_tok;
      a.pad = 0;
      aitems[e] = a;
    }
  }
  if (tid == 0) {
    hdr->split_pages = C;
    publish(tot_items, tot_cascade, tot_tiles, n_merge, tot_parts);
  }
}

cudaError_t launch_plan(const AttnParams& p, cudaStream_t stream, bool programmatic) {
  static_assert(sizeof(PlanSmem) < 200 * 1024, "planner shared memory");
  const bool scan = p.cascade_enabled && p.window <= 0 && p.num_seqs > kScanInPlanner;
  if (scan) {
    lcp_kernel<<<(p.num_seqs + kLcpWarps - 1) / kLcpWarps, kLcpWarps * 32, 0, stream>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // After the prefix scan (and only then: an earlier grid of the caller's
  // may write what phase 1 reads) the planner may be launched
  // programmatically, so that its launch and first phase overlap the scan.
  // One row per thread up to 1024 rows; fewer threads for small batches:
  // every phase ends in a CTA barrier, and barriers over 8 warps are cheaper
  // than over 32.
  const int B = p.num_seqs;
  LaunchCfg lc(dim3(1), dim3(B <= 256 ? 256 : B <= 512 ? 512 : 1024), sizeof(PlanSmem), stream, programmatic && scan);
  if (B <= 256) return cudaLaunchKernelEx(&lc.cfg, plan_kernel<256, 1>, p);
  if (B <= 512) return cudaLaunchKernelEx(&lc.cfg, plan_kernel<512, 1>, p);
  if (B <= 1024) return cudaLaunchKernelEx(&lc.cfg, plan_kernel<1024, 1>, p);
  return cudaLaunchKernelEx(&lc.cfg, plan_kernel<1024, 2>, p);
}

cudaError_t prepare_plan_kernel() {
  // every kernel of the library asks for the largest shared-memory carveout,
  // so an SM never has to be reconfigured between them and a decode CTA can
  // share an SM with an append CTA
  for (auto fn : {plan_kernel<256, 1>, plan_kernel<512, 1>, plan_kernel<1024, 1>, plan_kernel<1024, 2>}) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PlanSmem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mcpu
