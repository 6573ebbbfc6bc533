// Fused rotary embedding + KV append, and device-side growth of block tables.
//
// rope_append_kernel: for every query token t of row r at position
// p = S_r - L_r + i, rotates q[t] (all q heads, in place) and k_new[t] (all
// kv heads) by the angles of table row p, then writes the rotated k and the
// unrotated v into the row's page, as the plain KV append does. The rotation
// pairs dimension i with i + D/2 (half split):
//   y_i = x_i cos_i(p) - x_{i+D/2} sin_i(p),  y_{i+D/2} = x_{i+D/2} cos_i(p) + x_i sin_i(p)
// in fp32, rounded once to bf16. One warp per token, bound by HBM (q read and
// written: 16 KiB per token at 64 heads). A row of 64 dims is eight 16-byte
// vectors; a group of four lanes owns a row, lane c of it vectors c and c + 4
// (dims 8c .. 8c + 7 and the same + 32), so a warp moves eight rows at a time
// with 16-byte loads and stores, and a lane's 8 cosines and 8 sines stay in
// registers for all rows of its token. Measured at 35681 tokens, 64 / 8 heads
// (740 MB moved): 219 -> 102 us, 7.2 TB/s, against a CTA per token whose warps
// moved two bytes per lane.
//
// grow_tables_kernel: every logical page a row needs for its S_r tokens and
// whose block-table entry is negative gets a page popped from a device stack
// of free page ids; entries already set (shared prompt pages, earlier pages)
// are left alone. An empty stack sets kStatusPoolExhausted.
#include "common.cuh"

namespace mcpu {

constexpr int kRopeWarps = 8;

struct RopeParams {
  __nv_bfloat16* q;
  const __nv_bfloat16* k_new;
  const __nv_bfloat16* v_new;
  __nv_bfloat16* k_cache;
  __nv_bfloat16* v_cache;
  const int32_t* block_table;
  const int32_t* seq_lens;
  const int32_t* qsl;
  const float* cos_sin;  // [max_position, 64]: cos then sin
  int32_t* status;
  int32_t num_seqs, total_q, max_pages, num_pages, num_q_heads, num_kv_heads, max_position;
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Rotates 8 dims (x: dims i, y: dims i + 32) by the angles of cos c, sin s. One
// product of each sum is rounded to fp32, the other fused: which one is spelled
// out, so that no compilation changes the last bit.
__device__ __forceinline__ float rotate_lo(float a, float b, float c, float s) { return fmaf(a, c, -__fmul_rn(b, s)); }
__device__ __forceinline__ float rotate_hi(float a, float b, float c, float s) { return fmaf(a, s, __fmul_rn(b, c)); }
__device__ __forceinline__ void rotate8(uint4& x, uint4& y, const float (&c)[8], const float (&s)[8]) {
  uint32_t* xw = reinterpret_cast<uint32_t*>(&x);
  uint32_t* yw = reinterpret_cast<uint32_t*>(&y);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a0 = bf16_lo(xw[i]), a1 = bf16_hi(xw[i]), b0 = bf16_lo(yw[i]), b1 = bf16_hi(yw[i]);
    const float c0 = c[2 * i], c1 = c[2 * i + 1], s0 = s[2 * i], s1 = s[2 * i + 1];
    xw[i] = pack_bf16x2(rotate_lo(a0, b0, c0, s0), rotate_lo(a1, b1, c1, s1));
    yw[i] = pack_bf16x2(rotate_hi(a0, b0, c0, s0), rotate_hi(a1, b1, c1, s1));
  }
}

__global__ void __launch_bounds__(kRopeWarps * 32) rope_append_kernel(const RopeParams p) {
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * kRopeWarps + (threadIdx.x >> 5);
  if (t >= p.total_q) return;
  int pos;
  const int dst = append_slot_warp(p.qsl, p.seq_lens, p.block_table, p.num_seqs, p.total_q, p.max_pages, p.num_pages,
                                   p.status, p.max_position, t, &pos);
  if (pos < 0) return;
  const int sub = lane >> 2, col = lane & 3;  // row within the eight, vector within the row
  float c[8], s[8];
  const float* cs = p.cos_sin + (size_t)pos * kHeadDim + 8 * col;
  if ((reinterpret_cast<uintptr_t>(p.cos_sin) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < 8; i += 4) {
      const float4 cv = __ldg(reinterpret_cast<const float4*>(cs + i));
      const float4 sv = __ldg(reinterpret_cast<const float4*>(cs + 32 + i));
      c[i] = cv.x, c[i + 1] = cv.y, c[i + 2] = cv.z, c[i + 3] = cv.w;
      s[i] = sv.x, s[i + 1] = sv.y, s[i + 2] = sv.z, s[i + 3] = sv.w;
    }
  } else {  // the table need only be 4-byte aligned
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = __ldg(cs + i), s[i] = __ldg(cs + 32 + i);
  }
  const int Hq = p.num_q_heads, Hkv = p.num_kv_heads;
  // q rows, rotated in place; four steps of eight rows in flight
  uint4* q = reinterpret_cast<uint4*>(p.q + (size_t)t * Hq * kHeadDim) + col;
  constexpr int kSteps = 4;
  for (int r0 = 0; r0 < Hq; r0 += 8 * kSteps) {
    uint4 x[kSteps], y[kSteps];
#pragma unroll
    for (int u = 0; u < kSteps; ++u) {
      const int r = r0 + 8 * u + sub;
      if (r < Hq) x[u] = q[r * 8], y[u] = q[r * 8 + 4];
    }
#pragma unroll
    for (int u = 0; u < kSteps; ++u) {
      const int r = r0 + 8 * u + sub;
      if (r < Hq) {
        rotate8(x[u], y[u], c, s);
        q[r * 8] = x[u], q[r * 8 + 4] = y[u];
      }
    }
  }
  if (dst < 0) return;
  // k rotated and v as is, into the token's slot of its page
  const size_t block = (size_t)(dst / kPage) * Hkv;
  for (int h = sub; h < Hkv; h += 8) {
    const size_t src = ((size_t)t * Hkv + h) * 8 + col, at = ((block + h) * kPage + dst % kPage) * 8 + col;
    const uint4* kn = reinterpret_cast<const uint4*>(p.k_new) + src;
    const uint4* vn = reinterpret_cast<const uint4*>(p.v_new) + src;
    uint4 x = __ldg(kn), y = __ldg(kn + 4);
    const uint4 v0 = __ldg(vn), v1 = __ldg(vn + 4);
    rotate8(x, y, c, s);
    uint4* ko = reinterpret_cast<uint4*>(p.k_cache) + at;
    uint4* vo = reinterpret_cast<uint4*>(p.v_cache) + at;
    ko[0] = x, ko[4] = y;
    vo[0] = v0, vo[4] = v1;
  }
}

cudaError_t launch_rope_append(void* q, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                               const int32_t* block_table, const int32_t* seq_lens, const int32_t* qsl,
                               const float* cos_sin, int32_t max_position, int32_t* status, int32_t num_seqs,
                               int32_t total_q, int32_t max_pages, int32_t num_pages, int32_t num_q_heads,
                               int32_t num_kv_heads, cudaStream_t stream) {
  RopeParams p;
  p.q = static_cast<__nv_bfloat16*>(q);
  p.k_new = static_cast<const __nv_bfloat16*>(k_new);
  p.v_new = static_cast<const __nv_bfloat16*>(v_new);
  p.k_cache = static_cast<__nv_bfloat16*>(k_cache);
  p.v_cache = static_cast<__nv_bfloat16*>(v_cache);
  p.block_table = block_table;
  p.seq_lens = seq_lens;
  p.qsl = qsl;
  p.cos_sin = cos_sin;
  p.status = status;
  p.num_seqs = num_seqs;
  p.total_q = total_q;
  p.max_pages = max_pages;
  p.num_pages = num_pages;
  p.num_q_heads = num_q_heads;
  p.num_kv_heads = num_kv_heads;
  p.max_position = max_position;
  rope_append_kernel<<<(total_q + kRopeWarps - 1) / kRopeWarps, kRopeWarps * 32, 0, stream>>>(p);
  return cudaGetLastError();
}

// one warp per row: lanes take the row's logical pages 32 at a time
__global__ void __launch_bounds__(256) grow_tables_kernel(int32_t* block_table, const int32_t* seq_lens,
                                                          int32_t num_seqs, int32_t max_pages,
                                                          const int32_t* free_pages, int32_t* free_count,
                                                          int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= num_seqs) return;
  const int S = seq_lens[r];
  if (S < 0 || S > max_pages * kPage) {
    if (lane == 0) atomicOr(status, kStatusBadLengths);
    return;
  }
  const int need = (S + kPage - 1) / kPage;
  int32_t* row = block_table + (size_t)r * max_pages;
  for (int j = lane; j < need; j += 32) {
    if (row[j] >= 0) continue;
    const int top = atomicSub(free_count, 1);
    if (top <= 0) {
      atomicAdd(free_count, 1);  // give the slot back: the stack is empty
      atomicOr(status, kStatusPoolExhausted);
    } else {
      row[j] = free_pages[top - 1];
    }
  }
}

cudaError_t launch_grow_tables(int32_t* block_table, const int32_t* seq_lens, int32_t num_seqs, int32_t max_pages,
                               const int32_t* free_pages, int32_t* free_count, int32_t* status,
                               cudaStream_t stream) {
  const int warps_per_cta = 8;
  const int grid = (num_seqs + warps_per_cta - 1) / warps_per_cta;
  grow_tables_kernel<<<grid, warps_per_cta * 32, 0, stream>>>(block_table, seq_lens, num_seqs, max_pages,
                                                               free_pages, free_count, status);
  return cudaGetLastError();
}

}  // namespace mcpu
