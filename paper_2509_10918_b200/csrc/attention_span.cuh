// What the two tensor-core attention kernels (attention_two_tc.cu, attention_tc.cu) share: the work units and how they
// are cut into spans, the scratch of partial pieces and how the pieces of a row are added up.
//
// Work unit = (batch, head, 256 queries) = two 128-row query tiles that share every K/V tile; one iteration = one 64-key
// tile of a unit.  A launch is persistent, one CTA per SM, and the units' iterations, laid end to end, are cut into one
// contiguous span per CTA.  A span that covers only part of a unit's keys leaves the unnormalised accumulator, the
// reference and the row sum of its piece in global scratch; the warp that arrives last at the (unit, warp) ticket adds the
// pieces up and writes the output rows.  Nobody waits for another CTA.
#pragma once

#include "attention_core.cuh"
#include "common.cuh"
#include "tc.cuh"

namespace toma {
namespace attn {

constexpr int kUM = 2 * kBM;     // queries per work unit
constexpr int kMaxCtas = 160;    // scratch and the span table are sized for this many persistent CTAs (ids fit a byte)
constexpr int kTicketCols = 16;  // tickets per unit: one per softmax warp of the larger kernel

// The iterations [0, T) are cut into G contiguous spans, CTA g running [bounds[g], bounds[g + 1]).
// With whole units every bound is a multiple of nblk (no scratch traffic), which wins when the unit
// count happens to fill the CTAs evenly; otherwise the spans are cut at single key tiles so that the
// longest span is as short as possible when every piece is charged its pipeline drain and epilogue
// (plan_spans): a piece of one or two tiles costs its CTA more than the tiles it moves are worth.
struct Spans {
  int T, G, nblk, split;
  int longest;  // iterations of the longest span
  int bounds[kMaxCtas + 1];
  // Lowest and highest CTA among those whose spans hold key tiles of the unit CTA g's span starts in ([0][g])
  // and of the unit it ends in ([1][g]): the only units a CTA can share.  Filled in by the host, so that the
  // kernel does not search the bounds at the end of a piece.
  uint8_t unit_lo[2][kMaxCtas], unit_hi[2][kMaxCtas];
  __host__ __device__ int bound(int g) const { return bounds[g]; }
  // the CTA whose span holds iteration `it`
  __host__ __device__ int owner(int it) const {
    int lo = 0, hi = G - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (bounds[mid] <= it) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  }
};

// What the ends of a CTA's span need of the plan, in shared memory: at the end of a piece the parameter memory is cold, and
// its reads, one behind the other, cost a microsecond.  Filled in by lanes 0 and 1 of a warp at the start.
struct Edges {
  int lo[2], hi[2];  // lowest and highest CTA with key tiles of the unit the span starts in, and of the one it ends in
  int first_unit;    // the unit the span starts in
  int other_slot;    // scratch slot of the last unit's other contributor, where it has one
  __device__ __forceinline__ void fill(const Spans& sp, int it_begin, int it_end, int lane) {
    const int u = (lane ? it_end - 1 : it_begin) / sp.nblk;
    lo[lane] = sp.unit_lo[lane][blockIdx.x];
    hi[lane] = sp.unit_hi[lane][blockIdx.x];
    if (lane == 0) {
      first_unit = u;
    } else {  // a CTA's first piece sits in slot 0 of its two, a later partial piece in slot 1
      const int g = lo[1] == (int)blockIdx.x ? hi[1] : lo[1];
      other_slot = 2 * g + (u > sp.bound(g) / sp.nblk ? 1 : 0);
    }
  }
};

// One piece = the part of a span inside one unit: key tiles [k0, k0 + cnt) of unit u.
struct Piece {
  int u, k0, cnt;
};
__device__ __forceinline__ Piece piece_at(int it, int it_end, int nblk) {
  Piece p;
  p.u = it / nblk;
  p.k0 = it - p.u * nblk;
  const int left = it_end - it;
  p.cnt = left < nblk - p.k0 ? left : nblk - p.k0;
  return p;
}

// A position in the CTA's span for the single-thread roles: `n` counts key tiles across pieces (ring
// slots, S buffers and their barrier phases follow n), `pc` counts pieces (phases of the per-piece
// barriers), `j` is the tile inside the current piece of `cnt` tiles.
struct Cursor {
  int it, it_end, nblk, j, cnt, pc, n;
  __device__ __forceinline__ void load() {
    const int left = it_end - it, in_unit = nblk - it % nblk;
    cnt = left < in_unit ? left : in_unit;
  }
  __device__ __forceinline__ void init(int b, int e, int nb) {
    it = b, it_end = e, nblk = nb, j = 0, pc = 0, n = 0;
    load();
  }
  __device__ __forceinline__ bool valid() const { return it < it_end; }
  __device__ __forceinline__ bool last_of_piece() const { return j + 1 == cnt; }
  __device__ __forceinline__ void next() {
    ++n;
    if (++j == cnt) {
      it += cnt, ++pc, j = 0;
      load();
    }
  }
};

// Scratch of one piece: O as [DH / 4][256 rows] float4, then m[256], l[256].
template <int DH>
__host__ __device__ constexpr size_t piece_floats() { return (size_t)kUM * DH + 2 * kUM; }

// Where the output rows of unit u start for query row `row` (0..255) of the unit (nullptr past the sequence end).
template <int DH>
__device__ __forceinline__ __nv_bfloat16* out_row(__nv_bfloat16* o, int u, int row, int L, int heads) {
  const int nq = (L + kUM - 1) / kUM;
  const int bh = u / nq, qi = (u - bh * nq) * kUM + row, b = bh / heads, h = bh - b * heads;
  if (qi >= L) return nullptr;
  return o + ((size_t)b * L + qi) * ((size_t)heads * DH) + (size_t)h * DH;
}

// Scratch slot of the piece of unit u that CTA g left: its first piece sits in slot 0, a later
// partial piece (necessarily its last) in slot 1.
template <int DH>
__device__ __forceinline__ const float* slot_of(const float* pieces, const Spans& sp, int g, int u) {
  const int first_unit = sp.bound(g) / sp.nblk;
  return pieces + (size_t)(2 * g + (u > first_unit ? 1 : 0)) * piece_floats<DH>();
}

// Adds up the pieces of one query row of unit u (channels [ch, ch + kCh) of the head), left by CTAs g_first..g_last:
//   O = sum_i 2^(m_i - M) O_i / sum_i 2^(m_i - M) l_i,  M = max_i m_i  (m in the log2 domain).
// Contributors are taken two at a time so that their loads are in flight together, and summed in
// ascending CTA order with one fused multiply-add each, starting from zero: finish_partial's direct
// path follows the same order, so the result does not depend on which path a launch takes.  Loads bypass L1: the pieces
// were written by other SMs during this launch.  kStep: accumulator columns at a time, kQuads: float4 loads in flight per
// contributor.
template <int DH, int kCh, int kStep, int kQuads>
__device__ __noinline__ void combine_rows(const float* pieces, const Spans& sp, int u, int g_first, int g_last, int row, int ch,
                                          __nv_bfloat16* dst) {
  constexpr size_t kM = (size_t)kUM * DH, kL = (size_t)kUM * DH + kUM;
  float M = -INFINITY;
  for (int g = g_first; g <= g_last; g += 2) {
    const float* sa = slot_of<DH>(pieces, sp, g, u);
    const float* sb = g < g_last ? slot_of<DH>(pieces, sp, g + 1, u) : sa;
    M = max3(M, __ldcg(sa + kM + row), __ldcg(sb + kM + row));
  }
#pragma unroll 1
  for (int c0 = ch; c0 < ch + kCh; c0 += kStep) {
    float denom = 0.f;
    float acc[kStep];
#pragma unroll
    for (int e = 0; e < kStep; ++e) acc[e] = 0.f;
    for (int g = g_first; g <= g_last; g += 2) {
      const float* sa = slot_of<DH>(pieces, sp, g, u);
      const float* sb = g < g_last ? slot_of<DH>(pieces, sp, g + 1, u) : sa;
      const float ma = __ldcg(sa + kM + row), la = __ldcg(sa + kL + row);
      const float mb = __ldcg(sb + kM + row), lb = __ldcg(sb + kL + row);
      const float wa = ex2_mufu(ma - M), wb = g < g_last ? ex2_mufu(mb - M) : 0.f;
      denom = fmaf(wb, lb, fmaf(wa, la, denom));
      const float4* pa = reinterpret_cast<const float4*>(sa) + (size_t)(c0 >> 2) * kUM + row;  // the loads below at constant offsets
      const float4* pb = reinterpret_cast<const float4*>(sb) + (size_t)(c0 >> 2) * kUM + row;
#pragma unroll
      for (int s = 0; s < kStep; s += 4 * kQuads) {
        float4 va[kQuads], vb[kQuads];
#pragma unroll
        for (int q = 0; q < kQuads; ++q) {
          va[q] = __ldcg(pa + (size_t)(s / 4 + q) * kUM);
          vb[q] = __ldcg(pb + (size_t)(s / 4 + q) * kUM);
        }
#pragma unroll
        for (int q = 0; q < kQuads; ++q) {
          float* a4 = &acc[s + 4 * q];
          a4[0] = fmaf(wb, vb[q].x, fmaf(wa, va[q].x, a4[0]));
          a4[1] = fmaf(wb, vb[q].y, fmaf(wa, va[q].y, a4[1]));
          a4[2] = fmaf(wb, vb[q].z, fmaf(wa, va[q].z, a4[2]));
          a4[3] = fmaf(wb, vb[q].w, fmaf(wa, va[q].w, a4[3]));
        }
      }
    }
    if (!dst) continue;
    const float inv = 1.f / denom;
#pragma unroll
    for (int e = 0; e < kStep; e += 8)
      *reinterpret_cast<uint4*>(dst + c0 + e) =
          make_uint4(pack_bf16_rn(acc[e] * inv, acc[e + 1] * inv), pack_bf16_rn(acc[e + 2] * inv, acc[e + 3] * inv),
                     pack_bf16_rn(acc[e + 4] * inv, acc[e + 5] * inv), pack_bf16_rn(acc[e + 6] * inv, acc[e + 7] * inv));
  }
}

// Whether each of the kN tickets (a multiple of four, 16-byte aligned) has been drawn once; if so, what their drawers had
// written before is visible from here on.  (One fence behind all the loads: loads that acquire each wait for the one before,
// 10 us for sixteen.)
template <int kN>
__device__ __forceinline__ bool all_drawn_once(const uint32_t* tk) {
  uint32_t off = 0;
#pragma unroll
  for (int w = 0; w < kN; w += 4) {
    uint32_t v[4];
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "l"(tk + w) : "memory");
    off |= (v[0] ^ 1u) | (v[1] ^ 1u) | (v[2] ^ 1u) | (v[3] ^ 1u);
  }
  if (off) return false;
  __threadfence();
  return true;
}

__device__ __forceinline__ void st_release_cta(uint32_t* smem_word, uint32_t v) {
  asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(smem_word)), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire_cta(const uint32_t* smem_word) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(smem_word)) : "memory");
  return v;
}

// Publishes this warp's 32 rows of a piece and takes the (unit, warp) ticket.  Returns the number
// of contributors that had taken it before.  Called by whole warps only.
__device__ __forceinline__ uint32_t take_ticket(uint32_t* ticket, int lane) {
  __threadfence();
  __syncwarp();
  uint32_t t = 0;
  if (lane == 0) t = atomicAdd(ticket, 1u);
  return __shfl_sync(0xffffffffu, t, 0);
}

// Batch item, first channel and first token of the 32 rows of unit u that start at row `row0_in` of it.
template <int DH>
__device__ __forceinline__ void warp_rows_of(int u, int row0_in, int L, int heads, int& b, int& ch0, int& row0) {
  const int nq = (L + kUM - 1) / kUM;
  const int bh = u / nq;
  b = bh / heads;
  ch0 = (bh - b * heads) * DH;
  row0 = (u - bh * nq) * kUM + row0_in;
}

inline size_t ticket_bytes(int B, int L, int heads) {
  const size_t units = (size_t)B * heads * ((L + kUM - 1) / kUM);
  return (units * kTicketCols * sizeof(uint32_t) + 255) & ~(size_t)255;
}

// The two-group kernel (head_dim 64 or 128) on a plan; ws: tickets, zero where units are split, then the pieces.
cudaError_t launch_attention_two(int B, int L, int heads, int dh, const void* q, const void* k, const void* v, void* o, void* ws, const Spans& sp,
                                 uint32_t* dev_status, cudaStream_t s);

}  // namespace attn
}  // namespace toma
