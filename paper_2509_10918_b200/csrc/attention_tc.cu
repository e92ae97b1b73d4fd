// Attention core softmax(Q K^T / sqrt(dh)) V (Eq. 1 with tau = 1) on the sm_100a tensor
// cores, bf16 in / bf16 out, fp32 softmax and accumulation.
//
// Work unit = (batch, head, 256 queries) = two 128-row query tiles that share every K/V tile; one
// iteration = one 64-key tile of a unit.  The launch is persistent, one CTA per SM, and the units'
// iterations, laid end to end, are cut into one contiguous span per CTA, so that every CTA runs the
// same number of key tiles whatever the unit count.  A span that covers only part of a unit's keys
// leaves the unnormalised accumulator, the reference maximum and the row sum of its piece in global
// scratch; the warp that arrives last at the (unit, warp) ticket adds the pieces up and writes the
// output rows.  Nobody waits for another CTA.
//
// Inside a CTA (20 warps): warps 0..15 run the softmax as four pipelines of four warps, one per query tile q and parity h
// of the key tile (one thread per query row, straight out of tensor memory; so two threads share a row, each with every
// second key tile), warp 16 feeds Q, K and V through TMA rings, one elected thread of warp 17 issues the tcgen05 MMAs (at
// head_dim 128 those of query tile 0, and one of warp 19 those of query tile 1), warp 18 publishes a partial first piece
// (memory fence and tickets, off everybody else's path).
//   S_q,j = Q_q K_j^T      -> tensor memory, 64 columns per pipeline.  MMAs issued by one thread execute in order, so
//                             S_q,j+2 is issued right behind the product that reads P_q,j out of the same columns,
//                             without a round trip through a barrier.
//   P_q,j = 2^(S*c - m)    -> written back over S_q,j's first 32 columns as bf16 and used as the A operand (from tensor
//                             memory) of  O += P_q,j V_j
//   O                      -> at head_dim 64 every pipeline has an accumulator and a reference m of its own (four of 64
//                             columns beside four of S fill the tensor memory), added up at the end of a piece; at
//                             head_dim 128 the two pipelines of a query tile share one, and with it the reference
//   reference              -> set 2^32 above the piece's first scores and moved only when scores outgrow it (see
//                             chunk_exp_ref), so no row maximum stands before the exponentials
//   exponentials           -> one pair of columns in four goes through a degree-3 polynomial on the FMA pipe (relative
//                             error 7.5e-5, far below bf16 resolution of P), the rest through MUFU ex2; the scaling
//                             S*c - m and the polynomial run in packed f32x2 arithmetic
// What bounds it is the softmax (per 64 keys and row about 450 issue slots of a warp; the tensor pipe is busy 35 to 60 % of
// the time): with one pipeline per query tile a scheduler had two softmax warps, which left it idle whenever both waited
// for tensor memory or each other's dependencies.  Four pipelines: 960 -> 754 us at 4 x 8192 tokens and 10 heads of 64,
// 49.5 -> 41.6 us at 2 x 2048, 142 -> 136.5 us at 4 x 2048 tokens and 17 heads of 128.
// Keys past the sequence end are zero-filled by TMA and masked out; query rows past the end are
// computed on zeros and not written.
#include <mutex>

#include "attention_core.cuh"
#include "common.cuh"
#include "tc.cuh"

namespace toma {

using namespace tc;
using namespace attn;

namespace {

constexpr int kUM = 2 * kBM;  // queries per work unit
constexpr int kSoftWarps = 16;
constexpr int kThreads = (kSoftWarps + 4) * 32;

template <int DH>
struct AttCfg {
  static constexpr int kStages = DH == 64 ? 8 : 4;         // K/V ring depth (S runs two tiles ahead of P V)
  static constexpr int kQBufs = DH == 64 ? 2 : 1;          // Q buffers: the next unit's Q lands under this unit's tail
  static constexpr int kChunks = DH / 64;                  // 64-column (128-byte) slabs per row
  static constexpr int kQSlab = kBM * 128;                 // 128 query rows x 128 B
  static constexpr int kQTile = kChunks * kQSlab;          // one query tile
  static constexpr int kQBytes = 2 * kQTile;               // both query tiles of a unit
  static constexpr int kKvSlab = kBN * 128;                // 64 key rows x 128 B
  static constexpr int kKvBytes = kChunks * kKvSlab;       // one K or V tile
  static constexpr int kOutBytes = kSoftWarps * 32 * 64;   // per softmax warp: 32 output rows of 32 channels, staged for a TMA store
  static constexpr int kBarBytes = 512;
  static constexpr int kSmemBytes = 1024 + kQBufs * kQBytes + 2 * kStages * kKvBytes + kOutBytes + kBarBytes;
  static constexpr int kTmemCols = 512;
  // Threads that issue MMAs.  At head_dim 128 a tile is 12 MMAs and one thread for both query tiles keeps the tensor pipe
  // waiting; at head_dim 64 the softmax bounds and a second thread takes issue slots from it (752 -> 799 us at 4 x 8192
  // tokens, 10 heads).
  static constexpr int kIssuers = DH == 128 ? 2 : 1;
  // Tensor memory: a pipeline (query tile q, parity h) has 64 columns of S (P takes the first 32) and, at head_dim 64, an
  // accumulator of its own; at head_dim 128 the two pipelines of a query tile share one.
  static constexpr bool kOwnO = DH == 64;
  __device__ static constexpr uint32_t s_col(int q, int h) { return kOwnO ? (q * 2 + h) * 128 : q * 256 + h * 64; }
  __device__ static constexpr uint32_t o_col(int q, int h) { return kOwnO ? (q * 2 + h) * 128 + 64 : q * 256 + 128; }
};

struct Barriers {
  uint64_t q_full[2], q_empty[2];       // per piece: Q landed / every S MMA of the piece has read Q
  uint64_t k_full[8], kv_empty[8];      // per tile: K and V landed / every MMA that reads them is done
  uint64_t s_full[2][2], p_full[2][2];  // per tile and pipeline: S ready for the softmax / P ready for the PV MMAs
  uint64_t pv_done[2][2];               // the tile's PV MMAs are complete
  uint64_t o_free[2];                   // per piece and query tile: the epilogue has read the accumulators
  uint64_t pub_ready, pub_done;         // first partial piece: written by the softmax warps / published, tickets drawn
  uint32_t first_ticket[kSoftWarps];    // per softmax warp: ticket its first (partial) piece drew
  uint32_t move[8];                     // shared accumulator: a warp of this row group wants the reference moved
  uint32_t others_done;                 // set by the publisher when the span's last unit has all its other pieces in scratch
  uint32_t poll_stop[2];                // set by each softmax group when the answer is no longer needed
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(Barriers) <= 512, "barrier block outgrew its reservation");

constexpr int kSnapTiles = 2;
constexpr int kMaxCtas = 160;  // scratch and the span table are sized for this many persistent CTAs (ids fit a byte)

// The iterations [0, T) are cut into G contiguous spans, CTA g running [bounds[g], bounds[g + 1]).
// With whole units every bound is a multiple of nblk (no scratch traffic), which wins when the unit
// count happens to fill the CTAs evenly; otherwise the spans are cut at single key tiles so that the
// longest span is as short as possible when every piece is charged its pipeline drain and epilogue
// (plan_spans): a piece of one or two tiles costs its CTA more than the tiles it moves are worth.
struct Spans {
  int T, G, nblk, split;
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

// Adds up the pieces of one query row of unit u (channels [ch, ch + DH / 2) of the head), left by CTAs g_first..g_last:
//   O = sum_i 2^(m_i - M) O_i / sum_i 2^(m_i - M) l_i,  M = max_i m_i  (m in the log2 domain).
// Contributors are taken two at a time so that their loads are in flight together, and summed in
// ascending CTA order with one fused multiply-add each, starting from zero: finish_partial's direct
// path follows the same order, so the result does not depend on which path a launch takes.  Loads bypass L1: the pieces
// were written by other SMs during this launch.
template <int DH>
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
  for (int c0 = ch; c0 < ch + DH / 2; c0 += 16) {  // 16 accumulator columns at a time
    float denom = 0.f;
    float acc[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = 0.f;
    for (int g = g_first; g <= g_last; g += 2) {
      const float* sa = slot_of<DH>(pieces, sp, g, u);
      const float* sb = g < g_last ? slot_of<DH>(pieces, sp, g + 1, u) : sa;
      const float ma = __ldcg(sa + kM + row), la = __ldcg(sa + kL + row);
      const float mb = __ldcg(sb + kM + row), lb = __ldcg(sb + kL + row);
      const float wa = ex2_mufu(ma - M), wb = g < g_last ? ex2_mufu(mb - M) : 0.f;
      denom = fmaf(wb, lb, fmaf(wa, la, denom));
      float4 va[4], vb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        va[q] = __ldcg(reinterpret_cast<const float4*>(sa) + (size_t)(c0 / 4 + q) * kUM + row);
        vb[q] = __ldcg(reinterpret_cast<const float4*>(sb) + (size_t)(c0 / 4 + q) * kUM + row);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float* a4 = &acc[4 * q];
        a4[0] = fmaf(wb, vb[q].x, fmaf(wa, va[q].x, a4[0]));
        a4[1] = fmaf(wb, vb[q].y, fmaf(wa, va[q].y, a4[1]));
        a4[2] = fmaf(wb, vb[q].z, fmaf(wa, va[q].z, a4[2]));
        a4[3] = fmaf(wb, vb[q].w, fmaf(wa, va[q].w, a4[3]));
      }
    }
    if (!dst) continue;
    const float inv = 1.f / denom;
#pragma unroll
    for (int e = 0; e < 16; e += 8)
      *reinterpret_cast<uint4*>(dst + c0 + e) =
          make_uint4(pack_bf16_rn(acc[e] * inv, acc[e + 1] * inv), pack_bf16_rn(acc[e + 2] * inv, acc[e + 3] * inv),
                     pack_bf16_rn(acc[e + 4] * inv, acc[e + 5] * inv), pack_bf16_rn(acc[e + 6] * inv, acc[e + 7] * inv));
  }
}

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
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

// The per-thread view of a softmax thread.  Two threads share a query row, both on its tensor-memory lane: each has every
// second key tile (its pipeline, `half`) and, at the end of a piece, half of the head's channels.
struct Row {
  int q;        // query tile 0 or 1
  int half;
  int warp;     // softmax warp 0..15 = ticket column
  int lane;
  int row;      // query row inside the unit, 0..255
  uint32_t tm;  // this row's tensor-memory lane
};
// Both warps of a row group meet at a barrier of their own.
__device__ __forceinline__ int pair_of(const Row& t) { return t.q * 4 + (t.warp & 3); }
__device__ __forceinline__ void pair_sync(const Row& t) {
  __syncwarp();
  asm volatile("bar.sync %0, 64;" ::"r"(1 + pair_of(t)) : "memory");
}
// Where a softmax warp stages its output rows, and the map they are stored through: kept out of Row (the softmax
// loop holds a Row in registers) and derived where a piece ends.
struct OutStage {
  uint8_t* stage;           // this warp's 2 KB of the output staging area (it lies right below the barriers)
  const CUtensorMap* tm_o;  // output as (channel, token, batch), box = 32 channels x 32 tokens
};
template <int DH>
__device__ __forceinline__ uint8_t* stage_of(const void* bar, int warp) {
  return const_cast<uint8_t*>(reinterpret_cast<const uint8_t*>(bar)) - AttCfg<DH>::kOutBytes + warp * 2048;
}
// Two words of this thread's for the other thread of the row, through the (then idle) staging areas.
template <int DH>
__device__ __forceinline__ uint2 exchange(const Row& t, const void* bar, uint32_t a, uint32_t b) {
  volatile uint32_t* mine = reinterpret_cast<volatile uint32_t*>(stage_of<DH>(bar, t.warp)) + t.lane;
  const volatile uint32_t* other = reinterpret_cast<volatile uint32_t*>(stage_of<DH>(bar, t.warp ^ 4)) + t.lane;
  mine[0] = a;
  mine[32] = b;
  pair_sync(t);
  const uint2 o = make_uint2(other[0], other[32]);
  pair_sync(t);  // read: the areas may be written again
  return o;
}
// A row at the end of a piece: reference and row sum of both pipelines together, and what their accumulators count in it
// (own accumulators only; 0: nothing, not even if it is no number).
struct Joint {
  float m, l, w0, w1;
};
template <int DH>
__device__ __forceinline__ Joint join_halves(const Row& t, const void* bar, float m, float l) {
  const uint2 o = exchange<DH>(t, bar, __float_as_uint(m), __float_as_uint(l));
  const float mo = __uint_as_float(o.x), lo = __uint_as_float(o.y);
  Joint r;
  r.m = fmaxf(m, mo);
  const float own = ex2_mufu(m - r.m), oth = ex2_mufu(mo - r.m);  // a pipeline without a tile: 2^-inf = 0
  r.w0 = t.half ? oth : own;
  r.w1 = t.half ? own : oth;
  r.l = t.half ? fmaf(r.w1, l, r.w0 * lo) : fmaf(r.w1, lo, r.w0 * l);
  return r;
}
// 16 accumulator columns of the row, both pipelines' together.
template <int DH>
__device__ __forceinline__ void read_o16(const Row& t, const Joint& jn, int c, uint32_t (&r)[16]) {
  using C = AttCfg<DH>;
  tmem_ld16(t.tm + C::o_col(t.q, 0) + c, r);
  if constexpr (C::kOwnO) {
    uint32_t r1[16];
    tmem_ld16(t.tm + C::o_col(t.q, 1) + c, r1);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float a = jn.w0 != 0.f ? jn.w0 * __uint_as_float(r[e]) : 0.f;
      r[e] = __float_as_uint(jn.w1 != 0.f ? fmaf(jn.w1, __uint_as_float(r1[e]), a) : a);
    }
  } else {
    tmem_wait_ld();
  }
}
// The last products of both pipelines, in a piece of `cnt` tiles whose last is number `last_n` of the span.
__device__ __forceinline__ bool wait_o(const Row& t, Barriers* bar, int last_n, int cnt, uint32_t* dev_status) {
  bool ok = mbar_wait(&bar->pv_done[t.q][last_n & 1], (last_n >> 1) & 1, dev_status, &bar->abort_flag);
  if (cnt > 1) ok = ok && mbar_wait(&bar->pv_done[t.q][(last_n - 1) & 1], ((last_n - 1) >> 1) & 1, dev_status, &bar->abort_flag);
  return __all_sync(0xffffffffu, ok);
}

// Output rows leave through shared memory: a thread puts 16 channels of its row (scaled, bf16) into its warp's staged
// slab (32 channels x 32 rows, 64-byte swizzled = the output map's box), and when the slab is complete the
// warp stores it with one TMA store - whole sectors instead of 16-byte stores to 32 different rows per warp
// instruction.  Rows past the end of the sequence are clipped by the store.
__device__ __forceinline__ void stage16(const OutStage& os, int lane, int part, const uint32_t (&r)[16], float inv) {
#pragma unroll
  for (int e = 0; e < 16; e += 8) {
    uint4 v;
    v.x = pack_bf16_rn(__uint_as_float(r[e]) * inv, __uint_as_float(r[e + 1]) * inv);
    v.y = pack_bf16_rn(__uint_as_float(r[e + 2]) * inv, __uint_as_float(r[e + 3]) * inv);
    v.z = pack_bf16_rn(__uint_as_float(r[e + 4]) * inv, __uint_as_float(r[e + 5]) * inv);
    v.w = pack_bf16_rn(__uint_as_float(r[e + 6]) * inv, __uint_as_float(r[e + 7]) * inv);
    *reinterpret_cast<uint4*>(os.stage + lane * 64 + (((part * 2 + (e >> 3)) ^ ((lane >> 1) & 3)) << 4)) = v;
  }
}
// Whole warp.  (ch0, row0, b): first channel of the slab, first token of the warp's 32 rows, batch item.
__device__ __forceinline__ void flush_slab(const OutStage& os, int lane, int ch0, int row0, int b, int L) {
  fence_proxy_async();  // the staged rows are read by the TMA engine
  __syncwarp();
  if (lane == 0 && row0 < L) {
    tma_store_3d(os.tm_o, os.stage, ch0, row0, b);
    tma_store_commit();
    tma_store_wait_read();  // the slab is staged again right away
  }
  __syncwarp();
}
// Batch item, first channel and first token of the 32 rows that warp t.warp holds of unit u.
template <int DH>
__device__ __forceinline__ void warp_rows_of(int u, const Row& t, int L, int heads, int& b, int& ch0, int& row0) {
  const int nq = (L + kUM - 1) / kUM;
  const int bh = u / nq;
  b = bh / heads;
  ch0 = (bh - b * heads) * DH;
  row0 = (u - bh * nq) * kUM + (t.row & ~31);
}

// End of a piece that covers all keys of its unit (the only kind when units are kept whole), run by
// the softmax warps: wait for the accumulators, normalise, write the rows out.  Returns false when
// the wait ran out.
template <int DH>
__device__ __noinline__ bool finish_whole(Row t, Barriers* bar, Piece p, int last_n, Joint jn, const CUtensorMap* tm_o, int L, int heads,
                                          uint32_t* dev_status) {
  if (!wait_o(t, bar, last_n, p.cnt, dev_status)) return false;
  tc_fence_after();
  int b, ch0, row0;
  warp_rows_of<DH>(p.u, t, L, heads, b, ch0, row0);
  const OutStage os{stage_of<DH>(bar, t.warp), tm_o};
  const float inv = 1.f / jn.l;
  const int c0 = t.half * (DH / 2);
#pragma unroll 1
  for (int c = c0; c < c0 + DH / 2; c += 32) {
    uint32_t r[16];
    read_o16<DH>(t, jn, c, r);
    stage16(os, t.lane, 0, r, inv);
    read_o16<DH>(t, jn, c + 16, r);
    stage16(os, t.lane, 1, r, inv);
    if (c + 32 >= c0 + DH / 2) {
      tc_fence_before();
      __syncwarp();
      if (t.lane == 0) mbar_arrive(&bar->o_free[t.q]);  // the next piece's first PV product may overwrite the accumulator
    }
    flush_slab(os, t.lane, ch0 + c, row0, b, L);
  }
  return true;
}

// End of a piece that covers only part of its unit's keys, run by the softmax warps:
//   - the last piece of the CTA's span, when the unit's only other contributor has already
//     published (it ran at the start of its own span, so it normally has), is added to that
//     contributor's piece straight from tensor memory and written out: nothing of it goes through
//     scratch, and the other piece is fetched while the last MMAs drain;
//   - any other piece is left in scratch with its reference and row sum and a (unit, warp)
//     ticket is drawn; the warp that draws a unit's last ticket adds its pieces up.  A last piece
//     does that here; a first piece, with more of the span to come, hands the fence and the
//     tickets' round trips to the publisher thread and looks at the outcome in settle_first_piece.
// Every decision that ends in a warp-wide operation is taken once per warp (lane 0 reads, the warp
// gets the value by shuffle), so a warp always goes one way as a whole.  Both warps of a row write the row's reference
// and sum (the same values), so that each one's ticket covers what it needs.
// Out of line (it runs at most twice per CTA and is register-hungry).  Returns false when the wait
// ran out.
template <int DH>
__device__ __noinline__ bool finish_partial(Row t, Barriers* bar, Piece p, int pc, int last_n, bool last_of_span, Joint jn,
                                            __nv_bfloat16* o, const CUtensorMap* tm_o, int L, int heads, const Spans& sp,
                                            uint32_t* tickets, float* pieces, uint32_t* dev_status) {
  constexpr size_t kM = (size_t)kUM * DH, kL = (size_t)kUM * DH + kUM;
  const int row = t.row, lane = t.lane, c0 = t.half * (DH / 2);
  uint32_t* ticket = tickets + (size_t)p.u * kSoftWarps + t.warp;
  // a partial piece lies in the unit the span starts in or in the one it ends in
  const int which = p.u == sp.bound(blockIdx.x) / sp.nblk ? 0 : 1;
  const int g_first = sp.unit_lo[which][blockIdx.x], g_last = sp.unit_hi[which][blockIdx.x];
  bool own_first = false;  // this CTA is the lower of the two contributors
  const float4* other = nullptr;
  float m_o = 0.f, l_o = 0.f;
  float4 vo[4];  // 16 columns of the other piece, the next 16 on their way
  // the publisher warp watches the tickets of the span's last unit; its answer carries the
  // acquire that orders the loads below after the other contributor's writes
  uint32_t others = 0;
  if (last_of_span && g_last == g_first + 1) {
    if (lane == 0) others = ld_acquire_cta(&bar->others_done);
    __syncwarp();
    others = __shfl_sync(0xffffffffu, others, 0);
  }
  const bool direct = others == 1u;
  if (last_of_span && (row & (kBM - 1)) == 0 && t.half == 0) *(volatile uint32_t*)&bar->poll_stop[t.q] = 1u;
  if (direct) {
    own_first = (int)blockIdx.x == g_first;
    const float* slot = slot_of<DH>(pieces, sp, own_first ? g_last : g_first, p.u);
    m_o = __ldcg(slot + kM + row);
    l_o = __ldcg(slot + kL + row);
    other = reinterpret_cast<const float4*>(slot) + row;
#pragma unroll
    for (int q = 0; q < 4; ++q) vo[q] = __ldcg(other + (size_t)(c0 / 4 + q) * kUM);
  }
  if (!wait_o(t, bar, last_n, p.cnt, dev_status)) return false;
  tc_fence_after();
  int b_item, ch0, row0;
  warp_rows_of<DH>(p.u, t, L, heads, b_item, ch0, row0);
  float* slot = pieces + (size_t)(2 * blockIdx.x + (pc > 0 ? 1 : 0)) * piece_floats<DH>();
  if (direct) {
    const OutStage os{stage_of<DH>(bar, t.warp), tm_o};
    const float M = fmaxf(jn.m, m_o);
    const float w_own = ex2_mufu(jn.m - M), w_o = ex2_mufu(m_o - M);
    const float inv = 1.f / (own_first ? fmaf(w_o, l_o, w_own * jn.l) : fmaf(w_own, jn.l, w_o * l_o));
#pragma unroll 1
    for (int c = c0; c < c0 + DH / 2; c += 16) {
      float4 vc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) vc[q] = vo[q];
      if (c + 16 < c0 + DH / 2) {
#pragma unroll
        for (int q = 0; q < 4; ++q) vo[q] = __ldcg(other + (size_t)((c + 16) / 4 + q) * kUM);
      }
      uint32_t r[16];
      read_o16<DH>(t, jn, c, r);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float vv[4] = {vc[q].x, vc[q].y, vc[q].z, vc[q].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float own = __uint_as_float(r[4 * q + e]);
          r[4 * q + e] = __float_as_uint(own_first ? fmaf(w_o, vv[e], w_own * own) : fmaf(w_own, own, w_o * vv[e]));
        }
      }
      stage16(os, lane, (c >> 4) & 1, r, inv);
      if ((c >> 4) & 1) flush_slab(os, lane, ch0 + c - 16, row0, b_item, L);
    }
  } else {
#pragma unroll 1
    for (int c = c0; c < c0 + DH / 2; c += 16) {
      uint32_t r[16];
      read_o16<DH>(t, jn, c, r);
#pragma unroll
      for (int e = 0; e < 16; e += 4)
        reinterpret_cast<float4*>(slot)[(size_t)((c + e) / 4) * kUM + row] =
            make_float4(__uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
    }
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(&bar->o_free[t.q]);  // the next piece's first PV product may overwrite the accumulator
  if (direct) return true;
  slot[kM + row] = jn.m;
  slot[kL + row] = jn.l;
  if (!last_of_span) {  // the publisher thread fences, draws the tickets and leaves them for settle_first_piece
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar->pub_ready);
  } else if (take_ticket(ticket, lane) == (uint32_t)(g_last - g_first)) {
    __threadfence();
    combine_rows<DH>(pieces, sp, p.u, g_first, g_last, row, c0, out_row<DH>(o, p.u, row, L, heads));
  }
  return true;
}

// End of a CTA's span: if its first piece was partial and took the unit's last ticket (the other
// contributors, which run that unit at the end of their spans, are normally later), add the
// unit's pieces up now.
template <int DH>
__device__ __noinline__ void settle_first_piece(Barriers* bar, int it_begin, int it_end, Row t, __nv_bfloat16* o, int L,
                                                int heads, const Spans& sp, const float* pieces, uint32_t* dev_status) {
  const int nblk = sp.nblk, u = it_begin / nblk;
  const bool first_partial = it_begin > u * nblk || it_end < (u + 1) * nblk;
  if (!first_partial || it_end <= (u + 1) * nblk) return;  // whole, or also the span's last piece: settled already
  const int g_first = sp.unit_lo[0][blockIdx.x], g_last = sp.unit_hi[0][blockIdx.x];
  if (!mbar_wait(&bar->pub_done, 0, dev_status, &bar->abort_flag)) return;
  if (bar->first_ticket[t.warp] != (uint32_t)(g_last - g_first)) return;
  __threadfence();
  combine_rows<DH>(pieces, sp, u, g_first, g_last, t.row, t.half * (DH / 2), out_row<DH>(o, u, t.row, L, heads));
}

// Largest score (log2 domain) of this row in a tile, the first `valid` of its columns counting.
__device__ __noinline__ float tile_max(uint32_t s_addr, int valid, float scale_log2) {
  float mx = -INFINITY;
#pragma unroll 1
  for (int c = 0; c < valid; c += 16) {
    uint32_t r[16];
    tmem_ld16(s_addr + c, r);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) mx = c + e < valid ? fmaxf(mx, __uint_as_float(r[e])) : mx;
  }
  return mx * scale_log2;
}
// The reference for a row whose scores have reached `mx`.
__device__ __forceinline__ float reference(float mx, float m_used) { return mx > m_used + 1.f ? ceilf(mx) + kHeadroom : m_used; }
// Columns [c0, c1) of this row's accumulator times `factor` (a power of two: exact).
__device__ __forceinline__ void scale_o(uint32_t o_addr, int c0, int c1, float factor) {
#pragma unroll 1
  for (int c = c0; c < c1; c += 16) {
    uint32_t r[16];
    tmem_ld16(o_addr + c, r);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * factor);
    tmem_st16(o_addr + c, r);
  }
  tmem_wait_st();
}

// Own accumulators (head_dim 64): some row of this warp has scores that outgrew its reference.  Such rows get a new one,
// kHeadroom above the tile's largest score, and the pipeline's accumulator is multiplied by the power of two between the
// two (references are whole numbers).  Out of line, it hardly ever runs.  Returns the new reference.
template <int DH>
__device__ __noinline__ float move_reference(Row t, Barriers* bar, uint32_t s_addr, int valid, float scale_log2, float m_used, bool have_o, int n,
                                             uint32_t* dev_status) {
  const float m_new = reference(tile_max(s_addr, valid, scale_log2), m_used);
  // every product issued so far must have landed
  if (have_o && __all_sync(0xffffffffu, mbar_wait(&bar->pv_done[t.q][t.half], ((n >> 1) - 1) & 1, dev_status, &bar->abort_flag))) {
    tc_fence_after();
    scale_o(t.tm + AttCfg<DH>::o_col(t.q, t.half), 0, DH, ex2_mufu(m_used - m_new));
  }
  return m_new;
}

// Shared accumulator (head_dim 128): the two warps of a row group have one reference per row, and moving it takes both.
// Each brings the number of its next tile whose P it has not stored (`next`; kNoTile at the end of the piece), whether
// that tile's S lies ready (`have_s`; the warp that asks has it), and whether it asks.  Tiles below the smaller `next`
// have been multiplied or will be without further ado; the only other P there can be is that of tile min + 1, stored by
// the other warp and waiting behind it: it is rescaled where it lies.  Returns the new reference, and whether anybody
// asked (two warps at the end of their piece just meet here).
constexpr int kNoTile = 1 << 30;
struct Meeting {
  float m;
  bool asked;
};
template <int DH>
__device__ __noinline__ Meeting meet(Row t, Barriers* bar, uint32_t s_addr, int valid, float scale_log2, float m_used, bool ask, bool have_s, int next,
                                     int first_n, int last_n, uint32_t* dev_status) {
  using C = AttCfg<DH>;
  const float mx = have_s ? tile_max(s_addr, valid, scale_log2) : -INFINITY;
  const uint2 o = exchange<DH>(t, bar, __float_as_uint(mx), (uint32_t)next * 2u + (ask ? 1u : 0u));
  if (!ask && !(o.y & 1u)) return Meeting{m_used, false};
  const int other_next = (int)(o.y >> 1), low = min(next, other_next);
  const float m_new = reference(fmaxf(mx, __uint_as_float(o.x)), m_used);
  const float factor = ex2_mufu(m_used - m_new);
  if (low > first_n && low != kNoTile) {  // products of the piece's tiles below `low`: in order, so the last one tells
    const bool ok = mbar_wait(&bar->pv_done[t.q][(low - 1) & 1], ((low - 1) >> 1) & 1, dev_status, &bar->abort_flag);
    if (__all_sync(0xffffffffu, ok)) {
      tc_fence_after();
      scale_o(t.tm + C::o_col(t.q, 0), t.half * (DH / 2), (t.half + 1) * (DH / 2), factor);
    }
  }
  if ((low & 1) != t.half && next > low + 1 && low < last_n) {  // this warp has stored P of tile low + 1
#pragma unroll 1
    for (int c = 0; c < 32; c += 16) {
      uint32_t r[16];
      tmem_ld16(s_addr + c, r);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; ++e)
        r[e] = pack_bf16_rn(__uint_as_float(r[e] << 16) * factor, __uint_as_float(r[e] & 0xFFFF0000u) * factor);
      tmem_st16(s_addr + c, r);
    }
    tmem_wait_st();
  }
  tc_fence_before();
  if (t.lane == 0) *(volatile uint32_t*)&bar->move[pair_of(t)] = 0u;
  pair_sync(t);
  tc_fence_after();
  return Meeting{m_new, true};
}

// Waits for a tile's S, or for the row group's other warp to want the reference moved.  One answer per warp.
enum class Wait { kReady, kMove, kAborted };
__device__ __forceinline__ Wait wait_s_or_move(uint64_t* bar, uint32_t parity, const volatile uint32_t* move, uint32_t* dev_status,
                                               volatile int* abort_flag) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return Wait::kReady;
    if (__any_sync(0xffffffffu, *move != 0u)) return Wait::kMove;
    if ((it & 1023u) == 1023u && __any_sync(0xffffffffu, *abort_flag)) return Wait::kAborted;
  }
  *abort_flag = 1;
  if (dev_status) atomicOr(dev_status, kStatusTimeout);
  return Wait::kAborted;
}

template <int DH>
__global__ void __launch_bounds__(kThreads, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o,
                    __nv_bfloat16* __restrict__ o, int L, int heads,
                    float scale_log2, const __grid_constant__ Spans sp, uint32_t* __restrict__ tickets, float* __restrict__ pieces,
                    uint32_t* dev_status) {
  using C = AttCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + C::kQBufs * C::kQBytes;
  uint8_t* sV = sK + C::kStages * C::kKvBytes;
  uint8_t* sOut = sV + C::kStages * C::kKvBytes;
  Barriers* bar = reinterpret_cast<Barriers*>(sOut + C::kOutBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblk = sp.nblk;
  const int nq = (L + kUM - 1) / kUM;  // units per (batch, head)
  const int it_begin = sp.bound(blockIdx.x), it_end = sp.bound(blockIdx.x + 1);

  if (threadIdx.x == 0) {
    for (int q = 0; q < 2; ++q) {
      mbar_init(&bar->q_full[q], 1);
      mbar_init(&bar->q_empty[q], C::kIssuers);
      for (int h = 0; h < 2; ++h) {
        mbar_init(&bar->s_full[q][h], 1);
        mbar_init(&bar->p_full[q][h], 4);  // one arrival per softmax warp of the pipeline
        mbar_init(&bar->pv_done[q][h], 1);
      }
      mbar_init(&bar->o_free[q], 8);
      bar->poll_stop[q] = 0;
    }
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&bar->k_full[s], 1);
      mbar_init(&bar->kv_empty[s], C::kIssuers);
    }
    for (int g = 0; g < 8; ++g) bar->move[g] = 0;
    mbar_init(&bar->pub_ready, kSoftWarps);
    mbar_init(&bar->pub_done, 1);
    bar->others_done = 0;
    bar->abort_flag = 0;
    mbar_fence_init();
  }
  if (threadIdx.x == kSoftWarps * 32) {  // descriptor fetches overlap the previous kernel's tail
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    prefetch_tmap(&tm_o);
  }
  dependency_wait();
  if (threadIdx.x == 0) release_dependents();
  if (warp == 17) tmem_alloc(&bar->tmem_base, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int* abort_flag = &bar->abort_flag;

  if (warp == 16) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      Cursor c;
      int u = 0, key0 = 0, b = 0, ch0 = 0;
      for (c.init(it_begin, it_end, nblk); c.valid(); c.next(), key0 += kBN) {
        if (c.j == 0) {
          u = c.it / nblk, key0 = (c.it - u * nblk) * kBN;
          const int bh = u / nq, q0 = (u - bh * nq) * kUM, qb = c.pc % C::kQBufs;
          b = bh / heads, ch0 = (bh - b * heads) * DH;
          // a Q buffer is free once the S MMAs of the piece that used it have read it
          if (c.pc >= C::kQBufs && !mbar_wait(&bar->q_empty[qb], ((c.pc / C::kQBufs) - 1) & 1, dev_status, abort_flag)) break;
          mbar_expect_tx(&bar->q_full[qb], C::kQBytes);
          for (int t = 0; t < 2; ++t)
            for (int ch = 0; ch < C::kChunks; ++ch)
              tma_load_3d(sQ + qb * C::kQBytes + t * C::kQTile + ch * C::kQSlab, &tm_q, &bar->q_full[qb], ch0 + ch * 64, q0 + t * kBM, b);
        }
        const int s = c.n % C::kStages;
        if (c.n >= C::kStages && !mbar_wait(&bar->kv_empty[s], ((c.n / C::kStages) - 1) & 1, dev_status, abort_flag)) break;
        mbar_expect_tx(&bar->k_full[s], 2 * C::kKvBytes);  // K and V of a tile arrive under one barrier
        for (int ch = 0; ch < C::kChunks; ++ch)
          tma_load_3d(sK + s * C::kKvBytes + ch * C::kKvSlab, &tm_k, &bar->k_full[s], ch0 + ch * 64, key0, b);
        for (int ch = 0; ch < C::kChunks; ++ch)
          tma_load_3d(sV + s * C::kKvBytes + ch * C::kKvSlab, &tm_v, &bar->k_full[s], ch0 + ch * 64, key0, b);
      }
    }
  } else if (warp == 17 || (warp == 19 && C::kIssuers == 2)) {
    // ------------------------------------------------------------------ MMA issuer(s)
    // A thread's MMAs execute in the order it issues them: the S product of tile n+2 goes into the buffer whose
    // P the PV product of tile n, issued just before by the same thread, still reads.  The two query tiles'
    // products are independent of each other: one thread issues both, or each tile has its own thread
    // (query tiles [q_lo, q_hi) here); the barriers that both tiles' products free count one arrival per thread.
    const int q_lo = C::kIssuers == 2 && warp == 19 ? 1 : 0, q_hi = C::kIssuers == 2 && warp == 17 ? 1 : 2;
    if (elect_one()) {
      constexpr uint32_t idesc_s = idesc_f16(kFmtBF16, kFmtBF16, false, false, kBM, kBN);
      constexpr uint32_t idesc_o = idesc_f16(kFmtBF16, kFmtBF16, false, true, kBM, DH);
      // Descriptors are built once and advanced by adding a constant to the 14-bit start-address
      // field (no carry: all tiles live below 256 KB).
      const uint64_t q_desc0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);
      const uint64_t k_desc0 = smem_desc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t v_desc0 = smem_desc_sw128(smem_u32(sV), C::kKvSlab, 1024);
      Cursor cs, cp;  // the S products run two tiles ahead of the PV products
      cs.init(it_begin, it_end, nblk);
      cp.init(it_begin, it_end, nblk);
      // Q of the piece and K of the tile that `cs` points at have landed
      auto s_inputs = [&]() -> bool {
        if (cs.j == 0 && !mbar_wait(&bar->q_full[cs.pc % C::kQBufs], (cs.pc / C::kQBufs) & 1, dev_status, abort_flag)) return false;
        return mbar_wait(&bar->k_full[cs.n % C::kStages], (cs.n / C::kStages) & 1, dev_status, abort_flag);
      };
      auto issue_s = [&](int q) {
        const int s = cs.n % C::kStages, h = cs.n & 1, qb = cs.pc % C::kQBufs;
        const uint64_t qd = q_desc0 + (uint64_t)((qb * C::kQBytes + q * C::kQTile) >> 4);
        const uint64_t kd = k_desc0 + (uint64_t)((s * C::kKvBytes) >> 4);
        const uint32_t t_s = tmem + C::s_col(q, h);
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk) {
          const uint64_t qoff = (uint64_t)(((kk >> 2) * C::kQSlab + (kk & 3) * 32) >> 4);
          const uint64_t koff = (uint64_t)(((kk >> 2) * C::kKvSlab + (kk & 3) * 32) >> 4);
          mma_ss(t_s, qd + qoff, kd + koff, idesc_s, kk > 0);
        }
        mma_commit(&bar->s_full[q][h]);
      };
      bool ok = true;
      for (int pre = 0; pre < 2 && ok && cs.valid(); ++pre) {
        ok = s_inputs();
        if (!ok) break;
        tc_fence_after();
        for (int q = q_lo; q < q_hi; ++q) issue_s(q);
        if (cs.last_of_piece()) mma_commit(&bar->q_empty[cs.pc % C::kQBufs]);
        cs.next();
      }
      while (ok && cp.valid()) {
        const int s = cp.n % C::kStages, h = cp.n & 1;
        const bool more = cs.valid();
        const uint64_t vd = v_desc0 + (uint64_t)((s * C::kKvBytes) >> 4);
        const bool fresh = cp.j == 0 || (C::kOwnO && cp.j == 1);  // the accumulator's first product of the piece
#pragma unroll
        for (int q = q_lo; q < q_hi; ++q) {
          // P ready implies that the K/V tile has landed
          if (!mbar_wait(&bar->p_full[q][h], (cp.n >> 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          // the first product of a piece overwrites the accumulator the previous epilogue reads
          if (fresh && cp.pc > 0 && !mbar_wait(&bar->o_free[q], (cp.pc - 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t t_o = tmem + C::o_col(q, h), t_p = tmem + C::s_col(q, h);
#pragma unroll
          for (int kk = 0; kk < kBN / 16; ++kk)  // 16 keys per MMA: 8 packed columns of P, 16 rows of V
            mma_ts(t_o, t_p + kk * 8, vd + (uint64_t)((kk * 2048) >> 4), idesc_o, !fresh || kk > 0);
          mma_commit(&bar->pv_done[q][h]);
          if (q == q_hi - 1) mma_commit(&bar->kv_empty[s]);
          if (more) {
            if (q == q_lo) {
              ok = s_inputs();
              if (!ok) break;
              tc_fence_after();
            }
            issue_s(q);
          }
        }
        if (!ok) break;
        if (more) {
          if (cs.last_of_piece()) mma_commit(&bar->q_empty[cs.pc % C::kQBufs]);
          cs.next();
        }
        cp.next();
      }
    }
  } else if (warp == 18) {
    // ------------------------------------------------------------------ publisher
    if (lane == 0) {
      // When the span's first piece is partial and more pieces follow, make that piece
      // visible to the other CTAs and draw its tickets here, off the softmax warps' path.
      const int u = it_begin / nblk;
      const bool early = (it_begin > u * nblk || it_end < (u + 1) * nblk) && it_end > (u + 1) * nblk;
      if (early && mbar_wait(&bar->pub_ready, 0, dev_status, abort_flag)) {
        __threadfence();
        uint32_t t[kSoftWarps];
#pragma unroll
        for (int w = 0; w < kSoftWarps; ++w) t[w] = atomicAdd(&tickets[(size_t)u * kSoftWarps + w], 1u);
#pragma unroll
        for (int w = 0; w < kSoftWarps; ++w) bar->first_ticket[w] = t[w];
        mbar_arrive(&bar->pub_done);
      }
      // When the span ends inside a unit that one other CTA shares, that CTA ran its part at the
      // start of its span and has normally published it long since.  Watch its tickets (acquire)
      // and leave the answer in shared memory for the softmax warps: they add the two pieces up
      // straight from tensor memory if the answer is there when their last piece ends, and go
      // through scratch and tickets otherwise.  Polling keeps the ticket out of their registers.
      const int ul = (it_end - 1) / nblk;
      if (it_end < (ul + 1) * nblk && sp.unit_hi[1][blockIdx.x] == sp.unit_lo[1][blockIdx.x] + 1) {
        const uint32_t* tk = tickets + (size_t)ul * kSoftWarps;
        for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
          if ((*(volatile uint32_t*)&bar->poll_stop[0] && *(volatile uint32_t*)&bar->poll_stop[1]) || *abort_flag) break;
          bool all = true;
#pragma unroll
          for (int w = 0; w < kSoftWarps; ++w) all = all && ld_acquire_gpu(tk + w) == 1u;
          if (all) {
            st_release_cta(&bar->others_done, 1u);
            break;
          }
          __nanosleep(500);
        }
      }
    }
  } else if (warp < kSoftWarps) {
    // ------------------------------------------------------------------ softmax / epilogue
    Row t;
    t.q = warp >> 3, t.half = (warp >> 2) & 1, t.warp = warp, t.lane = lane;
    t.row = t.q * kBM + (warp & 3) * 32 + lane;  // query row inside the unit; (warp & 3) * 32 + lane is its tensor-memory lane
    t.tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_addr = t.tm + C::s_col(t.q, t.half);
    uint64_t* s_bar = &bar->s_full[t.q][t.half];
    volatile uint32_t* move = &bar->move[pair_of(t)];
    // A warp whose wait ran out goes on without waiting: the two warps of a row meet at barriers, and neither may
    // stay away (the results are void, and the status word says so).
    bool ok = true;
    int pc = 0;
    for (int it = it_begin; it < it_end; ++pc) {
      const Piece p = piece_at(it, it_end, nblk);
      // number of the piece's first tile: the tiles of this pipeline are those of its parity
      const int n0 = it - it_begin, last_n = n0 + p.cnt - 1;
      it += p.cnt;
      float m_used = -INFINITY;
      uint64_t l2 = 0;
      if constexpr (!C::kOwnO) {  // one reference for both pipelines: out of the piece's first tile
        float mx = -INFINITY;
        if ((n0 & 1) == t.half) {
          ok = ok && __all_sync(0xffffffffu, mbar_wait(s_bar, (n0 >> 1) & 1, dev_status, abort_flag));
          tc_fence_after();
          mx = tile_max(s_addr, min(32, L - p.k0 * kBN), scale_log2);
        }
        m_used = ceilf(fmaxf(mx, __uint_as_float(exchange<DH>(t, bar, __float_as_uint(mx), 0u).x))) + kHeadroom;
      }
      auto moved_to = [&](float m_new) {
        const float f = ex2_mufu(m_used - m_new);
        l2 = mul2(l2, pack2(f, f));
        m_used = m_new;
      };
      bool first = true;
      for (int j = (n0 ^ t.half) & 1; j < p.cnt; j += 2) {
        const int n = n0 + j, valid = min(kBN, L - (p.k0 + j) * kBN);  // keys of this tile inside the sequence
        if constexpr (C::kOwnO) {
          ok = ok && mbar_wait(s_bar, (n >> 1) & 1, dev_status, abort_flag);
          __syncwarp();
          tc_fence_after();
          if (first) m_used = ceilf(tile_max(s_addr, min(valid, 32), scale_log2)) + kHeadroom;
        } else {
          while (ok) {
            const Wait w = wait_s_or_move(s_bar, (n >> 1) & 1, move, dev_status, abort_flag);
            if (w == Wait::kReady) break;
            if (w == Wait::kAborted) ok = false;
            else moved_to(meet<DH>(t, bar, s_addr, valid, scale_log2, m_used, false, false, n, n0, last_n, dev_status).m);
          }
          tc_fence_after();
        }
        uint32_t pk[32];
        uint64_t sum2;
        bool asked = false;  // a second time would not help (scores that are no numbers)
#pragma unroll 1
        for (;;) {
          sum2 = 0;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t r[32];
            tmem_ld32(s_addr + c * 32, r);
            tmem_wait_ld(r);
            if (valid < (c + 1) * 32) {  // keys that are not there
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (c * 32 + e >= valid) r[e] = 0xFF800000u;  // -inf
            }
            chunk_exp_ref(r, *reinterpret_cast<uint32_t(*)[16]>(&pk[c * 16]), scale_log2, -m_used, sum2);
          }
          const bool grown = __any_sync(0xffffffffu, outgrown(sum2)) && !asked;
          if constexpr (C::kOwnO) {
            if (!grown) break;
            moved_to(move_reference<DH>(t, bar, s_addr, valid, scale_log2, m_used, !first, n, dev_status));
          } else {
            if (!grown && __all_sync(0xffffffffu, *move == 0u)) break;
            if (grown && lane == 0) *move = 1u;
            moved_to(meet<DH>(t, bar, s_addr, valid, scale_log2, m_used, grown, true, n, n0, last_n, dev_status).m);
          }
          asked = asked || grown;
        }
        first = false;
        tmem_st32(s_addr, pk);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar->p_full[t.q][t.half]);
        // the sum, while the tensor cores already multiply P
        float even, odd;
        unpack2(add2(l2, sum2), even, odd);
        if (__any_sync(0xffffffffu, may_dominate(sum2, even + odd))) {
          const bool dom = dominates(largest2(pk), even + odd);
          if (__any_sync(0xffffffffu, dom)) {
            const uint64_t rounded = rounded_sum2(pk);
            if (dom) sum2 = rounded;
          }
        }
        l2 = add2(l2, sum2);
      }
      if constexpr (!C::kOwnO) {  // the other warp may still want to move the reference
        for (;;) {
          const Meeting mt = meet<DH>(t, bar, s_addr, 0, scale_log2, m_used, false, false, kNoTile, n0, last_n, dev_status);
          if (!mt.asked) break;
          moved_to(mt.m);
        }
      }
      float l, l_odd;
      unpack2(l2, l, l_odd);
      const Joint jn = join_halves<DH>(t, bar, m_used, l + l_odd);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) continue;
      if (p.cnt == nblk) ok = finish_whole<DH>(t, bar, p, last_n, jn, &tm_o, L, heads, dev_status);
      else ok = finish_partial<DH>(t, bar, p, pc, last_n, it >= it_end, jn, o, &tm_o, L, heads, sp, tickets, pieces, dev_status);
    }
    if (__all_sync(0xffffffffu, ok)) settle_first_piece<DH>(bar, it_begin, it_end, t, o, L, heads, sp, pieces, dev_status);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 17) {
    tc_fence_after();
    tmem_dealloc(tmem, C::kTmemCols);
  }
}

size_t ticket_bytes(int B, int L, int heads) {
  const size_t units = (size_t)B * heads * ((L + kUM - 1) / kUM);
  return (units * kSoftWarps * sizeof(uint32_t) + 255) & ~(size_t)255;
}

int max_ctas() {
  const int sms = sm_count();
  int G = sms < kMaxCtas ? sms : kMaxCtas;
  const int v = g_tune_attention_ctas.load(std::memory_order_relaxed);  // test-only override
  if (v >= 1 && v <= kMaxCtas) G = v;
  return G;
}

// Key tiles a split costs a CTA, in units of one tile's time: writing, publishing and adding up the
// partial results at the end of its span.
constexpr int kSplitCostTiles = 4;

// What a piece costs its CTA beyond its key tiles, in half tiles: the pipeline drains, the accumulator is read
// out and (partial pieces) goes through scratch, tickets and the addition of the unit's pieces.
constexpr int kPieceCostWhole = 4, kPieceCostPartial = 8;

// The farthest end of a span that starts at iteration `start` and costs at most C half tiles
// (2 per key tile plus the piece costs above); `start` itself when not even one tile fits.
int span_end(int start, int T, int nblk, long long C) {
  long long cost = 0;
  int it = start;
  while (it < T) {
    const int k0 = it % nblk, room = nblk - k0;
    const long long rest_of_unit = 2LL * room + (k0 ? kPieceCostPartial : kPieceCostWhole);
    if (cost + rest_of_unit <= C) {
      cost += rest_of_unit;
      it += room;
      continue;
    }
    const long long cnt = (C - cost - kPieceCostPartial) / 2;  // a partial piece that ends inside the unit
    if (cnt >= 1) it += (int)(cnt < room - 1 ? cnt : room - 1);
    break;
  }
  return it;
}

// Spans of cost at most C, left to right; the number of spans, or 0 when C is too small for some span or more
// than `gmax` spans would be needed.
int cut_spans(int T, int nblk, long long C, int gmax, int* bounds) {
  int g = 0, it = 0;
  bounds[0] = 0;
  while (it < T) {
    if (g == gmax) return 0;
    const int end = span_end(it, T, nblk, C);
    if (end == it) return 0;
    bounds[++g] = it = end;
  }
  return g;
}

// Whole units per CTA when that is at most kSplitCostTiles tiles slower than a perfectly even cut;
// otherwise spans cut at single key tiles: evenly where a span holds two units or more (the pieces' costs are
// small beside it), else so that the longest span, pieces' costs included, is as short as possible (the
// smallest budget C for which a left-to-right cut needs no more spans than there are CTAs).
Spans make_spans(int units, int nblk, int gmax, int forced) {
  Spans sp = {};
  sp.nblk = nblk;
  sp.T = units * nblk;
  const int whole_tiles = ((units + gmax - 1) / gmax) * nblk;  // longest CTA with whole units
  const int even_tiles = (sp.T + gmax - 1) / gmax;             // longest CTA with an even cut
  int mode = whole_tiles <= even_tiles + kSplitCostTiles ? 0 : 1;
  if (forced == 0 || forced == 1) mode = forced;
  sp.split = mode;
  const int quantum = mode == 0 ? nblk : 1;
  const int quanta = sp.T / quantum;
  sp.G = quanta < gmax ? quanta : gmax;
  const int q = quanta / sp.G, r = quanta - q * sp.G;  // the first r spans hold q + 1 quanta, the others q
  for (int g = 0; g <= sp.G; ++g) sp.bounds[g] = (g * q + (g < r ? g : r)) * quantum;
  if (mode == 1 && q >= 2 * nblk) {
    // long spans: the even cut, with every bound that falls within kSnapTiles of a unit boundary moved onto it
    for (int g = 1; g < sp.G; ++g) {
      const int unit_edge = (sp.bounds[g] + nblk / 2) / nblk * nblk;
      const int off = sp.bounds[g] - unit_edge;
      if (off != 0 && off >= -kSnapTiles && off <= kSnapTiles) sp.bounds[g] = unit_edge;
    }
  } else if (mode == 1) {
    // spans of less than two units: the pieces' costs decide
    // (no budget below an even share of the tiles will do; the search climbs from there before it bisects)
    long long lo = 2LL * sp.T / gmax > 2 + kPieceCostPartial ? 2LL * sp.T / gmax : 2 + kPieceCostPartial, step = 4, hi = lo;
    while (!cut_spans(sp.T, nblk, hi, gmax, sp.bounds)) {
      lo = hi + 1;
      hi += step;
      step *= 2;
    }
    while (lo < hi) {  // cut_spans succeeds for every budget from some value on
      const long long mid = (lo + hi) / 2;
      if (cut_spans(sp.T, nblk, mid, gmax, sp.bounds)) hi = mid;
      else lo = mid + 1;
    }
    sp.G = cut_spans(sp.T, nblk, lo, gmax, sp.bounds);
  }
  for (int g = 0; g < sp.G; ++g) {
    const int unit[2] = {sp.bounds[g] / nblk, (sp.bounds[g + 1] - 1) / nblk};
    for (int e = 0; e < 2; ++e) {
      sp.unit_lo[e][g] = (uint8_t)sp.owner(unit[e] * nblk);
      sp.unit_hi[e][g] = (uint8_t)sp.owner((unit[e] + 1) * nblk - 1);
    }
  }
  return sp;
}

// The plan of a launch, kept from call to call: it depends on these four numbers alone, and working it out costs the
// host 15 to 40 us - as much as the kernel of a small call takes.  Bounded: the least recently used of 32 plans goes.
void plan_spans(int units, int nblk, Spans* out) {
  struct Entry {
    int units = 0, nblk = 0, gmax = 0, forced = 0;
    unsigned long long used = 0;
    Spans sp;
  };
  static std::mutex mu;
  static Entry cache[32];
  static unsigned long long clock = 0;
  const int gmax = max_ctas(), forced = g_tune_attention_split.load(std::memory_order_relaxed);  // test-only override
  {
    std::lock_guard<std::mutex> lock(mu);
    for (Entry& e : cache)
      if (e.used && e.units == units && e.nblk == nblk && e.gmax == gmax && e.forced == forced) {
        e.used = ++clock;
        *out = e.sp;
        return;
      }
  }
  *out = make_spans(units, nblk, gmax, forced);
  std::lock_guard<std::mutex> lock(mu);
  Entry* oldest = cache;
  for (Entry& e : cache)
    if (e.used < oldest->used) oldest = &e;
  oldest->units = units, oldest->nblk = nblk, oldest->gmax = gmax, oldest->forced = forced;
  oldest->used = ++clock;
  oldest->sp = *out;
}

template <int DH>
cudaError_t launch(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, void* ws,
                   bool tickets_clean, uint32_t* dev_status, cudaStream_t s) {
  using C = AttCfg<DH>;
  CUtensorMap tq, tk, tv, to;
  const uint64_t dims[3] = {(uint64_t)heads * DH, (uint64_t)L, (uint64_t)B};
  const uint64_t strides[2] = {(uint64_t)heads * DH * 2, (uint64_t)L * heads * DH * 2};
  const uint32_t box_q[3] = {64, kBM, 1};
  const uint32_t box_kv[3] = {64, kBN, 1};
  const uint32_t box_o[3] = {32, 32, 1};  // a softmax warp's 32 rows of 32 channels
  if (!encode_tmap_16bit(&tq, q, 3, dims, strides, box_q) || !encode_tmap_16bit(&tk, k, 3, dims, strides, box_kv) ||
      !encode_tmap_16bit(&tv, v, 3, dims, strides, box_kv) || !encode_tmap_16bit(&to, o, 3, dims, strides, box_o))
    return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> smem_raised{0};
  cudaError_t e = raise_dynamic_smem(attention_tc_kernel<DH>, C::kSmemBytes, smem_raised);
  if (e != cudaSuccess) return e;
  const long long units = (long long)B * heads * ((L + kUM - 1) / kUM);
  const int nblk = (L + kBN - 1) / kBN;
  if (units * nblk > 0x7fffffffLL) return cudaErrorInvalidValue;  // iteration indices are 32-bit
  Spans sp;
  plan_spans((int)units, nblk, &sp);
  const size_t tb = ticket_bytes(B, L, heads);
  if (sp.split && !tickets_clean) {  // units are split: their tickets start at zero
    e = cudaMemsetAsync(ws, 0, tb, s);
    if (e != cudaSuccess) return e;
  }
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)DH);
  e = launch_dependent(attention_tc_kernel<DH>, dim3(sp.G), dim3(kThreads), (size_t)C::kSmemBytes, s, tq, tk, tv, to,
                       (__nv_bfloat16*)o, L, heads, scale_log2, sp, (uint32_t*)ws, (float*)((char*)ws + tb), dev_status);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

size_t attention_tc_workspace_bytes(int B, int L, int heads, int dh) {
  const size_t piece = (dh == 64 ? piece_floats<64>() : piece_floats<128>()) * sizeof(float);
  return ticket_bytes(B, L, heads) + 2 * (size_t)kMaxCtas * piece;
}

size_t attention_tc_ticket_bytes(int B, int L, int heads) { return ticket_bytes(B, L, heads); }

int attention_tc_plan(int B, int L, int heads, int info[4], int* bounds, int* owner_first, int* owner_last, int capacity) {
  const long long units = (long long)B * heads * ((L + kUM - 1) / kUM);
  const int nblk = (L + kBN - 1) / kBN;
  if (units * nblk > 0x7fffffffLL) return 0;
  Spans sp;
  plan_spans((int)units, nblk, &sp);
  info[0] = sp.G;
  info[1] = sp.split;
  info[2] = (int)units;
  info[3] = nblk;
  for (int g = 0; g <= sp.G && g < capacity; ++g) {
    if (bounds) bounds[g] = sp.bound(g);
    if (g < sp.G && sp.split) {
      if (owner_first) owner_first[g] = sp.owner(sp.bound(g));
      if (owner_last) owner_last[g] = sp.owner(sp.bound(g + 1) - 1);
    }
  }
  return sp.G;
}

cudaError_t launch_attention_tc(int B, int L, int heads, int dh, const void* q, const void* k, const void* v, void* o,
                                void* ws, bool tickets_clean, uint32_t* dev_status, cudaStream_t s) {
  if (dh == 64) return launch<64>(B, L, heads, q, k, v, o, ws, tickets_clean, dev_status, s);
  if (dh == 128) return launch<128>(B, L, heads, q, k, v, o, ws, tickets_clean, dev_status, s);
  return cudaErrorInvalidValue;
}

}  // namespace toma
