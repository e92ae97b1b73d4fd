// Attention core softmax(Q K^T / sqrt(64)) V (Eq. 1 with tau = 1) on the sm_100a tensor cores, bf16 in / bf16 out, fp32
// softmax and accumulation: four softmax pipelines per CTA, for head_dim 64 (units, spans and pieces: attention_span.cuh),
// and the work plan and the choice between this kernel and attention_two_tc.cu's for every call.
//
// Inside a CTA (20 warps, the last one idle): warps 0..15 run the softmax as four pipelines of four warps, one per query tile q and parity h
// of the key tile (one thread per query row, straight out of tensor memory; so two threads share a row, each with every
// second key tile), warp 16 feeds Q, K and V through TMA rings, one elected thread of warp 17 issues the tcgen05 MMAs,
// warp 18 publishes a partial first piece (memory fence and tickets, off everybody else's path).
//   S_q,j = Q_q K_j^T      -> tensor memory, 64 columns per pipeline.  MMAs issued by one thread execute in order, so
//                             S_q,j+2 is issued right behind the product that reads P_q,j out of the same columns,
//                             without a round trip through a barrier.
//   P_q,j = 2^(S*c - m)    -> written back over S_q,j's first 32 columns as bf16 and used as the A operand (from tensor
//                             memory) of  O += P_q,j V_j
//   O                      -> every pipeline has an accumulator and a reference m of its own (four of 64 columns beside four
//                             of S fill the tensor memory), added up at the end of a piece
//   reference              -> set 2^32 above the piece's first tile and moved only when scores outgrow it (see
//                             chunk_exp_ref), so no row maximum stands before the exponentials
//   exponentials           -> one pair of columns in four goes through a degree-3 polynomial on the FMA pipe (relative
//                             error 7.5e-5, far below bf16 resolution of P), the rest through MUFU ex2; the scaling
//                             S*c - m and the polynomial run in packed f32x2 arithmetic
// What bounds it is the softmax: with one pipeline per query tile a scheduler has two softmax warps, which leaves it idle
// whenever both wait for tensor memory or each other's dependencies.  Four pipelines against the two groups of
// attention_two_tc.cu: 955 -> 740 us at 4 x 8192 tokens and 10 heads of 64, 42.0 -> 38.2 at 2 x 2048.  At head_dim 128 the
// pipelines of a query tile have to share an accumulator, and with it the reference: 4 % faster at 4 x 2048 tokens and 17
// heads, 2 to 10 % slower on shorter sequences, 6 to 12 % on peaked scores, and the results depended on the moment at
// which a reference moved.
// Keys past the sequence end are zero-filled by TMA and masked out; query rows past the end are
// computed on zeros and not written.
#include <mutex>

#include "attention_span.cuh"

namespace toma {

using namespace tc;
using namespace attn;

namespace {

constexpr int DH = 64;
constexpr int kSoftWarps = 16;
constexpr int kThreads = (kSoftWarps + 4) * 32;  // the last warp idles: a block of 19 was 0.5 % slower
static_assert(kSoftWarps <= kTicketCols, "tickets per unit");

constexpr int kStages = 8;                       // K/V ring depth (S runs two tiles ahead of P V)
constexpr int kQBufs = 2;                        // Q buffers: the next unit's Q lands under this unit's tail
constexpr int kQTile = kBM * 128;                // one query tile: 128 rows x 128 B
constexpr int kQBytes = 2 * kQTile;              // both query tiles of a unit
constexpr int kKvBytes = kBN * 128;              // one K or V tile: 64 rows x 128 B
constexpr int kOutBytes = kSoftWarps * 32 * 64;  // per softmax warp: 32 output rows of 32 channels, staged for a TMA store
constexpr int kBarBytes = 512;
constexpr int kSmemBytes = 1024 + kQBufs * kQBytes + 2 * kStages * kKvBytes + kOutBytes + kBarBytes;
constexpr int kTmemCols = 512;
// One thread issues the MMAs of both query tiles: the softmax bounds, and a second thread takes issue slots from it (752 ->
// 799 us at 4 x 8192 tokens, 10 heads).
// Tensor memory: a pipeline (query tile q, parity h) has 64 columns of S (P takes the first 32) and 64 of its accumulator.
__device__ __forceinline__ constexpr uint32_t s_col(int q, int h) { return (q * 2 + h) * 128; }
__device__ __forceinline__ constexpr uint32_t o_col(int q, int h) { return (q * 2 + h) * 128 + 64; }

struct Barriers {
  uint64_t q_full[2], q_empty[2];       // per piece: Q landed / every S MMA of the piece has read Q
  uint64_t k_full[kStages], kv_empty[kStages];  // per tile: K and V landed / every MMA that reads them is done
  uint64_t s_full[2][2], p_full[2][2];  // per tile and pipeline: S ready for the softmax / P ready for the PV MMAs
  uint64_t pv_done[2][2];               // the tile's PV MMAs are complete
  uint64_t o_free[2];                   // per piece and query tile: the epilogue has read the accumulators
  uint64_t pub_ready, pub_done;         // first partial piece: written by the softmax warps / published, tickets drawn
  uint32_t first_ticket[kSoftWarps];    // per softmax warp: ticket its first (partial) piece drew
  uint32_t others_done;                 // set by the publisher when the span's last unit has all its other pieces in scratch
  uint32_t poll_stop[2];                // set by each softmax group when the answer is no longer needed
  Edges edge;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(Barriers) <= kBarBytes, "barrier block outgrew its reservation");

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
__device__ __forceinline__ uint8_t* stage_of(const void* bar, int warp) {
  return const_cast<uint8_t*>(reinterpret_cast<const uint8_t*>(bar)) - kOutBytes + warp * 2048;
}
// Two words of this thread's for the other thread of the row, through the (then idle) staging areas.
__device__ __forceinline__ uint2 exchange(const Row& t, const void* bar, uint32_t a, uint32_t b) {
  volatile uint32_t* mine = reinterpret_cast<volatile uint32_t*>(stage_of(bar, t.warp)) + t.lane;
  const volatile uint32_t* other = reinterpret_cast<volatile uint32_t*>(stage_of(bar, t.warp ^ 4)) + t.lane;
  mine[0] = a;
  mine[32] = b;
  pair_sync(t);
  const uint2 o = make_uint2(other[0], other[32]);
  pair_sync(t);  // read: the areas may be written again
  return o;
}
// A row at the end of a piece: reference and row sum of both pipelines together, and what their accumulators count in it
// (0: nothing, not even if it is no number).
struct Joint {
  float m, l, w0, w1;
};
__device__ __forceinline__ Joint join_halves(const Row& t, const void* bar, float m, float l) {
  const uint2 o = exchange(t, bar, __float_as_uint(m), __float_as_uint(l));
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
__device__ __forceinline__ void read_o16(const Row& t, const Joint& jn, int c, uint32_t (&r)[16]) {
  uint32_t r1[16];
  tmem_ld16(t.tm + o_col(t.q, 0) + c, r);
  tmem_ld16(t.tm + o_col(t.q, 1) + c, r1);
  tmem_wait_ld();
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const float a = jn.w0 != 0.f ? jn.w0 * __uint_as_float(r[e]) : 0.f;
    r[e] = __float_as_uint(jn.w1 != 0.f ? fmaf(jn.w1, __uint_as_float(r1[e]), a) : a);
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
// Whole warp.  (ch0, row0, b): first channel of the slab, first token of the warp's 32 rows, batch item.  The slab is being
// read until staging_free().
__device__ __forceinline__ void flush_slab(const OutStage& os, int lane, int ch0, int row0, int b, int L) {
  fence_proxy_async();  // the staged rows are read by the TMA engine
  __syncwarp();
  if (lane == 0 && row0 < L) {
    tma_store_3d(os.tm_o, os.stage, ch0, row0, b);
    tma_store_commit();
  }
}
__device__ __forceinline__ void staging_free(int lane) {
  if (lane == 0) tma_store_wait_read();
  __syncwarp();
}
// End of a piece that covers all keys of its unit (the only kind when units are kept whole), run by
// the softmax warps: wait for the accumulators, normalise, write the rows out.  Returns false when
// the wait ran out.
__device__ __noinline__ bool finish_whole(Row t, Barriers* bar, Piece p, int last_n, Joint jn, const CUtensorMap* tm_o, int L, int heads,
                                          uint32_t* dev_status) {
  if (!wait_o(t, bar, last_n, p.cnt, dev_status)) return false;
  tc_fence_after();
  int b, ch0, row0;
  warp_rows_of<DH>(p.u, t.row & ~31, L, heads, b, ch0, row0);
  const OutStage os{stage_of(bar, t.warp), tm_o};
  const float inv = 1.f / jn.l;
  const int c0 = t.half * (DH / 2);
  static_assert(DH / 2 == 32, "a slab per warp and piece");
  uint32_t r[2][16];
  read_o16(t, jn, c0, r[0]);
  read_o16(t, jn, c0 + 16, r[1]);
  tc_fence_before();
  __syncwarp();
  if (t.lane == 0) mbar_arrive(&bar->o_free[t.q]);  // the next piece's first PV product may overwrite the accumulator
  stage16(os, t.lane, 0, r[0], inv);
  stage16(os, t.lane, 1, r[1], inv);
  flush_slab(os, t.lane, ch0 + c0, row0, b, L);
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
__device__ __noinline__ bool finish_partial(Row t, Barriers* bar, Piece p, int pc, int last_n, bool last_of_span, Joint jn,
                                            __nv_bfloat16* o, const CUtensorMap* tm_o, int L, int heads, const Spans& sp,
                                            uint32_t* tickets, float* pieces, uint32_t* dev_status) {
  constexpr size_t kM = (size_t)kUM * DH, kL = (size_t)kUM * DH + kUM;
  const int row = t.row, lane = t.lane, c0 = t.half * (DH / 2);
  uint32_t* ticket = tickets + (size_t)p.u * kTicketCols + t.warp;
  // a partial piece lies in the unit the span starts in or in the one it ends in
  const int which = p.u == bar->edge.first_unit ? 0 : 1;
  const int g_first = bar->edge.lo[which], g_last = bar->edge.hi[which];
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
    const float* slot = pieces + (size_t)bar->edge.other_slot * piece_floats<DH>();
    m_o = __ldcg(slot + kM + row);
    l_o = __ldcg(slot + kL + row);
    other = reinterpret_cast<const float4*>(slot) + row;
#pragma unroll
    for (int q = 0; q < 4; ++q) vo[q] = __ldcg(other + (size_t)(c0 / 4 + q) * kUM);
  }
  if (!wait_o(t, bar, last_n, p.cnt, dev_status)) return false;
  tc_fence_after();
  int b_item, ch0, row0;
  warp_rows_of<DH>(p.u, t.row & ~31, L, heads, b_item, ch0, row0);
  float* slot = pieces + (size_t)(2 * blockIdx.x + (pc > 0 ? 1 : 0)) * piece_floats<DH>();
  if (direct) {
    const OutStage os{stage_of(bar, t.warp), tm_o};
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
      read_o16(t, jn, c, r);
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
      read_o16(t, jn, c, r);
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
    combine_rows<DH, DH / 2, 16, 4>(pieces, sp, p.u, g_first, g_last, row, c0, out_row<DH>(o, p.u, row, L, heads));
  }
  return true;
}

// End of a CTA's span: if its first piece was partial and took the unit's last ticket (the other
// contributors, which run that unit at the end of their spans, are normally later), add the
// unit's pieces up now.
__device__ __noinline__ void settle_first_piece(Barriers* bar, int it_begin, int it_end, Row t, __nv_bfloat16* o, int L,
                                                int heads, const Spans& sp, const float* pieces, uint32_t* dev_status) {
  const int nblk = sp.nblk, u = it_begin / nblk;
  const bool first_partial = it_begin > u * nblk || it_end < (u + 1) * nblk;
  if (!first_partial || it_end <= (u + 1) * nblk) return;  // whole, or also the span's last piece: settled already
  const int g_first = bar->edge.lo[0], g_last = bar->edge.hi[0];
  if (!mbar_wait_warp(&bar->pub_done, 0, dev_status, &bar->abort_flag)) return;
  if (bar->first_ticket[t.warp] != (uint32_t)(g_last - g_first)) return;
  __threadfence();
  combine_rows<DH, DH / 2, 16, 4>(pieces, sp, u, g_first, g_last, t.row, t.half * (DH / 2), out_row<DH>(o, u, t.row, L, heads));
}

// Largest score (log2 domain) of this row in a tile, the first `valid` of its columns counting.
__device__ __noinline__ float tile_max(uint32_t s_addr, int valid, float scale_log2) {
  float even = -INFINITY, odd = -INFINITY;
#pragma unroll 1
  for (int c = 0; c < valid; c += 32) {
    uint32_t r[32];
    tmem_ld32(s_addr + c, r);
    tmem_wait_ld();
    if (valid - c < 32) {
#pragma unroll
      for (int e = 0; e < 32; ++e)
        if (c + e >= valid) r[e] = 0xFF800000u;  // -inf
    }
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      even = max3(even, __uint_as_float(r[e]), __uint_as_float(r[e + 2]));
      odd = max3(odd, __uint_as_float(r[e + 1]), __uint_as_float(r[e + 3]));
    }
  }
  return fmaxf(even, odd) * scale_log2;
}
// The reference for a row whose scores have reached `mx`.
__device__ __forceinline__ float reference(float mx, float m_used) { return mx > m_used ? mx + kHeadroom : m_used; }
// This row's accumulator times `factor`.
__device__ __forceinline__ void scale_o(uint32_t o_addr, float factor) {
#pragma unroll 1
  for (int c = 0; c < DH; c += 16) {
    uint32_t r[16];
    tmem_ld16(o_addr + c, r);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * factor);
    tmem_st16(o_addr + c, r);
  }
  tmem_wait_st();
}

// Some row of this warp has scores that outgrew its reference.  Such rows get a new one, kHeadroom above the tile's largest
// score, and the pipeline's accumulator is multiplied by what lies between the two.  Out of line, it hardly ever runs.
// Returns the new reference.
__device__ __noinline__ float move_reference(Row t, Barriers* bar, uint32_t s_addr, int valid, float scale_log2, float m_used, bool have_o, int n,
                                             uint32_t* dev_status) {
  const float m_new = reference(tile_max(s_addr, valid, scale_log2), m_used);
  // every product issued so far must have landed
  if (have_o && __all_sync(0xffffffffu, mbar_wait(&bar->pv_done[t.q][t.half], ((n >> 1) - 1) & 1, dev_status, &bar->abort_flag))) {
    tc_fence_after();
    scale_o(t.tm + o_col(t.q, t.half), ex2_mufu(m_used - m_new));
  }
  return m_new;
}

__global__ void __launch_bounds__(kThreads, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o,
                    __nv_bfloat16* __restrict__ o, int L, int heads,
                    float scale_log2, const __grid_constant__ Spans sp, uint32_t* __restrict__ tickets, float* __restrict__ pieces,
                    uint32_t* dev_status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + kQBufs * kQBytes;
  uint8_t* sV = sK + kStages * kKvBytes;
  uint8_t* sOut = sV + kStages * kKvBytes;
  Barriers* bar = reinterpret_cast<Barriers*>(sOut + kOutBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblk = sp.nblk;
  const int nq = (L + kUM - 1) / kUM;  // units per (batch, head)
  const int it_begin = sp.bound(blockIdx.x), it_end = sp.bound(blockIdx.x + 1);

  if (threadIdx.x == 0) {
    for (int q = 0; q < 2; ++q) {
      mbar_init(&bar->q_full[q], 1);
      mbar_init(&bar->q_empty[q], 1);
      for (int h = 0; h < 2; ++h) {
        mbar_init(&bar->s_full[q][h], 1);
        mbar_init(&bar->p_full[q][h], 4);  // one arrival per softmax warp of the pipeline
        mbar_init(&bar->pv_done[q][h], 1);
      }
      mbar_init(&bar->o_free[q], 8);
      bar->poll_stop[q] = 0;
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bar->k_full[s], 1);
      mbar_init(&bar->kv_empty[s], 1);
    }
    mbar_init(&bar->pub_ready, kSoftWarps);
    mbar_init(&bar->pub_done, 1);
    bar->others_done = 0;
    bar->abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == kSoftWarps + 3 && lane < 2) bar->edge.fill(sp, it_begin, it_end, lane);
  if (threadIdx.x == kSoftWarps * 32) {  // descriptor fetches overlap the previous kernel's tail
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    prefetch_tmap(&tm_o);
  }
  dependency_wait();
  if (threadIdx.x == 0) release_dependents();
  if (warp == 17) tmem_alloc(&bar->tmem_base, kTmemCols);
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
          const int bh = u / nq, q0 = (u - bh * nq) * kUM, qb = c.pc % kQBufs;
          b = bh / heads, ch0 = (bh - b * heads) * DH;
          // a Q buffer is free once the S MMAs of the piece that used it have read it
          if (c.pc >= kQBufs && !mbar_wait(&bar->q_empty[qb], ((c.pc / kQBufs) - 1) & 1, dev_status, abort_flag)) break;
          mbar_expect_tx(&bar->q_full[qb], kQBytes);
          for (int t = 0; t < 2; ++t) tma_load_3d(sQ + qb * kQBytes + t * kQTile, &tm_q, &bar->q_full[qb], ch0, q0 + t * kBM, b);
        }
        const int s = c.n % kStages;
        if (c.n >= kStages && !mbar_wait(&bar->kv_empty[s], ((c.n / kStages) - 1) & 1, dev_status, abort_flag)) break;
        mbar_expect_tx(&bar->k_full[s], 2 * kKvBytes);  // K and V of a tile arrive under one barrier
        tma_load_3d(sK + s * kKvBytes, &tm_k, &bar->k_full[s], ch0, key0, b);
        tma_load_3d(sV + s * kKvBytes, &tm_v, &bar->k_full[s], ch0, key0, b);
      }
    }
  } else if (warp == 17) {
    // ------------------------------------------------------------------ MMA issuer
    // A thread's MMAs execute in the order it issues them: the S product of tile n+2 goes into the buffer whose
    // P the PV product of tile n, issued just before by the same thread, still reads.
    if (elect_one()) {
      constexpr uint32_t idesc_s = idesc_f16(kFmtBF16, kFmtBF16, false, false, kBM, kBN);
      constexpr uint32_t idesc_o = idesc_f16(kFmtBF16, kFmtBF16, false, true, kBM, DH);
      // Descriptors are built once and advanced by adding a constant to the 14-bit start-address
      // field (no carry: all tiles live below 256 KB).
      const uint64_t q_desc0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);
      const uint64_t k_desc0 = smem_desc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t v_desc0 = smem_desc_sw128(smem_u32(sV), kKvBytes, 1024);
      Cursor cs, cp;  // the S products run two tiles ahead of the PV products
      cs.init(it_begin, it_end, nblk);
      cp.init(it_begin, it_end, nblk);
      // Q of the piece and K of the tile that `cs` points at have landed
      auto s_inputs = [&]() -> bool {
        if (cs.j == 0 && !mbar_wait(&bar->q_full[cs.pc % kQBufs], (cs.pc / kQBufs) & 1, dev_status, abort_flag)) return false;
        return mbar_wait(&bar->k_full[cs.n % kStages], (cs.n / kStages) & 1, dev_status, abort_flag);
      };
      auto issue_s = [&](int q) {
        const int s = cs.n % kStages, h = cs.n & 1, qb = cs.pc % kQBufs;
        const uint64_t qd = q_desc0 + (uint64_t)((qb * kQBytes + q * kQTile) >> 4);
        const uint64_t kd = k_desc0 + (uint64_t)((s * kKvBytes) >> 4);
        const uint32_t t_s = tmem + s_col(q, h);
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk) {
          const uint64_t off = (uint64_t)((kk * 32) >> 4);
          mma_ss(t_s, qd + off, kd + off, idesc_s, kk > 0);
        }
        mma_commit(&bar->s_full[q][h]);
      };
      bool ok = true;
      for (int pre = 0; pre < 2 && ok && cs.valid(); ++pre) {
        ok = s_inputs();
        if (!ok) break;
        tc_fence_after();
        for (int q = 0; q < 2; ++q) issue_s(q);
        if (cs.last_of_piece()) mma_commit(&bar->q_empty[cs.pc % kQBufs]);
        cs.next();
      }
      while (ok && cp.valid()) {
        const int s = cp.n % kStages, h = cp.n & 1;
        const bool more = cs.valid();
        const uint64_t vd = v_desc0 + (uint64_t)((s * kKvBytes) >> 4);
        const bool fresh = cp.j <= 1;  // the accumulator's first product of the piece
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          // P ready implies that the K/V tile has landed
          if (!mbar_wait(&bar->p_full[q][h], (cp.n >> 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          // the first product of a piece overwrites the accumulator the previous epilogue reads
          if (fresh && cp.pc > 0 && !mbar_wait(&bar->o_free[q], (cp.pc - 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t t_o = tmem + o_col(q, h), t_p = tmem + s_col(q, h);
#pragma unroll
          for (int kk = 0; kk < kBN / 16; ++kk)  // 16 keys per MMA: 8 packed columns of P, 16 rows of V
            mma_ts(t_o, t_p + kk * 8, vd + (uint64_t)((kk * 2048) >> 4), idesc_o, !fresh || kk > 0);
          mma_commit(&bar->pv_done[q][h]);
          if (q == 1) mma_commit(&bar->kv_empty[s]);
          if (more) {
            if (q == 0) {
              ok = s_inputs();
              if (!ok) break;
              tc_fence_after();
            }
            issue_s(q);
          }
        }
        if (!ok) break;
        if (more) {
          if (cs.last_of_piece()) mma_commit(&bar->q_empty[cs.pc % kQBufs]);
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
        for (int w = 0; w < kSoftWarps; ++w) t[w] = atomicAdd(&tickets[(size_t)u * kTicketCols + w], 1u);
#pragma unroll
        for (int w = 0; w < kSoftWarps; ++w) bar->first_ticket[w] = t[w];
        mbar_arrive(&bar->pub_done);
      }
      // When the span ends inside a unit that one other CTA shares, that CTA ran its part at the
      // start of its span and has normally published it long since.  Watch its tickets (plain loads, one fence behind them)
      // and leave the answer in shared memory for the softmax warps: they add the two pieces up
      // straight from tensor memory if the answer is there when their last piece ends, and go
      // through scratch and tickets otherwise.  Polling keeps the ticket out of their registers.
      const int ul = (it_end - 1) / nblk;
      if (it_end < (ul + 1) * nblk && sp.unit_hi[1][blockIdx.x] == sp.unit_lo[1][blockIdx.x] + 1) {
        const uint32_t* tk = tickets + (size_t)ul * kTicketCols;
        for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
          if ((*(volatile uint32_t*)&bar->poll_stop[0] && *(volatile uint32_t*)&bar->poll_stop[1]) || *abort_flag) break;
          if (all_drawn_once<kSoftWarps>(tk)) {
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
    const uint32_t s_addr = t.tm + s_col(t.q, t.half);
    uint64_t* s_bar = &bar->s_full[t.q][t.half];
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
      auto moved_to = [&](float m_new) {
        const float f = ex2_mufu(m_used - m_new);
        l2 = mul2(l2, pack2(f, f));
        m_used = m_new;
      };
      bool first = true;
      for (int j = (n0 ^ t.half) & 1; j < p.cnt; j += 2) {
        const int n = n0 + j, valid = min(kBN, L - (p.k0 + j) * kBN);  // keys of this tile inside the sequence
        ok = ok && mbar_wait(s_bar, (n >> 1) & 1, dev_status, abort_flag);
        __syncwarp();
        tc_fence_after();
        if (first) m_used = tile_max(s_addr, valid, scale_log2) + kHeadroom;
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
          if (!grown) break;
          moved_to(move_reference(t, bar, s_addr, valid, scale_log2, m_used, !first, n, dev_status));
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
      float l, l_odd;
      unpack2(l2, l, l_odd);
      staging_free(lane);
      const Joint jn = join_halves(t, bar, m_used, l + l_odd);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) continue;
      if (p.cnt == nblk) ok = finish_whole(t, bar, p, last_n, jn, &tm_o, L, heads, dev_status);
      else ok = finish_partial(t, bar, p, pc, last_n, it >= it_end, jn, o, &tm_o, L, heads, sp, tickets, pieces, dev_status);
    }
    if (__all_sync(0xffffffffu, ok)) settle_first_piece(bar, it_begin, it_end, t, o, L, heads, sp, pieces, dev_status);
    staging_free(lane);  // shared memory must outlive the engine's reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 17) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
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

// Bounds of long spans this close to a unit boundary move onto it.
constexpr int kSnapTiles = 2;

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
  sp.longest = 0;
  for (int g = 0; g < sp.G; ++g) {
    if (sp.bounds[g + 1] - sp.bounds[g] > sp.longest) sp.longest = sp.bounds[g + 1] - sp.bounds[g];
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

cudaError_t launch_four(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, void* ws, const Spans& sp,
                        uint32_t* dev_status, cudaStream_t s) {
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
  if (cudaError_t e = raise_dynamic_smem(attention_tc_kernel, kSmemBytes, smem_raised); e != cudaSuccess) return e;
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)DH);
  const cudaError_t e = launch_dependent(attention_tc_kernel, dim3(sp.G), dim3(kThreads), (size_t)kSmemBytes, s, tq, tk, tv, to, (__nv_bfloat16*)o, L,
                                         heads, scale_log2, sp, (uint32_t*)ws, (float*)((char*)ws + ticket_bytes(B, L, heads)), dev_status);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

// Key tiles of the longest span from which on four pipelines win at head_dim 64: their join at the end of a piece and the
// larger block cost a CTA what it gains in about six tiles (timed on 260 shapes: one to four tiles 0.85 to 1.0 times as
// fast, eight 1.01 to 1.12, sixteen 1.08, a hundred 1.15 to 1.2).
// Spans cut inside units end in pieces, whose reading and adding up costs four pipelines more: there it takes fourteen (4 x
// 512 tokens, 23 heads, spans of eleven: 24 us against 20).
constexpr int kFourFrom = 8, kFourFromSplit = 14;

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
  const long long units = (long long)B * heads * ((L + kUM - 1) / kUM);
  const int nblk = (L + kBN - 1) / kBN;
  if (units * nblk > 0x7fffffffLL) return cudaErrorInvalidValue;  // iteration indices are 32-bit
  Spans sp;
  plan_spans((int)units, nblk, &sp);
  if (sp.split && !tickets_clean)  // units are split: their tickets start at zero
    if (cudaError_t e = cudaMemsetAsync(ws, 0, ticket_bytes(B, L, heads), s); e != cudaSuccess) return e;
  if (dh == 64 && sp.longest >= (sp.split ? kFourFromSplit : kFourFrom)) return launch_four(B, L, heads, q, k, v, o, ws, sp, dev_status, s);
  return launch_attention_two(B, L, heads, dh, q, k, v, o, ws, sp, dev_status, s);
}

}  // namespace toma
