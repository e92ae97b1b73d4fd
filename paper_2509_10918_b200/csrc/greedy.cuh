// The rounds of the greedy selection (Algorithm 2) on one tile's fixed-point similarity matrix, exact and with
// ties to the lowest index.  Shared by the selection kernel and the one-kernel refresh of small tiles.
//
// Gains are kept incrementally: after a pick t only the columns j with S[t][j] > m[j] change the cached maximum,
// and for those
//   g_i += relu(S[i][j] - m_new[j]) - relu(S[i][j] - m_old[j])
//        = max(S[i][j], m_new) - max(S[i][j], m_old) - (m_new - m_old).
// All quantities are integers, so this equals recomputing g_i = sum_j relu(S[i][j] - m[j]) every round.  S is
// symmetric and always read as row j.
//
// Several picks per round.  A round is a chain of latencies (argmax, read the pick's row, find the changed columns,
// read their rows, update), so rounds are what costs.  Gains never grow, hence: if the candidate with the second
// largest key has no column in common with the pick - no j that both improve -, its gain is the same after the
// pick's update and it IS the next pick; likewise a third and a fourth against those before them.  A round takes
// the longest such prefix of the up to four largest keys.  On tiles of 256 correlated tokens with 128 destinations
// that makes 55 rounds out of 127, on 1024 tokens with 512 destinations 176 out of 511; the picks are the same.
//
// Thread = two tokens = one 32-bit word of every row (entries biased to be >= 0, see sq_pitch() in common.cuh): the
// update of both for one changed column is two 16x2 maxima.  The differences are non-negative and at most 8190 (|S| <=
// 4095), so eight columns add up in a word without a carry between the halves (65520).  Every warp posts its two best keys and its
// third; the four best of all posted keys are the four best of all as long as they exceed every third.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace toma {
namespace greedy {

constexpr int kPicks = 4;

__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Gain and candidate in one key, 0 = none: the largest key is the largest gain with the lowest index.  A gain is
// below 2^22: sum_j relu(S_ij - m_j) = (sum |S_ij - m_j| + sum (S_ij - m_j)) / 2, the second sum is not positive
// for the first pick's m (the largest row sum) and m only grows, so a gain is at most N_loc * 8190 / 2 < 2^22.
constexpr int kIdxBits = 10;
__device__ __forceinline__ uint32_t make_key(uint32_t gain, int i) { return ((gain << kIdxBits) | (uint32_t)(kMaxNloc - 1 - i)) + 1u; }
__device__ __forceinline__ int key_index(uint32_t key) { return kMaxNloc - 1 - (int)((key - 1u) & (kMaxNloc - 1)); }

// Shared memory of the rounds (kTok: the largest tile of the caller).
template <int kTok>
struct Shared {
  uint4 post[16];             // per warp: its three best keys
  uint2 info[16];             // per warp: picks that do not collide in its columns; its changed columns for 1..4 picks
  uint2 list[kTok + 32];      // changed columns: word offset of the row, new maximum << 16 | old one
};

// Predicated stores and loads that stay where they are written: a branch around each, or a load sunk to its use,
// costs a round more than the instruction itself.
__device__ __forceinline__ void store_if(bool p, uint2* smem, uint32_t x, uint32_t y) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.v2.u32 [%1], {%2, %3};\n\t}" ::"r"((uint32_t)p),
               "r"((uint32_t)__cvta_generic_to_shared(smem)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void store_if(bool p, int32_t* dst, int v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.u32 [%1], %2;\n\t}" ::"r"((uint32_t)p), "l"(dst), "r"(v)
               : "memory");
}
__device__ __forceinline__ uint2 load_entry(const uint2* smem) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"((uint32_t)__cvta_generic_to_shared(smem)));
  return v;
}
template <bool kGlobal>
__device__ __forceinline__ uint32_t load_word(const uint32_t* p) {
  uint32_t v;
  if constexpr (kGlobal) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
  else asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)));
  return v;
}

__device__ __forceinline__ void warps_sync(int n_warps) { asm volatile("bar.sync 1, %0;" ::"r"(n_warps * 32) : "memory"); }

// Called by `n_warps` whole warps, threads numbered tid = 0 .. 32 n_warps - 1 of them (kOne: one warp, no block
// barrier).  S: row 0 of the matrix, pitch_w words per row.  gain0 / gain1: initial gains of tokens 2 tid and 2 tid + 1
// against row `first` (already picked and written to out[0]); out: the D_loc picks (global or shared memory).
template <bool kOne, bool kGlobal, int kTok>
__device__ __forceinline__ void rounds(const uint32_t* S, int pitch_w, int Nloc, int Dloc, int n_warps, int tid, int first, uint32_t gain0,
                                       uint32_t gain1, Shared<kTok>& sh, int32_t* out) {
  const int warp = kOne ? 0 : tid >> 5, lane = tid & 31;
  const unsigned below = (1u << lane) - 1u;
  const int j0 = 2 * tid, j1 = j0 + 1;
  const bool have0 = j0 < Nloc, have1 = j1 < Nloc;
  const uint32_t* Sc = S + (have0 ? tid : 0);  // a thread without tokens reads somebody else's column and uses nothing of it
  auto word = [&](uint32_t off) { return load_word<kGlobal>(Sc + off); };
  uint32_t off = (!have0 || j0 == first ? 1u : 0u) | (!have1 || j1 == first ? 2u : 0u);  // tokens selected, or not there
  uint32_t k0 = off & 1u ? 0u : make_key(gain0, j0), k1 = off & 2u ? 0u : make_key(gain1, j1);
  uint32_t m = word((uint32_t)(first * pitch_w));
  if (!have0) m |= 0xFFFFu;  // never improves
  if (!have1) m |= 0xFFFF0000u;

  for (int r = 1; r < Dloc;) {
    // ---- the four best keys, in order; `valid` of them are certain to be the four best
    uint32_t hi = max(k0, k1), lo = min(k0, k1);
    uint32_t b[kPicks];
    int valid = kPicks;
    if constexpr (kOne) {
#pragma unroll
      for (int x = 0; x < kPicks; ++x) {
        b[x] = __reduce_max_sync(0xffffffffu, hi);
        if (hi == b[x]) hi = lo, lo = 0u;
      }
      valid = 1 + (b[1] > 0u) + (b[2] > 0u) + (b[3] > 0u);
    } else {
      uint4 p;
      p.x = __reduce_max_sync(0xffffffffu, hi);
      if (hi == p.x) hi = lo, lo = 0u;
      p.y = __reduce_max_sync(0xffffffffu, hi);
      if (hi == p.y) hi = lo;
      p.z = __reduce_max_sync(0xffffffffu, hi);
      if (lane == 0) sh.post[warp] = p;
      warps_sync(n_warps);
      const uint32_t* post = reinterpret_cast<const uint32_t*>(sh.post);
      uint32_t key = lane < 2 * n_warps ? post[(lane >> 1) * 4 + (lane & 1)] : 0u;
      const uint32_t third = __reduce_max_sync(0xffffffffu, lane < n_warps ? post[lane * 4 + 2] : 0u);
#pragma unroll
      for (int x = 0; x < kPicks; ++x) {
        b[x] = __reduce_max_sync(0xffffffffu, key);
        if (key == b[x]) key = 0u;
      }
      valid = 1 + (b[1] > third) + (b[2] > third) + (b[3] > third);
    }
    valid = min(valid, Dloc - r);
    // ---- what each of them would improve; d[x] > 0 where pick x raises the cached maximum of a column
    uint32_t d[kPicks];
    int i[kPicks];
#pragma unroll
    for (int x = 0; x < kPicks; ++x) {
      i[x] = b[x] ? key_index(b[x]) : 0;
      d[x] = word((uint32_t)(i[x] * pitch_w));
    }
#pragma unroll
    for (int x = 0; x < kPicks; ++x) d[x] = max_u16x2(d[x], m) - m;
    // two of them improve the same column <=> the maximum of the raises is not their sum
    const uint32_t d01 = d[0] + d[1], d012 = d01 + d[2];
    const bool c1 = max_u16x2(d[0], d[1]) != d01, c2 = max_u16x2(d01, d[2]) != d012, c3 = max_u16x2(d012, d[3]) != d012 + d[3];
    const unsigned a1 = __ballot_sync(0xffffffffu, c1), a2 = __ballot_sync(0xffffffffu, c2), a3 = __ballot_sync(0xffffffffu, c3);
    int n = a1 ? 1 : a2 ? 2 : a3 ? 3 : 4;
    int base = 0, total;
    if constexpr (!kOne) {
      uint32_t cnt = 0, sum = 0;
#pragma unroll
      for (int x = 0; x < kPicks; ++x) {
        cnt += __popc(__ballot_sync(0xffffffffu, (d[x] & 0xFFFFu) != 0u)) + __popc(__ballot_sync(0xffffffffu, d[x] > 0xFFFFu));
        sum |= min(cnt, 255u) << (8 * x);  // beyond 64 only for prefixes that collide anyway
      }
      if (lane == 0) sh.info[warp] = make_uint2((uint32_t)n, sum);
      warps_sync(n_warps);
      const uint2 in = lane < n_warps ? sh.info[lane] : make_uint2((uint32_t)kPicks, 0u);
      n = min(valid, (int)__reduce_min_sync(0xffffffffu, in.x));
      const uint32_t c = (in.y >> (8 * (n - 1))) & 255u;
      base = (int)__reduce_add_sync(0xffffffffu, lane < warp ? c : 0u);
      total = (int)__reduce_add_sync(0xffffffffu, c);
    } else {
      n = min(valid, n);
      total = 0;
    }
    // ---- the n picks: their changed columns (disjoint) as one list
    uint32_t raise = d[0];
#pragma unroll
    for (int x = 1; x < kPicks; ++x) raise += x < n ? d[x] : 0u;
    const bool up0 = (raise & 0xFFFFu) != 0u, up1 = raise > 0xFFFFu;
    const unsigned u0 = __ballot_sync(0xffffffffu, up0), u1 = __ballot_sync(0xffffffffu, up1);
    const uint32_t mn = m + raise;
    if (kOne) total = __popc(u0) + __popc(u1);
    store_if(up0, &sh.list[base + __popc(u0 & below)], (uint32_t)(j0 * pitch_w), __byte_perm(m, mn, 0x5410));
    store_if(up1, &sh.list[base + __popc(u0) + __popc(u1 & below)], (uint32_t)(j1 * pitch_w), __byte_perm(m, mn, 0x7632));
    store_if(tid < 32, &sh.list[total + lane], 0u, 0u);  // neutral: new = old
    m = mn;
    if constexpr (kOne) __syncwarp();
    else warps_sync(n_warps);
    // ---- their effect on this thread's two gains: kBatch columns' rows in flight, added up eight at a time.  Rows in
    // shared memory: eight; in L2 or DRAM: up to 32, but no more than there are - late picks change one or two columns
    // each, and 32 for everybody took 830 us instead of 733 us (64 tiles of 1024 tokens, 512 destinations).
    auto batch = [&](int e, auto rows) {
      constexpr int kBatch = decltype(rows)::value;
      uint2 c[kBatch];
      uint32_t v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) c[u] = load_entry(&sh.list[e + u]);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) v[u] = word(c[u].x);
#pragma unroll
      for (int u0 = 0; u0 < kBatch; u0 += 8) {
        uint32_t g = 0u, y = 0u;
#pragma unroll
        for (int u = u0; u < u0 + 8; ++u) {
          g += max_u16x2(v[u], __byte_perm(c[u].y, 0u, 0x3232)) - max_u16x2(v[u], __byte_perm(c[u].y, 0u, 0x1010));
          y += c[u].y;
        }
        const uint32_t step = (y >> 16) - (y & 0xFFFFu);
        k0 += ((g & 0xFFFFu) - step) << kIdxBits;
        k1 += ((g >> 16) - step) << kIdxBits;
      }
    };
    int e = 0;
    if constexpr (kGlobal) {
      for (; total - e > 16; e += 32) batch(e, std::integral_constant<int, 32>{});
      if (total - e > 8) {
        batch(e, std::integral_constant<int, 16>{});
        e += 16;
      }
    }
    if constexpr (!kGlobal && !kOne)  // two loads in flight for one (2 x 4096 tokens of 256-token regions: 60.2 us, now 59.5)
      for (; total - e > 8; e += 16) batch(e, std::integral_constant<int, 16>{});
    for (; e < total; e += 8) batch(e, std::integral_constant<int, 8>{});
    store_if(tid < n, out + r + tid, tid == 0 ? i[0] : tid == 1 ? i[1] : tid == 2 ? i[2] : i[3]);
    uint32_t hit = 0u;  // bit 0 / 1: this thread's first / second token was picked
#pragma unroll
    for (int x = 0; x < kPicks; ++x) hit |= (uint32_t)(i[x] ^ j0) < (x < n ? 2u : 0u) ? 1u << (i[x] & 1) : 0u;
    off |= hit;
    r += n;
    if (kOne) __syncwarp();
    if (off & 1u) k0 = 0u;
    if (off & 2u) k1 = 0u;
  }
}

}  // namespace greedy
}  // namespace toma
