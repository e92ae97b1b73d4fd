// Device helpers of the tensor-core attention kernels, for one query row straight out of tensor memory: the online softmax
// of a 64-key tile (attention_two_tc.cu and, in its one instance without a mask at head_dim 64, block_fused_tc.cu) and the
// exponentials against a reference with headroom (attention_tc.cu).
#pragma once

#include "common.cuh"
#include "tc.cuh"

namespace toma {
namespace attn {

using namespace tc;

constexpr int kBM = 128;  // rows of one query tile = threads of one softmax warp group
constexpr int kBN = 64;   // keys per tile
constexpr float kRescaleThreshold = 8.0f;

// 2^x for x <= 127 on the FMA pipe, two at a time: round to nearest integer with the 1.5*2^23 trick, degree-3
// near-minimax polynomial for 2^f on [-0.5, 0.5], exponent patched in with an integer add.  Below -126 the result is
// 2^-126; above 127 the add runs into the sign bit and wraps, so callers whose x has no upper bound clamp it.
__device__ __forceinline__ void ex2_poly2(uint64_t x2, float& p0, float& p1) {
  float x0, x1;
  unpack2(x2, x0, x1);
  x2 = pack2(fmaxf(x0, -126.f), fmaxf(x1, -126.f));
  const uint64_t k2 = pack2(12582912.f, 12582912.f);
  const uint64_t t2 = add2(x2, k2);
  const uint64_t f2 = sub2(x2, sub2(t2, k2));
  uint64_t q2 = fma2(pack2(0.0551716648f, 0.0551716648f), f2, pack2(0.2426111251f, 0.2426111251f));
  q2 = fma2(q2, f2, pack2(0.6932609677f, 0.6932609677f));
  q2 = fma2(q2, f2, pack2(0.9999280572f, 0.9999280572f));
  float q0, q1, t0, t1;
  unpack2(q2, q0, q1);
  unpack2(t2, t0, t1);
  p0 = __int_as_float(__float_as_int(q0) + (int)((unsigned)__float_as_int(t0) << 23));
  p1 = __int_as_float(__float_as_int(q1) + (int)((unsigned)__float_as_int(t1) << 23));
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint32_t pack_bf16_rn(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t pack_bf16_trunc(float lo, float hi) {  // upper halves of both words
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// View of 32 consecutive registers of a larger per-thread array (all indices are compile-time).
template <int kOff, int kN>
__device__ __forceinline__ uint32_t (&sub32(uint32_t (&r)[kN]))[32] {
  return *reinterpret_cast<uint32_t(*)[32]>(&r[kOff]);
}

// Maximum of 32 tensor-memory words (columns first .. first+31 of this row; columns >= valid ignored).
template <bool kMask>
__device__ __forceinline__ float chunk_max(const uint32_t (&r)[32], float mx, int first, int valid) {
  if (kMask) {
#pragma unroll
    for (int e = 0; e < 32; ++e) mx = fmaxf(mx, (first + e < valid) ? __uint_as_float(r[e]) : -INFINITY);
  } else {
#pragma unroll
    for (int e = 0; e < 32; e += 2) mx = max3(mx, __uint_as_float(r[e]), __uint_as_float(r[e + 1]));
  }
  return mx;
}

// P for 32 columns as packed bf16 pairs in pk[16]; sum2: fp32 sums of the even and the odd columns, when sums stay in
// registers (one packed addition per pair, and two chains; one sum of single values was 1 instruction in 9 of the tile's:
// 4608 tokens, 24 heads of 128 channels 225.9 -> 221.8 us).
// kMorePoly: three pairs of columns in eight instead of two take the polynomial (timed: 1-2 % faster at head_dim
// 128, where the sums add to the FMA pipe's load anyway, 4 % slower at head_dim 64).
template <bool kMask, bool kRegSum, bool kMorePoly>
__device__ __forceinline__ void chunk_exp(const uint32_t (&r)[32], uint32_t (&pk)[16], float scale, float neg_m, int first, int valid,
                                          uint64_t& sum2) {
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    // S * c - m for a pair of columns in one packed multiply-add
    const uint64_t x2 = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), pack2(scale, scale), pack2(neg_m, neg_m));
    float p0, p1;
    const bool poly = kMorePoly ? ((e & 14) == 6 || (e & 14) == 10 || (e & 14) == 14) : (e & 6) == 6;
    if (poly) {  // this pair of exponentials on the FMA pipe
      ex2_poly2(x2, p0, p1);
    } else {
      float x0, x1;
      unpack2(x2, x0, x1);
      p0 = ex2_mufu(x0);
      p1 = ex2_mufu(x1);
    }
    if (kMask) {
      if (first + e >= valid) p0 = 0.f;
      if (first + e + 1 >= valid) p1 = 0.f;
    }
    if (kRegSum) {
      sum2 = add2(sum2, pack2(p0, p1));
      pk[e >> 1] = pack_bf16_rn(p0, p1);
    } else {
      pk[e >> 1] = pack_bf16_trunc(p0, p1);
    }
  }
}

// One 64-key tile of the online softmax for one query row.
template <int DH, bool kSumMma, bool kMask>
__device__ __forceinline__ void softmax_tile(uint32_t sb, uint32_t ob, float scale_log2, int valid, int j, float& m_used,
                                             float& l, uint64_t* pv_done, uint32_t pv_parity, uint32_t* dev_status, volatile int* abort_flag) {
  uint32_t sr[64];
  tmem_ld32(sb, sub32<0>(sr));
  tmem_ld32(sb + 32, sub32<32>(sr));
  tmem_wait_ld();
  float mx = -INFINITY;
  mx = chunk_max<kMask>(sub32<0>(sr), mx, 0, valid);
  mx = chunk_max<kMask>(sub32<32>(sr), mx, 32, valid);
  mx *= scale_log2;
  float factor = 1.f;
  bool rescale = false;
  if (j == 0) {
    m_used = mx;
  } else if (mx > m_used + kRescaleThreshold) {
    factor = ex2_mufu(m_used - mx);
    m_used = mx;
    rescale = true;
  }
  if (__any_sync(0xffffffffu, rescale)) {
    // O holds every PV product issued so far; the last one (tile j-1) must have landed
    mbar_wait(pv_done, pv_parity, dev_status, abort_flag);  // ran out: the results are void, but all lanes go the same way
    tc_fence_after();
    l *= factor;
#pragma unroll
    for (int c = 0; c < DH / 32; ++c) {
      uint32_t t[32];
      tmem_ld32(ob + c * 32, t);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 32; ++e) t[e] = __float_as_uint(__uint_as_float(t[e]) * factor);
      tmem_st32(ob + c * 32, t);
    }
    if (kSumMma) {
      uint32_t rs[16];
      tmem_ld16(ob + DH, rs);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; ++e) rs[e] = __float_as_uint(__uint_as_float(rs[e]) * factor);
      tmem_st16(ob + DH, rs);
    }
  }
  // P = 2^(S*c - m) as packed bf16 over the first 32 columns of this S buffer
  const float neg_m = -m_used;
  constexpr bool kRegSum = !kSumMma;
  uint32_t pk[16];
  uint64_t sum2 = 0;
  chunk_exp<kMask, kRegSum, DH == 128>(sub32<0>(sr), pk, scale_log2, neg_m, 0, valid, sum2);
  tmem_st16(sb, pk);
  chunk_exp<kMask, kRegSum, DH == 128>(sub32<32>(sr), pk, scale_log2, neg_m, 32, valid, sum2);
  tmem_st16(sb + 16, pk);
  tmem_wait_st();
  if (kRegSum) {
    float even, odd;
    unpack2(sum2, even, odd);
    l += even + odd;
  }
}

// ------------------------------------------------------------------ softmax against a reference with headroom
// P = 2^(S c - m) of 32 columns as packed bf16 for a reference m that lies 2^kHeadroom above the largest score seen when it
// was set.  Everything is floating point, so the common factor costs no precision (a power of two exactly: the largest P
// stay just below a power of two, where their 8 bits are worth most); what it buys is that the reference need
// not follow the row maximum: no maximum is taken before the exponentials.  Instead the sum of the tile's P is looked at
// (sum2: fp32 sums of the even and the odd columns): one of kOutgrown or more, or none at all, says that the scores have
// outgrown the headroom, and the caller moves the reference.  Scores may climb 44 nats before that: every row of
// self-attention climbs on its way to its own key, and a move costs its warp about a microsecond (tokens of variance 4, 4 x
// 512, 23 heads: 27.9 us with 22 nats).  Products of P and V stay in range for |V| from 2^-94 to 2^87.
// One pair of columns in four takes the polynomial of ex2_poly2 on the FMA pipe, the others MUFU (timed: one in eight to
// three in eight are within 2 % of each other).
constexpr float kHeadroom = 32.f;
constexpr float kOutgrown = 0x1p33f;

__device__ __forceinline__ void chunk_exp_ref(const uint32_t (&r)[32], uint32_t (&pk)[16], float scale, float neg_m, uint64_t& sum2) {
  const uint64_t c2 = pack2(scale, scale), m2 = pack2(neg_m, neg_m);
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    const uint64_t x2 = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), c2, m2);
    float p0, p1, x0, x1;
    unpack2(x2, x0, x1);
    if ((e & 6) == 6) {
      // a score may lie any distance above the reference: 2^126 stands for all that is larger, for outgrown() to see
      ex2_poly2(pack2(fminf(x0, 126.f), fminf(x1, 126.f)), p0, p1);
    } else {
      p0 = ex2_mufu(x0);
      p1 = ex2_mufu(x1);
    }
    sum2 = add2(sum2, pack2(p0, p1));
    pk[e >> 1] = pack_bf16_rn(p0, p1);
  }
}
// The largest P of a tile, even and odd columns (P is not negative, so packed bf16 compare as whole numbers).
__device__ __forceinline__ uint32_t largest2(const uint32_t (&pk)[32]) {
  uint32_t top = 0;
#pragma unroll
  for (int e = 0; e < 32; e += 2) top = __vimax3_u16x2(pk[e], pk[e + 1], top);
  return top;
}
__device__ __forceinline__ bool outgrown(uint64_t sum2) {
  float even, odd;
  unpack2(sum2, even, odd);
  return !(even + odd < kOutgrown);
}
// sum2 adds up P before its rounding to bf16: one instruction per pair of columns, where the rounded values take three
// (735 us against 825 us at 4 x 8192 tokens, 10 heads of 64).  Rounding errors of many keys cancel; that of a key which
// makes up most of its row would scale the whole output row by up to 2^-9.  In a tile where some P is more than a quarter
// of the row's sum so far, the row therefore counts what the product really multiplies.  Where the whole tile is less than
// a quarter no P can be: the largest is looked for in the other tiles only, a row's first few and the odd one later.
__device__ __forceinline__ bool may_dominate(uint64_t sum2, float sum) {
  float even, odd;
  unpack2(sum2, even, odd);
  return 4.f * (even + odd) > sum;
}
__device__ __forceinline__ bool dominates(uint32_t top, float sum) {
  return 4.f * fmaxf(__uint_as_float(top << 16), __uint_as_float(top & 0xFFFF0000u)) > sum;
}
__device__ __forceinline__ uint64_t rounded_sum2(const uint32_t (&pk)[32]) {
  uint64_t sum2 = 0;
#pragma unroll
  for (int e = 0; e < 32; ++e) sum2 = add2(sum2, pack2(__uint_as_float(pk[e] << 16), __uint_as_float(pk[e] & 0xFFFF0000u)));
  return sum2;
}

}  // namespace attn
}  // namespace toma
