// FFMA attention core softmax(Q K^T / sqrt(dh)) V (Eq. 1 with tau = 1) with an
// online softmax.  Used for the fp32 mode and for head sizes the tensor-core
// kernel does not cover.
//
// A CTA takes 32 or 64 queries of a head and walks the keys 64 at a time, K and V double buffered in shared memory
// (16-byte asynchronous copies).  Sixteen lanes share four query rows: a thread computes 4 x 4 scores (keys tx, tx + 16,
// tx + 32, tx + 48, whose rows of DH + 4 floats fall into different banks) and 4 x DH / 16 outputs, four contraction
// steps per 16-byte shared read, so that 64 multiply-adds go with eight reads.  Scores become probabilities in
// registers (row maxima and sums by shuffles within the sixteen lanes) and pass through shared memory once, between
// lanes of one half warp.  Bound by the FMA pipe where there are queries enough to fill it (16 warps per SM).  Where there are
// not, the four warps of 32 queries wait for their own latencies - 10 heads x 512 tokens x 64 channels, fp32: 46 us, 9 of
// them multiply-adds -, and so two to four groups of warps share the queries, each with every second to fourth key tile, a
// reference and sums of its own, added up at the end (KG): 28 us.  512 tokens of 20 heads of 128 223 -> 206, bound by reads of
// shared memory, as are all (2.8 cycles for each of them, eight for 32 packed multiply-adds).
#include <float.h>

#include <type_traits>

#include "common.cuh"
#include "spread.cuh"
#include "tc.cuh"

namespace toma {

namespace {

constexpr int kKeys = 64;

__device__ __forceinline__ void copy16(float* dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
// Four elements of a bf16 row widened into shared memory (the asynchronous copy cannot convert).
__device__ __forceinline__ void copy16(float* dst, const __nv_bfloat16* src, bool in) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (in) {
    const uint2 q = *reinterpret_cast<const uint2*>(src);
    v = make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u), __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xFFFF0000u));
  }
  *reinterpret_cast<float4*>(dst) = v;
}

// KG groups of BQ * 4 threads.  One group: K and V double buffered; several: one buffer of each per group, the next K on its
// way from the scores on, the next V from the outputs on.
template <int DH, int BQ, int KG>
struct SimtCfg {
  static constexpr int kPitch = DH + 4;
  static constexpr int kTile = kKeys * kPitch;
  static constexpr int kPPitch = kKeys + 4;
  static constexpr int kBufs = KG == 1 ? 2 : 1;
  static constexpr bool kByTile = KG <= 2 && BQ == 32;
  static constexpr int kGroup = 2 * kBufs * kTile + BQ * kPPitch;
  static constexpr size_t kSmem = ((size_t)BQ * kPitch + (size_t)KG * kGroup) * 4;
  static_assert(BQ * DH <= kTile && 2 * BQ <= kPPitch * BQ, "a group's outputs and sums fit where its tiles were");
};

template <bool kSecond, typename A>
__device__ __forceinline__ A& select_sum(A& first, A& second) {
  if constexpr (kSecond) return second;
  else return first;
}

template <typename T, int DH, int BQ, int KG>
__global__ void __launch_bounds__(BQ * 4 * KG) attention_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                                                     T* __restrict__ o, int L, int heads, float scale) {
  using C = SimtCfg<DH, BQ, KG>;
  constexpr int kThreads = BQ * 4, DV = DH / 16;
  extern __shared__ __align__(16) float att_smem[];
  const int group = KG == 1 ? 0 : threadIdx.x / kThreads, tid = KG == 1 ? threadIdx.x : threadIdx.x % kThreads;
  float* Qs = att_smem;                                // [BQ][pitch], scaled
  float* Ks = Qs + BQ * C::kPitch + group * C::kGroup; // [bufs][64][pitch]
  float* Vs = Ks + C::kBufs * C::kTile;                // [bufs][64][pitch]
  float* Ps = Vs + C::kBufs * C::kTile;                // [BQ][64 + 4]
  const int b = blockIdx.z, h = blockIdx.y, q0 = blockIdx.x * BQ;
  const int tx = tid & 15, r0 = (tid >> 4) * 4;
  const size_t row_stride = (size_t)heads * DH;
  const size_t base = (size_t)b * L * row_stride + (size_t)h * DH;
  auto load_one = [&](float* dst, const T* src, int k0) {
#pragma unroll 4
    for (int e = tid; e < kKeys * (DH / 4); e += kThreads) {
      const int r = e / (DH / 4), c = (e % (DH / 4)) * 4;
      const bool in = k0 + r < L;
      copy16(dst + r * C::kPitch + c, src + base + (size_t)(in ? k0 + r : 0) * row_stride + c, in);
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
  auto load_tile = [&](int k0, int st) {
    if constexpr (sizeof(T) == 4) {
      load_one(Ks + st * C::kTile, k, k0);
      load_one(Vs + st * C::kTile, v, k0);
    } else {  // bf16 packets pass through registers: in one loop twice as many are on their way
#pragma unroll 4
      for (int e = tid; e < kKeys * (DH / 4); e += kThreads) {
        const int r = e / (DH / 4), c = (e % (DH / 4)) * 4, dst = st * C::kTile + r * C::kPitch + c;
        const bool in = k0 + r < L;
        const size_t off = base + (size_t)(in ? k0 + r : 0) * row_stride + c;
        copy16(Ks + dst, k + off, in);
        copy16(Vs + dst, v + off, in);
      }
    }
    commit();
  };
  auto group_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kThreads) : "memory"); };
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (threadIdx.x == 0) tc::release_dependents();
  if constexpr (KG == 1) {
    load_tile(0, 0);
  } else if constexpr (sizeof(T) == 2) {
    load_tile(group * kKeys, 0);
    commit();
  } else {
    load_one(Ks, k, group * kKeys);
    commit();
    load_one(Vs, v, group * kKeys);
    commit();
  }
  for (int e = threadIdx.x; e < BQ * DH; e += kThreads * KG) {
    const int r = e / DH, c = e % DH;
    Qs[r * C::kPitch + c] = q0 + r < L ? to_f32(q[base + (size_t)(q0 + r) * row_stride + c]) * scale : 0.f;
  }
  // outputs of two channels in a register pair; a single one (DV = 1) in a register
  constexpr int kPairs = (DV + 1) / 2;
  using Acc = std::conditional_t<DV == 1, float, uint64_t>;
  Acc acc[4][kPairs] = {};
  float m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = KG > 1 ? -FLT_MAX : -INFINITY, l[i] = 0.f;  // one group's keys may all be at -infinity
  int st = 0;
  if constexpr (KG > 1) __syncthreads();  // the queries
  for (int k0 = group * kKeys; k0 < L; k0 += KG * kKeys, st ^= C::kBufs - 1) {
    if constexpr (KG > 1) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");  // K; V may still be on its way
      group_sync();
    } else {
      if (k0 + kKeys < L) {
        load_tile(k0 + kKeys, st ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
    }
    const float* Kt = Ks + st * C::kTile + tx * C::kPitch;
    const float* Qt = Qs + r0 * C::kPitch;
    // eight chains of DH / 8 channels instead of one of DH (a third of the rounding error of a score), the even and the odd
    // channels of a quarter in one packed multiply-add
    float s[4][4] = {};
#pragma unroll 1
    for (int c0 = 0; c0 < DH; c0 += DH / 4) {
      uint64_t part[4][4] = {};
#pragma unroll 8
      for (int c = c0; c < c0 + DH / 4; c += 4) {
        ulonglong2 a[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(Qt + i * C::kPitch + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const ulonglong2*>(Kt + j * 16 * C::kPitch + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) part[i][j] = tc::fma2(a[i].y, w[j].y, tc::fma2(a[i].x, w[j].x, part[i][j]));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float even, odd;
          tc::unpack2(part[i][j], even, odd);
          s[i][j] += even + odd;
        }
    }
    if (k0 + kKeys > L) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (k0 + tx + 16 * j >= L)
#pragma unroll
          for (int i = 0; i < 4; ++i) s[i][j] = -INFINITY;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float mx = fmaxf(fmaxf(s[i][0], s[i][1]), fmaxf(s[i][2], s[i][3]));
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      const float m_new = fmaxf(m[i], mx);
      const float corr = expf(m[i] - m_new);  // m = -inf on the first tile gives 0
      m[i] = m_new;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = expf(s[i][j] - m_new);
        sum += p;
        Ps[(r0 + i) * C::kPPitch + tx + 16 * j] = p;
      }
      l[i] = l[i] * corr + sum;  // this lane's keys; the sixteen lanes' sums meet at the end
#pragma unroll
      for (int c = 0; c < kPairs; ++c) {
        if constexpr (DV == 1) acc[i][c] *= corr;
        else acc[i][c] = tc::mul2(acc[i][c], tc::pack2(corr, corr));
      }
    }
    if constexpr (KG > 1) {
      group_sync();  // K has been read
      if (k0 + KG * kKeys < L) load_one(Ks, k, k0 + KG * kKeys);
      commit();
      asm volatile("cp.async.wait_group 1;" ::: "memory");  // V
      group_sync();
    } else {
      __syncwarp();  // a row's probabilities are written and read by the same half warp
    }
    // One or two groups with 32 queries: a tile's outputs are summed by themselves and added to the others'.  Chains of 64 keys and one
    // of tiles, instead of one of a group's keys, take a third off the error of an output, so that fewer groups (longer
    // chains) lose nothing against four; a query's registers have no room for it with more threads to an SM.
    [[maybe_unused]] Acc part[4][kPairs] = {};
    Acc(&sum)[4][kPairs] = select_sum<C::kByTile>(acc, part);
    const float* Vt = Vs + st * C::kTile;
#pragma unroll 4
    for (int kk = 0; kk < kKeys; kk += 4) {
      float4 p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4*>(Ps + (r0 + i) * C::kPPitch + kk);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float* vr = Vt + (kk + u) * C::kPitch;
        Acc vv[kPairs];  // channels tx DV .. (DV <= 4), or tx 4 .. and 64 + tx 4 ..
        if constexpr (DV >= 4) {
#pragma unroll
          for (int g = 0; g < DV / 4; ++g) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(vr + g * 64 + tx * 4);
            vv[2 * g] = t.x, vv[2 * g + 1] = t.y;
          }
        } else if constexpr (DV == 2) {
          vv[0] = *reinterpret_cast<const uint64_t*>(vr + tx * 2);
        } else {
          vv[0] = vr[tx];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float pu = u == 0 ? p[i].x : u == 1 ? p[i].y : u == 2 ? p[i].z : p[i].w;
#pragma unroll
          for (int c = 0; c < kPairs; ++c) {
            if constexpr (DV == 1) sum[i][c] = fmaf(pu, vv[c], sum[i][c]);
            else sum[i][c] = tc::fma2(tc::pack2(pu, pu), vv[c], sum[i][c]);
          }
        }
      }
    }
    if constexpr (C::kByTile) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < kPairs; ++c) {
          if constexpr (DV == 1) acc[i][c] += part[i][c];
          else acc[i][c] = tc::add2(acc[i][c], part[i][c]);
        }
    }
    if constexpr (KG > 1) {
      group_sync();  // V and the probabilities have been read
      if (k0 + KG * kKeys < L) load_one(Vs, v, k0 + KG * kKeys);
      commit();
    } else {
      __syncthreads();  // this stage's tiles are overwritten next
    }
  }
  float out[4][2 * kPairs];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < kPairs; ++c) {
      if constexpr (DV == 1) out[i][c] = acc[i][c];
      else tc::unpack2(acc[i][c], out[i][2 * c], out[i][2 * c + 1]);
    }
  if constexpr (KG > 1) {
    // the groups' outputs and sums, to where their tiles were, and from there into one
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // a group without a tile has fetched zeros
    group_sync();
    float* mine = Ks;  // [BQ][DH]
    float* ml = Ps;    // m[BQ], l[BQ]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float sum = l[i];
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, x);
      if (tx == 0) ml[r0 + i] = m[i], ml[BQ + r0 + i] = sum;
#pragma unroll
      for (int c = 0; c < DV; ++c) mine[(r0 + i) * DH + (DV >= 4 ? (c / 4) * 64 + tx * 4 + c % 4 : tx * DV + c)] = out[i][c];
    }
    __syncthreads();
    const float* all = att_smem + BQ * C::kPitch;
    for (int e = threadIdx.x; e < BQ * DH / 4; e += kThreads * KG) {
      const int r = e / (DH / 4), c = (e % (DH / 4)) * 4;
      float M = -INFINITY, sum = 0.f;
#pragma unroll
      for (int g = 0; g < KG; ++g) M = fmaxf(M, all[g * C::kGroup + 2 * C::kBufs * C::kTile + r]);
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int g = 0; g < KG; ++g) {
        const float* p = all + g * C::kGroup;
        const float w = expf(p[2 * C::kBufs * C::kTile + r] - M);  // a group without a tile: 0
        sum = fmaf(w, p[2 * C::kBufs * C::kTile + BQ + r], sum);
        const float4 a = *reinterpret_cast<const float4*>(p + r * DH + c);
        t.x = fmaf(w, a.x, t.x), t.y = fmaf(w, a.y, t.y), t.z = fmaf(w, a.z, t.z), t.w = fmaf(w, a.w, t.w);
      }
      const float inv = 1.f / sum;
      if (q0 + r < L) {
        T* dst = o + base + (size_t)(q0 + r) * row_stride + c;
        from_f32(dst[0], t.x * inv), from_f32(dst[1], t.y * inv), from_f32(dst[2], t.z * inv), from_f32(dst[3], t.w * inv);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float sum = l[i];
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, x);
      const float inv = 1.f / sum;
      if (q0 + r0 + i < L) {
        T* dst = o + base + (size_t)(q0 + r0 + i) * row_stride;
#pragma unroll
        for (int c = 0; c < DV; ++c) from_f32(dst[DV >= 4 ? (c / 4) * 64 + tx * 4 + c % 4 : tx * DV + c], out[i][c] * inv);
      }
    }
  }
}

template <typename T, int DH, int BQ, int KG>
cudaError_t run_one(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, cudaStream_t s) {
  using C = SimtCfg<DH, BQ, KG>;
  static SpreadState state;
  const dim3 grid((L + BQ - 1) / BQ, heads, B);
  count_launch();
  return launch_spread(attention_simt_kernel<T, DH, BQ, KG>, state, false, grid, dim3(BQ * 4 * KG), 0, (int)C::kSmem, s, (const T*)q, (const T*)k, (const T*)v,
                       (T*)o, L, heads, 1.0f / sqrtf((float)DH));
}

template <typename T, int DH>
cudaError_t run(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, cudaStream_t s) {
  // Queries per CTA and groups of warps that share them, timed in all forms on 300 shapes, 32 to 2300 tokens, 0.05 to 27 CTAs of 32
  // queries per SM (us; fp32).  64 queries read K and V half as often: from two CTAs of them per SM on, which fill it.
  auto per_sm = [&](int bq) { return (double)((long long)((L + bq - 1) / bq) * heads * B) / sm_count(); };
  if (per_sm(64) >= 2) return run_one<T, DH, 64, 1>(B, L, heads, q, k, v, o, s);
  if constexpr (DH == 128) {
    // bound by shared-memory reads, and two groups would not have a second K and V: one group, 64 queries where the fullest SM
    // has no more of them so (3 x 300 tokens, 7 heads: 60 with 32, 46 with 64)
    const bool wide = ceil(per_sm(64)) * 64 <= ceil(per_sm(32)) * 32;
    return wide ? run_one<T, DH, 64, 1>(B, L, heads, q, k, v, o, s) : run_one<T, DH, 32, 1>(B, L, heads, q, k, v, o, s);
  } else {
    // Groups hide latencies while an SM has one CTA: four (head_dim 64, 260 tokens: 18.8 with one group, 15.6 with four), or
    // three with 40 queries where 32 would leave one more CTA to some SMs (705 tokens, 0.85 per SM: 59 and 37; 2271 tokens, 1.95
    // per SM: 198, two groups of 32 235; 1986 tokens, 2.7 per SM: 265 and 273, but 343 tokens, 2.8 per SM: 63 and 59; not at head_dim
    // 16, 386 tokens, 1.55 per SM: 23.6, one group of 32 22.2).  With more
    // CTAs two groups (652 tokens, 2.7 of 32 queries per SM: one 92, two 79, four 85).  Below head_dim 64 there is too little to a key tile
    // for that to pay in the long run: two groups for four tiles and two CTAs per SM at most, else one (head_dim 16,
    // 450 tokens, 3.65 per SM: one 30.9, two 31.4, three 37.4).
    if (per_sm(32) <= 1) return run_one<T, DH, 32, 4>(B, L, heads, q, k, v, o, s);
    const bool rounds = (per_sm(32) > 2 && per_sm(40) <= 2) || (L > 1024 && per_sm(32) > 3 && per_sm(40) <= 3);
    if (per_sm(40) <= 1 || (DH > 16 && rounds)) return run_one<T, DH, 40, 3>(B, L, heads, q, k, v, o, s);
    if constexpr (DH < 64)
      if (L > 4 * kKeys || per_sm(32) > 2) return run_one<T, DH, 32, 1>(B, L, heads, q, k, v, o, s);
    return run_one<T, DH, 32, 2>(B, L, heads, q, k, v, o, s);
  }
}

template <typename T>
cudaError_t run_dtype(int B, int L, int heads, int dh, const void* q, const void* k, const void* v, void* o, cudaStream_t s) {
  switch (dh) {
    case 16: return run<T, 16>(B, L, heads, q, k, v, o, s);
    case 32: return run<T, 32>(B, L, heads, q, k, v, o, s);
  }
  if constexpr (sizeof(T) == 4) {  // bf16: on the tensor cores
    if (dh == 64) return run<T, 64>(B, L, heads, q, k, v, o, s);
    if (dh == 128) return run<T, 128>(B, L, heads, q, k, v, o, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_attention_simt(int B, int L, int heads, int dh, bool f32, const void* q, const void* k,
                                  const void* v, void* o, cudaStream_t s) {
  return f32 ? run_dtype<float>(B, L, heads, dh, q, k, v, o, s) : run_dtype<__nv_bfloat16>(B, L, heads, dh, q, k, v, o, s);
}

}  // namespace toma
