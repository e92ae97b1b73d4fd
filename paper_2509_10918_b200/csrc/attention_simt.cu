// FFMA attention core softmax(Q K^T / sqrt(dh)) V (Eq. 1 with tau = 1) with an
// online softmax.  Used for the fp32 mode and for head sizes the tensor-core
// kernel does not cover.
//
// A CTA takes 32 or 64 queries of a head and walks the keys 64 at a time, K and V double buffered in shared memory
// (16-byte asynchronous copies).  Sixteen lanes share four query rows: a thread computes 4 x 4 scores (keys tx, tx + 16,
// tx + 32, tx + 48, whose rows of DH + 4 floats fall into different banks) and 4 x DH / 16 outputs, four contraction
// steps per 16-byte shared read, so that 64 multiply-adds go with eight reads.  Scores become probabilities in
// registers (row maxima and sums by shuffles within the sixteen lanes) and pass through shared memory once, between
// lanes of one half warp.  Bound by the FMA pipe; 10 heads x 512 tokens x 64 channels, fp32: 159 us with one thread
// per query and quarter row before.
#include "common.cuh"

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

template <int DH, int BQ>
struct SimtCfg {
  static constexpr int kPitch = DH + 4;
  static constexpr int kTile = kKeys * kPitch;
  static constexpr int kPPitch = kKeys + 4;
  static constexpr size_t kSmem = ((size_t)BQ * kPitch + 4 * kTile + (size_t)BQ * kPPitch) * 4;
};

template <typename T, int DH, int BQ>
__global__ void __launch_bounds__(BQ * 4) attention_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                                                T* __restrict__ o, int L, int heads, float scale) {
  using C = SimtCfg<DH, BQ>;
  constexpr int kThreads = BQ * 4, DV = DH / 16;
  extern __shared__ __align__(16) float att_smem[];
  float* Qs = att_smem;                  // [BQ][pitch], scaled
  float* Ks = Qs + BQ * C::kPitch;       // [2][64][pitch]
  float* Vs = Ks + 2 * C::kTile;         // [2][64][pitch]
  float* Ps = Vs + 2 * C::kTile;         // [BQ][64 + 4]
  const int b = blockIdx.z, h = blockIdx.y, q0 = blockIdx.x * BQ, tid = threadIdx.x;
  const int tx = tid & 15, r0 = (tid >> 4) * 4;
  const size_t row_stride = (size_t)heads * DH;
  const size_t base = (size_t)b * L * row_stride + (size_t)h * DH;
  auto load_tile = [&](int k0, int st) {
#pragma unroll 4
    for (int e = tid; e < kKeys * (DH / 4); e += kThreads) {
      const int r = e / (DH / 4), c = (e % (DH / 4)) * 4;
      const bool in = k0 + r < L;
      const size_t off = base + (size_t)(in ? k0 + r : 0) * row_stride + c;
      copy16(Ks + st * C::kTile + r * C::kPitch + c, k + off, in);
      copy16(Vs + st * C::kTile + r * C::kPitch + c, v + off, in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  load_tile(0, 0);
  for (int e = tid; e < BQ * DH; e += kThreads) {
    const int r = e / DH, c = e % DH;
    Qs[r * C::kPitch + c] = q0 + r < L ? to_f32(q[base + (size_t)(q0 + r) * row_stride + c]) * scale : 0.f;
  }
  float acc[4][DV] = {}, m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = -INFINITY, l[i] = 0.f;
  int st = 0;
  for (int k0 = 0; k0 < L; k0 += kKeys, st ^= 1) {
    if (k0 + kKeys < L) {
      load_tile(k0 + kKeys, st ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* Kt = Ks + st * C::kTile + tx * C::kPitch;
    const float* Qt = Qs + r0 * C::kPitch;
    // four chains of DH / 4 channels instead of one of DH: half the rounding error of a score
    float s[4][4] = {};
#pragma unroll 1
    for (int c0 = 0; c0 < DH; c0 += DH / 4) {
      float part[4][4] = {};
#pragma unroll 4
      for (int c = c0; c < c0 + DH / 4; c += 4) {
        float4 a[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(Qt + i * C::kPitch + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4*>(Kt + j * 16 * C::kPitch + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            part[i][j] = fmaf(a[i].w, w[j].w, fmaf(a[i].z, w[j].z, fmaf(a[i].y, w[j].y, fmaf(a[i].x, w[j].x, part[i][j]))));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] += part[i][j];
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
      for (int c = 0; c < DV; ++c) acc[i][c] *= corr;
    }
    __syncwarp();  // a row's probabilities are written and read by the same half warp
    const float* Vt = Vs + st * C::kTile;
#pragma unroll 2
    for (int kk = 0; kk < kKeys; kk += 4) {
      float4 p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4*>(Ps + (r0 + i) * C::kPPitch + kk);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float* vr = Vt + (kk + u) * C::kPitch;
        float vv[DV];  // channels tx DV .. (DV <= 4), or tx 4 .. and 64 + tx 4 ..
        if constexpr (DV >= 4) {
#pragma unroll
          for (int g = 0; g < DV / 4; ++g) {
            const float4 t = *reinterpret_cast<const float4*>(vr + g * 64 + tx * 4);
            vv[4 * g] = t.x; vv[4 * g + 1] = t.y; vv[4 * g + 2] = t.z; vv[4 * g + 3] = t.w;
          }
        } else {
#pragma unroll
          for (int c = 0; c < DV; ++c) vv[c] = vr[tx * DV + c];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float pu = u == 0 ? p[i].x : u == 1 ? p[i].y : u == 2 ? p[i].z : p[i].w;
#pragma unroll
          for (int c = 0; c < DV; ++c) acc[i][c] = fmaf(pu, vv[c], acc[i][c]);
        }
      }
    }
    __syncthreads();  // this stage's tiles are overwritten next
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float sum = l[i];
#pragma unroll
    for (int x = 8; x > 0; x >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, x);
    const float inv = 1.f / sum;
    if (q0 + r0 + i < L) {
      T* dst = o + base + (size_t)(q0 + r0 + i) * row_stride;
#pragma unroll
      for (int c = 0; c < DV; ++c) from_f32(dst[DV >= 4 ? (c / 4) * 64 + tx * 4 + c % 4 : tx * DV + c], acc[i][c] * inv);
    }
  }
}

template <typename T, int DH, int BQ>
cudaError_t run_one(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, cudaStream_t s) {
  static std::atomic<unsigned long long> raised{0};
  if (cudaError_t e = raise_dynamic_smem(attention_simt_kernel<T, DH, BQ>, (int)SimtCfg<DH, BQ>::kSmem, raised); e != cudaSuccess) return e;
  const dim3 grid((L + BQ - 1) / BQ, heads, B);
  attention_simt_kernel<T, DH, BQ><<<grid, BQ * 4, SimtCfg<DH, BQ>::kSmem, s>>>((const T*)q, (const T*)k, (const T*)v, (T*)o, L, heads,
                                                                              1.0f / sqrtf((float)DH));
  count_launch();
  return cudaGetLastError();
}

template <typename T, int DH>
cudaError_t run(int B, int L, int heads, const void* q, const void* k, const void* v, void* o, cudaStream_t s) {
  // 64 queries per CTA read K and V half as often; 32 while that would not give every SM two CTAs
  const long long ctas64 = (long long)((L + 63) / 64) * heads * B;
  return ctas64 >= 2LL * sm_count() ? run_one<T, DH, 64>(B, L, heads, q, k, v, o, s) : run_one<T, DH, 32>(B, L, heads, q, k, v, o, s);
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
