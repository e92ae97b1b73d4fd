// FFMA versions of the merge-weight logits, the column softmax / row
// normalisation (Sec. 4.2.1), the merge X_m = A~ X and the unmerge A~^T X'
// (Sec. 4.2.2).  They serve the fp32 mode (whose 1e-4 tolerance rules out
// reduced-precision tensor-core inputs) and every shape the tensor-core kernels do not
// cover.
#include <math.h>

#include "common.cuh"
#include "spread.cuh"
#include "tc.cuh"

namespace toma {

// Four consecutive elements as floats; `vec`: the address is aligned for one load of all four.
__device__ __forceinline__ float4 load4(const float* p, int n, bool vec) {
  if (vec && n >= 4) return *reinterpret_cast<const float4*>(p);
  return make_float4(n > 0 ? p[0] : 0.f, n > 1 ? p[1] : 0.f, n > 2 ? p[2] : 0.f, n > 3 ? p[3] : 0.f);
}
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p, int n, bool vec) {
  if (vec && n >= 4) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u), __uint_as_float(q.y << 16),
                       __uint_as_float(q.y & 0xFFFF0000u));
  }
  return make_float4(n > 0 ? to_f32(p[0]) : 0.f, n > 1 ? to_f32(p[1]) : 0.f, n > 2 ? to_f32(p[2]) : 0.f, n > 3 ? to_f32(p[3]) : 0.f);
}

// Two columns of a row of sums: two floats in a 64-bit register, so that one packed fma (one issue slot) serves both.
struct Sum2f {
  unsigned long long v;
  __device__ __forceinline__ void fma(unsigned long long a2, unsigned long long b2) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(a2), "l"(b2)); }
  __device__ __forceinline__ void get(float* o) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(o[0]), "=f"(o[1]) : "l"(v)); }
};

// C[m][n] = sum_k A(m,k) B(k,n) for one batch entry (blockIdx.z), every sum one chain of fused multiply-adds in
// ascending k (the result does not depend on the tile form).  Tile BM x BN, TM x TN outputs per thread, 16
// contraction steps per stage: the next stage's operands are on their way into registers (16-byte loads along the
// operand's contiguous axis) while the current one is multiplied out of shared memory, two stages deep.  Both
// operands lie there as [k][row], rows swizzled by 8 ((k / 4) % 4), which keeps groups of eight together for the
// 16-byte reads and the transposing stores free of bank conflicts.
// `Op`: a_ptr / b_ptr give the contiguous line of an operand (a row m or n if k runs along it, else a row k).
constexpr int kBK = 16;
template <int kRows>
__device__ __forceinline__ constexpr int swz(int k4) { return 8 * (k4 & 3 & (kRows / 8 - 1)); }

template <class Op, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), BM == 128 ? 2 : 4) simt_gemm_kernel(const Op op) {
  constexpr int kThreads = (BM / TM) * (BN / TN);
  constexpr int kPackA = BM * kBK / 4, kPackB = BN * kBK / 4;  // 4-element packets of a stage
  constexpr int kVecA = (kPackA + kThreads - 1) / kThreads, kVecB = (kPackB + kThreads - 1) / kThreads;
  __shared__ __align__(16) float As[2][kBK][BM];
  __shared__ __align__(16) float Bs[2][kBK][BN];
  const int batch = blockIdx.z, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, tid = threadIdx.x;
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (tid == 0) tc::release_dependents();
  const int tn = tid % (BN / TN) * 4, tm = tid / (BN / TN) * TM;  // columns tn .. + 3, and with TN = 8 BN / 2 further on
  // packet e of an operand: k along the line: line e / 4, k 4 (e % 4); else: k e / (rows / 4), rows 4 (e % (rows / 4))
  float4 ra[kVecA], rb[kVecB];
  typename Op::APtr pa[kVecA];  // lines of an operand with k along them stay the same for the whole sum
  bool ha[kVecA];               // ... and are there
  if (Op::a_k_contig) {
#pragma unroll
    for (int v = 0; v < kVecA; ++v) {
      const int r = m0 + (tid + v * kThreads) / 4;
      ha[v] = r < op.M && tid + v * kThreads < kPackA;
      pa[v] = op.a_ptr(batch, ha[v] ? r : 0);
    }
  }
  auto fetch = [&](int k0) {
#pragma unroll
    for (int v = 0; v < kVecA; ++v) {
      const int e = tid + v * kThreads;
      if (Op::a_k_contig) {
        const int k = k0 + 4 * (e & 3);
        ra[v] = ha[v] ? load4(pa[v] + k, op.K - k, op.a_vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        const int k = k0 + e / (BM / 4), r = m0 + 4 * (e % (BM / 4));
        ra[v] = e < kPackA && k < op.K && r < op.M ? load4(op.a_ptr(batch, k) + r, op.M - r, op.a_vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int v = 0; v < kVecB; ++v) {
      const int e = tid + v * kThreads;
      const int k = k0 + e / (BN / 4), r = n0 + 4 * (e % (BN / 4));
      rb[v] = e < kPackB && k < op.K && r < op.N ? load4(op.b_ptr(batch, k) + r, op.N - r, op.b_vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto put = [&](int st) {
#pragma unroll
    for (int v = 0; v < kVecA; ++v) {
      const int e = tid + v * kThreads;
      if (kPackA % kThreads && e >= kPackA) continue;
      if (Op::a_k_contig) {
        const int r = e / 4, k = 4 * (e & 3), c = r ^ swz<BM>(e & 3);
        As[st][k][c] = ra[v].x;
        As[st][k + 1][c] = ra[v].y;
        As[st][k + 2][c] = ra[v].z;
        As[st][k + 3][c] = ra[v].w;
      } else {
        const int k = e / (BM / 4), r = 4 * (e % (BM / 4));
        *reinterpret_cast<float4*>(&As[st][k][r ^ swz<BM>(k >> 2)]) = ra[v];
      }
    }
#pragma unroll
    for (int v = 0; v < kVecB; ++v) {
      const int e = tid + v * kThreads;
      if (kPackB % kThreads && e >= kPackB) continue;
      const int k = e / (BN / 4), r = 4 * (e % (BN / 4));
      *reinterpret_cast<float4*>(&Bs[st][k][r ^ swz<BN>(k >> 2)]) = rb[v];
    }
  };
  Sum2f acc[TM][TN / 2] = {};
  fetch(0);
  put(0);
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < op.K; k0 += kBK, st ^= 1) {
    const bool more = k0 + kBK < op.K;
    if (more) fetch(k0 + kBK);
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      float4 a[TM / 4];
      ulonglong2 b[TN / 4];
#pragma unroll
      for (int u = 0; u < TM / 4; ++u) a[u] = *reinterpret_cast<const float4*>(&As[st][k][(tm + 4 * u) ^ swz<BM>(k >> 2)]);
#pragma unroll
      for (int u = 0; u < TN / 4; ++u) b[u] = *reinterpret_cast<const ulonglong2*>(&Bs[st][k][(tn + u * (BN / 2)) ^ swz<BN>(k >> 2)]);
#pragma unroll
      for (int u = 0; u < TM / 4; ++u) {
        const float av[4] = {a[u].x, a[u].y, a[u].z, a[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          unsigned long long a2;
          asm("mov.b64 %0, {%1, %1};" : "=l"(a2) : "f"(av[e]));
#pragma unroll
          for (int q = 0; q < TN / 4; ++q) {
            acc[4 * u + e][2 * q].fma(a2, b[q].x);
            acc[4 * u + e][2 * q + 1].fma(a2, b[q].y);
          }
        }
      }
    }
    if (more) {
      put(st ^ 1);  // last read before the previous barrier
      __syncthreads();
    }
  }
#pragma unroll
  for (int u = 0; u < TM; ++u) {
    const int m = m0 + tm + u;
    if (m >= op.M) break;
#pragma unroll
    for (int q = 0; q < TN / 4; ++q) {
      const int n = n0 + tn + q * (BN / 2);
      float v[4];
      acc[u][2 * q].get(v);
      acc[u][2 * q + 1].get(v + 2);
      if (n < op.N) op.store4(batch, m, n, op.N - n, v);
    }
  }
}

// Four consecutive outputs of a row, `n` of them real.
template <typename T>
__device__ __forceinline__ void put4(T* p, int n, bool vec, const float (&v)[4]) {
  if (vec && n >= 4) {
    if constexpr (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      __align__(8) __nv_bfloat16 h[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) from_f32(h[e], v[e]);
      *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(h);
    }
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < n) from_f32(p[e], v[e]);
  }
}

struct TileMap {
  int P, tiles_x, th, tw, W, Nloc, Dloc, d, n_all, Lm;
  __device__ __forceinline__ size_t x_row(int batch, int l) const {  // row of X for tile-local slot l
    const int b = batch / P, p = batch - b * P;
    return (size_t)b * n_all + tile_token(p, l, tiles_x, th, tw, W);
  }
  __device__ __forceinline__ size_t m_row(int batch, int i) const {  // row of the merged tensor
    const int b = batch / P, p = batch - b * P;
    return (size_t)b * Lm + (size_t)p * Dloc + i;
  }
};

// Stored weights A~^T of one tile: fp32 mode keeps one fp32 plane [N_loc][D_loc]; bf16 mode keeps
// the value split into two bf16 planes, hi = bf16(v) and lo = bf16(v - hi), hi plane first, so that
// the tensor-core kernels can feed both planes as bf16 operands and still carry ~16 mantissa bits.
__device__ __forceinline__ float w_load(const float* w, int batch, size_t off, size_t plane) {
  return w[(size_t)batch * plane + off];
}
__device__ __forceinline__ float w_load(const __nv_bfloat16* w, int batch, size_t off, size_t plane) {
  const __nv_bfloat16* t = w + (size_t)batch * 2 * plane;
  return __bfloat162float(t[off]) + __bfloat162float(t[plane + off]);
}
__device__ __forceinline__ void w_store(float* w, int batch, size_t off, size_t plane, float v) {
  w[(size_t)batch * plane + off] = v;
}
__device__ __forceinline__ void w_store(__nv_bfloat16* w, int batch, size_t off, size_t plane, float v) {
  __nv_bfloat16* t = w + (size_t)batch * 2 * plane;
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  t[off] = hi;
  t[plane + off] = __float2bfloat16_rn(v - __bfloat162float(hi));
}

static TileMap make_map(const Geom& g) {
  return TileMap{g.P, g.tiles_x, g.th, g.tw, g.W, g.Nloc, g.Dloc, g.d, (int)g.tokens_all(), g.Lm};
}

// Stored weights A~^T as an operand: the fp32 plane, or the sum of the two bf16 planes.
struct SplitW {
  const __nv_bfloat16* hi;
  size_t plane;
  __device__ __forceinline__ SplitW operator+(int e) const { return SplitW{hi + e, plane}; }
};
__device__ __forceinline__ float4 load4(const SplitW& p, int n, bool) {
  float v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = e < n ? to_f32(p.hi[e]) + to_f32(p.hi[p.plane + e]) : 0.f;
  return make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ const float* w_line(const float* w, int batch, size_t off, size_t plane) { return w + batch * plane + off; }
__device__ __forceinline__ SplitW w_line(const __nv_bfloat16* w, int batch, size_t off, size_t plane) {
  return SplitW{w + batch * 2 * plane + off, plane};
}
template <typename WT> struct WLine { typedef const float* Ptr; };
template <> struct WLine<__nv_bfloat16> { typedef SplitW Ptr; };

// logits[batch][i][k] = <X[idx_i], X_k> * scale
template <typename T>
struct LogitsOp {
  int M, N, K;
  TileMap tm;
  const T* x;
  const int32_t* idx;
  float* logits;
  float scale;
  __device__ __forceinline__ const T* a_ptr(int batch, int i) const { return x + tm.x_row(batch, idx[(size_t)batch * tm.Dloc + i]) * tm.d; }
  __device__ __forceinline__ const T* b_ptr(int batch, int k) const { return x + tm.x_row(batch, k) * tm.d; }
};

// xm[m_row(i)][c] = sum_k w[batch][k][i] x[x_row(k)][c]
template <typename T, typename WT>
struct MergeOp {
  static constexpr bool a_k_contig = false;
  typedef typename WLine<WT>::Ptr APtr;
  int M, N, K;
  bool a_vec, b_vec;
  TileMap tm;
  const WT* w;
  const T* x;
  T* xm;
  __device__ __forceinline__ APtr a_ptr(int batch, int k) const { return w_line(w, batch, (size_t)k * tm.Dloc, (size_t)tm.Nloc * tm.Dloc); }
  __device__ __forceinline__ const T* b_ptr(int batch, int k) const { return x + tm.x_row(batch, k) * tm.d; }
  __device__ __forceinline__ void store4(int batch, int i, int c, int n, const float* v) const {
    const float f[4] = {v[0], v[1], v[2], v[3]};
    put4(xm + tm.m_row(batch, i) * tm.d + c, n, true, f);
  }
};

// out[x_row(k)][c] = sum_i w[batch][k][i] y[m_row(i)][c]
template <typename T, typename WT>
struct UnmergeOp {
  static constexpr bool a_k_contig = true;
  typedef typename WLine<WT>::Ptr APtr;
  int M, N, K;
  bool a_vec, b_vec;
  TileMap tm;
  const WT* w;
  const T* y;
  T* out;
  __device__ __forceinline__ APtr a_ptr(int batch, int k) const { return w_line(w, batch, (size_t)k * tm.Dloc, (size_t)tm.Nloc * tm.Dloc); }
  __device__ __forceinline__ const T* b_ptr(int batch, int i) const { return y + tm.m_row(batch, i) * tm.d; }
  __device__ __forceinline__ void store4(int batch, int k, int c, int n, const float* v) const {
    const float f[4] = {v[0], v[1], v[2], v[3]};
    put4(out + tm.x_row(batch, k) * tm.d + c, n, true, f);
  }
};

template <class Op, int BM, int BN, int TM, int TN>
static void run_tile(const Op& op, int batches, cudaStream_t s) {
  const dim3 grid((op.N + BN - 1) / BN, (op.M + BM - 1) / BM, batches);
  static SpreadState state;
  count_launch();
  launch_spread(simt_gemm_kernel<Op, BM, BN, TM, TN>, state, true, grid, dim3((BM / TM) * (BN / TN)), 2 * kBK * (BM + BN) * 4, 0, s, op);  // errors: cudaGetLastError
}

// Tile form: the least work on the fullest SM, padding included.  A larger tile reads its operands less often per
// multiply-add (rel: its measured rate per SM against the 128 x 128 form once eight warps or more are resident); with
// fewer warps an SM cannot hide its latencies and runs in proportion slower.
struct TileForm {
  int bm, bn, warps;
  double rel;
};
static int pick_form(const TileForm* f, int n, int M, int N, int batches) {
  int best = 0;
  double best_cost = 0.0;
  for (int i = 0; i < n; ++i) {
    const double ctas = (double)((M + f[i].bm - 1) / f[i].bm) * ((N + f[i].bn - 1) / f[i].bn) * batches;
    const double per_sm = ceil(ctas / sm_count()), warps = per_sm * f[i].warps;
    const double cost = per_sm * f[i].bm * f[i].bn / f[i].rel * (warps < 8 ? 8 / warps : 1.0);
    if (i == 0 || cost < best_cost) best = i, best_cost = cost;
  }
  return best;
}

template <class Op>
static void run_gemm(const Op& op, int batches, cudaStream_t s) {
  static constexpr TileForm forms[] = {{128, 128, 8, 1.0}, {64, 64, 4, 0.85}, {32, 64, 4, 0.6}};
  switch (pick_form(forms, 3, op.M, op.N, batches)) {
    case 0: run_tile<Op, 128, 128, 8, 8>(op, batches, s); break;
    case 1: run_tile<Op, 64, 64, 4, 8>(op, batches, s); break;
    default: run_tile<Op, 32, 64, 4, 4>(op, batches, s);
  }
}

// Softmax over the destination axis for every source token (a token's shares sum to 1); logits[batch][i][k] is
// overwritten with A_ik.  A CTA takes 32 source tokens: maxima and exponentials by all its threads (eight rows of 128
// bytes at a time), the denominator of a token by one thread in destination order, out of shared memory.
constexpr int kSoftTok = 32, kSoftThreads = 512;
__global__ void __launch_bounds__(kSoftThreads) softmax_dest_kernel(float* __restrict__ logits, int Nloc, int Dloc) {
  extern __shared__ float e_smem[];  // [D_loc][32] exponentials
  __shared__ float red[kSoftThreads / 32][kSoftTok];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = blockIdx.x * kSoftTok + lane;
  constexpr int kWarps = kSoftThreads / 32;
  const bool live = k < Nloc;
  tc::dependency_wait();
  if (threadIdx.x == 0) tc::release_dependents();
  float* L = logits + (size_t)blockIdx.y * Dloc * Nloc + (live ? k : 0);
  float mx = -INFINITY;
#pragma unroll 8
  for (int i = warp; i < Dloc; i += kWarps) {
    const float v = L[(size_t)i * Nloc];
    e_smem[i * kSoftTok + lane] = v;
    mx = fmaxf(mx, v);
  }
  red[warp][lane] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) mx = fmaxf(mx, red[w][lane]);
#pragma unroll 4
  for (int i = warp; i < Dloc; i += kWarps) e_smem[i * kSoftTok + lane] = expf(e_smem[i * kSoftTok + lane] - mx);
  __syncthreads();
  if (warp == 0) {
    float sum = 0.f;
#pragma unroll 16
    for (int i = 0; i < Dloc; ++i) sum += e_smem[i * kSoftTok + lane];
    red[0][lane] = 1.f / sum;
  }
  __syncthreads();
  const float inv = red[0][lane];
  if (live) {
#pragma unroll 4
    for (int i = warp; i < Dloc; i += kWarps) L[(size_t)i * Nloc] = e_smem[i * kSoftTok + lane] * inv;
  }
}
// The same for more destinations than shared memory holds (global merge): the exponentials stay where the logits were.  The same
// sums in the same order.  (One thread per source token took three passes of its own over them: a millisecond of latencies in
// 30 to 90 CTAs, whose time depended on where a dependent launch had placed them - 2 x 4416 tokens of 256 channels, the weights
// as a whole 1407 us launched by itself, 1615 behind its predecessor; 3528 tokens of 640 channels 1461 and 1200.)
__global__ void __launch_bounds__(kSoftThreads) softmax_dest_long_kernel(float* __restrict__ logits, int Nloc, int Dloc) {
  __shared__ float red[kSoftThreads / 32][kSoftTok];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = blockIdx.x * kSoftTok + lane;
  constexpr int kWarps = kSoftThreads / 32;
  const bool live = k < Nloc;
  tc::dependency_wait();
  if (threadIdx.x == 0) tc::release_dependents();
  float* L = logits + (size_t)blockIdx.y * Dloc * Nloc + (live ? k : 0);
  float mx = -INFINITY;
#pragma unroll 8
  for (int i = warp; i < Dloc; i += kWarps) mx = fmaxf(mx, L[(size_t)i * Nloc]);
  red[warp][lane] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) mx = fmaxf(mx, red[w][lane]);
  if (live) {
#pragma unroll 8
    for (int i = warp; i < Dloc; i += kWarps) L[(size_t)i * Nloc] = expf(L[(size_t)i * Nloc] - mx);
  }
  __syncthreads();  // the block's exponentials are in memory, and red has been read
  if (warp == 0 && live) {
    float sum = 0.f;
    int i = 0;
    for (; i + 32 <= Dloc; i += 32) {  // 32 loads on their way, added up in destination order
      float e[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) e[u] = L[(size_t)(i + u) * Nloc];
#pragma unroll
      for (int u = 0; u < 32; ++u) sum += e[u];
    }
    for (; i < Dloc; ++i) sum += L[(size_t)i * Nloc];
    red[0][lane] = 1.f / sum;
  }
  __syncthreads();
  const float inv = red[0][lane];
  if (live) {
#pragma unroll 8
    for (int i = warp; i < Dloc; i += kWarps) L[(size_t)i * Nloc] *= inv;
  }
}

// Row normalisation of 32 destinations of a region: A~^T[k][i] = A_ik / sum_k' A_ik' and, when wu is given, the shares
// themselves, A^T[k][i] = A_ik, in the same layout.  A row's sum is a warp's (32 strided partial sums, then a tree); the
// planes are written through a 32 x 32 transpose in shared memory, so that consecutive lanes write consecutive weights.
template <typename WT>
__global__ void __launch_bounds__(256) rownorm_kernel(const float* __restrict__ A, WT* __restrict__ w, WT* __restrict__ wu,
                                                      int Nloc, int Dloc) {
  __shared__ float inv[32];
  __shared__ float tr[8][32][33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int batch = blockIdx.y, i0 = blockIdx.x * 32;
  const int ni = min(32, Dloc - i0);
  tc::dependency_wait();
  if (threadIdx.x == 0) tc::release_dependents();
  const float* a = A + ((size_t)batch * Dloc + i0) * Nloc;
  {  // a warp's four rows side by side
    const int r0 = warp * 4;
    float z[4] = {};
#pragma unroll 4
    for (int k = lane; k < Nloc; k += 32)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r0 + u < ni) z[u] += a[(size_t)(r0 + u) * Nloc + k];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z[u] += __shfl_xor_sync(0xffffffffu, z[u], o);
      if (lane == 0 && r0 + u < ni) inv[r0 + u] = z[u] > 0.f ? 1.f / z[u] : 0.f;
    }
  }
  __syncthreads();
  const size_t plane = (size_t)Nloc * Dloc;
  for (int k0 = (blockIdx.z * 8 + warp) * 32; k0 < Nloc; k0 += gridDim.z * 256) {
    const int nk = min(32, Nloc - k0);
#pragma unroll
    for (int r = 0; r < 32; ++r) tr[warp][lane][r] = r < ni && lane < nk ? a[(size_t)r * Nloc + k0 + lane] : 0.f;
    __syncwarp();
    if (lane < ni) {
      const float f = inv[lane];
#pragma unroll 8
      for (int k = 0; k < nk; ++k) {
        const float v = tr[warp][k][lane];
        const size_t off = (size_t)(k0 + k) * Dloc + i0 + lane;
        w_store(w, batch, off, plane, v * f);
        if (wu) w_store(wu, batch, off, plane, v);
      }
    }
    __syncwarp();
  }
}

// Logits of bf16 tokens, <X[idx_i], X_k> * scale, every sum one chain of fused multiply-adds in ascending channels, whatever the
// tile form.  What bounds it is the FMA pipe (a product is 2 N_loc D_loc d operations of the
// 75 TFLOP/s it has) as long as operands keep coming, and those of the general kernel above, which made them once, did not: its stages of 16 channels, one
// ahead, cover a third of a load's latency, and it converts and transposes them on the way.  Here the rows travel as they
// are, by cp.async, kStages - 1 stages of 64 channels ahead, and are widened in registers as they are read (a shift or a mask,
// on the ALU pipe beside the FMAs).  Rows lie 144 bytes apart, so that eight threads read eight rows' 16 bytes at once.
// Thread = TM x TN outputs, rows tm + u BM / TM and columns tn + u BN / TN.  Logits, softmax and normalisation of 384 regions of
// 96 tokens of 1280 channels 355 -> 163 us, of 32 of 252 tokens of 640 channels 92 -> 55, of 3 of 126 tokens 53 -> 18.
constexpr int kLogitK = 64, kLogitPitch = kLogitK * 2 + 16;
template <int BM, int BN>
constexpr int logit_stages() { return BM + BN > 64 ? 4 : 6; }
template <int BM, int BN>
constexpr int logit_smem() { return logit_stages<BM, BN>() * (BM + BN) * kLogitPitch + (BM + BN) * 8; }

__device__ __forceinline__ void cp_async16(uint32_t smem, const void* src, bool real) {  // zeros where nothing is read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem), "l"(src), "r"(real ? 16 : 0) : "memory");
}

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN)) logits_kernel(const LogitsOp<__nv_bfloat16> op) {
  constexpr int kStages = logit_stages<BM, BN>(), kRows = BM + BN, kStageBytes = kRows * kLogitPitch;
  constexpr int kGm = BM / TM, kGn = BN / TN, kThreads = kGm * kGn, kPackets = kRows * 8 / kThreads;
  static_assert(kRows * 8 % kThreads == 0, "tile form");
  extern __shared__ __align__(16) uint8_t logit_smem_raw[];
  const __nv_bfloat16** row = reinterpret_cast<const __nv_bfloat16**>(logit_smem_raw + kStages * kStageBytes);
  const int tid = threadIdx.x, batch = blockIdx.z, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int tn = tid % kGn, tm = tid / kGn;
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (tid == 0) tc::release_dependents();
  for (int e = tid; e < kRows; e += kThreads) {
    const int i = e < BM ? m0 + e : n0 + e - BM;
    row[e] = i < (e < BM ? op.M : op.N) ? (e < BM ? op.a_ptr(batch, i) : op.b_ptr(batch, i)) : nullptr;
  }
  __syncthreads();
  const uint32_t base = tc::smem_u32(logit_smem_raw);
  const int nk = (op.K + kLogitK - 1) / kLogitK;
  auto fetch = [&](int ks) {
    if (ks < nk) {
#pragma unroll
      for (int v = 0; v < kPackets; ++v) {
        const int e = tid + v * kThreads, r = e >> 3, c = ks * kLogitK + (e & 7) * 8;
        const __nv_bfloat16* p = row[r];
        const bool real = p != nullptr && c < op.K;
        cp_async16(base + (ks % kStages) * kStageBytes + r * kLogitPitch + (e & 7) * 16, real ? p + c : op.x, real);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  Sum2f acc[TM][TN / 2] = {};
#pragma unroll 1
  for (int ks = 0; ks < kStages - 1; ++ks) fetch(ks);
#pragma unroll 1
  for (int ks = 0; ks < nk; ++ks) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();         // stage ks is there for all, stage ks - 1 read by all
    fetch(ks + kStages - 1);
    const uint8_t* st = logit_smem_raw + (ks % kStages) * kStageBytes;
#pragma unroll 2
    for (int c = 0; c < 8; ++c) {
      uint4 a[TM], b[TN];
#pragma unroll
      for (int u = 0; u < TM; ++u) a[u] = *reinterpret_cast<const uint4*>(st + (tm + u * kGm) * kLogitPitch + c * 16);
#pragma unroll
      for (int u = 0; u < TN; ++u) b[u] = *reinterpret_cast<const uint4*>(st + (BM + tn + u * kGn) * kLogitPitch + c * 16);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        auto wide = [&](const uint4& q) {
          const uint32_t h = (e >> 1) == 0 ? q.x : (e >> 1) == 1 ? q.y : (e >> 1) == 2 ? q.z : q.w;
          return __uint_as_float(e & 1 ? h & 0xFFFF0000u : h << 16);
        };
        uint64_t b2[TN / 2];
#pragma unroll
        for (int u = 0; u < TN / 2; ++u) b2[u] = tc::pack2(wide(b[2 * u]), wide(b[2 * u + 1]));
#pragma unroll
        for (int u = 0; u < TM; ++u) {
          const float av = wide(a[u]);
          const uint64_t a2 = tc::pack2(av, av);
#pragma unroll
          for (int q = 0; q < TN / 2; ++q) acc[u][q].fma(a2, b2[q]);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < TM; ++u) {
    const int m = m0 + tm + u * kGm;
    if (m >= op.M) break;
    float* dst = op.logits + ((size_t)batch * op.M + m) * op.N;
#pragma unroll
    for (int q = 0; q < TN / 2; ++q) {
      float v[2];
      acc[u][q].get(v);
      const int n = n0 + tn + 2 * q * kGn;
      if (n < op.N) dst[n] = v[0] * op.scale;
      if (n + kGn < op.N) dst[n + kGn] = v[1] * op.scale;
    }
  }
}

template <int BM, int BN, int TM, int TN>
static cudaError_t run_logits(const LogitsOp<__nv_bfloat16>& op, int batches, cudaStream_t s) {
  static SpreadState state;
  const dim3 grid((op.N + BN - 1) / BN, (op.M + BM - 1) / BM, batches);
  count_launch();
  return launch_spread(logits_kernel<BM, BN, TM, TN>, state, false, grid, dim3((BM / TM) * (BN / TN)), 0, logit_smem<BM, BN>(), s, op);
}
// The same of fp32 tokens, summed in double: one chain with 64 x 64 tiles, eight with 16 x 16, so that a logit within some
// 2^-50 of the middle between two fp32 numbers may round either way with the form, which depends on the number of regions.  Their way into double
// is the bound where there is enough to do (eight conversions, at a quarter of the rate, for sixteen multiply-adds); few and
// small regions wait for loads instead, and so KG groups of threads share a tile, each with every KG-th four channels of a
// stage of 32, and add up through shared memory at the end.  Thread = 4 x 4 outputs.
constexpr int kLogit64K = 32, kLogit64Pitch = kLogit64K * 4 + 16;
template <int BM, int BN>
constexpr int logit64_stages() { return BM + BN > 32 ? 4 : 8; }
template <int BM, int BN, int KG>
constexpr int logit64_smem() {
  constexpr int ring = logit64_stages<BM, BN>() * (BM + BN) * kLogit64Pitch, parts = (KG - 1) * BM * BN * 8;
  return (ring > parts ? ring : parts) + (BM + BN) * 8;
}

template <int BM, int BN, int KG>
__global__ void __launch_bounds__(BM / 4 * (BN / 4) * KG) logits64_kernel(const LogitsOp<float> op) {
  constexpr int kStages = logit64_stages<BM, BN>(), kRows = BM + BN, kStageBytes = kRows * kLogit64Pitch;
  constexpr int kGm = BM / 4, kGn = BN / 4, kGroup = kGm * kGn, kThreads = kGroup * KG, kPackets = kRows * 8 / kThreads;
  static_assert(kRows * 8 % kThreads == 0 && 8 % KG == 0, "tile form");
  extern __shared__ __align__(16) uint8_t logit_smem_raw[];
  const float** row = reinterpret_cast<const float**>(logit_smem_raw + logit64_smem<BM, BN, KG>() - kRows * 8);
  const int tid = threadIdx.x, batch = blockIdx.z, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int in_group = tid % kGroup, kg = tid / kGroup, tn = in_group % kGn, tm = in_group / kGn;
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (tid == 0) tc::release_dependents();
  for (int e = tid; e < kRows; e += kThreads) {
    const int i = e < BM ? m0 + e : n0 + e - BM;
    row[e] = i < (e < BM ? op.M : op.N) ? (e < BM ? op.a_ptr(batch, i) : op.b_ptr(batch, i)) : nullptr;
  }
  __syncthreads();
  const uint32_t base = tc::smem_u32(logit_smem_raw);
  const int nk = (op.K + kLogit64K - 1) / kLogit64K;
  auto fetch = [&](int ks) {
    if (ks < nk) {
#pragma unroll
      for (int v = 0; v < kPackets; ++v) {
        const int e = tid + v * kThreads, r = e >> 3, c = ks * kLogit64K + (e & 7) * 4;
        const float* p = row[r];
        const bool real = p != nullptr && c < op.K;
        cp_async16(base + (ks % kStages) * kStageBytes + r * kLogit64Pitch + (e & 7) * 16, real ? p + c : op.x, real);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  double acc[4][4] = {};
#pragma unroll 1
  for (int ks = 0; ks < kStages - 1; ++ks) fetch(ks);
#pragma unroll 1
  for (int ks = 0; ks < nk; ++ks) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();         // stage ks is there for all, stage ks - 1 read by all
    fetch(ks + kStages - 1);
    const uint8_t* st = logit_smem_raw + (ks % kStages) * kStageBytes;
#pragma unroll 1
    for (int c = kg; c < 8; c += KG) {
      float4 a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = *reinterpret_cast<const float4*>(st + (tm + u * kGm) * kLogit64Pitch + c * 16);
#pragma unroll
      for (int u = 0; u < 4; ++u) b[u] = *reinterpret_cast<const float4*>(st + (BM + tn + u * kGn) * kLogit64Pitch + c * 16);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        auto wide = [&](const float4& q) { return (double)(e == 0 ? q.x : e == 1 ? q.y : e == 2 ? q.z : q.w); };
        double bd[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) bd[u] = wide(b[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double ad = wide(a[u]);
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[u][q] = fma(ad, bd[q], acc[u][q]);
        }
      }
    }
  }
  if constexpr (KG > 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the last stages have been read
    double* part = reinterpret_cast<double*>(logit_smem_raw);  // [KG - 1][16][kGroup]
    if (kg > 0) {
#pragma unroll
      for (int e = 0; e < 16; ++e) part[((kg - 1) * 16 + e) * kGroup + in_group] = acc[e >> 2][e & 3];
    }
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int e = 0; e < 16; ++e)
#pragma unroll
      for (int g = 0; g < KG - 1; ++g) acc[e >> 2][e & 3] += part[(g * 16 + e) * kGroup + in_group];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int m = m0 + tm + u * kGm;
    if (m >= op.M) break;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = n0 + tn + q * kGn;
      if (n < op.N) op.logits[((size_t)batch * op.M + m) * op.N + n] = (float)(acc[u][q] * (double)op.scale);
    }
  }
}

template <int BM, int BN, int KG>
static cudaError_t run_logits64(const LogitsOp<float>& op, int batches, cudaStream_t s) {
  static SpreadState state;
  const dim3 grid((op.N + BN - 1) / BN, (op.M + BM - 1) / BM, batches);
  count_launch();
  return launch_spread(logits64_kernel<BM, BN, KG>, state, false, grid, dim3(BM / 4 * (BN / 4) * KG), 0, logit64_smem<BM, BN, KG>(), s, op);
}
// Timed on thirteen shapes (microseconds per tile and 640 channels on the fullest SM): 16 x 16 takes 3.2 among many; 64 x 64
// takes 44, one or two of them 90, and wins where every SM has several.  The weights as a whole (with logits in stages of 16
// channels, one ahead, before): 16 regions of 64 tokens, 640 channels 27 -> 15 us, of 256 tokens 100 -> 65, 256 of those 769
// -> 698.  32 x 32 in four groups was between the two, and 4 % better than both at 4 regions of 1024 tokens.
static cudaError_t launch_logits64(const LogitsOp<float>& op, int batches, cudaStream_t s) {
  auto on_an_sm = [&](int b) {
    const long long ctas = (long long)((op.M + b - 1) / b) * ((op.N + b - 1) / b) * batches;
    return (double)((ctas + sm_count() - 1) / sm_count());
  };
  return fmax(90.0, 44.0 * on_an_sm(64)) < 3.2 * on_an_sm(16) ? run_logits64<64, 64, 1>(op, batches, s) : run_logits64<16, 16, 8>(op, batches, s);
}
// The form that is through first.  Timed on thirteen shapes (microseconds per tile and 640 channels on the fullest SM): 64 x 64
// takes 18 while an SM has few of them and 14.5 among many; 64 x 32 by 64 threads takes 8, but 18 where there is nothing
// beside it; 32 x 32 by 128 threads 5.3, alone as well.
static cudaError_t launch_logits(const LogitsOp<__nv_bfloat16>& op, int batches, cudaStream_t s) {
  auto on_an_sm = [&](int bm, int bn) {
    const long long ctas = (long long)((op.M + bm - 1) / bm) * ((op.N + bn - 1) / bn) * batches;
    return (double)((ctas + sm_count() - 1) / sm_count());
  };
  const double n = on_an_sm(64, 64), large = n * (n > 4 ? 14.5 : 18.0), tall = fmax(18.0, 8.0 * on_an_sm(64, 32)), small = 5.3 * on_an_sm(32, 32);
  if (large <= tall && large <= small) return run_logits<64, 64, 4, 8>(op, batches, s);
  return tall <= small ? run_logits<64, 32, 4, 8>(op, batches, s) : run_logits<32, 32, 2, 4>(op, batches, s);
}

cudaError_t launch_weights_simt(const Geom& g, const void* x, const int32_t* idx, void* w, void* wu, float* logits,
                                cudaStream_t s) {
  const int batches = g.B * g.P;
  cudaError_t e;
  if (g.f32) {  // fp32 mode sums the logits in double: a logit of some hundreds has to be right to its last fp32 bit
    LogitsOp<float> op{g.Dloc, g.Nloc, g.d, make_map(g), (const float*)x, idx, logits, g.logit_scale};
    if ((e = launch_logits64(op, batches, s)) != cudaSuccess) return e;
  } else {
    LogitsOp<__nv_bfloat16> op{g.Dloc, g.Nloc, g.d, make_map(g), (const __nv_bfloat16*)x, idx, logits, g.logit_scale};
    if ((e = launch_logits(op, batches, s)) != cudaSuccess) return e;
  }
  const size_t smem = (size_t)g.Dloc * kSoftTok * 4;
  if (smem <= 200 * 1024) {
    static SpreadState state;
    e = launch_spread(softmax_dest_kernel, state, false, dim3((g.Nloc + kSoftTok - 1) / kSoftTok, batches), dim3(kSoftThreads), kSoftThreads * 4, (int)smem, s, logits,
                      g.Nloc, g.Dloc);
  } else {
    static SpreadState state;
    e = launch_spread(softmax_dest_long_kernel, state, false, dim3((g.Nloc + kSoftTok - 1) / kSoftTok, batches), dim3(kSoftThreads), kSoftThreads * 4, 0, s,
                      logits, g.Nloc, g.Dloc);
  }
  if (e != cudaSuccess) return e;
  count_launch();
  // a CTA per 32 destinations, their source tokens split further where that leaves SMs idle (each part sums the rows anew)
  const int blocks = (g.Dloc + 31) / 32;
  int row_parts = 1;
  while (row_parts < 8 && (long long)blocks * batches * row_parts < sm_count() && row_parts * 256 < g.Nloc) row_parts *= 2;
  const dim3 grid(blocks, batches, row_parts);
  // (Not spread: what counts is that its CTAs are there when the softmax ends.  21 regions of 264 tokens, 1536 channels: 100 us for the
  // weights as a whole, 137 spread.)
  e = g.f32 ? launch_dependent(rownorm_kernel<float>, grid, dim3(256), 0, s, logits, (float*)w, (float*)wu, g.Nloc, g.Dloc)
            : launch_dependent(rownorm_kernel<__nv_bfloat16>, grid, dim3(256), 0, s, logits, (__nv_bfloat16*)w, (__nv_bfloat16*)wu, g.Nloc, g.Dloc);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Copy of the un-merged trailing tokens (rows [src_row0, src_row0 + n_extra) of every batch item).
template <typename T>
__global__ void copy_rows_kernel(const T* __restrict__ src, T* __restrict__ dst, int n_extra, int d, size_t src_stride,
                                 size_t dst_stride, size_t src_row0, size_t dst_row0) {
  const size_t per = (size_t)n_extra * d;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= per) return;
  const int b = blockIdx.y;
  dst[(size_t)b * dst_stride + dst_row0 * d + e] = src[(size_t)b * src_stride + src_row0 * d + e];
}

// Rows of bf16 packets (the tensor-core kernels' text tokens), where too few threads of theirs would copy them.
__global__ void __launch_bounds__(256) copy_packets_kernel(const RowCopy c) {
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (threadIdx.x == 0) tc::release_dependents();
  copy_part(c, (size_t)blockIdx.x * 256 + threadIdx.x, (size_t)gridDim.x * 256);
}
cudaError_t launch_copy_rows(const RowCopy& c, cudaStream_t s) {
  const size_t want = (c.per + 4 * 256 - 1) / (4 * 256), most = (size_t)sm_count() * 8;  // four packets per thread, a full chip at most
  const cudaError_t e = launch_dependent(copy_packets_kernel, dim3((unsigned)(want < most ? want : most)), dim3(256), 0, s, c);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
static void copy_extra(const Geom& g, const T* src, T* dst, bool merging, cudaStream_t s) {
  if (g.n_extra == 0) return;
  const size_t per = (size_t)g.n_extra * g.d;
  const size_t full = (size_t)g.tokens_all() * g.d, mrg = (size_t)g.Lm * g.d;
  dim3 grid((unsigned)((per + 255) / 256), g.B);
  if (merging)
    copy_rows_kernel<T><<<grid, 256, 0, s>>>(src, dst, g.n_extra, g.d, full, mrg, (size_t)g.N, (size_t)g.D);
  else
    copy_rows_kernel<T><<<grid, 256, 0, s>>>(src, dst, g.n_extra, g.d, mrg, full, (size_t)g.D, (size_t)g.N);
  count_launch();
}

cudaError_t launch_merge_simt(const Geom& g, const void* w, const void* x, void* xm, cudaStream_t s) {
  const int batches = g.B * g.P;
  if (g.f32) {
    MergeOp<float, float> op{g.Dloc, g.d, g.Nloc, g.Dloc % 4 == 0, true, make_map(g), (const float*)w, (const float*)x, (float*)xm};
    run_gemm<MergeOp<float, float>>(op, batches, s);
    copy_extra<float>(g, (const float*)x, (float*)xm, true, s);
  } else {
    MergeOp<__nv_bfloat16, __nv_bfloat16> op{g.Dloc, g.d, g.Nloc, false, true, make_map(g), (const __nv_bfloat16*)w, (const __nv_bfloat16*)x,
                                      (__nv_bfloat16*)xm};
    run_gemm<MergeOp<__nv_bfloat16, __nv_bfloat16>>(op, batches, s);
    copy_extra<__nv_bfloat16>(g, (const __nv_bfloat16*)x, (__nv_bfloat16*)xm, true, s);
  }
  return cudaGetLastError();
}

cudaError_t launch_unmerge_simt(const Geom& g, const void* w, const void* y, void* out, cudaStream_t s) {
  const int batches = g.B * g.P;
  if (g.f32) {
    UnmergeOp<float, float> op{g.Nloc, g.d, g.Dloc, g.Dloc % 4 == 0, true, make_map(g), (const float*)w, (const float*)y, (float*)out};
    run_gemm<UnmergeOp<float, float>>(op, batches, s);
    copy_extra<float>(g, (const float*)y, (float*)out, false, s);
  } else {
    UnmergeOp<__nv_bfloat16, __nv_bfloat16> op{g.Nloc, g.d, g.Dloc, false, true, make_map(g), (const __nv_bfloat16*)w, (const __nv_bfloat16*)y,
                                        (__nv_bfloat16*)out};
    run_gemm<UnmergeOp<__nv_bfloat16, __nv_bfloat16>>(op, batches, s);
    copy_extra<__nv_bfloat16>(g, (const __nv_bfloat16*)y, (__nv_bfloat16*)out, false, s);
  }
  return cudaGetLastError();
}

// c[m][n] = sum_k a[m][k] w[k][n] (plain projection; fp32 mode and shapes the tensor-core kernel does not take).
template <typename T>
struct LinearOp {
  static constexpr bool a_k_contig = true;
  typedef const T* APtr;
  int M, N, K;
  bool a_vec, b_vec;
  const T* a_;
  const T* w_;
  T* c_;
  int act;
  __device__ __forceinline__ const T* a_ptr(int, int m) const { return a_ + (size_t)m * K; }
  __device__ __forceinline__ const T* b_ptr(int, int k) const { return w_ + (size_t)k * N; }
  __device__ __forceinline__ void store4(int, int m, int n, int left, const float* v) const {
    float f[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) f[e] = act == kActGelu ? gelu(v[e]) : v[e];
    put4(c_ + (size_t)m * N + n, left, N % 4 == 0, f);
  }
};

cudaError_t launch_linear_simt(int M, int N, int K, bool f32, const void* a, const void* w, void* c, int act, cudaStream_t s) {
  if (f32) {
    LinearOp<float> op{M, N, K, K % 4 == 0, N % 4 == 0, (const float*)a, (const float*)w, (float*)c, act};
    run_gemm<LinearOp<float>>(op, 1, s);
  } else {
    LinearOp<__nv_bfloat16> op{M, N, K, K % 4 == 0, N % 4 == 0, (const __nv_bfloat16*)a, (const __nv_bfloat16*)w, (__nv_bfloat16*)c, act};
    run_gemm<LinearOp<__nv_bfloat16>>(op, 1, s);
  }
  return cudaGetLastError();
}

// gidx[b][p * D_loc + k] = image token of tile p's k-th pick.
__global__ void global_idx_kernel(const int32_t* __restrict__ idx, int32_t* __restrict__ gidx, int P, int Dloc, int tiles_x,
                                  int th, int tw, int W, int total) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (threadIdx.x == 0) tc::release_dependents();
  if (e >= total) return;
  const int p = (e / Dloc) % P;
  gidx[e] = tile_token(p, idx[e], tiles_x, th, tw, W);
}

cudaError_t launch_global_idx(const Geom& g, const int32_t* idx, int32_t* gidx, cudaStream_t s) {
  const int total = g.B * g.D;
  count_launch();
  return launch_dependent(global_idx_kernel, dim3((total + 255) / 256), dim3(256), 0, s, idx, gidx, g.P, g.Dloc, g.tiles_x, g.th, g.tw, g.W, total);
}

// Dense fp32 A~ [batch][P][D_loc][N_loc]  <->  stored A~^T [batch][P][N_loc][D_loc].
template <typename WT, bool kExport>
__global__ void weights_convert_kernel(WT* __restrict__ w, float* __restrict__ dense, int Nloc, int Dloc, size_t total) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const size_t per = (size_t)Nloc * Dloc;
  const size_t batch = e / per, r = e - batch * per;
  const int k = (int)(r / Dloc), i = (int)(r - (size_t)k * Dloc);
  float* dp = dense + batch * per + (size_t)i * Nloc + k;
  if (kExport) *dp = w_load(w, (int)batch, r, per); else w_store(w, (int)batch, r, per, *dp);
}

cudaError_t launch_weights_export(const Geom& g, const void* w, float* dense, cudaStream_t s) {
  const size_t total = (size_t)g.B * g.P * g.Nloc * g.Dloc;
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if (g.f32) weights_convert_kernel<float, true><<<blocks, 256, 0, s>>>((float*)w, dense, g.Nloc, g.Dloc, total);
  else weights_convert_kernel<__nv_bfloat16, true><<<blocks, 256, 0, s>>>((__nv_bfloat16*)w, dense, g.Nloc, g.Dloc, total);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_weights_import(const Geom& g, const float* dense, void* w, cudaStream_t s) {
  const size_t total = (size_t)g.B * g.P * g.Nloc * g.Dloc;
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if (g.f32) weights_convert_kernel<float, false><<<blocks, 256, 0, s>>>((float*)w, (float*)dense, g.Nloc, g.Dloc, total);
  else weights_convert_kernel<__nv_bfloat16, false><<<blocks, 256, 0, s>>>((__nv_bfloat16*)w, (float*)dense, g.Nloc, g.Dloc, total);
  count_launch();
  return cudaGetLastError();
}

}  // namespace toma
