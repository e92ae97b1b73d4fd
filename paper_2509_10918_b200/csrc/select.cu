// Destination selection (Sec. 4.1, Algorithm 2): token quantisation and the greedy
// facility-location argmax with exact incremental integer gains (the fixed-point Gram
// matrix between the two is gram_tc.cu's).
#include "common.cuh"
#include "greedy.cuh"
#include "tc.cuh"

namespace toma {

// ---------------------------------------------------------------------------
// Quantise: one warp per image token.  y = bf16(rint(x * 0.99*4096/|x|) * 2^-12)
// written tile-major: row (b*P + p)*N_loc + l.  Defined in fp64 (the squares added up per lane in channel order, then by
// the tree below; scale, product and rounding), so that the CPU definition can be matched bit for bit.
// The fp64 pipe and its conversions bounded this kernel (4 x 16384 tokens of 640 channels: 65 us, where reading and writing
// them takes 26; now 49).  bf16 tokens therefore get their squares' sum from the same fp64 additions, but of doubles put together
// from the bits, and the products as pairs of floats: x * scale = hi + lo to about 2^-45 of it, and what is not within 2^-20
// of the middle between two integers rounds as the fp64 product does.  A token with a channel that is (one in four
// hundred of 640 to 3072 normally distributed channels), or with a norm far from 1, is done again in fp64.
// ---------------------------------------------------------------------------
// Eight consecutive elements as floats (16-byte aligned source).
__device__ __forceinline__ void widen8(const uint4& raw, float (&v)[8]) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    v[2 * e] = __uint_as_float(w[e] << 16);
    v[2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) { widen8(*reinterpret_cast<const uint4*>(p), v); }
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&k)[8]) {  // k: integers of up to 13 bits
  __align__(16) __nv_bfloat162 q[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) q[e] = __floats2bfloat162_rn(k[2 * e] * (1.0f / 4096.0f), k[2 * e + 1] * (1.0f / 4096.0f));
  *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(q);
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// The definition, eight channels (16 or 32 contiguous bytes) per lane and trip; dim is a multiple of 8.
template <typename T>
__device__ __forceinline__ void quantise_f64(const T* row, __nv_bfloat16* out, int d, int lane) {
  double ss = 0.0;
  for (int c = lane * 8; c < d; c += 256) {
    float v[8];
    load8(row + c, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) ss += (double)v[e] * (double)v[e];
  }
  const double scale = kCosScaleTimesOne / fmax(sqrt(warp_sum(ss)), 1e-30);
  for (int c = lane * 8; c < d; c += 256) {  // second read of the row: an L1/L2 hit
    float v[8];
    load8(row + c, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = (float)rint((double)v[e] * scale);
    store8(out + c, v);
  }
}
// A bf16 value (as a float's bits) as the same double; 2^-127 or so instead of zero and of denormals.
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = __float_as_uint(v);
  return __hiloint2double((int)(((b & 0x7FFFFFFFu) >> 3) + 0x38000000u), 0);  // without the sign: it is squared
}
// kTrips > 0: the warp's trips over the token's channels, all on their way before the first is used and kept in registers for
// the products.  0: one at a time, read twice.  False: not this way.  (quantise_kernel, kTrips < 0: never this way.)
template <int kTrips>
__device__ __forceinline__ bool quantise_fast(const __nv_bfloat16* row, __nv_bfloat16* out, int d, int lane) {
  double ss = 0.0;
  auto add_squares = [&](const uint4& raw) {
    float v[8];
    widen8(raw, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const double x = widen(v[e]);
      ss = fma(x, x, ss);  // the square is exact
    }
  };
  float s_hi, s_lo, off = 0.f;  // the scale; largest distance from an integer
  auto set_scale = [&] {
    ss = warp_sum(ss);
    // no infinities, no sum that 2^-254 for a zero could change, no scale whose parts leave the range of floats
    if (!(ss > 1e-40 && ss < 1e40)) return false;
    const double scale = kCosScaleTimesOne / sqrt(ss);
    s_hi = (float)scale, s_lo = (float)(scale - (double)s_hi);
    return true;
  };
  auto write = [&](const uint4& raw, int c) {
    float v[8];
    widen8(raw, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      // rounded one by one whatever the compiler would fuse: lo is what the product p has lost (p - k of the unrounded product
      // would count it twice, 2^-13 at most, and let wrong roundings pass)
      const float p = __fmul_rn(v[e], s_hi);
      const float lo = fmaf(v[e], s_lo, fmaf(v[e], s_hi, -p));
      const float k = __fsub_rn(__fadd_rn(p, 12582912.f), 12582912.f);  // |p| <= 4056: the nearest integer
      off = fmaxf(off, fabsf(__fadd_rn(__fsub_rn(p, k), lo)));
      v[e] = k;
    }
    store8(out + c, v);
  };
  auto at = [&](int c) { return *reinterpret_cast<const uint4*>(row + c); };
  if constexpr (kTrips > 0) {
    uint4 raw[kTrips];
#pragma unroll
    for (int t = 0; t < kTrips; ++t)
      if (t * 256 + lane * 8 < d) raw[t] = at(t * 256 + lane * 8);
#pragma unroll
    for (int t = 0; t < kTrips; ++t)
      if (t * 256 + lane * 8 < d) add_squares(raw[t]);
    if (!set_scale()) return false;
#pragma unroll
    for (int t = 0; t < kTrips; ++t)
      if (t * 256 + lane * 8 < d) write(raw[t], t * 256 + lane * 8);
  } else {
    for (int c = lane * 8; c < d; c += 256) add_squares(at(c));
    if (!set_scale()) return false;
    for (int c = lane * 8; c < d; c += 256) write(at(c), c);  // second read of the row: an L1/L2 hit
  }
  return !__any_sync(0xffffffffu, off > 0.5f - 0x1p-20f);
}

template <typename T, int kTrips>
__global__ void __launch_bounds__(256) quantise_kernel(const T* __restrict__ x, __nv_bfloat16* __restrict__ y, int B,
                                                       int N, int n_all, int d, int W, int th, int tw, int tiles_x,
                                                       int P, int Nloc) {
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (threadIdx.x == 0) tc::release_dependents();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= B * N) return;
  const int b = warp / N, n = warp - b * N;
  const int yy = n / W, xx = n - yy * W;
  const int p = (yy / th) * tiles_x + xx / tw;
  const int l = (yy % th) * tw + xx % tw;
  const T* row = x + ((size_t)b * n_all + n) * d;
  __nv_bfloat16* out = y + ((size_t)(b * P + p) * Nloc + l) * d;
  if constexpr (sizeof(T) == 2 && kTrips >= 0) {
    if (quantise_fast<kTrips>(row, out, d, lane)) return;
  }
  quantise_f64(row, out, d, lane);
}

cudaError_t launch_quantise(const Geom& g, const void* x, __nv_bfloat16* y, cudaStream_t s) {
  const long long warps = (long long)g.B * g.N;
  const int blocks = (int)((warps * 32 + 255) / 256);
  auto launch = [&](auto kernel, auto* tokens) {
    return launch_dependent(kernel, dim3(blocks), dim3(256), 0, s, tokens, y, g.B, g.N, (int)g.tokens_all(), g.d, g.W, g.th, g.tw, g.tiles_x, g.P, g.Nloc);
  };
  // Channels kept in registers: 4096 tokens of 3072 channels 6 us less, 2 x 4096 of 640 1.5 less.  Where a warp runs once, the long
  // straight code of more than four trips costs more than that gains (2048 tokens of 1280 channels: 1 us), and where an SM has
  // one CTA the fp64 pipe is not the bound and the definition's short code is through first (selection of 1024 tokens of 1088
  // channels 21.5 us, 22.3 by floats; of 672 of 1280 17.1 and 17.7; of 2048 of 1280 24.4 and 24.1).
  const __nv_bfloat16* h = (const __nv_bfloat16*)x;
  const bool few = warps <= 8LL * sm_count(), once = warps <= 16LL * sm_count();
  static_assert(kMaxDim <= 16 * 256, "sixteen trips hold a token's channels");
  const cudaError_t e = g.f32 ? launch(quantise_kernel<float, -1>, (const float*)x)
                        : few ? launch(quantise_kernel<__nv_bfloat16, -1>, h)
                        : g.d <= 1024 ? launch(quantise_kernel<__nv_bfloat16, 4>, h)
                        : once ? launch(quantise_kernel<__nv_bfloat16, 0>, h)
                        : g.d <= 2048 ? launch(quantise_kernel<__nv_bfloat16, 8>, h) : launch(quantise_kernel<__nv_bfloat16, 16>, h);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Greedy (Algorithm 2), one CTA per tile; the rounds are greedy.cuh's.  The two passes over the whole matrix (row
// sums for the first pick, initial gains) run on all warps with 16-byte reads; then the warps that own tokens
// (64 each) go on.  kSmem: the matrix is copied to shared memory during the first pass (up to 336 tokens), which
// turns the two dependent reads of a round from an L2 round trip into a shared-memory latency.
// Measured against one pick per round and one thread per token (kernel time, launch included): 32 tiles of 256
// tokens with 128 destinations 72.8 -> 50.8 us, 256 such tiles 140 -> 94 us, 64 tiles of 1024 tokens with 512
// destinations 1783 -> 695 us (there the rows come from L2 and DRAM, 32 of them in flight per thread; with 8 it
// was 837 us).
// ---------------------------------------------------------------------------
constexpr int kGreedyThreads = 512;  // at most
constexpr int kGreedySmemTok = 336;  // 336 x 336 entries and the lists below fill an SM's shared memory

template <bool kOne, bool kSmem>
__global__ void __launch_bounds__(kOne ? 64 : kGreedyThreads, 1) greedy_kernel(const uint16_t* __restrict__ sq, int32_t* __restrict__ idx, int Nloc,
                                                                int Dloc) {
  constexpr int kTok = kOne ? 64 : kSmem ? kGreedySmemTok : kMaxNloc;
  extern __shared__ __align__(16) uint32_t greedy_smem[];
  __shared__ greedy::Shared<kTok> sh;
  __shared__ int total[kTok];  // row sums (biased alike), then initial gains + msum
  __shared__ int msum;
  __shared__ int2 best[16];
  const int threads = blockDim.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int pitch = sq_pitch(Nloc), vecs = pitch / 8;  // 16-byte packets per row
  const uint4* src = reinterpret_cast<const uint4*>(sq + (size_t)blockIdx.x * Nloc * pitch);
  for (int e = tid; e < kTok; e += threads) total[e] = 0;
  if (tid == 0) msum = 0;
  tc::dependency_wait();  // launched with programmatic stream serialisation
  if (tid == 0) tc::release_dependents();
  __syncthreads();
  const int v = tid % vecs, n_rg = threads / vecs, rg = tid / vecs;  // this thread's packet of a row, and its rows
  const uint4* S4 = kSmem ? reinterpret_cast<const uint4*>(greedy_smem) : src;
  int acc[8];
  auto add8 = [&](const uint32_t (&t)[4]) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      acc[2 * w] += (int)(t[w] & 0xFFFFu);
      acc[2 * w + 1] += (int)(t[w] >> 16);
    }
  };
  auto post8 = [&] {
    if (rg < n_rg)
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (8 * v + c < Nloc) atomicAdd(&total[8 * v + c], acc[c]);
  };
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = 0;
  if (rg < n_rg)
    for (int r0 = rg; r0 < Nloc; r0 += 8 * n_rg) {
      uint4 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = r0 + u * n_rg < Nloc ? src[(size_t)(r0 + u * n_rg) * vecs + v] : make_uint4(0u, 0u, 0u, 0u);
      uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (kSmem && r0 + u * n_rg < Nloc) reinterpret_cast<uint4*>(greedy_smem)[(r0 + u * n_rg) * vecs + v] = q[u];
        t[0] += q[u].x; t[1] += q[u].y; t[2] += q[u].z; t[3] += q[u].w;  // eight entries below 2^13 per half: no carry
      }
      add8(t);
    }
  post8();
  __syncthreads();

  // ---- first pick: the largest row sum, the lowest index on ties
  {
    int s = -1, i = kMaxNloc;
    for (int e = tid; e < Nloc; e += threads)
      if (total[e] > s) s = total[e], i = e;
    const int bs = __reduce_max_sync(0xffffffffu, s);
    const int bi = __reduce_min_sync(0xffffffffu, s == bs ? i : kMaxNloc);
    if (lane == 0) best[warp] = make_int2(bs, bi);
  }
  __syncthreads();
  int first;
  {
    const int2 b = lane < threads / 32 ? best[lane] : make_int2(-1, kMaxNloc);
    const int bs = __reduce_max_sync(0xffffffffu, b.x);
    first = __reduce_min_sync(0xffffffffu, b.x == bs ? b.y : kMaxNloc);
  }
  for (int e = tid; e < kTok; e += threads) total[e] = 0;
  __syncthreads();

  // ---- initial gains: g_i = sum_j max(S[j][i], m_j) - sum_j m_j with m = the first pick's row
  const uint16_t* mrow = reinterpret_cast<const uint16_t*>(S4 + (size_t)first * vecs);
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = 0;
  if (rg < n_rg)
    for (int r0 = rg; r0 < Nloc; r0 += 8 * n_rg) {
      uint4 q[8];
      uint32_t mj[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = r0 + u * n_rg < Nloc;
        q[u] = in ? S4[(size_t)(r0 + u * n_rg) * vecs + v] : make_uint4(0u, 0u, 0u, 0u);
        mj[u] = in ? mrow[r0 + u * n_rg] * 0x10001u : 0u;
      }
      uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        t[0] += greedy::max_u16x2(q[u].x, mj[u]);
        t[1] += greedy::max_u16x2(q[u].y, mj[u]);
        t[2] += greedy::max_u16x2(q[u].z, mj[u]);
        t[3] += greedy::max_u16x2(q[u].w, mj[u]);
      }
      add8(t);
    }
  post8();
  {
    int ms = 0;
    for (int e = tid; e < Nloc; e += threads) ms += mrow[e];
    ms = __reduce_add_sync(0xffffffffu, ms);
    if (lane == 0 && ms) atomicAdd(&msum, ms);
  }
  __syncthreads();

  const int n_warps = kOne ? 1 : (Nloc + 63) / 64;
  if (warp >= n_warps) return;
  int32_t* out = idx + (size_t)blockIdx.x * Dloc;
  if (tid == 0) out[0] = first;
  const int j0 = 2 * tid;
  greedy::rounds<kOne, !kSmem, kTok>(reinterpret_cast<const uint32_t*>(S4), pitch / 2, Nloc, Dloc, n_warps, tid, first,
                                     j0 < Nloc ? (uint32_t)(total[j0] - msum) : 0u, j0 + 1 < Nloc ? (uint32_t)(total[j0 + 1] - msum) : 0u, sh, out);
}

template <bool kOne, bool kSmem>
static cudaError_t run_greedy(const Geom& g, const uint16_t* sq, int32_t* idx, cudaStream_t s) {
  const size_t smem = kSmem ? (size_t)g.Nloc * sq_pitch(g.Nloc) * 2 : 0;
  static std::atomic<unsigned long long> raised{0};
  if (kSmem)
    if (cudaError_t e = raise_dynamic_smem(greedy_kernel<kOne, kSmem>, kOne ? 64 * 64 * 2 : kGreedySmemTok * kGreedySmemTok * 2, raised); e != cudaSuccess)
      return e;
  // A region's threads: enough for its two passes over the matrix, few enough that many small regions share an SM (with 512
  // for every size selection of 408 regions of 64 tokens took 53 us and takes 34, of 644 regions of 16 tokens 33 and 16).
  const int threads = g.Nloc <= 64 ? 64 : g.Nloc <= 128 ? 128 : g.Nloc <= 192 ? 256 : kGreedyThreads;
  // Rows in global memory, and few threads in no more regions than there are SMs: not launched before the predecessor ends.
  // CTAs placed then are spread over the chip, those placed beside the predecessor's last ones crowd where there is room
  // first, and share the paths to L2 that bound the rounds (64 tiles of 1024 tokens: 600 us against 543 us), or an SM's
  // issue slots (144 of 128 tokens: 90 us against 60).
  if (!kSmem || (threads < kGreedyThreads && g.B * g.P <= sm_count())) {
    greedy_kernel<kOne, kSmem><<<g.B * g.P, threads, smem, s>>>(sq, idx, g.Nloc, g.Dloc);
    return cudaGetLastError();
  }
  return launch_dependent(greedy_kernel<kOne, kSmem>, dim3(g.B * g.P), dim3(threads), smem, s, sq, idx, g.Nloc, g.Dloc);
}

cudaError_t launch_greedy(const Geom& g, const uint16_t* sq, int32_t* idx, cudaStream_t s) {
  const cudaError_t e = g.Nloc <= 64               ? run_greedy<true, true>(g, sq, idx, s)
                        : g.Nloc <= kGreedySmemTok ? run_greedy<false, true>(g, sq, idx, s)
                                                   : run_greedy<false, false>(g, sq, idx, s);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace toma
