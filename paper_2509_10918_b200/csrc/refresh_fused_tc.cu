// Destination selection and merge weights of a 64-token tile in one kernel (Sec. 4.1, Algorithm 2 and
// Sec. 4.2.1), for the refresh steps of the small-tile block: instead of a Gram kernel, a greedy kernel, a
// gather and a weights kernel - four launches of a few microseconds of work each - one CTA per tile
//   1. streams the tile's quantised tokens y and its raw tokens x (64-channel slabs, TMA ring) through one
//      Gram product of all 128 on the tensor cores: S = y y^T (exact in fp32: every partial sum is a multiple of 2^-24
//      below 1) and G = x x^T are 64 x 64 each of its accumulator.  (Two products of 64 rows, with 64 more that are not
//      there, read 12 KB of shared memory per 16 channels where this one reads 8, and took 5.7 us of 20 for 1280 channels.)
//   2. rounds S to the fixed-point S_q in shared memory and runs the greedy rounds on it in ONE warp (two
//      candidates and two cached maxima per lane, no block barrier; several picks per round: greedy.cuh);
//   3. takes the logits of Sec. 4.2.1 out of G - the logit of source k and destination i is G[idx_i][k] scaled,
//      so no second contraction and no gathered copy of the destinations is needed -, softmax over the
//      destinations per source, row sums per destination in a fixed order, and writes A~^T as hi and lo planes.
// The quantised tokens come from quantise_kernel (fp64 arithmetic over 148 SMs; one CTA per tile would take
// longer over it than the kernel takes as a whole).
// Warp 2: TMA producer; warp 3: MMA issuer.  Then warps 0, 1: thread = token = tensor-memory lane of S (warp 0 runs the greedy
// rounds); warps 2, 3: the same of G; all four write the weights.
#include "common.cuh"
#include "greedy.cuh"
#include "tc.cuh"

namespace toma {

using namespace tc;

namespace {

constexpr int kTok = 64;            // tokens per tile this kernel is written for
constexpr int kSlab = kTok * 128;   // one 64-channel slab of 64 tokens
constexpr int kStageBytes = 2 * kSlab;  // y slab, then x slab
constexpr int kRing = 8;            // stages: 128 KB in flight per CTA (few CTAs: bytes in flight are what counts)
constexpr int kPitch = kTok + 1;    // fp32 row pitch of G and of the shares in shared memory (conflict-free both ways)

struct RBars {
  uint64_t full[kRing], empty[kRing], done;
  uint32_t tmem_base;
  int abort_flag;
};

struct RParams {
  int P, tiles_x, th, tw, d, Dloc;
  float scale_log2;  // log2(e) / (tau * sqrt(d))
  int32_t* idx;      // [tile][D_loc]
  __nv_bfloat16* w;  // A~^T planes: [tile][hi, lo][64 tokens][D_loc]
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Algorithm 2 on a 64 x 64 S_q (biased, two tokens to a word) in shared memory, by one warp; the rounds are
// greedy.cuh's.  Lane l owns tokens 2 l and 2 l + 1.
__device__ __forceinline__ void greedy_one_warp(const uint32_t* S, int Dloc, int lane, greedy::Shared<kTok>& sh, int* sel, int32_t* out) {
  constexpr int kPitchW = kTok / 2;
  uint32_t sum0 = 0, sum1 = 0;
#pragma unroll
  for (int j0 = 0; j0 < kTok; j0 += 8) {
    uint32_t t = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) t += S[(j0 + u) * kPitchW + lane];  // eight entries below 2^13 per half: no carry
    sum0 += t & 0xFFFFu;
    sum1 += t >> 16;
  }
  // first pick: the largest column sum, lowest index on ties
  const uint32_t first_key = __reduce_max_sync(0xffffffffu, max(greedy::make_key(sum0, 2 * lane), greedy::make_key(sum1, 2 * lane + 1)));
  const int first = greedy::key_index(first_key);
  const uint16_t* mrow = reinterpret_cast<const uint16_t*>(S + first * kPitchW);
  uint32_t g0 = 0, g1 = 0, ms = 0;
#pragma unroll
  for (int j0 = 0; j0 < kTok; j0 += 8) {
    uint32_t t = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t mj = mrow[j0 + u];
      ms += mj;
      t += greedy::max_u16x2(S[(j0 + u) * kPitchW + lane], mj * 0x10001u);
    }
    g0 += t & 0xFFFFu;
    g1 += t >> 16;
  }
  if (lane == 0) sel[0] = first;
  greedy::rounds<true, false, kTok>(S, kPitchW, kTok, Dloc, 1, lane, first, g0 - ms, g1 - ms, sh, sel);
  __syncwarp();
  for (int r = lane; r < Dloc; r += 32) out[r] = sel[r];
}

__device__ __forceinline__ void rows_sync() { asm volatile("bar.sync 1, 64;" ::: "memory"); }  // warps 0 and 1

__global__ void __launch_bounds__(128, 1)
refresh_small_kernel(const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_x, const RParams p,
                     uint32_t* dev_status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* ring = smem;
  uint16_t* S = reinterpret_cast<uint16_t*>(ring + kRing * kStageBytes);        // [64][64]
  float* G = reinterpret_cast<float*>(S + kTok * kTok);                         // [64][kPitch]
  float* A = G + kTok * kPitch;                                                 // shares [D_loc][kPitch]
  float* zinv = A + kTok * kPitch;                                              // [64]
  int* sel = reinterpret_cast<int*>(zinv + kTok);                               // [64]
  greedy::Shared<kTok>* lists = reinterpret_cast<greedy::Shared<kTok>*>(sel + kTok);
  RBars* bar = reinterpret_cast<RBars*>(lists + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile_b = blockIdx.x, b = tile_b / p.P, tile = tile_b - b * p.P;
  const int ty = tile / p.tiles_x, tx = tile - ty * p.tiles_x;
  const int nk = p.d / 64;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&bar->full[s], 1);
      mbar_init(&bar->empty[s], 1);
    }
    mbar_init(&bar->done, 1);
    bar->abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&tm_y);
    prefetch_tmap(&tm_x);
  }
  dependency_wait();  // before tensor memory is held and before any global access
  if (threadIdx.x == 0) release_dependents();
  if (warp == 3) tmem_alloc(&bar->tmem_base, 128);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int* abort_flag = &bar->abort_flag;

  if (warp == 2) {
    if (elect_one()) {
      for (int k = 0; k < nk; ++k) {
        const int s = k % kRing;
        if (k >= kRing && !mbar_wait(&bar->empty[s], ((k / kRing) - 1) & 1, dev_status, abort_flag)) break;
        uint8_t* st = ring + s * kStageBytes;
        mbar_expect_tx(&bar->full[s], kStageBytes);
        tma_load_3d(st, &tm_y, &bar->full[s], k * 64, 0, tile_b);
        tma_load_4d(st + kSlab, &tm_x, &bar->full[s], k * 64, tx * p.tw, ty * p.th, b);
      }
    }
  } else if (warp == 3) {
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_f16(kFmtBF16, kFmtBF16, false, false, 2 * kTok, 2 * kTok);
      bool ok = true;
      for (int k = 0; k < nk; ++k) {
        const int s = k % kRing;
        if (!mbar_wait(&bar->full[s], (k / kRing) & 1, dev_status, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t ya = smem_u32(ring + s * kStageBytes);  // 64 rows of y, 64 of x
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {  // 16 channels per MMA
          const uint64_t yd = smem_desc_sw128(ya + kk * 32, 16, 1024);
          mma_ss(tmem, yd, yd, idesc, k > 0 || kk > 0);
        }
        mma_commit(&bar->empty[s]);
      }
      if (ok) mma_commit(&bar->done);
    }
  }
  __syncwarp();
  const int r = threadIdx.x & (kTok - 1);  // token; threadIdx.x = its tensor-memory lane
  if (mbar_wait_warp(&bar->done, 0, dev_status, abort_flag)) {
    tc_fence_after();
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (warp < 2 ? 0 : kTok);
#pragma unroll
    for (int c0 = 0; c0 < kTok; c0 += 32) {
      uint32_t v[32];
      tmem_ld32(taddr + c0, v);
      tmem_wait_ld();
      if (warp < 2) {  // S_q[r][c] = rint(<y_r, y_c> * 4096), the diagonal by definition
#pragma unroll
        for (int e = 0; e < 32; ++e)
          S[(c0 + e) * kTok + r] = (uint16_t)((c0 + e == r ? kDiagQ : __float2int_rn(__uint_as_float(v[e]) * 4096.f)) + kSqBias);
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) G[r * kPitch + c0 + e] = __uint_as_float(v[e]);
      }
    }
  }
  __syncthreads();  // S_q and G are complete in shared memory - or somebody's wait ran out, the last of them
  const bool go = *abort_flag == 0;
  const int Dl = p.Dloc;
  if (go && warp < 2) {
    // ---- Algorithm 2
    if (warp == 0) greedy_one_warp(reinterpret_cast<const uint32_t*>(S), Dl, lane, *lists, sel, p.idx + (size_t)tile_b * Dl);
    rows_sync();
    // ---- Sec. 4.2.1: thread = source token k; logit of destination i is G[idx_i][k] / (tau sqrt(d)).  Eight at a time, so that
    // their reads are in flight together (one behind the other: 2.5 us).
    float mx = -INFINITY;
    for (int i0 = 0; i0 < Dl; i0 += 8) {
      float g[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) g[e] = G[sel[i0 + e] * kPitch + r];
#pragma unroll
      for (int e = 0; e < 8; ++e) mx = fmaxf(mx, g[e]);
    }
    const float neg_m = -mx * p.scale_log2;
    float sum = 0.f;
    for (int i0 = 0; i0 < Dl; i0 += 8) {
      float g[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) g[e] = G[sel[i0 + e] * kPitch + r];
#pragma unroll
      for (int e = 0; e < 8; ++e) g[e] = ex2(fmaf(g[e], p.scale_log2, neg_m));
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        A[(i0 + e) * kPitch + r] = g[e];
        sum += g[e];
      }
    }
    const float inv = 1.f / sum;
    for (int i0 = 0; i0 < Dl; i0 += 8) {
      float g[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) g[e] = A[(i0 + e) * kPitch + r];
#pragma unroll
      for (int e = 0; e < 8; ++e) A[(i0 + e) * kPitch + r] = g[e] * inv;
    }
    rows_sync();
    if (r < Dl) {  // row sum of destination r over the tile's sources, in source order
      float z = 0.f;
      for (int k = 0; k < kTok; ++k) z += A[r * kPitch + k];
      zinv[r] = z > 0.f ? 1.f / z : 0.f;  // a row sum that underflowed to 0 gives a zero row
    }
  }
  __syncthreads();
  if (go) {
    // A~^T[k][i] = A[i][k] / Z_i as hi + lo bf16 planes; a source's D_loc weights are contiguous (D_loc % 8 == 0), and two
    // threads take every second eight of them
    __nv_bfloat16* hi_row = p.w + ((size_t)tile_b * 2 * kTok + r) * Dl;
    __nv_bfloat16* lo_row = hi_row + (size_t)kTok * Dl;
    for (int i0 = (warp >> 1) * 8; i0 < Dl; i0 += 16) {
      __align__(16) __nv_bfloat16 hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float v = A[(i0 + e) * kPitch + r] * zinv[i0 + e];
        hi[e] = __float2bfloat16_rn(v);
        lo[e] = __float2bfloat16_rn(v - __bfloat162float(hi[e]));
      }
      *reinterpret_cast<uint4*>(hi_row + i0) = *reinterpret_cast<const uint4*>(hi);
      *reinterpret_cast<uint4*>(lo_row + i0) = *reinterpret_cast<const uint4*>(lo);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 3) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

constexpr int kRefreshSmem = 1024 + kRing * kStageBytes + kTok * kTok * 2 + 2 * kTok * kPitch * 4 + 2 * kTok * 4 + (int)sizeof(greedy::Shared<kTok>) + 256;
static_assert(sizeof(RBars) <= 256, "barrier block outgrew its reservation");

}  // namespace

// Shapes the one-kernel selection + weights covers: bf16 tokens, tile-local merge, tiles of 64 tokens that are one
// 4-D TMA box, destinations in whole 16-byte rows of the weight planes, whole 64-channel slabs, and no second
// (shares) matrix behind the weights.
bool refresh_fused_supported(const Geom& g) {
  if (g.f32 || g.global_merge || g.unmerge_mode != TOMA_UNMERGE_TRANSPOSE) return false;
  if (g.Nloc != kTok || g.tw > 64 || 64 % g.tw != 0 || g.th != 64 / g.tw) return false;
  if (g.Dloc < 1 || g.Dloc > kTok || g.Dloc % 8 != 0 || g.d % 64 != 0) return false;
  return true;
}

// `y`: the tile-major quantised tokens (launch_quantise).  Writes idx and the weight planes.
cudaError_t launch_refresh_fused(const Geom& g, const __nv_bfloat16* y, const void* x, int32_t* idx, void* w, uint32_t* dev_status,
                                 cudaStream_t s) {
  CUtensorMap ty, tx;
  const uint64_t ydims[3] = {(uint64_t)g.d, (uint64_t)g.Nloc, (uint64_t)g.B * g.P};
  const uint64_t ystrides[2] = {(uint64_t)g.d * 2, (uint64_t)g.Nloc * g.d * 2};
  const uint32_t ybox[3] = {64, (uint32_t)kTok, 1};
  const uint64_t xdims[4] = {(uint64_t)g.d, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.B};
  const uint64_t xstrides[3] = {(uint64_t)g.d * 2, (uint64_t)g.W * g.d * 2, (uint64_t)g.tokens_all() * g.d * 2};
  const uint32_t xbox[4] = {64, (uint32_t)g.tw, (uint32_t)g.th, 1};
  if (!encode_tmap_16bit(&ty, y, 3, ydims, ystrides, ybox) || !encode_tmap_16bit(&tx, x, 4, xdims, xstrides, xbox))
    return cudaErrorInvalidValue;
  RParams p;
  p.P = g.P; p.tiles_x = g.tiles_x; p.th = g.th; p.tw = g.tw; p.d = g.d; p.Dloc = g.Dloc;
  p.scale_log2 = g.logit_scale * 1.4426950408889634f;
  p.idx = idx;
  p.w = (__nv_bfloat16*)w;
  static std::atomic<unsigned long long> raised{0};
  cudaError_t e = raise_dynamic_smem(refresh_small_kernel, kRefreshSmem, raised);
  if (e != cudaSuccess) return e;
  e = launch_dependent(refresh_small_kernel, dim3(g.B * g.P), dim3(128), (size_t)kRefreshSmem, s, ty, tx, p, dev_status);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace toma
