// Dense projection C[m][n] = sum_k A[m][k] W[k][n] on the sm_100a tensor cores (bf16 in, fp32
// accumulation in tensor memory, bf16 out): the QKV and output projections of the attention module
// that ToMA wraps (Algorithm 3's core module F; App. C counts them as the 4 d^2 N term).
//
// Rows of A (tokens) sit on the MMA M dimension.  A is the K-major operand exactly as stored ([m][k] row-major),
// W the MN-major one exactly as stored ([k][n] row-major), so neither is transposed or copied.  Up to three weight /
// output pairs share A (Q, K and V in one launch).  Warp 0 feeds a TMA ring, warp 1 issues the MMAs, the other warps take
// the accumulators out of tensor memory (through the activation when one is asked for: the first layer of the MLP, the
// other module ToMA wraps), stage their 32 rows in shared memory as 64-column slabs in the layout of the output tensor
// map's box and store them with one TMA store per warp and slab: whole lines, asynchronous, instead of 16-byte stores to
// 32 different rows per warp instruction.
#include <climits>

#include "common.cuh"
#include "tc.cuh"

namespace toma {

using namespace tc;

namespace {

constexpr int kKC = 64;                  // contraction elements per stage
constexpr int kSlab = kKC * 128;         // [64 k][64 n] slab of W, 128-byte rows
constexpr int kABytes = 128 * 128;       // [128 m][64 k] slab of A

// GELU(v) = v Phi(v) = max(v, 0) - |v| Phi(-|v|) of two values, for results that are rounded to bf16.
// Phi(-a) = erfcx(a / sqrt 2) / 2 * 2^(-a^2 log2(e) / 2), and erfcx(x) / 2 = t (c0 + c1 t + ... + c7 t^7) with
// t = 1 / (1 + 0.33 x): the coefficients are the minimax fit of the relative error on x in [0, 10] (9.4e-8; with fp32
// arithmetic the result is within 5e-7 of the exact one for v > -1 and 8e-6 down to -13, where v (1 + erff) loses all
// digits).  Eleven issue slots and two MUFU operations per value against about 45 slots with erff, which made the first
// layer of an MLP of 4096 x 2560 x 640 a matter of its epilogue (34 us of which 13 us the activation).
__device__ __forceinline__ float rcp_mufu(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float min_nan(float a, float b) {  // a number that is none stays one
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ uint64_t both(float v) { return pack2(v, v); }
__device__ __forceinline__ void gelu2(uint32_t& v0, uint32_t& v1) {
  const float x0 = __uint_as_float(v0), x1 = __uint_as_float(v1);
  const uint64_t a = pack2(min_nan(fabsf(x0), 30.f), min_nan(fabsf(x1), 30.f));
  float d0, d1, e0, e1;
  unpack2(fma2(a, both(0.233345238f), both(1.f)), d0, d1);
  const uint64_t t = pack2(rcp_mufu(d0), rcp_mufu(d1));
  uint64_t q = fma2(both(-0.0676728131f), t, both(0.230118425f));
  q = fma2(q, t, both(-0.175574611f));
  q = fma2(q, t, both(0.204249755f));
  q = fma2(q, t, both(0.0236104601f));
  q = fma2(q, t, both(0.100611901f));
  q = fma2(q, t, both(0.0914779779f));
  q = fma2(q, t, both(0.0931789011f));
  unpack2(mul2(mul2(a, both(-0.72134752f)), a), e0, e1);
  q = mul2(mul2(mul2(q, t), a), pack2(ex2_mufu(e0), ex2_mufu(e1)));
  float g0, g1;
  unpack2(sub2(pack2(fmaxf(x0, 0.f), fmaxf(x1, 0.f)), q), g0, g1);
  v0 = __float_as_uint(g0);
  v1 = __float_as_uint(g1);
}

// ------------------------------------------------------------------------------------------------
// Persistent form: one CTA per SM walks over tiles of 128 rows x kCols columns.  The ring runs on across tiles, and two
// accumulators in tensor memory alternate, so that a tile's epilogue (eight warps: a GELU per element is as long as the
// tile's MMAs at K = 640) runs under the next tile's loads and MMAs.  Against one tile per CTA, four epilogue warps and
// nothing overlapped: 4096 x 2560 x 640 with GELU 34 -> 22 us, without 20.3 -> 15.9 us, 4096 x 640 x 2560
// 20.5 -> 16.1 us, 8192 x 4096 x 1024 64 -> 53.9 us, 6144 x 640 x 640 8.1 -> 7.8 us (rows x columns x contraction).
// ------------------------------------------------------------------------------------------------
constexpr int kMaxStages = 6;
constexpr int kEpiWarps = 8;

struct PersistBars {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

template <int kCols>
struct PersistCfg {
  static constexpr int kStageBytes = kABytes + kCols / 64 * kSlab;
  static constexpr int kStages = kCols == 128 ? 6 : 4;
  static constexpr int kStaging = kEpiWarps * 32 * 128;  // per epilogue warp: 32 rows of a 64-column slab
  static constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kStaging + 256;
  static constexpr uint32_t kAccCols = kCols == 128 ? 128 : 256;
};

// A warp's 32 rows of a tile, every second 64-column slab from `half` on: out of tensor memory, through the activation, staged
// in `mine` (32 rows of 128 B) and stored.
__device__ __forceinline__ void tile_out(uint32_t taddr, uint8_t* mine, int lane, const CUtensorMap* tm_c, int half, int slabs, int n0, int m0, int M,
                                         int act) {
#pragma unroll 1
  for (int j = half; j < slabs; j += 2) {
    if (lane == 0) tma_store_wait_read();  // the slab staged before has been read
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < 64; c += 32) {
      uint32_t r[32];
      tmem_ld32(taddr + j * 64 + c, r);
      tmem_wait_ld();
      if (act == kActGelu) {
#pragma unroll
        for (int e = 0; e < 32; e += 2) gelu2(r[e], r[e + 1]);
      }
#pragma unroll
      for (int e = 0; e < 32; e += 8) {
        __align__(16) __nv_bfloat162 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = __floats2bfloat162_rn(__uint_as_float(r[e + 2 * u]), __uint_as_float(r[e + 2 * u + 1]));
        *reinterpret_cast<uint4*>(mine + sw128_offset(lane, (c + e) >> 3)) = *reinterpret_cast<const uint4*>(q);
      }
    }
    fence_proxy_async();  // the staged rows are read by the TMA engine
    __syncwarp();
    if (lane == 0 && m0 < M) {  // rows past M and columns past N inside a box are clipped by the store
      tma_store_2d(tm_c, mine, n0 + j * 64, m0);
      tma_store_commit();
    }
  }
}

template <int kCols>
__global__ void __launch_bounds__((2 + kEpiWarps) * 32, 1)
linear_persistent_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w0,
                         const __grid_constant__ CUtensorMap tm_w1, const __grid_constant__ CUtensorMap tm_w2,
                         const __grid_constant__ CUtensorMap tm_c0, const __grid_constant__ CUtensorMap tm_c1,
                         const __grid_constant__ CUtensorMap tm_c2, int M, int N, int K, int n_items, int act, uint32_t* dev_status) {
  using C = PersistCfg<kCols>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* staging = smem + C::kStages * C::kStageBytes;
  PersistBars* bar = reinterpret_cast<PersistBars*>(staging + C::kStaging);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = (K + kKC - 1) / kKC;
  const int mb = (M + 127) / 128, nb = (N + kCols - 1) / kCols;
  // item -> row block (fastest: CTAs that run together share W slabs), column block, matrix
  auto m_of = [&](int item) { return item % mb * 128; };
  auto n_of = [&](int item) { return item / mb % nb * kCols; };
  auto z_of = [&](int item) { return item / mb / nb; };
  auto slabs_at = [&](int n0) { return (min(kCols, N - n0) + 63) / 64; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&bar->full[s], 1);
      mbar_init(&bar->empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&bar->acc_full[a], 1);
      mbar_init(&bar->acc_empty[a], kEpiWarps);
    }
    bar->abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_w0);
    prefetch_tmap(&tm_c0);
  }
  dependency_wait();
  if (threadIdx.x == 0) release_dependents();
  if (warp == 1) tmem_alloc(&bar->tmem_base, 2 * C::kAccCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int* abort_flag = &bar->abort_flag;

  if (warp == 0) {
    if (elect_one()) {
      int kc = 0;  // k-steps so far, over all items: ring slot and phase follow it
      bool ok = true;
      for (int item = blockIdx.x; ok && item < n_items; item += gridDim.x) {
        const int m0 = m_of(item), n0 = n_of(item), z = z_of(item), slabs = slabs_at(n0);
        const CUtensorMap* tm_w = z == 0 ? &tm_w0 : z == 1 ? &tm_w1 : &tm_w2;
        for (int k = 0; k < nk; ++k, ++kc) {
          const int s = kc % C::kStages;
          if (kc >= C::kStages && !mbar_wait(&bar->empty[s], ((kc / C::kStages) - 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          uint8_t* sa = smem + s * C::kStageBytes;
          mbar_expect_tx(&bar->full[s], kABytes + slabs * kSlab);
          tma_load_2d(sa, &tm_a, &bar->full[s], k * kKC, m0);
          for (int j = 0; j < slabs; ++j) tma_load_2d(sa + kABytes + j * kSlab, tm_w, &bar->full[s], n0 + j * 64, k * kKC);
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      int kc = 0, n = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++n) {
        const int a = n & 1;
        if (n >= 2 && !mbar_wait(&bar->acc_empty[a], ((n >> 1) - 1) & 1, dev_status, abort_flag)) break;
        tc_fence_after();
        const uint32_t t_acc = tmem + a * C::kAccCols;
        const uint32_t idesc = idesc_f16(kFmtBF16, kFmtBF16, false, true, 128, slabs_at(n_of(item)) * 64);
        for (int k = 0; k < nk; ++k, ++kc) {
          const int s = kc % C::kStages;
          if (!mbar_wait(&bar->full[s], (kc / C::kStages) & 1, dev_status, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t aa = smem_u32(smem + s * C::kStageBytes), wa = aa + kABytes;
          const int ksteps = min(kKC, K - k * kKC + 15) / 16;  // 16 contraction elements per MMA (zero filled past K)
          for (int kk = 0; kk < ksteps; ++kk)
            mma_ss(t_acc, smem_desc_sw128(aa + kk * 32, 16, 1024), smem_desc_sw128(wa + kk * 2048, kSlab, 1024), idesc, k > 0 || kk > 0);
          mma_commit(&bar->empty[s]);
        }
        if (!ok) break;
        mma_commit(&bar->acc_full[a]);
      }
    }
  } else {
    // two warps per quarter of the rows, each with every second 64-column slab
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* mine = staging + (warp - 2) * 4096;
    int n = 0;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++n) {
      const int a = n & 1, m0 = m_of(item) + quarter * 32, n0 = n_of(item), z = z_of(item), slabs = slabs_at(n0);
      const CUtensorMap* tm_c = z == 0 ? &tm_c0 : z == 1 ? &tm_c1 : &tm_c2;
      // one answer per warp: the tensor-memory loads below are warp-wide operations
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->acc_full[a], (n >> 1) & 1, dev_status, abort_flag))) break;
      tc_fence_after();
      const uint32_t taddr = tmem + a * C::kAccCols + ((uint32_t)(quarter * 32) << 16);
      tile_out(taddr, mine, lane, tm_c, half, slabs, n0, m0, M, act);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->acc_empty[a]);
    }
    if (lane == 0) tma_store_wait_read();  // shared memory must outlive the engine's reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * C::kAccCols);
  }
}

// ------------------------------------------------------------------------------------------------
// The same by pairs of SMs: a cluster of two CTAs walks over tiles of 256 rows x 256 columns.  Each CTA loads and keeps 128 of
// the rows of A and 128 of the columns of W, the first one's thread issues the MMAs of both (cta_group::2).  An SM then takes
// in 32 KB and reads 32 KB out of shared memory per 128 x 256 x 64 multiply-adds (512 cycles) where one working alone takes in
// and reads 48 KB each, which is more than the 128 bytes a cycle that shared memory has.  4096 x 2560 x 640 16.5 -> 15.0 us,
// 8192 x 1280 x 1280 25.6 -> 23.9, 16384 x 8192 x 4096 1092 -> 925 (rows x columns x contraction; against 256 x 256 by one CTA
// for the last).  A k-step still takes about 650 cycles: six stages do not quite cover the way from a free slot to its loads.
// Both CTAs' loads count on the first one's barrier; MMA completion is committed to both.
// ------------------------------------------------------------------------------------------------
constexpr int kPairRows = 256, kPairCols = 256, kPairStages = 6;
// Row blocks that are walked over together.  The 74 tiles under way then need 12 row blocks of A and six or seven column blocks
// of W at a time, which they read in step; with all rows of A first (61 blocks and one) every k-step came out of DRAM where A is
// larger than L2.  Panels of 4 to 16 timed on 23 shapes: 12 takes 0.95 to 1.0 of the time of all rows first (1.01 once), 8 and 16 up
// to 1 and 2 % more than 12.  Twelve at most, all panels of a matrix alike: a last one of a few rows shares nothing (6585 x 8448 x 2112 and
// others of 13 to 37 row blocks 3 % slower with panels of twelve and a rest).
constexpr int kPanel = 12;
constexpr int kPairStageBytes = kABytes + 2 * kSlab;     // a CTA's half
constexpr int kPairStaging = kEpiWarps * 32 * 128;
constexpr int kPairSmem = 1024 + kPairStages * kPairStageBytes + kPairStaging + 256;
struct PairBars {
  uint64_t full[kPairStages], empty[kPairStages];  // (full: of the first CTA)
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(PairBars) <= 256, "barrier block outgrew its reservation");

__global__ void __launch_bounds__((2 + kEpiWarps) * 32, 1)
linear_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w0,
                   const __grid_constant__ CUtensorMap tm_w1, const __grid_constant__ CUtensorMap tm_w2,
                   const __grid_constant__ CUtensorMap tm_c0, const __grid_constant__ CUtensorMap tm_c1,
                   const __grid_constant__ CUtensorMap tm_c2, int M, int N, int K, int n_items, int act, uint32_t* dev_status) {
  extern __shared__ uint8_t smem_raw[];
  // (the same offset in both CTAs: they are launched alike)
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* staging = smem + kPairStages * kPairStageBytes;
  PairBars* bar = reinterpret_cast<PairBars*>(staging + kPairStaging);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int nk = (K + kKC - 1) / kKC;
  const int mb = (M + kPairRows - 1) / kPairRows, nb = (N + kPairCols - 1) / kPairCols;
  const int pair = blockIdx.x / 2, pairs = gridDim.x / 2;
  const int panels = (mb + kPanel - 1) / kPanel, panel = (mb + panels - 1) / panels;  // row blocks of a panel, alike but for the last
  // item -> matrix, panel, column block, row block (fastest)
  auto place = [&](int item, int& m0, int& n0, int& z) {
    z = item / (mb * nb);
    const int in_z = item - z * mb * nb, first = in_z / (panel * nb) * panel, in_panel = in_z - first * nb, rows = min(panel, mb - first);
    n0 = in_panel / rows * kPairCols;
    m0 = (first + in_panel % rows) * kPairRows;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(&bar->full[s], 1);
      mbar_init(&bar->empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&bar->acc_full[a], 1);
      mbar_init(&bar->acc_empty[a], 2 * kEpiWarps);
    }
    bar->abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_w0);
    prefetch_tmap(&tm_c0);
  }
  cluster_sync();  // both CTAs' barriers are there
  dependency_wait();
  if (threadIdx.x == 0) release_dependents();
  if (warp == 1) tmem_alloc_pair(&bar->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int* abort_flag = &bar->abort_flag;

  if (warp == 0) {
    if (elect_one()) {
      int kc = 0;  // k-steps so far, over all items: ring slot and phase follow it
      bool ok = true;
      for (int item = pair; ok && item < n_items; item += pairs) {
        int m0, n0, z;
        place(item, m0, n0, z);
        m0 += rank * 128, n0 += rank * 128;  // this CTA's rows and columns
        const CUtensorMap* tm_w = z == 0 ? &tm_w0 : z == 1 ? &tm_w1 : &tm_w2;
        for (int k = 0; k < nk; ++k, ++kc) {
          const int s = kc % kPairStages;
          if (kc >= kPairStages && !mbar_wait(&bar->empty[s], ((kc / kPairStages) - 1) & 1, dev_status, abort_flag)) { ok = false; break; }
          uint8_t* sa = smem + s * kPairStageBytes;
          if (rank == 0) mbar_expect_tx(&bar->full[s], 2 * kPairStageBytes);  // what lies past M or N comes as zeros and counts
          tma_load_2d_pair(sa, &tm_a, &bar->full[s], k * kKC, m0);
          for (int j = 0; j < 2; ++j) tma_load_2d_pair(sa + kABytes + j * kSlab, tm_w, &bar->full[s], n0 + j * 64, k * kKC);
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      if (elect_one()) {
        constexpr uint32_t idesc = idesc_f16(kFmtBF16, kFmtBF16, false, true, kPairRows, kPairCols);
        int kc = 0, n = 0;
        bool ok = true;
        for (int item = pair; ok && item < n_items; item += pairs, ++n) {
          const int a = n & 1;
          if (n >= 2 && !mbar_wait(&bar->acc_empty[a], ((n >> 1) - 1) & 1, dev_status, abort_flag)) break;
          tc_fence_after();
          for (int k = 0; k < nk; ++k, ++kc) {
            const int s = kc % kPairStages;
            if (!mbar_wait(&bar->full[s], (kc / kPairStages) & 1, dev_status, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t aa = smem_u32(smem + s * kPairStageBytes), wa = aa + kABytes;
            const int ksteps = min(kKC, K - k * kKC + 15) / 16;  // 16 contraction elements per MMA (zero filled past K)
            for (int kk = 0; kk < ksteps; ++kk)
              mma_ss_pair(tmem + a * 256, smem_desc_sw128(aa + kk * 32, 16, 1024), smem_desc_sw128(wa + kk * 2048, kSlab, 1024), idesc, k > 0 || kk > 0);
            mma_commit_pair(&bar->empty[s]);
          }
          if (ok) mma_commit_pair(&bar->acc_full[a]);
        }
      }
    }
  } else {
    // two warps per quarter of the CTA's rows, each with every second 64-column slab
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* mine = staging + (warp - 2) * 4096;
    int n = 0;
    for (int item = pair; item < n_items; item += pairs, ++n) {
      int m0, n0, z;
      place(item, m0, n0, z);
      m0 += rank * 128 + quarter * 32;
      const int a = n & 1, slabs = (min(kPairCols, N - n0) + 63) / 64;
      const CUtensorMap* tm_c = z == 0 ? &tm_c0 : z == 1 ? &tm_c1 : &tm_c2;
      // one answer per warp: the tensor-memory loads below are warp-wide operations
      if (!__all_sync(0xffffffffu, mbar_wait(&bar->acc_full[a], (n >> 1) & 1, dev_status, abort_flag))) break;
      tc_fence_after();
      tile_out(tmem + a * 256 + ((uint32_t)(quarter * 32) << 16), mine, lane, tm_c, half, slabs, n0, m0, M, act);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_at(peer_addr(smem_u32(&bar->acc_empty[a]), 0));  // of the issuing CTA, which may be this one
    }
    if (lane == 0) tma_store_wait_read();  // shared memory must outlive the engine's reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
  cluster_sync();  // neither leaves while the other's MMAs read its shared memory or its arrivals are under way
}

template <int kCols>
cudaError_t run_persistent(int M, int N, int K, int n_mats, const CUtensorMap& ta, const CUtensorMap (&tw)[3], const CUtensorMap (&tc)[3], int act,
                           uint32_t* dev_status, cudaStream_t s) {
  using C = PersistCfg<kCols>;
  static std::atomic<unsigned long long> raised{0};
  if (cudaError_t e = raise_dynamic_smem(linear_persistent_kernel<kCols>, C::kSmemBytes, raised); e != cudaSuccess) return e;
  const long long items = (long long)((M + 127) / 128) * ((N + kCols - 1) / kCols) * n_mats;
  if (items > INT32_MAX / 2) return cudaErrorInvalidValue;
  const int grid = items < sm_count() ? (int)items : sm_count();
  return launch_dependent(linear_persistent_kernel<kCols>, dim3(grid), dim3((2 + kEpiWarps) * 32), (size_t)C::kSmemBytes, s, ta, tw[0], tw[1], tw[2],
                          tc[0], tc[1], tc[2], M, N, K, (int)items, act, dev_status);
}

// How many pairs the device holds at once: 0 where it places no cluster of this size (asked once per device; the other forms
// need none).
int pairs_at_once() {
  static std::atomic<unsigned long long> raised{0};
  static std::atomic<int> known[64];  // per device: 0 unknown, else the answer + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (const int k = known[dev].load(std::memory_order_relaxed)) return k - 1;
  int clusters = 0;
  bool ok = raise_dynamic_smem(linear_pair_kernel, kPairSmem, raised) == cudaSuccess;
  if (ok) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3((2 + kEpiWarps) * 32);
    cfg.dynamicSmemBytes = kPairSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ok = cudaOccupancyMaxActiveClusters(&clusters, linear_pair_kernel, &cfg) == cudaSuccess;
  }
  if (!ok) (void)cudaGetLastError();  // a failed query is an answer, not an error of the caller's stream
  if (!ok || clusters < 0) clusters = 0;
  known[dev].store(clusters + 1, std::memory_order_relaxed);
  return clusters;
}

}  // namespace

// Tile form: the one with the least serial work per SM, i.e. tiles per SM (rounded up) times the time of one, which was
// timed on seventeen shapes between 200 x 640 x 640 and 16384 x 8192 x 4096: a tile of 128 x 192 takes 1.2 times, one of
// 128 x 256 1.35 times as long as one of 128 x 128 (they read fewer operand bytes per multiply-add), a pair's of 256 x 256
// 1.25 times - 1.1 from about 2048 contraction elements on - and a fifth more per launch for the cluster's start and end.
// Returns 128 x 256 (1), 128 x 192 (2), 256 x 256 by pairs (3) or 128 x 128 (4).
int linear_tc_form(int M, int N, int K, int n_mats, int sms, int pairs) {
  auto cost = [&](int rows, int cols, int tile, int at_once) {
    const long long tiles = (long long)((M + rows - 1) / rows) * ((N + cols - 1) / cols) * n_mats;
    return (tiles + at_once - 1) / at_once * tile;
  };
  const long long cost128 = cost(128, 128, 20, sms), cost192 = cost(128, 192, 24, sms), cost256 = cost(128, 256, 27, sms);
  const long long cost_pair = M > 128 && pairs > 0 ? cost(kPairRows, kPairCols, K >= 2048 ? 22 : 25, pairs) + 4 : LLONG_MAX;
  if (cost_pair < cost128 && cost_pair < cost192 && cost_pair < cost256) return 3;
  return cost128 <= cost192 && cost128 <= cost256 ? 4 : cost192 <= cost256 ? 2 : 1;
}

bool linear_tc_shape_ok(int M, int N, int K) { return M >= 1 && N >= 8 && K >= 8 && N % 8 == 0 && K % 8 == 0; }

// c[i] = a * w[i] for i < n_mats (1..3); a [M][K], w[i] [K][N], c[i] [M][N], all bf16 row-major.
cudaError_t launch_linear_tc(int M, int N, int K, const void* a, const void* const* w, void* const* c, int n_mats, int act,
                             uint32_t* dev_status, cudaStream_t s) {
  CUtensorMap ta, tw[3], tc_[3];
  const uint64_t adims[2] = {(uint64_t)K, (uint64_t)M};
  const uint64_t astr[1] = {(uint64_t)K * 2};
  const uint32_t abox[2] = {64, 128};
  if (!encode_tmap_16bit(&ta, a, 2, adims, astr, abox)) return cudaErrorInvalidValue;
  const uint64_t wdims[2] = {(uint64_t)N, (uint64_t)K};
  const uint64_t wstr[1] = {(uint64_t)N * 2};
  const uint32_t wbox[2] = {64, 64};
  const uint64_t cdims[2] = {(uint64_t)N, (uint64_t)M};
  const uint32_t cbox[2] = {64, 32};  // a warp's 32 rows of one 64-column slab
  for (int i = 0; i < 3; ++i) {
    const int j = i < n_mats ? i : 0;
    if (!encode_tmap_16bit(&tw[i], w[j], 2, wdims, wstr, wbox) || !encode_tmap_16bit(&tc_[i], c[j], 2, cdims, wstr, cbox))
      return cudaErrorInvalidValue;
  }
  const int at_once = pairs_at_once();
  int form = linear_tc_form(M, N, K, n_mats, sm_count(), at_once);
  // test-only override
  if (const int v = g_tune_linear_tile.load(std::memory_order_relaxed); v && (v != 3 || (M > 128 && at_once > 0))) form = v;
  cudaError_t e;
  if (form == 3) {
    const long long items = (long long)((M + kPairRows - 1) / kPairRows) * ((N + kPairCols - 1) / kPairCols) * n_mats;
    if (items > INT32_MAX / 2) return cudaErrorInvalidValue;
    const int pairs = items < at_once ? (int)items : at_once;
    e = launch_dependent_cluster(linear_pair_kernel, dim3(2 * pairs), dim3((2 + kEpiWarps) * 32), (size_t)kPairSmem, 2, s, ta, tw[0], tw[1], tw[2],
                                 tc_[0], tc_[1], tc_[2], M, N, K, (int)items, act, dev_status);
  } else {
    e = form == 4   ? run_persistent<128>(M, N, K, n_mats, ta, tw, tc_, act, dev_status, s)
        : form == 2 ? run_persistent<192>(M, N, K, n_mats, ta, tw, tc_, act, dev_status, s)
                    : run_persistent<256>(M, N, K, n_mats, ta, tw, tc_, act, dev_status, s);
  }
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace toma
