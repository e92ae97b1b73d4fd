// Merge X_m = A~ X (Sec. 4.2.1) and unmerge A~^T X' (Sec. 4.2.2) on the sm_100a tensor cores for regions of any
// shape: N_loc no multiple of 64, D_loc no multiple of 16 - what divides an image whose sides are no powers of
// two.  (Regions that are whole 64-token boxes take linear_tc.cu.)
//
// Two things stand in the way of feeding such regions through TMA alone, and decide the design:
//   * A region's tokens are rows of tile_w tokens.  A TMA box takes r whole tile rows, r tile_w <= 64 (or 128) tokens
//     of consecutive slots; the last box of a region is a map of its own with the rows that are left, so that no
//     token of a neighbouring region is ever read.  The contraction is padded to 16 with zero weights.
//   * The weight planes [N_loc][D_loc] have rows of 2 D_loc bytes, which are neither 16-byte aligned nor a legal
//     TMA stride.  They are gathered instead: eight warps read the aligned 16-byte packets that cover eight weights,
//     shift them into place and write the 128-byte-swizzled operand tile; the same warps are the epilogue later.
// The weights are the A operand of both (destinations on M for the merge, MN-major; tokens on M for the unmerge,
// K-major), the tokens / attended rows the MN-major B operand with up to 320 channels: a weight block is then
// gathered once per 320 channels, and every thread of the epilogue holds one output row.
// Per CTA: warp 0 TMA, warp 1 MMA, warps 2..9 gather and epilogue.
#include <climits>

#include "common.cuh"
#include "tc.cuh"

namespace toma {

using namespace tc;

namespace {

constexpr int kWorkers = 256;       // threads of the gather / epilogue warps
constexpr int kMaxStages = 4;

struct RgBars {
  uint64_t full[kMaxStages], empty[kMaxStages], done;
  uint32_t tmem_base;
  int abort_flag;
};

struct RgParams {
  int P, tiles_x, th, tw, Nloc, Dloc, d;
  int rows;        // tile rows of a full box
  int nch;         // channels per CTA (a multiple of 64, at most 320)
  int stages;
  int kc;          // contraction rows of a stage (64 or 128; unmerge: 64)
  const __nv_bfloat16* w;
  const uint8_t* w_end;
  uint32_t* zero;  // merge only: words cleared on the side (the attention kernel's tickets)
  int zero_words;
  RowCopy extra;
};

// Eight consecutive weights starting `off` elements into a plane, the first `n` of them real and the rest 0.
__device__ __forceinline__ void funnel8(const uint4& lo, const uint4& hi, uint32_t sh, int n, uint32_t (&v)[4]) {
  uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  if (sh & 8u) {
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
  }
  if (sh & 4u) {
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = (sh & 2u) ? __funnelshift_r(w[i], w[i + 1], 16) : w[i];
    if (2 * i >= n) v[i] = 0u;
    else if (2 * i + 1 >= n) v[i] &= 0xFFFFu;
  }
}

// One weight block into its swizzled operand tile(s): `rows_total` rows starting at plane row `row0` (rows >= n_rows
// become 0), kChunks groups of eight columns starting at `col0` (columns >= D_loc become 0), both planes.  Slab s holds
// columns 64 s .. 64 s + 63; `slab_bytes` apart, planes `plane_bytes` apart.  In two halves, so that a block's packets
// are in flight while the block before waits for its buffer: load() takes four of the thread's rows, store() writes them.
template <int kChunks>
struct Gather {
  static constexpr int kRowStep = kWorkers / kChunks, kPass = 4 * kRowStep;  // rows between a thread's, rows of a pass
  uint4 lo[2][4], hi[2][4];
  uint32_t sh[2][4];

  __device__ __forceinline__ void load(const RgParams& p, const uint8_t* plane0, int t, int first, int row0, int n_rows, int col0) {
    const int ch = t % kChunks, n = min(8, p.Dloc - (col0 + ch * 8));
    const size_t plane_stride = (size_t)p.Nloc * p.Dloc * 2;
    const bool aligned = ((p.Dloc & 7) == 0);  // then every packet starts on 16 bytes
#pragma unroll
    for (int pl = 0; pl < 2; ++pl)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int row = first + t / kChunks + u * kRowStep;
        lo[pl][u] = hi[pl][u] = make_uint4(0u, 0u, 0u, 0u);
        sh[pl][u] = 0u;
        if (row < n_rows && n > 0) {
          const uint8_t* a = plane0 + pl * plane_stride + ((size_t)(row0 + row) * p.Dloc + col0 + ch * 8) * 2;
          const uint32_t s = (uint32_t)(reinterpret_cast<uintptr_t>(a) & 15);
          const uint4* q = reinterpret_cast<const uint4*>(a - s);
          sh[pl][u] = s;
          if (aligned) {
            lo[pl][u] = __ldg(q);
          } else if (reinterpret_cast<const uint8_t*>(q + 2) <= p.w_end) {
            lo[pl][u] = __ldg(q);
            if (s + 2 * n > 16) hi[pl][u] = __ldg(q + 1);
          } else {  // the last packets of the buffer: nothing behind its end is read
            __align__(16) __nv_bfloat16 e[8];
            for (int i = 0; i < 8; ++i) e[i] = i < n ? reinterpret_cast<const __nv_bfloat16*>(a)[i] : __float2bfloat16_rn(0.f);
            lo[pl][u] = *reinterpret_cast<const uint4*>(e);
            sh[pl][u] = 0u;
          }
        }
      }
  }
  __device__ __forceinline__ void store(const RgParams& p, int t, int first, int rows_total, int col0, uint8_t* dst, int slab_bytes,
                                        int plane_bytes) const {
    const int ch = t % kChunks, n = min(8, p.Dloc - (col0 + ch * 8));
    if (n <= 0) return;  // zero since the start
    uint8_t* out = dst + (ch >> 3) * slab_bytes;
#pragma unroll
    for (int pl = 0; pl < 2; ++pl)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int row = first + t / kChunks + u * kRowStep;
        if (row < rows_total) {
          uint32_t v[4];
          funnel8(lo[pl][u], hi[pl][u], sh[pl][u], n, v);
          *reinterpret_cast<uint4*>(out + pl * plane_bytes + sw128_offset(row, ch & 7)) = make_uint4(v[0], v[1], v[2], v[3]);
        }
      }
  }
};

// Epilogue: this warp's 32 accumulator rows (tensor-memory lanes 32 (warp & 3) ..), columns [c_lo, c_hi), as bf16 into
// the staged slabs [128 rows][64 channels], the layout of the output map's box.
__device__ __forceinline__ void stage_rows(uint8_t* so, uint32_t taddr, int row, int c_lo, int c_hi) {
  for (int c = c_lo; c < c_hi; c += 32) {
    uint32_t r[32];
    tmem_ld32(taddr + c, r);
    tmem_wait_ld();
    uint8_t* slab = so + (c >> 6) * (128 * 128);
#pragma unroll
    for (int e = 0; e < 32; e += 8) {
      __align__(16) __nv_bfloat162 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = __floats2bfloat162_rn(__uint_as_float(r[e + 2 * u]), __uint_as_float(r[e + 2 * u + 1]));
      *reinterpret_cast<uint4*>(slab + sw128_offset(row, ((c & 63) + e) >> 3)) = *reinterpret_cast<const uint4*>(q);
    }
  }
}

// kMerge: M = destinations, contraction over the region's tokens, box by box.  Otherwise M = one box of tokens,
// contraction over the destinations, 64 at a time.
//   grid: (channel block, M block, region)
//   tm_b / tm_b_tail: the B operand (merge: tokens, a full box and the region's last box; unmerge: attended rows, once)
//   tm_o / tm_o_tail: the output (merge: merged rows, once; unmerge: tokens, a full box and the region's last box)
template <bool kMerge>
__global__ void __launch_bounds__(64 + kWorkers, 1)
ragged_kernel(const __grid_constant__ CUtensorMap tm_b, const __grid_constant__ CUtensorMap tm_b_tail,
              const __grid_constant__ CUtensorMap tm_o, const __grid_constant__ CUtensorMap tm_o_tail, const RgParams p, uint32_t* dev_status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int batch = blockIdx.z, mb = blockIdx.y, c0 = blockIdx.x * p.nch;
  const int b = batch / p.P, tile = batch - b * p.P;
  const int ty = tile / p.tiles_x, tx = tile - ty * p.tiles_x;
  const int n_ch = min(p.nch, p.d - c0), slabs = (n_ch + 63) / 64, n_mma = slabs * 64;
  const int n_boxes = (p.th + p.rows - 1) / p.rows, tail_rows = p.th - (n_boxes - 1) * p.rows;
  // A: merge [2 planes][2 slabs of 64 destinations][kc tokens][128 B]; unmerge [2 planes][128 tokens][64 destinations]
  const int a_slab = kMerge ? p.kc * 128 : 128 * 128, a_plane = kMerge ? 2 * a_slab : a_slab;
  const int b_slab = p.kc * 128;
  const int stage_bytes = 2 * a_plane + (p.nch / 64) * b_slab;
  RgBars* bar = reinterpret_cast<RgBars*>(smem + p.stages * stage_bytes);
  const int nk = kMerge ? n_boxes : (p.Dloc + 63) / 64;
  const uint32_t ncols = p.nch > 256 ? 512u : p.nch > 128 ? 256u : p.nch > 64 ? 128u : 64u;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&bar->full[s], 1 + kWorkers / 32);
      mbar_init(&bar->empty[s], 1);
    }
    mbar_init(&bar->done, 1);
    bar->abort_flag = 0;
    mbar_fence_init();
    prefetch_tmap(&tm_b);
    prefetch_tmap(&tm_b_tail);
    prefetch_tmap(&tm_o);
    prefetch_tmap(&tm_o_tail);
  }
  // what no load ever writes has to be a finite number: padding rows of the B operand, padding columns of A
  for (int e = threadIdx.x; e < p.stages * stage_bytes / 16; e += blockDim.x) reinterpret_cast<uint4*>(smem)[e] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async();
  __syncthreads();
  dependency_wait();
  if (threadIdx.x == 0) release_dependents();
  if (kMerge && p.zero_words > 0) {
    const int cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const int n_thr = gridDim.x * gridDim.y * gridDim.z * blockDim.x;
    for (int i = cta * blockDim.x + threadIdx.x; i < p.zero_words; i += n_thr) p.zero[i] = 0u;
  }
  volatile int* abort_flag = &bar->abort_flag;
  // All meet once more when the tensor memory is there; the first loads, of tokens and of weights, do not wait for that. (With
  // the stores by slabs below: 384 regions of 96 tokens, 1280 channels, merge 97.4 -> 92.2 us, unmerge 81.6 -> 73.8.)
  if (warp == 0) {
    const int early = min(nk, p.stages);
    auto load = [&](int k) {
      const int s = k % p.stages;
      uint8_t* sb = smem + s * stage_bytes + 2 * a_plane;
      if (kMerge) {
        const bool tail = k == n_boxes - 1;
        mbar_expect_tx(&bar->full[s], slabs * (tail ? tail_rows : p.rows) * p.tw * 128);
        for (int c = 0; c < slabs; ++c)
          tma_load_4d(sb + c * b_slab, tail ? &tm_b_tail : &tm_b, &bar->full[s], c0 + c * 64, tx * p.tw, ty * p.th + k * p.rows, b);
      } else {
        mbar_expect_tx(&bar->full[s], slabs * b_slab);
        for (int c = 0; c < slabs; ++c) tma_load_4d(sb + c * b_slab, &tm_b, &bar->full[s], c0 + c * 64, k * 64, tile, b);
      }
    };
    if (elect_one())
      for (int k = 0; k < early; ++k) load(k);
    __syncwarp();
    __syncthreads();
    if (elect_one()) {
      for (int k = early; k < nk; ++k) {
        if (!mbar_wait(&bar->empty[k % p.stages], ((k / p.stages) - 1) & 1, dev_status, abort_flag)) break;
        load(k);
      }
    }
  } else if (warp == 1) {
    tmem_alloc(&bar->tmem_base, ncols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bar->tmem_base;
    if (elect_one()) {
      const int n_a = min(n_mma, 256), n_b = n_mma - n_a;
      const uint32_t idesc_a = idesc_f16(kFmtBF16, kFmtBF16, kMerge, true, 128, n_a);
      const uint32_t idesc_b = idesc_f16(kFmtBF16, kFmtBF16, kMerge, true, 128, n_b > 0 ? n_b : 64);
      bool ok = true;
      for (int k = 0; k < nk; ++k) {
        const int s = k % p.stages;
        if (!mbar_wait(&bar->full[s], (k / p.stages) & 1, dev_status, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t aa = smem_u32(smem + s * stage_bytes), ba = aa + 2 * a_plane;
        const int len = kMerge ? (k == n_boxes - 1 ? tail_rows : p.rows) * p.tw : min(64, p.Dloc - k * 64);
        const int ksteps = (len + 15) / 16;
        for (int kk = 0; kk < ksteps; ++kk) {
          const uint64_t bd = smem_desc_sw128(ba + kk * 2048, b_slab, 1024);
#pragma unroll
          for (int pl = 0; pl < 2; ++pl) {
            const uint64_t ad = kMerge ? smem_desc_sw128(aa + pl * a_plane + kk * 2048, a_slab, 1024)
                                       : smem_desc_sw128(aa + pl * a_plane + kk * 32, 16, 1024);
            mma_ss(tmem, ad, bd, idesc_a, k > 0 || kk > 0 || pl > 0);
            if (n_b > 0) mma_ss(tmem + 256, ad, smem_desc_sw128(ba + 4 * b_slab + kk * 2048, b_slab, 1024), idesc_b, k > 0 || kk > 0 || pl > 0);
          }
        }
        mma_commit(&bar->empty[s]);
      }
      if (ok) mma_commit(&bar->done);
    }
  } else {
    const int t = threadIdx.x - 64;
    const uint8_t* plane0 = reinterpret_cast<const uint8_t*>(p.w) + (size_t)batch * 2 * p.Nloc * p.Dloc * 2;
    const int box_tok = p.rows * p.tw;
    // block k of the weights: its first row, rows, padded rows and first column
    const int m_len = (mb == n_boxes - 1 ? tail_rows : p.rows) * p.tw;
    auto row0_of = [&](int k) { return kMerge ? k * box_tok : mb * box_tok; };
    auto rows_of = [&](int k) { return kMerge ? (k == n_boxes - 1 ? tail_rows : p.rows) * p.tw : m_len; };
    auto col0_of = [&](int k) { return kMerge ? mb * 128 : k * 64; };
    const int rows_total = kMerge ? (box_tok + 15) & ~15 : m_len;
    Gather<kMerge ? 16 : 8> gather;
    constexpr int kPass = Gather<kMerge ? 16 : 8>::kPass;
    gather.load(p, plane0, t, 0, row0_of(0), rows_of(0), col0_of(0));
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bar->tmem_base;
    bool ok = true;
    for (int k = 0; k < nk; ++k) {
      const int s = k % p.stages;
      // one answer per warp
      if (k >= p.stages) ok = __all_sync(0xffffffffu, mbar_wait(&bar->empty[s], ((k / p.stages) - 1) & 1, dev_status, abort_flag));
      if (!ok) break;
      uint8_t* sa = smem + s * stage_bytes;
      gather.store(p, t, 0, rows_total, col0_of(k), sa, a_slab, a_plane);
      for (int first = kPass; first < rows_total; first += kPass) {
        gather.load(p, plane0, t, first, row0_of(k), rows_of(k), col0_of(k));
        gather.store(p, t, first, rows_total, col0_of(k), sa, a_slab, a_plane);
      }
      if (k + 1 < nk) gather.load(p, plane0, t, 0, row0_of(k + 1), rows_of(k + 1), col0_of(k + 1));
      if (!kMerge) {
        if (k == nk - 1 && k >= p.stages) {  // columns past D_loc still hold an earlier block's weights
          const int first = (p.Dloc - k * 64 + 7) / 8, last = ((p.Dloc - k * 64 + 15) / 16) * 2;
          for (int e = t; e < (last - first) * 256; e += kWorkers) {
            const int ch = first + e / 256, pl = (e >> 7) & 1, row = e & 127;
            *reinterpret_cast<uint4*>(sa + pl * a_plane + sw128_offset(row, ch)) = make_uint4(0u, 0u, 0u, 0u);
          }
        }
      }
      fence_proxy_async();  // the MMA reads what these threads wrote
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->full[s]);
    }
    if (p.extra.per)
      copy_part(p.extra, (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * kWorkers + t,
                (size_t)gridDim.x * gridDim.y * gridDim.z * kWorkers);
    // every load has been consumed: the stages are the output's staging area (a wait that ran out: the results are void, the
    // way is the same: four warps meet at barriers)
    mbar_wait_warp(&bar->done, 0, dev_status, abort_flag);
    tc_fence_after();
    const int quarter = warp & 3, half = (warp - 2) >> 2, row = quarter * 32 + lane;
    // four warps take every second slab, which is stored as soon as they have staged it
    for (int c = half; c < slabs; c += 2) {
      stage_rows(smem, tmem + ((uint32_t)(quarter * 32) << 16), row, c * 64, c * 64 + 64);
      fence_proxy_async();  // the staged rows are read by the TMA engine
      asm volatile("bar.sync %0, %1;" ::"r"(1 + half), "n"(kWorkers / 2) : "memory");
      if ((t & 127) == 0) {
        const void* src = smem + c * (128 * 128);
        if (kMerge) tma_store_4d(&tm_o, src, c0 + c * 64, mb * 128, tile, b);  // rows past the region's D_loc are clipped
        else tma_store_4d(mb == n_boxes - 1 ? &tm_o_tail : &tm_o, src, c0 + c * 64, tx * p.tw, ty * p.th + mb * p.rows, b);
        tma_store_commit();
      }
    }
    if ((t & 127) == 0) tma_store_wait_read();  // shared memory must outlive the engine's reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(bar->tmem_base, ncols);
  }
}

bool token_map(const Geom& g, const void* x, int rows, CUtensorMap* tm) {
  const uint64_t dims[4] = {(uint64_t)g.d, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.B};
  const uint64_t strides[3] = {(uint64_t)g.d * 2, (uint64_t)g.W * g.d * 2, (uint64_t)g.tokens_all() * g.d * 2};
  const uint32_t box[4] = {64, (uint32_t)g.tw, (uint32_t)rows, 1};
  return encode_tmap_16bit(tm, x, 4, dims, strides, box);
}

// merged / attended rows as (channel, destination, region, batch): a box never reaches into the next region's rows
bool merged_map(const Geom& g, const void* m, int rows, CUtensorMap* tm) {
  const uint64_t dims[4] = {(uint64_t)g.d, (uint64_t)g.Dloc, (uint64_t)g.P, (uint64_t)g.B};
  const uint64_t strides[3] = {(uint64_t)g.d * 2, (uint64_t)g.Dloc * g.d * 2, (uint64_t)g.Lm * g.d * 2};
  const uint32_t box[4] = {64, (uint32_t)rows, 1, 1};
  return encode_tmap_16bit(tm, m, 4, dims, strides, box);
}

template <bool kMerge>
cudaError_t launch_ragged(const Geom& g, const void* w, const void* in, void* out, void* zero, size_t zero_bytes, uint32_t* dev_status,
                          cudaStream_t s) {
  RgParams p;
  p.P = g.P; p.tiles_x = g.tiles_x; p.th = g.th; p.tw = g.tw; p.Nloc = g.Nloc; p.Dloc = g.Dloc; p.d = g.d;
  // merge: boxes of at most 64 tokens keep a stage small (rows wider than that: 128); unmerge: a box is the M block
  p.kc = kMerge && g.tw > 64 ? 128 : 64;
  const int box_max = kMerge ? p.kc : 128;
  p.rows = box_max / g.tw < g.th ? box_max / g.tw : g.th;
  const int n_boxes = (g.th + p.rows - 1) / p.rows, tail = g.th - (n_boxes - 1) * p.rows;
  const int m_blocks = kMerge ? (g.Dloc + 127) / 128 : n_boxes;
  // Channels per CTA: the fewer CTAs per SM (rounded up) the better, then the fewer channels - a CTA's time is that of
  // gathering its weights, about what 600 channels' multiplications take, plus that of its channels (timed with 64 to 320
  // channels on nine shapes: one wave of 320 takes 42 us where one of 192 takes 35; 2 x 4032 tokens in regions of 18 x 14,
  // 640 channels: merge 22.0 -> 13.3 us, unmerge 17.9 -> 9.9 us against 128 and 256 channels without the prefetch).
  long long best = LLONG_MAX;
  for (int nch = 64; nch <= 320; nch += 64) {
    if (nch > 64 && nch - 64 >= g.d) break;
    const long long ctas = (long long)g.B * g.P * m_blocks * ((g.d + nch - 1) / nch);
    const long long cost = (ctas + sm_count() - 1) / sm_count() * (600 + nch);
    if (cost < best) best = cost, p.nch = nch;
  }
  p.w = (const __nv_bfloat16*)w;
  p.w_end = (const uint8_t*)w + (size_t)g.B * g.P * g.Nloc * g.Dloc * 4;
  p.zero = (uint32_t*)zero;
  p.zero_words = (int)(zero_bytes / 4);
  const RowCopy rows = extra_rows(g, in, out, kMerge);
  CUtensorMap tb, tbt, to, tot;
  bool ok;
  if (kMerge) ok = token_map(g, in, p.rows, &tb) && token_map(g, in, tail, &tbt) && merged_map(g, out, 128, &to);
  else ok = merged_map(g, in, 64, &tb) && token_map(g, out, p.rows, &to) && token_map(g, out, tail, &tot);
  if (!ok) return cudaErrorInvalidValue;
  if (kMerge) tot = to;
  else tbt = tb;
  const int a_plane = kMerge ? 2 * p.kc * 128 : 128 * 128;
  const int stage_bytes = 2 * a_plane + (p.nch / 64) * p.kc * 128;
  const int nk = kMerge ? n_boxes : (g.Dloc + 63) / 64;
  p.stages = (220 * 1024) / stage_bytes;
  p.stages = p.stages > 3 ? 3 : p.stages;
  if (p.stages > nk) p.stages = nk;
  int ring = p.stages * stage_bytes;
  const int staging = (p.nch / 64) * 128 * 128;
  if (ring < staging) {  // a single stage: as many as the staged output needs
    p.stages = (staging + stage_bytes - 1) / stage_bytes;
    ring = p.stages * stage_bytes;
  }
  const int smem = 1024 + ring + 256;
  static std::atomic<unsigned long long> raised{0};
  if (cudaError_t e = raise_dynamic_smem(ragged_kernel<kMerge>, 227 * 1024, raised); e != cudaSuccess) return e;
  const dim3 grid((unsigned)((g.d + p.nch - 1) / p.nch), (unsigned)m_blocks, (unsigned)(g.B * g.P));
  if (copied_beside(rows, (long long)grid.x * grid.y * grid.z * kWorkers)) p.extra = rows;
  const cudaError_t e = launch_dependent(ragged_kernel<kMerge>, grid, dim3(64 + kWorkers), (size_t)smem, s, tb, tbt, to, tot, p, dev_status);
  return finish_launch(e, rows, p.extra, s);
}

}  // namespace

// bf16 regions whose rows fit a TMA box of 128 tokens (grid z holds 65535 regions).
bool ragged_tc_supported(const Geom& g) { return !g.f32 && g.tw <= 128 && (long long)g.B * g.P <= 65535; }

cudaError_t launch_merge_ragged(const Geom& g, const void* w, const void* x, void* xm, void* zero, size_t zero_bytes, uint32_t* dev_status,
                                cudaStream_t s) {
  return launch_ragged<true>(g, w, x, xm, zero, zero_bytes, dev_status, s);
}

cudaError_t launch_unmerge_ragged(const Geom& g, const void* w, const void* y, void* out, uint32_t* dev_status, cudaStream_t s) {
  return launch_ragged<false>(g, w, y, out, nullptr, 0, dev_status, s);
}

}  // namespace toma
