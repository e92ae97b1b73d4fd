// Launches of the FFMA kernels: several CTAs of them fit an SM.
//
// CTAs of a dependent launch (launch_dependent()) are placed while the predecessor's retire, all that fit on the first SM that
// comes free.  432 CTAs of a kernel four of which fit an SM came to lie four on some SMs and two on others instead of three on
// each (fp32 projection of 373 x 4608 x 1152: 126 us so, 100 us evenly; of 1750 x 704 x 704 79 and 62), 18 of a softmax on a few
// SMs (fp32 weights of a region of 572 tokens, 384 channels: 43 and 34).  So a launch asks for as much shared memory as
// makes an SM hold no more of its CTAs than an even distribution gives it.  Not where it follows its like and fits beside it: nothing
// is uneven then, and an SM of its own for every CTA costs (projection of 103 x 2304 x 2304, 144 CTAs: 93 us, 101 so).
#pragma once

#include "common.cuh"
#include "tc.cuh"

namespace toma {

// What launch_spread() keeps of a kernel.
struct SpreadState {
  std::atomic<unsigned long long> raised{0};
  std::atomic<int> regs{0};  // registers per thread
};

// Dynamic shared memory to ask for.  `fixed`: the kernel's static shared memory; `dynamic`: what it uses of the dynamic one;
// `chained`: the predecessor is taken to be a launch of the same kind and size.
inline int spread_smem(long long ctas, int sms, int threads, int regs, int fixed, int dynamic, bool chained) {
  constexpr int kSmem = 228 * 1024, kCtaSmem = 1024;  // of an SM; what every CTA takes besides
  const int warps = (threads + 31) / 32, by_smem = kSmem / (fixed + dynamic + kCtaSmem), by_regs = 65536 / ((regs * 32 + 255) / 256 * 256 * warps);
  int slots = 64 / warps < 32 ? 64 / warps : 32;  // CTAs that fit an SM
  slots = slots < by_smem ? slots : by_smem;
  slots = slots < by_regs ? slots : by_regs;
  const long long per_sm = (ctas + sms - 1) / sms;
  if (per_sm >= slots || (chained && slots >= 2 * per_sm)) return dynamic;
  const int own = kSmem / ((int)per_sm + 1) - kCtaSmem + 128;  // one CTA more does not fit
  return own > fixed + dynamic ? own - fixed : dynamic;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_spread(void (*kernel)(KArgs...), SpreadState& st, bool chained, dim3 grid, dim3 block, int fixed, int dynamic, cudaStream_t s,
                          Args... args) {
  if (cudaError_t e = raise_dynamic_smem(kernel, 227 * 1024 - fixed, st.raised); e != cudaSuccess) return e;
  int regs = st.regs.load(std::memory_order_relaxed);
  if (regs == 0) {
    cudaFuncAttributes a;
    if (cudaError_t e = cudaFuncGetAttributes(&a, kernel); e != cudaSuccess) return e;
    st.regs.store(regs = a.numRegs > 0 ? a.numRegs : 1, std::memory_order_relaxed);
  }
  const int smem = spread_smem((long long)grid.x * grid.y * grid.z, sm_count(), (int)(block.x * block.y * block.z), regs, fixed, dynamic, chained);
  return launch_dependent(kernel, grid, block, (size_t)smem, s, args...);
}

}  // namespace toma
