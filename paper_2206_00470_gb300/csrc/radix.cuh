// Device helpers of the radix sorts (sort.cu, sort_small.cu).
#pragma once

#include "internal.cuh"

namespace adapm {
namespace {

constexpr int kRadixBits = 9;
constexpr int kDigits = 1 << kRadixBits;           // 512

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Lanes of the warp whose `valid` flag and low `nbits` digit bits equal this
// lane's (one ballot per bit: a warp-level multi-split).
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool valid, int nbits) {
  const uint32_t v = __ballot_sync(0xFFFFFFFFu, valid);
  uint32_t peers = valid ? v : ~v;
  for (int b = 0; b < nbits; ++b) {
    const bool bit = (d >> b) & 1u;
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, bit);
    peers &= bit ? bal : ~bal;
  }
  return peers;
}

// Exclusive scan of one value per thread over a block of NT threads.
template <int NT>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total,
                                                         uint32_t* sm /* NT/32 words */) {
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t s = lane < NT / 32 ? sm[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < NT / 32) sm[lane] = s;
  }
  __syncthreads();
  const uint32_t before = warp > 0 ? sm[warp - 1] : 0u;
  *total = sm[NT / 32 - 1];
  __syncthreads();
  return before + x - v;
}

struct PassPlan {
  int passes;
  int per;
};

PassPlan plan_for(int bits) {
  PassPlan p;
  p.passes = (bits + kRadixBits - 1) / kRadixBits;
  if (p.passes < 1) p.passes = 1;
  p.per = (bits + p.passes - 1) / p.passes;
  return p;
}

}  // namespace
}  // namespace adapm
