// Stable sort of up to kSmallSort keys with their positions by one block, in
// shared memory: the same order as the grid sort (sort.cu), for batches whose
// grid sort is all launches and grid barriers.  One ordinary launch also does
// what the callers of a small sort need beside it: copies the keys as given
// (a push plan), lists the distinct ones (an intent), or compares the keys
// with a plan's first and stops if they match (a push).
//
// Measured (pull + push + read back of n keys of 64 floats, no intents, grid
// sort -> this): 1000 keys 51 -> 34 us, 4000 keys 55 -> 45 us, 8000 keys 57 ->
// 53 us.  Bound by its own latency (one SM): per pass a warp ranks its keys by a
// ballot multi-split, 32 at a time, and the warps' digit counts are scanned;
// keys and positions stay in registers between passes and change places
// through shared memory.
#include "internal.cuh"
#include "radix.cuh"

namespace adapm {

namespace {

constexpr int kThreadsS = 1024;
constexpr int kWarpsS = kThreadsS / 32;

struct SmallArgs {
  SmallSort a;
  int passes, per, bits;
};

// Dynamic shared memory: the warps' digit counts, then keys and positions.
template <int ITEMS>
constexpr size_t small_smem() {
  return (size_t)kWarpsS * kDigits * sizeof(uint16_t) + (size_t)kThreadsS * ITEMS * (sizeof(uint32_t) + sizeof(uint16_t));
}

template <int ITEMS>
__global__ void __launch_bounds__(kThreadsS, 1) sort_small_kernel(SmallArgs sa) {
  after_previous();
  const SmallSort& a = sa.a;
  extern __shared__ __align__(16) unsigned char dsm[];
  uint16_t(*wcnt)[kDigits] = reinterpret_cast<uint16_t(*)[kDigits]>(dsm);
  uint32_t* sk = reinterpret_cast<uint32_t*>(dsm + kWarpsS * kDigits * sizeof(uint16_t));
  uint16_t* sp = reinterpret_cast<uint16_t*>(sk + kThreadsS * ITEMS);
  __shared__ uint32_t base[kDigits];
  __shared__ uint32_t scan[kWarpsS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    if (a.clear0) *a.clear0 = 0u;
    if (a.clear1) *a.clear1 = 0u;
  }
  if (sort_failed(a.st)) return;   // an earlier grid sort gave up: nothing may follow
  uint32_t key[ITEMS], pos[ITEMS];
  bool bad = false, miss = false;
  // warp w owns positions [w * 32 * ITEMS, ...), 32 at a time
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const uint32_t i = (uint32_t)((warp * ITEMS + it) * 32 + lane);
    key[it] = i < a.n ? a.raw[i] : kNoKey;
    pos[it] = i;
  }
  if (a.plan_keys) {
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      if (pos[it] >= a.n) continue;
      const uint32_t x = a.plan_keys[pos[it]];
      miss |= (key[it] < a.K ? key[it] : kNoKey) != (x < a.K ? x : kNoKey);
    }
  }
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    if (a.copy_out && pos[it] < a.n) a.copy_out[pos[it]] = key[it];
    if (key[it] >= a.K) {
      if (pos[it] < a.n && !(a.allow_nokey && key[it] == kNoKey)) bad = true;
      key[it] = kNoKey;
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) set_error(a.st, ERR_KEY_RANGE);
  if (a.plan_keys) {
    if (!__syncthreads_or(miss)) return;   // the plan holds this sort's result
    if (threadIdx.x == 0) {
      *a.plan_word = a.plan_seq;
      atomicAdd(&a.st->plan_misses, 1ull);
    }
  }
  const uint32_t lt = lanemask_lt();
  int shift = 0;
  for (int p = 0; p < sa.passes; ++p) {
    const int nbits = sa.per < sa.bits - shift ? sa.per : sa.bits - shift;
    const uint32_t mask = (1u << nbits) - 1u;
    const int words = (int)((mask + 2) / 2);   // of a warp's counts
    for (int i = threadIdx.x; i < kWarpsS * words; i += kThreadsS)
      reinterpret_cast<uint32_t*>(wcnt[i / words])[i % words] = 0u;
    __syncthreads();
    uint32_t rank[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const uint32_t d = (key[it] >> shift) & mask;
      const uint32_t peers = digit_peers(d, true, nbits);
      const uint32_t prior = wcnt[warp][d];
      rank[it] = prior + __popc(peers & lt);
      __syncwarp();
      if (lane == __ffs(peers) - 1) wcnt[warp][d] = (uint16_t)(prior + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    // per digit: exclusive prefix over the warps, then over the digits
    uint32_t run = 0;
    if (threadIdx.x <= mask) {
#pragma unroll 8
      for (int w = 0; w < kWarpsS; ++w) {
        const uint32_t c = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = (uint16_t)run;
        run += c;
      }
    }
    uint32_t total;
    const uint32_t ex = block_exclusive_scan<kThreadsS>(run, &total, scan);
    if (threadIdx.x <= mask) base[threadIdx.x] = ex;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const uint32_t d = (key[it] >> shift) & mask;
      const uint32_t to = base[d] + wcnt[warp][d] + rank[it];
      sk[to] = key[it];
      sp[to] = (uint16_t)pos[it];
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const uint32_t i = (uint32_t)((warp * ITEMS + it) * 32 + lane);
      key[it] = sk[i];
      pos[it] = sp[i];
    }
    shift += nbits;
  }
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const uint32_t i = (uint32_t)((warp * ITEMS + it) * 32 + lane);
    if (i < a.n && a.keys_out) {
      a.keys_out[i] = key[it];
      a.pos_out[i] = pos[it];
    }
  }
  if (!a.heads_out) return;
  // the distinct keys, ascending
  bool first[ITEMS];
  uint32_t mine = 0;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const uint32_t i = (uint32_t)((warp * ITEMS + it) * 32 + lane);
    first[it] = key[it] != kNoKey && (i == 0 || sk[i - 1] != key[it]);
    mine += __popc(__ballot_sync(0xFFFFFFFFu, first[it]));   // of the warp
  }
  uint32_t total;
  uint32_t at = block_exclusive_scan<kThreadsS>(lane == 0 ? mine : 0u, &total, scan);
  at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, first[it]);
    if (first[it]) a.heads_out[at + __popc(bal & lt)] = key[it];
    at += __popc(bal);
  }
  if (threadIdx.x == 0) *a.heads_count = total;
}

template <int ITEMS>
cudaError_t launch(const SmallArgs& sa, cudaStream_t stream) {
  constexpr size_t smem = small_smem<ITEMS>();
  // the kernel's dynamic shared-memory limit is a per-device attribute
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    const cudaError_t e =
        cudaFuncSetAttribute(sort_small_kernel<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  note_launches(1);
  launch_after(sort_small_kernel<ITEMS>, 1, kThreadsS, smem, stream, sa);
  return cudaGetLastError();
}

}  // namespace

cudaError_t sort_small(const SmallSort& a, int bits, cudaStream_t stream) {
  const PassPlan pl = plan_for(bits);
  const SmallArgs sa{a, pl.passes, pl.per, bits};
  if (a.n <= kThreadsS) return launch<1>(sa, stream);
  if (a.n <= 2 * kThreadsS) return launch<2>(sa, stream);
  if (a.n <= 4 * kThreadsS) return launch<4>(sa, stream);
  return launch<8>(sa, stream);
}

}  // namespace adapm
