// adapm_push's scatter: delta rows from the caller's array (push_kernels.cuh).
#include "push_kernels.cuh"

namespace adapm {

uint64_t push_chunk_rows(uint32_t D, uint64_t n, int sms) {
  // one span per resident block where the span fits in shared memory, else
  // as few full waves of resident blocks as do: rows per group = n / (groups
  // per block x resident blocks x waves), in [8, kPushSpan / groups].  (Spans
  // of kPushSpan rows whatever the last wave holds: 2.1M rows of 300 floats of
  // the SGNS step make 696 blocks, 2.3 waves of the 304 that run at a time, and
  // take 475 us against 410 us for 912, three full waves.)  The blocks counted
  // are those of rows from an array: AdaGrad sources of 65 to 96 vectors, four
  // per lane, and sources with scalars (push_blocks_per_sm) run fewer at a
  // time, so that their last wave can be partly empty.
  uint64_t ch = 0;
  dispatch_push_gc(D / 4, false, [&](auto Gc, auto Cc) {
    constexpr int G = decltype(Gc)::value, C = decltype(Cc)::value;
    constexpr uint64_t NG = kThreads / G;
    const uint64_t groups = NG * (uint64_t)sms * push_blocks_per_sm(C);
    const uint64_t most = kPushSpan / NG;
    const uint64_t waves = (n + groups * most - 1) / (groups * most);
    ch = waves ? (n + groups * waves - 1) / (groups * waves) : 8;
    if (ch < 8) ch = 8;
    if (ch > most) ch = most;
  });
  return ch;
}

uint64_t push_span_part_rows(uint64_t nchunks) { return 2 * (nchunks / 8 + 2); }

void launch_push(const Store& s, const PushArgs& a, int sms, cudaStream_t stream) {
  if (a.n == 0) return;
  if (a.coef != nullptr) return launch_push_factors(s, a, sms, stream);
  launch_push_source<kSrcRows>(s, a, sms, stream);
}

}  // namespace adapm
