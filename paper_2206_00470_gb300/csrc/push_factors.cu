// The training steps' scatter: delta rows formed from their factors
// (push_kernels.cuh).
#include "push_kernels.cuh"

namespace adapm {

void launch_push_factors(const Store& s, const PushArgs& a, int sms, cudaStream_t stream) {
  if (a.adagrad) launch_push_source<kSrcAda>(s, a, sms, stream);
  else launch_push_source<kSrcSgd>(s, a, sms, stream);
}

}  // namespace adapm
