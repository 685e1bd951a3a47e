// Kernel instantiation: per-term queues of g g -> t tbar g.
#include "me_kernels.cuh"
namespace me {
cudaError_t launch_terms_gg(bool mixed, const LaunchArgs& a, const TermBufs& tb, cudaStream_t st) {
  return launch_terms_one<P_GG_TTG>(mixed, a, tb, st);
}
}  // namespace me
