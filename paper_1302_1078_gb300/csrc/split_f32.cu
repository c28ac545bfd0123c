// SPLIT-variant launcher for float values (see split_kernel.cuh).
#include "split_impl.cuh"

namespace gbs {
cudaError_t launch_split_f32(const CsrView& A, const SplitIndex& I, const DenseView& D, bool vec16, int threads,
                             int share, const SplitScratch& S, cudaStream_t s) {
  return launch_split_t<float>(A, I, D, vec16, threads, share, S, s);
}
}  // namespace gbs
