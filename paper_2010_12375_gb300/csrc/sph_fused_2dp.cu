// The one-launch step of 2D tanks with a periodic axis (sph_fused_step.cuh); a translation unit
// of its own so that the four compile in parallel.
#include "sph_fused_step.cuh"

namespace sph {
cudaError_t launch_fused_2dp(const Buffers& b, int n_steps, int clear_counts, int follow, cudaStream_t s) {
  return launch_d<2, true>(b, n_steps, clear_counts, follow, s);
}
}  // namespace sph
