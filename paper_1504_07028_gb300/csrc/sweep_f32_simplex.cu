// FP32 instantiations of the fused sweep kernel with g4 as the probability simplex
// indicator.
#include "launch.h"

namespace sgs {
template <typename T>
cudaError_t launch_sweep_simplex(const SweepArgs<T>& a, int M, int G, int nt, bool diag, int tiles, size_t smem,
                                 cudaStream_t st) {
  return launch_sweep_variant<T, true, false>(a, M, G, nt, diag, tiles, smem, st);
}
template cudaError_t launch_sweep_simplex<float>(const SweepArgs<float>&, int, int, int, bool, int, size_t, cudaStream_t);
}  // namespace sgs
