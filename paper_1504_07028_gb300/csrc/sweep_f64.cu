// FP64 instantiations of the fused sweep kernel (g4 on the affine set, eq. 10).
#include "launch.h"

namespace sgs {
template <typename T>
cudaError_t launch_sweep(const SweepArgs<T>& a, int M, int G, int nt, bool diag, int tiles, size_t smem,
                         cudaStream_t st) {
  return launch_sweep_variant<T, false, false>(a, M, G, nt, diag, tiles, smem, st);
}
template cudaError_t launch_sweep<double>(const SweepArgs<double>&, int, int, int, bool, int, size_t, cudaStream_t);
}  // namespace sgs
