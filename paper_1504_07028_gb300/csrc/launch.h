// Launch entry points of the fused sweep, compiled in their own translation units per
// precision so that the build runs in parallel.
#pragma once

#include <cuda_runtime.h>

#include "sweep.cuh"

namespace sgs {

// nt: threads of a CTA (256 or 64); tiles = 0 only grants the dynamic shared memory, before any
// launch (so that graph capture never changes kernel attributes).
template <typename T>
cudaError_t launch_sweep(const SweepArgs<T>& a, int M, int G, int nt, bool diag, int tiles, size_t smem,
                         cudaStream_t st);
// The same for K equal to the lane count G and full-width tiles (NC = nt / G): compile-time
// class strides and z-tile stride.
template <typename T>
cudaError_t launch_sweep_keq(const SweepArgs<T>& a, int M, int G, int nt, bool diag, int tiles,
                             size_t smem, cudaStream_t st);
// The same with g4 as the probability simplex indicator.
template <typename T>
cudaError_t launch_sweep_simplex(const SweepArgs<T>& a, int M, int G, int nt, bool diag, int tiles,
                                 size_t smem, cudaStream_t st);

#define SGS_SWEEP_EXTERN(NAME, T) \
  extern template cudaError_t NAME<T>(const SweepArgs<T>&, int, int, int, bool, int, size_t, cudaStream_t);
SGS_SWEEP_EXTERN(launch_sweep, float)
SGS_SWEEP_EXTERN(launch_sweep, double)
SGS_SWEEP_EXTERN(launch_sweep_keq, float)
SGS_SWEEP_EXTERN(launch_sweep_keq, double)
SGS_SWEEP_EXTERN(launch_sweep_simplex, float)
SGS_SWEEP_EXTERN(launch_sweep_simplex, double)
#undef SGS_SWEEP_EXTERN

}  // namespace sgs
