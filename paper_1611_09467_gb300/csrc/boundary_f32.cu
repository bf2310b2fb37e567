// k_boundary in FP32 (a translation unit per precision: they compile side by side).
#include "boundary.cuh"

namespace peps {
PEPS_BOUNDARY_INST(float)
}  // namespace peps

#ifdef PEPS_PHASE_TIMING
// Diagnostic build only: copies the truncation's phase counters (cycles
// summed over CTAs, see PEPS_PHASE) to out[16] and optionally clears them.
extern "C" int peps_phase_read(unsigned long long* out, int reset) {
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  if (cudaMemcpyFromSymbol(out, ::peps_phase_cyc, 16 * sizeof(unsigned long long)) != cudaSuccess) return 1;
  if (reset) {
    const unsigned long long z[16] = {0};
    if (cudaMemcpyToSymbol(::peps_phase_cyc, z, sizeof(z)) != cudaSuccess) return 1;
  }
  return 0;
}
#endif
