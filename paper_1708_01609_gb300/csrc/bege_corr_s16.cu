// Correlate kernels for S = 16 columns (N = 2^17).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s16(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                 bool halfz, cudaStream_t s) {
  if (c.nc == 2 && c.threads == 256) return unit::launch_unit<16, 1>(p, a, halfz, s);
  if (c.nc == 4 && c.threads == 512) return unit::launch_unit<16, 2>(p, a, halfz, s);
  return cudaErrorInvalidValue;
}

}  // namespace bege
