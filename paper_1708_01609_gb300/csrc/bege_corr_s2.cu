// Correlate kernels for S = 2 columns (N = 2^14).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s2(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                 bool halfz, cudaStream_t s) {
  if (c.nc == 2 && c.threads == 256) return unit::launch_unit<2, 1>(p, a, halfz, s);
  return cudaErrorInvalidValue;
}

}  // namespace bege
