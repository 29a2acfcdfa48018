// Correlate kernels for S = 16 columns (N = 2^17).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s16(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                 cudaStream_t s) {
  return c.nc == 2 ? unit::launch_unit<16, 1>(p, a, s) : unit::launch_unit<16, 2>(p, a, s);
}

cudaError_t launch_range_s16(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  return unit::launch_range<16>(p, a, s);
}

}  // namespace bege
