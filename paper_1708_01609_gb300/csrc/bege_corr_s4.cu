// Correlate kernels for S = 4 columns (N = 2^15).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s4(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                 cudaStream_t s) {
  return c.nc == 2 ? unit::launch_unit<4, 1>(p, a, s) : unit::launch_unit<4, 2>(p, a, s);
}

cudaError_t launch_range_s4(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  return unit::launch_range<4>(p, a, s);
}

}  // namespace bege
