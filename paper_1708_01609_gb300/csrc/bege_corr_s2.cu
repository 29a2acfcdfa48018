// Correlate kernels for N = 2^14 (two columns of 4096 points).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s2(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  return a.Lp <= unit::kF ? unit::launch_short<unit::kF, true>(p, a, s)
                          : unit::launch_short<unit::kF, false>(p, a, s);
}

cudaError_t launch_range_s2(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  return a.Lp <= unit::kF ? unit::launch_range_short<unit::kF, true>(p, a, s)
                          : unit::launch_range_short<unit::kF, false>(p, a, s);
}

}  // namespace bege
