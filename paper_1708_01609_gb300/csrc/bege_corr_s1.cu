// Correlate kernels for N = 2^10 .. 2^13 (two columns of N / 4 points).
#include "bege_unit.cuh"

namespace bege {

cudaError_t launch_correlate_s1(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  switch (unit_geo(p.g).F) {
    case 256: return unit::launch_short<256, false>(p, a, s);
    case 512: return unit::launch_short<512, false>(p, a, s);
    case 1024: return unit::launch_short<1024, false>(p, a, s);
    case 2048: return unit::launch_short<2048, false>(p, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_range_s1(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  switch (unit_geo(p.g).F) {
    case 256: return unit::launch_range_short<256, false>(p, a, s);
    case 512: return unit::launch_range_short<512, false>(p, a, s);
    case 1024: return unit::launch_range_short<1024, false>(p, a, s);
    case 2048: return unit::launch_range_short<2048, false>(p, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bege
