// Correlate kernel for several segments of one length against the same
// templates.  The paper computes a template's transform once for a block of
// segments (Sec. 3.2 ii-iv); here a CTA runs the forward half of a template
// once, keeps its part of the spectrum (32 values per thread) in an
// L2-resident scratch, and then, for each segment, the product with that
// segment's coefficients, the inverse transform, sigma and the tails, with
// exactly the single-segment kernel's arithmetic.
#include "bege_unit.cuh"

namespace bege {

namespace {

using namespace unit;

constexpr int kMinB = 2;

template <int S>
__global__ void __launch_bounds__(kT, kMinB) correlate_multi_kernel(PlanDev p, MultiArgs a) {
  constexpr int C = S / 2;
  using SM = Sm<1>;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cluster.block_rank();
  unit::setup_common<1>(p);
  setup_unit<1>(p, S, rank, 0);
  if constexpr (C > 1) {
    if (threadIdx.x < C)
      SM::rowptr()[threadIdx.x] = cluster.map_shared_rank(SM::rows(0), (unsigned)threadIdx.x);
    cluster_arrive();  // paired with the wait of the first stage 1
  }
  __syncthreads();

  const int cid = blockIdx.x / C;
  const int ncl = gridDim.x / C;
  const int nz = (int)(a.Lp / 2);
  float2* const scratch = a.scratch + (size_t)blockIdx.x * 32 * kT;

  for (int64_t k = a.k0 + cid; k < a.k1; k += ncl) {
    // S2: forward stages 1-2 (stage 3 runs inside the middle for m = 0)
    stage1<1, true, (C > 1)>(0, S, rank, a.bank + k * a.Lp, nz, 1);
    unit_sync<1>(0);
    stage2<1>(0);
    mid_enter<1>(0, rank);
    const int64_t krow = k - a.k0;
    for (int m = 0; m < a.M; ++m) {
      // S3-S5 for segment m: product, sigma share, inverse transform
      if (m == 0) {
        middle<1, 1, true, false>(0, rank, a.AB[0], a.M > 1 ? scratch : nullptr, false);
      } else {
        // the rows are rewritten: after the cluster's reads (S = 2: after
        // every thread has read its own rows)
        if constexpr (C == 1) __syncthreads();
        middle<1, 1, true, (C > 1)>(0, rank, a.AB[m], scratch, true);
      }
      mid_leave<1>(0, rank);
      stage2i<1>(0);
      unit_sync<1>(0);
      const TailOut out{a.recs[m], a.cap[m], a.counter[m], nullptr};
      if constexpr (S == 2) {
        const float share = unit_power<1>(0);
        const float sigma = sigma_of(&share, 1, S * 2 * kF);
        if (threadIdx.x == 0) a.sigma[m][krow] = sigma;
        finish_s2<false>(p.uc, a.kappa * sigma, (uint32_t)k, krow, out, sigma);
      } else {
        stage1i<1>(0);
        if (threadIdx.x == 0) {
          const float share = unit_power<1>(0);
#pragma unroll
          for (int q = 0; q < C; ++q)
            *cluster.map_shared_rank(SM::sigall() + rank, (unsigned)q) = share;
        }
        cluster_arrive();
        Combine<S, 1> cb;
        cb.twiddles(p.uc, rank);
        cluster_wait();  // every row and share of the cluster is ready
        const float sigma = sigma_of(SM::sigall(), S / 2, S * 2 * kF);
        if (rank == 0 && threadIdx.x == 0) a.sigma[m][krow] = sigma;
        cb.template emit<false>(SM::rowptr(), p.uc, rank, a.kappa * sigma, (uint32_t)k, krow, out,
                                sigma);
        __syncwarp();
        cluster_arrive_relaxed();  // every remote value has fed a vote: the reads are done
      }
    }
  }
  if constexpr (C > 1) cluster_wait();  // the cluster's last reads of this CTA's rows
}

template <int S>
cudaError_t launch_multi_t(const PlanDev& p, const MultiArgs& a, cudaStream_t s) {
  constexpr int C = S / 2;
  constexpr size_t smem = unit::Lay<1>::total;
  auto kern = correlate_multi_kernel<S>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(kT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3((unsigned)(sms / C * C * kMinB), 1, 1);
  int max_clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&max_clusters, kern, &cfg);
  if (e != cudaSuccess) return e;
  if (max_clusters < 1) return cudaErrorInvalidConfiguration;
  int64_t want = a.k1 - a.k0;
  if (want > max_clusters) want = max_clusters;
  // the scratch holds kMinB CTAs per SM: the grid never exceeds that
  if (want * C > (int64_t)sms * kMinB) want = (int64_t)sms * kMinB / C;
  cfg.gridDim = dim3((unsigned)(want * C), 1, 1);
  return cudaLaunchKernelEx(&cfg, kern, p, a);
}

}  // namespace

size_t multi_scratch_bytes(int sms) { return (size_t)sms * kMinB * kT * 32 * sizeof(float2); }

cudaError_t launch_correlate_multi(const PlanDev& p, const MultiArgs& a, cudaStream_t s) {
  if (a.k1 <= a.k0 || a.M < 1) return cudaSuccess;
  if (p.g.F != kF || p.g.S < 2 || a.Lp > kF || a.M > kMaxMulti) return cudaErrorInvalidValue;
  switch (p.g.S) {
    case 2: return launch_multi_t<2>(p, a, s);
    case 4: return launch_multi_t<4>(p, a, s);
    case 8: return launch_multi_t<8>(p, a, s);
    case 16: return launch_multi_t<16>(p, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bege
