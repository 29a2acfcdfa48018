// Correlate kernel for several segments of one length against the same
// templates.  The paper computes a template's transform once for a block of
// segments (Sec. 3.2 ii-iv); here a CTA runs the forward half of a template
// once, keeps its part of the spectrum (32 values per thread) in an
// L2-resident scratch, and then, for each segment, the product with that
// segment's coefficients, the inverse transform, sigma and the tails, with
// exactly the single-segment kernel's arithmetic.  Bound by latency beside the
// single kernel's FP32 work: a segment begins with 64 KB of spectrum and 96 KB
// of coefficients per unit from L2, as 16-byte loads (as 8-byte ones 199 ns per
// correlation at N = 2^16 and M = 8, now 151; the single kernel 165).
#include "bege_unit.cuh"

namespace bege {

namespace {

using namespace unit;

template <int S, int U>
__global__ void __launch_bounds__(256 * U, U == 1 ? 2 : 1) correlate_multi_kernel(PlanDev p, MultiArgs a) {
  constexpr int C = S / 2 / U;
  constexpr int kT = Geo<kF>::T;
  constexpr int kAhead = S <= 4 ? 3 : S == 8 ? 2 : 1;  // the reload has nothing to hide behind
  using SM = Sm<kF, U>;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cluster.block_rank();
  const int ui = (int)threadIdx.x / kT;
  const int ug = rank * U + ui;
  unit::setup_common<SM, kT * U>(p);
  setup_unit<SM>(p, S, ug, ui);
  if (threadIdx.x < S / 2) {
    const int c = (int)threadIdx.x / U, u = (int)threadIdx.x % U;
    float4* const rows = C == 1 ? SM::rows(0) : cluster.map_shared_rank(SM::rows(0), (unsigned)c);
    SM::rowptr()[threadIdx.x] = rows + u * (SM::L::unit_bytes / 16);
  }
  if constexpr (C > 1) cluster_arrive();  // paired with the wait of the first stage 1
  __syncthreads();

  const int cid = blockIdx.x / C;
  const int ncl = gridDim.x / C;
  const int nz = (int)(a.Lp / 2);
  float4* const scratch = a.scratch + ((size_t)blockIdx.x * U + ui) * 16 * kT;

  for (int64_t k = a.k0 + cid; k < a.k1; k += ncl) {
    // S2: forward stages 1-2 (stage 3 runs inside the middle for m = 0)
    stage1<SM, true, false, (C > 1)>(ui, S, ug, a.bank + k * a.Lp, nz, 1);
    SM::sync(ui);
    stage2<SM>(ui);
    mid_enter<SM, U>(ui, ug);
    const int64_t krow = k - a.k0;
    for (int m = 0; m < a.M; ++m) {
      // S3-S5 for segment m: product, sigma share, inverse transform
      if (m == 0)
        middle<SM, kAhead, true, false>(ui, ug, a.AB[0], a.M > 1 ? scratch : nullptr, false);
      else  // the rows are rewritten after the cluster's reads
        middle<SM, kAhead, true, (C > 1)>(ui, ug, a.AB[m], scratch, true);
      mid_leave<SM, U>(ui, ug);
      stage2i<SM>(ui);
      SM::sync(ui);
      const TailOut out{a.recs[m], a.cap[m], a.counter[m], nullptr};
      if constexpr (S == 2) {
        const float share = unit_power<SM>(0);
        const float sigma = sigma_of(&share, 1, S * 2 * kF);
        if (threadIdx.x == 0) a.sigma[m][krow] = sigma;
        finish_s2<SM, false>(0, p.uc, a.kappa * sigma, (uint32_t)k, krow, out, sigma);
        // every thread has read its rows before the next middle rewrites them
        if (m + 1 < a.M) __syncthreads();
      } else {
        {
          float2 va[1][16], vb[1][16];
          stage1i<SM>(ui, va, vb);
          store_blocks<SM>(ui, va, vb);
        }
        if (SM::tid() == 0) {
          const float share = unit_power<SM>(ui);
#pragma unroll
          for (int q = 0; q < C; ++q) {
            if constexpr (C > 1)
              *cluster.map_shared_rank(SM::sigall() + ug, (unsigned)q) = share;
            else
              SM::sigall()[ug] = share;
          }
        }
        if constexpr (C > 1) cluster_arrive();
        Combine<S, U> cb;
        cb.twiddles(p.uc, rank);
        if constexpr (C > 1)
          cluster_wait();  // every row and share of the cluster is ready
        else
          __syncthreads();
        const float sigma = sigma_of(SM::sigall(), S / 2, S * 2 * kF);
        if (rank == 0 && threadIdx.x == 0) a.sigma[m][krow] = sigma;
        cb.template emit<false>(typename Combine<S, U>::Shared{SM::rowptr()}, p.uc, rank, a.kappa * sigma, (uint32_t)k, krow, out,
                                sigma);
        if constexpr (C > 1) {
          __syncwarp();
          cluster_arrive_relaxed();  // every remote value has fed a vote: the reads are done
        } else {
          __syncthreads();
        }
      }
    }
  }
  if constexpr (C > 1) cluster_wait();  // the cluster's last reads of this CTA's rows
}

template <int S, int U>
cudaError_t launch_multi_t(const PlanDev& p, const MultiArgs& a, cudaStream_t s) {
  constexpr int C = S / 2 / U;
  constexpr size_t smem = unit::Lay<kF, U, false>::total;
  constexpr int kMinB = U == 1 ? 2 : 1;
  auto kern = correlate_multi_kernel<S, U>;
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
  cfg.blockDim = dim3(256 * U, 1, 1);
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

size_t multi_scratch_bytes(int sms) { return (size_t)sms * 2 * 256 * 16 * sizeof(float4); }

cudaError_t launch_correlate_multi(const PlanDev& p, const MultiArgs& a, cudaStream_t s) {
  if (a.k1 <= a.k0 || a.M < 1) return cudaSuccess;
  if (p.g.F != kF || p.g.S < 2 || a.Lp > kF || a.M > kMaxMulti) return cudaErrorInvalidValue;
  // Units per CTA: one where the reload of the spectrum, not the cluster, is
  // waited for (8 segments, ns per correlation, one / two units: N = 2^15 64.4 /
  // 58.5, 2^16 148.6 / 150.5, 2^17 333 / 351).
  switch (p.g.S) {
    case 2: return launch_multi_t<2, 1>(p, a, s);
    case 4: return launch_multi_t<4, 2>(p, a, s);
    case 8: return launch_multi_t<8, 1>(p, a, s);
    case 16: return launch_multi_t<16, 1>(p, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bege
