// Batching form: many segments of different lengths N (2^14 .. 2^17), each
// against its own range of a bank, in one persistent launch.
//
// Every CTA holds two columns (256 threads, two CTAs per SM) and clusters
// have 8 CTAs.  A segment with S = N / 8192 columns needs C = S/2 CTAs per
// template, so a cluster splits into G = 8/C groups that correlate G
// templates of the same segment side by side.  Clusters take work items
// (segment, template range) from a queue in global memory; all CTAs of a
// cluster take the same item, rebuild the column twiddles for its N and run
// the templates with the same per-template body as the single-segment
// kernel (identical arithmetic, hence identical results).  The queue is a
// counter that the batch zeroes before each launch; clusters leave when it
// passes the last item, so nothing waits on anything else.
#include "bege_batch.h"
#include "bege_unit.cuh"

namespace bege {

namespace {

using namespace unit;

constexpr int kNC = 2;          // columns of a CTA (one unit)
constexpr int kT = Geo<kF>::T;
constexpr int kCluster = 8;

__device__ __forceinline__ int plan_index(int S) {
  return S == 2 ? 0 : S == 4 ? 1 : S == 8 ? 2 : 3;
}

// Per-item state lives in shared memory: kept in registers across the
// template loop it would push the 128-register budget of the FFT into spills.
struct ItemState {
  BatchSeg sg;
  int64_t k_begin, k_end;
};

template <int S>
__device__ __forceinline__ void combine_group(const float2* uc, int grank, float thr, uint32_t tmpl,
                                              int64_t krow, const TailOut& out) {
  Combine<S, 1> cb;
  cb.twiddles(uc, grank);
  cb.template emit<false>(typename Combine<S, 1>::Shared{Sm<kF, 1>::rowptr()}, uc, grank, thr, tmpl, krow, out, 0.f);
}

// One work item.  The stages do not depend on the column count S = N/8192, so
// one copy of them serves every segment length; only the tables and the
// S-point combine (compiled per S) do.
__device__ __forceinline__ void run_item(const BatchArgs& b, const ItemState* st, int rank) {
  const int S = st->sg.S;
  const int C = S / kNC;
  const int G = kCluster / C;
  using SM = Sm<kF, 1>;
  cg::cluster_group cluster = cg::this_cluster();
  const int group = rank / C, grank = rank - group * C, gbase = group * C;
  const PlanDev& p = b.plans[plan_index(S)];
  setup_unit<SM>(p, S, grank, 0);
  if (threadIdx.x < C)
    SM::rowptr()[threadIdx.x] = cluster.map_shared_rank(SM::rows(0), (unsigned)(gbase + threadIdx.x));
  __syncthreads();
  const int64_t iters = (st->k_end - st->k_begin + G - 1) / G;
  for (int64_t i = 0; i < iters; ++i) {
    const int64_t k = st->k_begin + i * G + group;
    const bool active = k < st->k_end;  // uniform over the CTAs of a group
    const int64_t krow = k - st->sg.k0;
    const TailOut out{st->sg.recs, st->sg.cap, st->sg.counter, nullptr};
    if (active) {
      stage1<SM, true, false, false>(0, S, grank, st->sg.bank + k * st->sg.Lp, (int)(st->sg.Lp / 2), 1);
      SM::sync(0);
      stage2<SM>(0);
      mid_enter<SM, 1>(0, grank);
      middle<SM, 1>(0, grank, st->sg.AB);
      mid_leave<SM, 1>(0, grank);
      stage2i<SM>(0);
      SM::sync(0);
      if (C == 1) {  // one CTA holds the template: no other CTA is waited for
        const float share = unit_power<SM>(0);
        const float sigma = sigma_of(&share, 1, S * 2 * kF);
        if (threadIdx.x == 0) st->sg.sigma[krow] = sigma;
        finish_s2<SM, false>(0, p.uc, st->sg.kappa * sigma, (uint32_t)k, krow, out, sigma);
      } else {
        float2 va[1][16], vb[1][16];
        stage1i<SM>(0, va, vb);
        store_blocks<SM>(0, va, vb);
        if (threadIdx.x == 0) {
          const float share = unit_power<SM>(0);
          for (int q = 0; q < C; ++q)
            *cluster.map_shared_rank(SM::sigall() + grank, (unsigned)(gbase + q)) = share;
        }
      }
    }
    if (C == 1) continue;
    cluster_arrive();
    cluster_wait();  // every row and share of the group is ready
    if (active) {
      const float sigma = sigma_of(SM::sigall(), C, S * 2 * kF);
      if (grank == 0 && threadIdx.x == 0) st->sg.sigma[krow] = sigma;
      const float thr = st->sg.kappa * sigma;
      switch (S) {
        case 4: combine_group<4>(p.uc, grank, thr, (uint32_t)k, krow, out); break;
        case 8: combine_group<8>(p.uc, grank, thr, (uint32_t)k, krow, out); break;
        default: combine_group<16>(p.uc, grank, thr, (uint32_t)k, krow, out); break;
      }
    }
    __syncwarp();
    cluster_arrive_relaxed();  // every remote value has fed a vote: the reads are done
    cluster_wait();
  }
}

__global__ void __launch_bounds__(kT, 2) batch_kernel(BatchArgs b) {
  __shared__ int item_slot;
  __shared__ ItemState st;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  unit::setup_common<Sm<kF, 1>, kT>(b.plans[0]);  // F-only tables: the same for every N
  for (;;) {
    if (rank == 0 && threadIdx.x == 0) item_slot = (int)atomicAdd(b.queue, 1u);
    cluster.sync();
    const int idx = *cluster.map_shared_rank(&item_slot, 0u);
    cluster.sync();  // every CTA has read the index before rank 0 takes the next
    if (idx >= b.n_items) break;
    if (threadIdx.x == 0) {
      const BatchItem item = b.items[idx];
      st.sg = b.segs[item.seg];
      st.k_begin = item.k_begin;
      st.k_end = item.k_end;
    }
    __syncthreads();
    run_item(b, &st, rank);
  }
}

// S1 for every segment of the batch: block i computes rank jobs[i].rank of
// segment jobs[i] (S/2 blocks per segment).
__global__ void __launch_bounds__(2 * kT, 1) segment_batch_kernel(BatchArgs b,
                                                             const SegJob* __restrict__ jobs) {
  const SegJob j = jobs[blockIdx.x];
  segment_unit<Sm<kF, 1>, false>(b.plans[plan_index(j.S)], j.S, j.rank, j.y, j.D, j.AB, false);
}

}  // namespace

int batch_max_clusters() {
  static int cached = -1;
  if (cached >= 0) return cached;
  constexpr size_t smem = unit::Lay<kF, 1, false>::total;
  if (cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(kT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cfg.gridDim = dim3((unsigned)(sms * 2 / kCluster * kCluster), 1, 1);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, batch_kernel, &cfg) != cudaSuccess) n = 0;
  cached = n;
  return n;
}

cudaError_t launch_batch(const BatchArgs& b, int clusters, cudaStream_t s) {
  constexpr size_t smem = unit::Lay<kF, 1, false>::total;
  cudaError_t e = cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(kT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.gridDim = dim3((unsigned)(clusters * kCluster), 1, 1);
  return cudaLaunchKernelEx(&cfg, batch_kernel, b);
}

cudaError_t launch_segment_batch(const BatchArgs& b, const SegJob* jobs, int njobs,
                                 cudaStream_t s) {
  constexpr size_t smem = unit::Lay<kF, 1, false>::total;
  cudaError_t e = cudaFuncSetAttribute(segment_batch_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (njobs <= 0) return cudaSuccess;
  segment_batch_kernel<<<njobs, 2 * kT, smem, s>>>(b, jobs);
  return cudaGetLastError();
}

}  // namespace bege
