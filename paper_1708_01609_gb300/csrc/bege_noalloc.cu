// bege_search_noalloc: the whole search (segment spectrum, correlation,
// sigma, tails) for callers that are not allowed to allocate device memory.
//
// Some programs hand every byte of device memory to one allocator of their
// own (a framework's caching pool, or an arena reserved once at start-up so
// that a latency-critical loop never pays for cudaMalloc/cudaFree, which
// synchronise the device and fragment the heap).  Such a caller can pass its
// own input and output buffers, but the library must not allocate the
// intermediates behind its back.  This entry point keeps them in one
// file-scope device array of fixed size instead:
//   - the product coefficients A, B and the segment spectrum D of the
//     segment (at most N = 2^16 samples),
//   - the FP32 twiddle tables for that N (computed on the device in FP64
//     by every call, ahead of the call's own kernels on its stream, so no
//     call depends on what an earlier call left in the array).
// Every CUDA context that loads the library has such an array until it ends
// (about 1.2 MiB).  All calls in a context share it and it keeps the
// contents of the last call, so two calls whose work overlaps on the GPU
// (for example on two streams) corrupt each other; callers serialise them.
#include <mutex>
#include <string>

#include "bege_internal.h"

namespace bege {

namespace {

constexpr int64_t kMaxN = 1 << 16;
constexpr int64_t kMaxH = kMaxN / 2;

constexpr size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

// Byte offsets of the regions of the scratch array (sized for N = 2^16).
constexpr size_t kOffAB = 0;
constexpr size_t kOffD = kOffAB + al256(kMaxH * sizeof(float4));
constexpr size_t kOffTables = kOffD + al256((kMaxH + 1) * sizeof(float2));
constexpr Geometry kMaxGeometry{(int)kMaxN, (int)kMaxH, 4096, (int)(kMaxH / 4096)};
constexpr size_t kScratchBytes = kOffTables + al256(plan_floats2(kMaxGeometry) * sizeof(float2));

static __device__ __align__(256) unsigned char g_search_scratch[kScratchBytes];

// Held while one call enqueues its kernels.
std::mutex g_mu;

}  // namespace

}  // namespace bege

extern "C" int bege_search_noalloc(const float* strain_dev, int64_t n, const float* bank_dev,
                                   int64_t ld, int64_t k_begin, int64_t k_end, float kappa,
                                   float* sigma_dev, bege_tail* tails_dev,
                                   uint64_t tail_capacity, unsigned long long* tail_count_dev,
                                   void* stream) {
  using namespace bege;
  if (!strain_dev || !bank_dev || !sigma_dev || !tail_count_dev || (tail_capacity && !tails_dev))
    return set_last_error(BEGE_EINVAL, "bege_search_noalloc: NULL pointer");
  if (n < 1024 || n > kMaxN || (n & (n - 1)))
    return set_last_error(BEGE_EINVAL,
                          "bege_search_noalloc: n must be a power of two in [2^10, 2^16]; "
                          "the fixed scratch array holds segments of at most 2^16 samples");
  if (ld < 8 || ld % 8 != 0 || ld > n)
    return set_last_error(BEGE_EINVAL,
                          "bege_search_noalloc: ld must be a multiple of 8 in [8, n]");
  if (k_begin < 0 || k_end <= k_begin)
    return set_last_error(BEGE_EINVAL, "bege_search_noalloc: empty template range");
  if (!(kappa >= 0.f) || kappa > 3.0e38f)
    return set_last_error(BEGE_EINVAL, "bege_search_noalloc: kappa must be finite and >= 0");
  if (reinterpret_cast<uintptr_t>(strain_dev) % 8 || reinterpret_cast<uintptr_t>(bank_dev) % 32 ||
      reinterpret_cast<uintptr_t>(tail_count_dev) % 8 ||
      reinterpret_cast<uintptr_t>(sigma_dev) % 4 || reinterpret_cast<uintptr_t>(tails_dev) % 4)
    return set_last_error(BEGE_EINVAL, "bege_search_noalloc: misaligned buffer");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Geometry g = make_geometry(n);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    // every CUDA context has a scratch array of its own: the current one's
    void* scratch = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&scratch, g_search_scratch);
    if (e != cudaSuccess)
      return set_last_error(BEGE_ECUDA,
                            std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    unsigned char* const base = static_cast<unsigned char*>(scratch);
    // The tables are rebuilt on every call, in stream order before this
    // call's kernels: the host keeps no record of which n the array holds,
    // which could disagree with the device's order of work.
    float2* const tables = reinterpret_cast<float2*>(base + kOffTables);
    e = launch_plan_tables(g, tables, s, tail_count_dev);
    if (e != cudaSuccess) return set_last_error(BEGE_ECUDA, cudaGetErrorString(e));
    const PlanDev p = plan_at(g, tables);
    float4* AB = reinterpret_cast<float4*>(base + kOffAB);
    float2* D = reinterpret_cast<float2*>(base + kOffD);
    e = launch_segment(p, strain_dev, D, AB, false, s);
    if (e == cudaSuccess) {
      CorrelateArgs a{};
      a.AB = AB;
      a.bank = bank_dev;
      a.Lp = ld;
      a.k0 = k_begin;
      a.k1 = k_end;
      a.kappa = kappa;
      a.sigma = sigma_dev;  // row k writes sigma_dev[k - k_begin]
      a.recs = tails_dev;
      a.cap = tail_capacity;
      a.counter = tail_count_dev;
      a.dump = nullptr;
      a.max_clusters = 0;
      e = launch_correlate(p, a, default_config(g), s);
      if (e == cudaSuccess) e = launch_range(p, a, s);
    }
    if (e != cudaSuccess) return set_last_error(BEGE_ECUDA, cudaGetErrorString(e));
  }
  return BEGE_OK;
}
