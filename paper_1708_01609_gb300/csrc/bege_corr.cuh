// Kernels of the matched-filter hot path, templated on the geometry.
//
// Matched filtering by FFT (van Putten, arXiv:1708.01609, Eq. 3S): for a
// real segment y (N samples) and a real template w (L <= N samples,
// zero-padded),
//     rho[n] = sum_m w[m] y[(n+m) mod N]               (Eq. A1, circular)
//            = (1/N) sum_j conj(W_j) D_j e^{+2 pi i j n/N}
// with sigma predicted by Parseval (Eq. PT) and tails |rho| > kappa sigma
// (Eq. tail).
//
// Real transforms as half-length complex transforms.  With H = N/2 and
// z[m] = w[2m] + i w[2m+1], Z = DFT_H(z) gives the template spectrum
//     W_j = (Z_j + conj Z_{H-j})/2 - (i/2) wN^j (Z_j - conj Z_{H-j}).
// The output is packed the same way, yo[n] = rho[2n] + i rho[2n+1], whose
// H-point spectrum is
//     Y_j = (P_j + conj P_{H-j})/2 + (i/2) wN^-j (P_j - conj P_{H-j}),
// P_j = conj(W_j) D_j.  Substituting W gives
//     Y_j = conj(Z_j) A_j + Z_{H-j} B_j,
//     A_j = g_j^2 D_j + d_j^2 conj D_{H-j},  B_j = g_j d_j (D_j + conj D_{H-j}),
//     g_j = (1 + i wN^-j)/2,  d_j = (1 - i wN^-j)/2,
// where A, B depend on the segment only and are computed once per segment
// (segment_kernel in bege_unit.cuh).  By Parseval on the packed spectrum
//     sigma^2 = (1/N) sum_n rho_n^2 = 2 sum_{j<H} |Y_j|^2 / N^2,
// the same quantity as Eq. PT's sum over the spectrum of rho.
//
// Residue columns (four-step with a pruned first step).  Bin j = S a + b,
// a < F, b < S, H = S F.  Forward:
//     Z_{Sa+b} = FFT_F(u_b)[a],  u_b[m1] = wH^(b m1) sum_{m2<S} z[m1+F m2] wS^(b m2);
// a template of L <= 2F samples has z = 0 beyond F, so only m2 = 0 remains
// (and with L <= F the upper half of u_b is zero as well).  Inverse, with
// n = n1 + F n2,
//     yo[n1 + F n2] = (1/H) sum_b wS^(-b n2) T_b[n1],
//     T_b[n1] = wH^(-b n1) IFFT_F(Y_{S.+b})[n1].
// Column b pairs with column S-b (bins j and H-j); columns {0, S/2} and
// {i, S-i} form units.  A CTA owns whole units; the CTAs of a thread-block
// cluster hold all S columns and exchange them only for the final S-point
// combine, through distributed shared memory or, by default for N >= 2^16,
// through a buffer in L2.
//
// This file: column maps, the tail epilogue and the launch; bege_unit.cuh has
// the segment and correlate kernels, bege_corr_tc.cu the tensor-core form.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>

#include "bege_fft.cuh"
#include "bege_internal.h"

namespace bege {

namespace cg = cooperative_groups;

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

extern __shared__ __align__(16) unsigned char smem_raw[];

// Column ownership for S >= 2 columns split over C = S/NC CTAs (this and the
// pair items: the tensor-core form).
template <int S, int NC>
struct ColMap {
  static_assert(NC % 2 == 0 && S % NC == 0, "column split");
  static constexpr int C = S / NC;
  static constexpr int UPC = NC / 2;
  // column held by local slot c of CTA `rank`: unit u (u < S/2) holds columns
  // u and S-u, unit 0 columns 0 and S/2; a CTA holds NC/2 consecutive units
  static __device__ __forceinline__ int slot_column(int rank, int c) {
    const int ug = rank * (NC / 2) + (c >> 1);
    const int second = c & 1;
    if (ug == 0) return second ? S / 2 : 0;
    return second ? S - ug : ug;
  }
  // owner rank and local slot of column b
  static __device__ __forceinline__ void home(int b, int* owner, int* slot) {
    int unit = 0, second = 0;
    if (b == S / 2)
      second = 1;
    else if (b < S / 2)
      unit = b;
    else {
      unit = S - b;
      second = 1;
    }
    *owner = unit / UPC;
    *slot = 2 * (unit % UPC) + second;
  }
};

// The bin pairs (j, H-j) held by a unit.  Unit 0 holds column 0 (pairs
// a <-> (F-a) mod F, with a = 0 and a = F/2 paired with themselves) and
// column S/2 (pairs a <-> F-1-a); unit i holds columns i and S-i (pairs
// (i, a) <-> (S-i, F-1-a)).
struct PairItem {
  int b, a, bp, ap, sj, sp;  // columns, rows, local slots
};

template <int F, int S>
__device__ __forceinline__ int unit_items(int ug) {
  return ug == 0 ? F + 1 : F;
}

template <int F, int S>
__device__ __forceinline__ PairItem pair_item(int ug, int ui, int it) {
  PairItem p;
  if (ug == 0) {
    if (it <= F / 2) {
      p.b = 0; p.a = it; p.bp = 0; p.ap = (F - it) & (F - 1);
      p.sj = p.sp = 2 * ui;
    } else {
      p.b = S / 2; p.a = it - (F / 2 + 1); p.bp = p.b; p.ap = F - 1 - p.a;
      p.sj = p.sp = 2 * ui + 1;
    }
  } else {
    p.b = ug; p.a = it; p.bp = S - ug; p.ap = F - 1 - it;
    p.sj = 2 * ui; p.sp = 2 * ui + 1;
  }
  return p;
}

// Y = conj(x) A + y B with ab = {A, B}: the spectral product of Eq. 3S in
// the packed form.  (Written as two chains of fused multiply-adds it needs
// two instructions fewer per value, but the longer chains make the fused
// middle stage spill.)
__device__ __forceinline__ float2 packed_product(float2 x, float2 y, float2 A, float2 B) {
  const float2 xa = make_float2(fmaf(x.x, A.x, x.y * A.y), fmaf(x.x, A.y, -x.y * A.x));
  return cadd(xa, cmul(y, B));
}
__device__ __forceinline__ float2 packed_product(float2 x, float2 y, float4 ab) {
  return packed_product(x, y, make_float2(ab.x, ab.y), make_float2(ab.z, ab.w));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// S2-S6: template spectrum, product, sigma, inverse FFT, threshold, compaction
// ---------------------------------------------------------------------------
// Where one correlation's tails (and optional full dump) go.
struct TailOut {
  bege_tail* recs;
  uint64_t cap;
  unsigned long long* counter;
  float* dump;
  // optional per-lag maximum over the bank (Eq. Ak): one 64-bit word per
  // lag, (bits of rho/sigma) << 32 | ~template, raised with atomicMax
  unsigned long long* proj = nullptr;
  // optional upper end of a tail band (Sec. 5): keep |rho| < kappa_hi sigma
  // as well; 0 = no upper end
  float kappa_hi = 0.f;
  // optional overlap-save mask: tails only at lags n < lag_end (the lags
  // whose template window does not wrap); all N lags by default
  uint32_t lag_end = 0xffffffffu;
};

// EXT: the extended epilogue, the per-lag maximum a.proj, the band's upper
// end a.kappa_hi and the lag mask a.lag_end (compiled only into the kernels
// that serve bege_correlate_max, bege_correlate_band and bege_correlate_ex,
// so the others keep their code unchanged).  sigma: the template's sigma (thr = kappa sigma).
//
// emit_row: the S values t[n2] (unscaled, natural order) of row n1, i.e. the
// lags 2 (n1 + F n2) and the next of each.  All lanes of the warp call it.
template <int S, int F, bool EXT>
__device__ __forceinline__ void emit_row(const float2 (&t)[S], int n1, int H, float thr,
                                         uint32_t tmpl, int64_t krow, const TailOut& a,
                                         float sigma) {
  const int lane = threadIdx.x & 31;
  // rho = t / H with H a power of two: |t / H| > thr exactly when |t| > thr H,
  // so the unscaled values are tested and only the emitted ones are scaled
  const float invH = 1.0f / (float)H;
  const float thrH = thr * (float)H;
  // |t / H| < kappa_hi sigma exactly when |t| < kappa_hi sigma H (H a power of two)
  const float hiH = (EXT && a.kappa_hi > 0.f) ? a.kappa_hi * sigma * (float)H : INFINITY;
  float big = 0.f;
#pragma unroll
  for (int n2 = 0; n2 < S; ++n2) big = fmaxf(big, fmaxf(fabsf(t[n2].x), fabsf(t[n2].y)));
  if (a.dump) {
    float2* row = reinterpret_cast<float2*>(a.dump) + krow * (int64_t)H;
#pragma unroll
    for (int n2 = 0; n2 < S; ++n2) row[n1 + F * n2] = cscale(t[n2], invH);
  }
  if (__any_sync(0xffffffffu, big > thrH)) {
    uint32_t mask = 0;
#pragma unroll
    for (int n2 = 0; n2 < S; ++n2) {
      if constexpr (EXT) {
        const float ax = fabsf(t[n2].x), ay = fabsf(t[n2].y);
        const uint32_t lag = (uint32_t)(2 * (n1 + F * n2));
        mask |= (ax > thrH && ax < hiH && lag < a.lag_end ? 1u : 0u) << (2 * n2);
        mask |= (ay > thrH && ay < hiH && lag + 1u < a.lag_end ? 1u : 0u) << (2 * n2 + 1);
      } else {
        mask |= (fabsf(t[n2].x) > thrH ? 1u : 0u) << (2 * n2);
        mask |= (fabsf(t[n2].y) > thrH ? 1u : 0u) << (2 * n2 + 1);
      }
    }
    const int cnt = __popc(mask);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(a.counter, (unsigned long long)total);
    base = __shfl_sync(0xffffffffu, base, 31);
    unsigned long long pos = base + (unsigned long long)(incl - cnt);
#pragma unroll
    for (int n2 = 0; n2 < S; ++n2) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if ((mask >> (2 * n2 + e)) & 1u) {
          if (pos < a.cap) {
            bege_tail* r = a.recs + pos;
            r->tmpl = tmpl;
            r->lag = (uint32_t)(2 * (n1 + F * n2) + e);
            r->value = (e ? t[n2].y : t[n2].x) * invH;
          }
          ++pos;
          if constexpr (EXT) {
            // positive values above the threshold: v > thr > 0, so the
            // bits of v / sigma order like the values; equal values keep
            // the smaller template (larger ~tmpl)
            const float v = (e ? t[n2].y : t[n2].x) * invH;
            if (a.proj && v > thr)
              atomicMax(a.proj + (2 * (n1 + F * n2) + e),
                        ((unsigned long long)__float_as_uint(v * (1.0f / sigma)) << 32) |
                            (unsigned long long)(~tmpl));
          }
        }
      }
    }
  }
}

// The tensor-core form's S-point DFT across columns (column b at colptr[b],
// padded rows) and the tails, in the extended epilogue, of CTA `rank`'s rows, thread `tix` of T.
template <int F, int S, int NC, int T>
__device__ __forceinline__ void combine_and_emit(float2* const* colptr, int H, int rank, float thr,
                                                 uint32_t tmpl, int64_t krow, const TailOut& a,
                                                 float sigma, int tix = threadIdx.x) {
  constexpr int C = ColMap<S, NC>::C;
  constexpr int per = F / C;
  static_assert(per % T == 0, "combine rounds");
#pragma unroll 1
  for (int it = 0; it < per / T; ++it) {
    const int n1 = rank * per + it * T + tix;
    const int pn1 = pad(n1);
    float2 t[S];
#pragma unroll
    for (int b = 0; b < S; ++b) t[b] = colptr[b][pn1];
    dft<S, true>(t);
    emit_row<S, F, true>(t, n1, H, thr, tmpl, krow, a, sigma);
  }
}

// ---------------------------------------------------------------------------
// Launch helpers
// ---------------------------------------------------------------------------
template <typename K>
static cudaError_t ensure_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Clusters of C CTAs of `kern` that fit on the current device at once.  The
// answer does not change, so each kernel keeps it per device (attribute and
// query take 0.4 us together).  The runtime keeps the attribute with the
// kernel, also over a reset of the device and in other contexts.
template <auto kern>
static cudaError_t resident_clusters(int C, int threads, size_t smem, int minb, int* out) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < kDevices && (*out = known[dev].load(std::memory_order_acquire)) > 0) return cudaSuccess;
  e = ensure_smem(kern, smem);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.gridDim = dim3((unsigned)(sms / C * C * minb), 1, 1);
  cfg.dynamicSmemBytes = smem;
  e = cudaOccupancyMaxActiveClusters(out, kern, &cfg);
  if (e != cudaSuccess) return e;
  if (*out < 1) return cudaErrorInvalidConfiguration;
  if (dev < kDevices) known[dev].store(*out, std::memory_order_release);
  return cudaSuccess;
}

// Launches `kern` with clusters of C CTAs (minb CTAs per SM), as many as fit
// and are needed for the templates of a, `each` at a time per cluster.  BEHIND:
// the kernel is made ready while the one before it runs, for which it waits
// itself (cudaGridDependencySynchronize): 2 to 3 us less for a range kernel.
template <auto kern, bool BEHIND = false>
static cudaError_t launch_clusters(int C, int threads, size_t smem, int minb, int each,
                                   const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  int clusters = 0;
  cudaError_t e = resident_clusters<kern>(C, threads, smem, minb, &clusters);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  int64_t want = (a.k1 - a.k0 + each - 1) / each;
  if (a.max_clusters > 0 && want > a.max_clusters) want = a.max_clusters;
  if (want > clusters) want = clusters;
  cfg.gridDim = dim3((unsigned)(want * C), 1, 1);
  if (BEHIND) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, kern, p, a);
}

}  // namespace bege
