// Geometry, plan tables, launch shapes, the segment-spectrum launcher and
// chirp-bank synthesis.
#include <algorithm>

#include "bege_unit.cuh"

namespace bege {

Geometry make_geometry(int64_t n) {
  Geometry g{};
  g.N = (int)n;
  g.H = g.N / 2;
  g.F = g.H < 4096 ? g.H : 4096;
  g.S = g.H / g.F;
  return g;
}

PlanDev plan_at(const Geometry& g, float2* base) {
  PlanDev p{};
  p.g = g;
  const UnitGeo u = unit_geo(g);
  const float2** const table[kUnitTables] = {&p.t1, &p.t2, &p.t3, &p.u2, &p.u1, &p.uc};
  for (int t = 0; t < kUnitTables; ++t) {
    *table[t] = base;
    base += unit_table_size(u, t);
  }
  p.wS = base;
  p.wN = base + u.S;
  return p;
}

// One table entry per thread (plan_at's order).
__global__ void __launch_bounds__(256)
plan_tables_kernel(Geometry g, float2* __restrict__ base, unsigned long long* zero) {
  int i = blockIdx.x * 256 + threadIdx.x;
  if (i == 0 && zero) *zero = 0;
  if (i >= plan_floats2(g)) return;
  float2* const out = base + i;
  const UnitGeo u = unit_geo(g);
  double s, c;
  for (int t = 0; t < kUnitTables; ++t) {
    if (i < unit_table_size(u, t)) {
      const Turn a = unit_table_turn(u, t, i);
      sincospi(2.0 * (double)a.num / (double)a.den, &s, &c);
      *out = rot_entry(c, s);
      return;
    }
    i -= unit_table_size(u, t);
  }
  const bool ws = i < u.S;  // exp(-2 pi i k / S), then exp(-2 pi i j / N)
  sincospi(-2.0 * (double)(ws ? i : i - u.S) / (double)(ws ? u.S : g.N), &s, &c);
  *out = make_float2((float)c, (float)s);
}

cudaError_t launch_plan_tables(const Geometry& g, float2* base, cudaStream_t s,
                               unsigned long long* zero) {
  plan_tables_kernel<<<(plan_floats2(g) + 255) / 256, 256, 0, s>>>(g, base, zero);
  return cudaGetLastError();
}

int correlate_configs(const Geometry& g, CorrConfig* out, int max) {
  CorrConfig all[4];
  int n = 0;
  if (g.S == 1) {
    all[n++] = {1, 256};
  } else if (g.S == 2) {
    all[n++] = {2, 256};
  } else {
    all[n++] = {2, 256};
    all[n++] = {4, 512};
  }
  for (int i = 0; i < n && i < max; ++i) out[i] = all[i];
  return n;
}

bool config_valid(const Geometry& g, CorrConfig c) {
  CorrConfig all[4];
  const int n = correlate_configs(g, all, 4);
  for (int i = 0; i < n; ++i)
    if (all[i].nc == c.nc && all[i].threads == c.threads) return true;
  return false;
}

// Default launch shape.  S >= 4: two units (512 threads) a CTA, one CTA per
// SM, so half as many CTAs meet in a cluster and a unit's neighbour in the
// CTA needs no distributed shared memory; S = 2 has one unit a template and
// two CTAs per SM.  Per template (65536 chirps, GB300), 4 x 512 against 2 x
// 256: N = 2^15 78 / 83 ns, 2^16 171 / 189, 2^17 405 / 420 (and 165 and 354 with
// the exchange through L2, which takes this shape).
CorrConfig default_config(const Geometry& g) {
  if (g.S == 1) return {1, 256};
  if (g.S == 2) return {2, 256};
  return {4, 512};
}

size_t exchange_bytes(const Geometry& g, CorrConfig cfg, int64_t count, int sms) {
  if (g.S < 8 || cfg.nc != 4) return 0;
  // one CTA of 4 columns per SM: no more than sms / (S / 4) clusters are resident
  const int64_t clusters = std::min<int64_t>(count, sms / (g.S / 4));
  return (size_t)clusters * g.S * 4096 * sizeof(float4);
}

cudaError_t launch_segment(const PlanDev& p, const float* y, float2* D, float4* AB, bool natural,
                           cudaStream_t s) {
  switch (unit_geo(p.g).F) {
    case 256: return unit::launch_segment_t<256, true>(p, y, D, AB, natural, s);
    case 512: return unit::launch_segment_t<512, true>(p, y, D, AB, natural, s);
    case 1024: return unit::launch_segment_t<1024, true>(p, y, D, AB, natural, s);
    case 2048: return unit::launch_segment_t<2048, true>(p, y, D, AB, natural, s);
    case 4096: return unit::launch_segment_t<4096, false>(p, y, D, AB, natural, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_correlate(const PlanDev& p, const CorrelateArgs& a, CorrConfig cfg,
                             cudaStream_t s) {
  if (a.k1 <= a.k0) return cudaSuccess;
  const Geometry& g = p.g;
  if (!config_valid(g, cfg)) return cudaErrorInvalidValue;
  switch (g.S) {
    case 1: return launch_correlate_s1(p, a, s);
    case 2: return launch_correlate_s2(p, a, s);
    case 4: return launch_correlate_s4(p, a, cfg, s);
    case 8: return launch_correlate_s8(p, a, cfg, s);
    case 16: return launch_correlate_s16(p, a, cfg, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_range(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  if (a.k1 <= a.k0) return cudaSuccess;
  switch (p.g.S) {
    case 1: return launch_range_s1(p, a, s);
    case 2: return launch_range_s2(p, a, s);
    case 4: return launch_range_s4(p, a, s);
    case 8: return launch_range_s8(p, a, s);
    case 16: return launch_range_s16(p, a, s);
    default: return cudaErrorInvalidValue;
  }
}

// Bound by the read of the bank from HBM, once after its upload.
__global__ void __launch_bounds__(256)
bank_large_kernel(const float4* __restrict__ w, int64_t n, int* __restrict__ flag) {
  bool large = false;
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
    const float4 v = __ldg(w + i);
    large |= !(fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))) <= kLargeSample);
  }
  if (large) *flag = 1;
}

cudaError_t launch_bank_large(const float* samples, int64_t n, int* flag, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  const int64_t blocks = std::min<int64_t>((n / 4 + 255) / 256, 152 * 8);
  bank_large_kernel<<<(unsigned)blocks, 256, 0, s>>>(reinterpret_cast<const float4*>(samples), n / 4,
                                                     flag);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Bank synthesis: w[m] = T(m) sin(2 pi phase(m)), unit L2 norm; time-
// symmetric banks (Fig. 2 caption): w[m] = T(m) (sin(2 pi phase(m)) +
// sin(2 pi phase(L - 1 - m))), the chirp forward and backward in time.
// ---------------------------------------------------------------------------
// sin(2 pi phase / 2^64) at kKeep samples m0, m0 + d, m0 + 2 d, ...: the phase
// alpha m + beta m^2 (cycles * 2^64, exact modulo one cycle) is quadratic in m,
// so the unit phasor advances by a factor that itself advances by the constant
// factor `turn` = exp(2 pi i 2 beta d^2).  The start values have exact phases.
// After i <= 15 steps a sample holds i (i - 1) / 2 times the error of `turn`, i
// times that of the first step and i (i + 1) / 2 roundings of a product, below
// 1e-13 in all (1.2e-14 is the largest of 200000 random chirps): far below half
// an FP32 ulp of a unit sine, so only rounding ties can differ.
constexpr int kChirpThreads = 256;
constexpr int kKeep = 16;

struct Phasor {
  double c, s;
};
__device__ __forceinline__ Phasor phasor(unsigned long long cycles) {
  Phasor p;
  sincospi((double)(long long)cycles * 0x1p-63, &p.s, &p.c);  // half turns in [-1, 1)
  return p;
}
__device__ __forceinline__ Phasor turned(Phasor a, Phasor b) {
  return {fma(a.c, b.c, -a.s * b.s), fma(a.c, b.s, a.s * b.c)};
}
__device__ __forceinline__ void add_chirp(unsigned long long alpha, unsigned long long beta,
                                          int64_t m0, int64_t d, Phasor turn, double (&v)[kKeep]) {
  const unsigned long long m = (unsigned long long)m0, e = (unsigned long long)d;
  Phasor p = phasor(alpha * m + beta * (m * m));
  Phasor step = phasor(alpha * e + beta * (2 * m * e + e * e));
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    v[i] += p.s;
    p = turned(p, step);
    step = turned(step, turn);
  }
}

// Samples base + 256 i of thread threadIdx.x, unscaled (0 from L on).
__device__ __forceinline__ void chirp_samples(unsigned long long alpha, unsigned long long beta,
                                              int64_t base, int64_t L, int width, double denom,
                                              bool symmetric, Phasor turn, double (&v)[kKeep]) {
  const int64_t m0 = base + threadIdx.x;
#pragma unroll
  for (int i = 0; i < kKeep; ++i) v[i] = 0.0;
  if (m0 >= L) return;
  add_chirp(alpha, beta, m0, kChirpThreads, turn, v);
  if (symmetric) add_chirp(alpha, beta, L - 1 - m0, -kChirpThreads, turn, v);
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int64_t m = m0 + (int64_t)kChirpThreads * i;
    const int64_t mm = m < L - 1 - m ? m : L - 1 - m;
    if (m >= L)
      v[i] = 0.0;
    else if (mm <= width)
      v[i] *= 0.5 * (1.0 - cospi(2.0 * (double)mm / denom));
  }
}

// One CTA per row.  Bound: FP64 (two lanes' worth per SM and cycle).  Rows of
// up to 4096 samples are evaluated once and kept in registers between the
// norm and the store; a sample costs two complex products and its share of
// the start values, about 14 FP64 instructions, where two evaluations of sinpi
// took about 60 (2^20 rows of 4096 samples: 415 -> 148 ms).
__global__ void __launch_bounds__(kChirpThreads)
bank_chirp_kernel(const unsigned long long* __restrict__ ab, int64_t L, int64_t Lp, double frac,
                  bool symmetric, float* __restrict__ bank) {
  __shared__ double red[8];
  __shared__ Phasor shared_turn;
  const int64_t k = blockIdx.x;
  const unsigned long long alpha = ab[2 * k], beta = ab[2 * k + 1];
  const int width = (frac > 0.0 && L >= 2) ? (int)floor(frac * (double)(L - 1) / 2.0) : -1;
  const double denom = frac * (double)(L - 1);
  if (threadIdx.x == 0)
    shared_turn = phasor(beta * (2ull * kChirpThreads * kChirpThreads));
  __syncthreads();
  const Phasor turn = shared_turn;
  constexpr int64_t kChunk = kChirpThreads * kKeep;
  double v[kKeep];
  double acc = 0.0;
  for (int64_t base = 0; base < L; base += kChunk) {
    chirp_samples(alpha, beta, base, L, width, denom, symmetric, turn, v);
#pragma unroll
    for (int i = 0; i < kKeep; ++i) acc = fma(v[i], v[i], acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  double norm = 0.0;
  for (int w = 0; w < kChirpThreads / 32; ++w) norm += red[w];
  const double scale = norm > 0.0 ? 1.0 / sqrt(norm) : 0.0;
  float* row = bank + k * Lp;
  for (int64_t base = 0; base < Lp; base += kChunk) {
    if (L > kChunk) chirp_samples(alpha, beta, base, L, width, denom, symmetric, turn, v);
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
      const int64_t m = base + threadIdx.x + (int64_t)kChirpThreads * i;
      if (m < Lp) row[m] = (float)(v[i] * scale);
    }
  }
}

cudaError_t launch_bank_chirp(const unsigned long long* alpha_beta, int64_t count, int64_t L,
                              int64_t Lp, double taper_frac, bool symmetric, float* bank,
                              cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  bank_chirp_kernel<<<(unsigned)count, kChirpThreads, 0, s>>>(alpha_beta, L, Lp, taper_frac, symmetric,
                                                    bank);
  return cudaGetLastError();
}

}  // namespace bege
