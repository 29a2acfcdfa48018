// Internal interface between the C-ABI host layer (bege_api.cpp) and the
// CUDA kernels (the .cu files).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/bege.h"

namespace bege {

// Geometry of the length-N correlation (N = 2H real samples).
//
// The real N-point transforms are carried by H-point complex transforms of
// the even/odd packed sequence z[m] = x[2m] + i x[2m+1].  The H-point
// transform is split by residue: bin j = S a + b (a < F, b < S) lives in
// "column" b, an F-point FFT of a twiddled, folded input (a four-step whose
// first step is pruned by the template's support).  Columns b and S-b hold
// the bins j and H-j that the real-FFT unpacking couples, so they form a
// "unit" of one CTA; the CTAs of a thread-block cluster share the S columns and
// exchange them only for the final S-point combine, through distributed shared
// memory or (exchange_bytes) through L2.  H <= 4096 counts as one column here;
// the FP32 kernels then work on two of half the length (UnitGeo).
struct Geometry {
  int N;    // real samples
  int H;    // N / 2 complex samples
  int F;    // min(H, 4096): the column length for N >= 2^14
  int S;    // H / F (1..16)
};

// Launch shape of the correlate kernel: columns per CTA (the cluster has
// S / nc CTAs) and threads per CTA.  Chosen per N by default or by the
// autotuner.  S = 1 has one shape, listed as {1, 256}: 256 threads, as many
// templates as they have units for.
struct CorrConfig {
  int nc;
  int threads;
};

// Device tables for one N (plan_tables_kernel: FP64, rounded to FP32 once).  wX^k means exp(-2 pi i k / X).
struct PlanDev {
  Geometry g;
  const float2* wS;    // [S of UnitGeo] wS^q
  const float2* wN;    // [H]            wN^j
  // tables of bege_unit.cuh for its columns (UnitGeo), {cos, tan} pairs
  // (rot_entry, unit_table_turn)
  const float2* t1;    // [S][R/2]     stage 1: column b
  const float2* t2;    // [S][8][R]    stage 2: column b, k0
  const float2* t3;    // [S/2][8][T]  stage 3: unit, thread
  const float2* u2;    // [8][16]      stage 2': n0
  const float2* u1;    // [R/2][256]   stage 1': n0 + 16 n1
  const float2* uc;    // [S/2][F]     stage c: n
};

// The correlation's columns: S >= 2 of F points, R = F / 256 and T = F / 16
// threads for two of them.
struct UnitGeo {
  int F, S, R, T;
};
constexpr __host__ __device__ UnitGeo unit_geo(const Geometry& g) {
  return g.S == 1 ? UnitGeo{g.F / 2, 2, g.F / 512, g.F / 32} : UnitGeo{g.F, g.S, g.F / 256, g.F / 16};
}

// Sizes (in float2) of the pair tables, in the order t1, t2, t3, u2, u1, uc.
constexpr int kUnitTables = 6;
constexpr __host__ __device__ int unit_table_size(const UnitGeo& g, int table) {
  switch (table) {
    case 0: return g.S * (g.R / 2);
    case 1: return g.S * 8 * g.R;
    case 2: return g.S / 2 * 8 * g.T;
    case 3: return 128;
    case 4: return g.R / 2 * 256;
    default: return g.S / 2 * g.F;
  }
}

// Entry i of a table: the angle it holds, num / den of a turn.
struct Turn {
  int64_t num, den;
};
// Pair q of an R-point DFT with twiddle base x / M turns: the levels one
// after the other, level l with (R / 2^(l+1)) x base + e / 2^(l+1), e < max(1, 2^(l-1)).
inline __host__ __device__ Turn dft_pair_turn(int R, int q, int64_t x, int64_t M) {
  int l = 0, n = 1;
  while (q >= n) {
    q -= n;
    ++l;
    n = l > 1 ? 1 << (l - 1) : 1;
  }
  const int64_t den = M << (l + 1);
  return {((x * (R >> (l + 1)) << (l + 1)) + q * M) % den, den};
}
inline __host__ __device__ Turn unit_table_turn(const UnitGeo& g, int table, int i) {
  const int R = g.R, S = g.S, T = g.T;
  const int64_t H = (int64_t)S * g.F;
  switch (table) {
    case 0: return dft_pair_turn(R, i % (R / 2), i / (R / 2), R * S);
    case 1: return dft_pair_turn(16, i / R % 8, (int64_t)S * (i % R) + i / (8 * R), 16 * R * S);
    case 2: {
      // thread t of the middle of unit u holds butterfly (k0, k1) of column b
      const int u = i / (8 * T), t = i % T, l = t & 15, w = t >> 5;
      int b = u, k0, k1 = l;
      if (u > 0) {
        k0 = (t & 16) ? R - 1 - w : w;
      } else if (R == 1 ? l >= 8 : (t & 16) != 0) {
        b = S / 2; k0 = w;
        if (R == 1) k1 = l - 8;
      } else if (w > 0) {
        k0 = w;
      } else {
        k0 = l < 8 ? 0 : R / 2; k1 = l & 7;
      }
      return dft_pair_turn(16, i / T % 8, (int64_t)S * (k0 + R * k1) + b, H);
    }
    case 3: return dft_pair_turn(16, i >> 4, i & 15, 256);
    case 4: return dft_pair_turn(R, i >> 8, i & 255, g.F);
    default: return dft_pair_turn(S, i / g.F, i % g.F, H);
  }
}

// {cos, tan} of an angle with FP64 cosine c and sine s, rounded so that
// cos * tan is the sine to FP32 also where the cosine is (nearly) zero.
inline __host__ __device__ float2 rot_entry(double c, double s) {
  float cf = (float)c;
  const float least = 9.31322574615478515625e-10f;  // 2^-30
  if (cf < least && cf > -least) cf = cf < 0.f ? -least : least;
  return make_float2(cf, (float)(s / (double)cf));
}

Geometry make_geometry(int64_t n);

// The tables of geometry g in an array of plan_floats2(g) float2 at `base`,
// and the kernel that writes them there, and 0 to *zero if given.
constexpr __host__ __device__ int plan_floats2(const Geometry& g) {
  const UnitGeo u = unit_geo(g);
  int n = u.S + g.H;
  for (int t = 0; t < kUnitTables; ++t) n += unit_table_size(u, t);
  return n;
}
PlanDev plan_at(const Geometry& g, float2* base);
cudaError_t launch_plan_tables(const Geometry& g, float2* base, cudaStream_t s,
                               unsigned long long* zero = nullptr);

// Record `msg` as the calling thread's last error (bege_last_error) and
// return `code`.
int set_last_error(int code, const std::string& msg);

// CUDA device of a context, and the row count of one of its banks (0 if the
// handle is unknown).
int ctx_device(const bege_ctx* ctx);
// Frees the idle buffers that the context keeps for later calls.
void ctx_drop_spare(bege_ctx* ctx);
int64_t bank_count(bege_ctx* ctx, int32_t bank_id);

// Stop every serving-form server of a context.
void serve_destroy_all(bege_ctx* ctx);

// Launch shapes compiled for geometry g (at most `max`); returns the count.
int correlate_configs(const Geometry& g, CorrConfig* out, int max);
CorrConfig default_config(const Geometry& g);
bool config_valid(const Geometry& g, CorrConfig c);

// S1: segment spectrum.  y: N floats (device).  D: H+1 complex (natural
// order).  AB: H float4 {A_j, B_j}, in residue-major order [b*F + a] (natural:
// the tensor-core kernel) or in the order the FP32 kernels read them.
cudaError_t launch_segment(const PlanDev& p, const float* y, float2* D, float4* AB, bool natural,
                           cudaStream_t s);

// S2..S6 over bank rows [k0, k1).  bank: rows of Lp floats (zero-padded
// beyond L, Lp a multiple of 8).  sigma: k1-k0 floats.  recs/cap/counter:
// tail records.  dump: optional (k1-k0) x N floats of rho.
struct CorrelateArgs {
  const float4* AB;
  const float* bank;
  int64_t Lp;
  int64_t k0, k1;
  float kappa;
  float* sigma;
  bege_tail* recs;
  uint64_t cap;
  unsigned long long* counter;
  float* dump;
  int max_clusters;      // 0 = as many as fit
  unsigned int* status;  // optional: set non-zero by a kernel whose bounded wait gave up
  unsigned long long* proj = nullptr;  // optional: per-lag maximum over the bank (Eq. Ak)
  float kappa_hi = 0.f;                // optional: tails only below kappa_hi sigma (0 = none)
  uint32_t lag_end = 0xffffffffu;      // optional: tails only at lags < lag_end (overlap-save)
  float4* exch = nullptr;              // optional: exchange_bytes, for this launch alone
};
// Bytes of the buffer through which a correlation of `count` templates in
// launch shape cfg can exchange its columns on a GPU of `sms` SMs (two
// templates per resident cluster); 0 where it has no use for one.
size_t exchange_bytes(const Geometry& g, CorrConfig cfg, int64_t count, int sms);
cudaError_t launch_correlate(const PlanDev& p, const CorrelateArgs& a, CorrConfig cfg,
                             cudaStream_t s);
// Behind the FP32 correlation of one segment in any form (single, block,
// batch): the templates whose sigma came out not finite once more in a wider
// range, where that gives another result.  Of use only for a bank that holds
// a sample above kLargeSample (or none that is known).
constexpr float kLargeSample = 0x1p64f;
cudaError_t launch_range(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
// *flag = 1 if one of the n samples (a multiple of 8) is above kLargeSample, else 0.
cudaError_t launch_bank_large(const float* samples, int64_t n, int* flag, cudaStream_t s);

// Several segments of one length against the same templates (Sec. 3.2: a
// template's transform serves a block of segments): per template the
// forward transform runs once, then the product, inverse, sigma and tails
// for each segment m < M into its own outputs.  F = 4096 (N >= 2^14) and
// Lp <= 4096 only.
constexpr int kMaxMulti = 8;
struct MultiArgs {
  const float* bank;
  int64_t Lp;
  int64_t k0, k1;
  float kappa;
  int M;
  const float4* AB[kMaxMulti];
  float* sigma[kMaxMulti];
  bege_tail* recs[kMaxMulti];
  uint64_t cap[kMaxMulti];
  unsigned long long* counter[kMaxMulti];
  float4* scratch;  // multi_scratch_bytes(): the template spectrum of each CTA
};
size_t multi_scratch_bytes(int sms);
cudaError_t launch_correlate_multi(const PlanDev& p, const MultiArgs& a, cudaStream_t s);

// Per-S launchers (one translation unit each).
cudaError_t launch_correlate_s1(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_correlate_s2(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_correlate_s4(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                cudaStream_t s);
cudaError_t launch_correlate_s8(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                cudaStream_t s);
cudaError_t launch_correlate_s16(const PlanDev& p, const CorrelateArgs& a, CorrConfig c,
                                 cudaStream_t s);
cudaError_t launch_range_s1(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_range_s2(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_range_s4(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_range_s8(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);
cudaError_t launch_range_s16(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s);

// Precision form: S2-S6 with the column FFTs on tcgen05 tensor cores.
// precision 1 = BF16x3, 2 = FP16x3.  Needs F = 4096 (N >= 2^14) and
// Lp <= 4096.
cudaError_t launch_correlate_tc(const PlanDev& p, const CorrelateArgs& a, int precision,
                                cudaStream_t s);

// Bank synthesis: count chirps, phase coefficients alpha/beta as unsigned
// 64-bit fixed point (cycles * 2^64), L samples, taper fraction; rows of Lp;
// symmetric: the chirp plus its time reversal (Fig. 2 caption).
cudaError_t launch_bank_chirp(const unsigned long long* alpha_beta, int64_t count, int64_t L,
                              int64_t Lp, double taper_frac, bool symmetric, float* bank,
                              cudaStream_t s);

}  // namespace bege
