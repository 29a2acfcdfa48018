// Internal interface between the C-ABI host layer (bege_api.cpp) and the
// CUDA kernels (bege_kernels.cu).  Not part of the public ABI.
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
// "unit" processed by one CTA; the CTAs of a thread-block cluster share the
// S columns and exchange them through distributed shared memory only for
// the final S-point combine.
struct Geometry {
  int N;    // real samples
  int H;    // N / 2 complex samples
  int F;    // column FFT length (512..4096)
  int S;    // columns = H / F (1..16)
  int R0;   // radix of the first Stockham pass = F / 256
};

// Launch shape of the correlate kernel: columns per CTA (the cluster has
// S / nc CTAs) and threads per CTA.  Chosen per N by default or by the
// autotuner.
struct CorrConfig {
  int nc;
  int threads;
};

// Device twiddle tables for one N (computed in FP64 on the host, rounded to
// FP32 once).  wX^k means exp(-2 pi i k / X).
struct PlanDev {
  Geometry g;
  const float2* tw2;   // [16*R0]  Stockham pass 2: [r*R0 + k] = w(16 R0)^(k r)
  const float2* tw3;   // [F]      Stockham pass 3: [r*(F/16) + k] = wF^(k r)
  const float2* wH;    // [256*S]  wH^k
  const float2* wR0S;  // [R0*S]   w(R0 S)^q
  const float2* wS;    // [S]      wS^q
  const float2* wN;    // [H]      wN^j
  // S >= 2, {cos, tan} sets of bege_unit.cuh (rot_entry, set_turns):
  const float2* t1;    // [S][8]         stage 1: column b
  const float2* t2;    // [S][8][16]     stage 2: column b, k0
  const float2* t3;    // [S/2][8][256]  stage 3: unit, thread
  const float2* u2;    // [8][16]        stage 2': n0
  const float2* u1;    // [8][256]       stage 1': n0 + 16 n1
  const float2* uc;    // [S/2][4096]    stage c: n
};

// Sizes (in float2) of the sets of an S-column plan, in the order t1, t2, t3,
// u2, u1, uc; all 0 for S = 1.
constexpr int kUnitTables = 6;
constexpr __host__ __device__ int unit_table_size(int S, int table) {
  if (S < 2) return 0;
  switch (table) {
    case 0: return 8 * S;
    case 1: return 128 * S;
    case 2: return 1024 * S;
    case 3: return 128;
    case 4: return 2048;
    default: return 2048 * S;
  }
}

// Entry i of a table: the angle it holds, num / den of a turn.
struct Turn {
  int64_t num, den;
};
inline __host__ __device__ Turn unit_table_turn(int S, int table, int i) {
  int64_t x = 0, M = 1;  // base x / M turns
  int q = 0;             // place in the 16-point set
  switch (table) {
    case 0: q = i & 7; x = i >> 3; M = 16 * S; break;
    case 1: {
      const int b = i >> 7, k0 = i & 15;
      q = (i >> 4) & 7; x = S * k0 + b; M = 256 * S;
      break;
    }
    case 2: {
      // thread t of the middle of unit u holds butterfly (k0, k1) of column b
      const int u = i >> 11, t = i & 255, l = t & 15;
      int b = u, k0, k1 = l;
      if (u > 0) {
        k0 = (t & 16) ? 15 - (t >> 5) : t >> 5;
      } else if (t & 16) {
        b = S / 2; k0 = t >> 5;
      } else if (t >= 32) {
        k0 = t >> 5;
      } else {
        k0 = l < 8 ? 0 : 8; k1 = l & 7;
      }
      q = (i >> 8) & 7; x = (int64_t)S * (k0 + 16 * k1) + b; M = 4096 * (int64_t)S;
      break;
    }
    case 3: q = i >> 4; x = i & 15; M = 256; break;
    case 4: q = i >> 8; x = i & 255; M = 4096; break;
    default: {
      // the S-point DFT uses the end of the set: S = 2 {base}, 4 {2 x base,
      // base}, 8 {4 x, 2 x, base, base + 1/8}, 16 the whole set
      const int e = i >> 12;
      x = i & 4095; M = 4096 * (int64_t)S;
      const int64_t den = 16 * M;
      if (S == 16) { q = e; break; }
      if (S == 8 && e == 3) return {(16 * x + 2 * M) % den, den};
      const int levels = S == 8 ? 2 : S == 4 ? 1 : 0;
      return {(16 * x << (levels - e)) % den, den};
    }
  }
  const int64_t den = 16 * M;
  switch (q) {
    case 0: return {128 * x % den, den};
    case 1: return {64 * x % den, den};
    case 2: return {32 * x % den, den};
    case 3: return {(32 * x + 2 * M) % den, den};
    default: return {(16 * x + (q - 4) * M) % den, den};
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

// Record `msg` as the calling thread's last error (bege_last_error) and
// return `code`.
int set_last_error(int code, const std::string& msg);

// CUDA device of a context, and the row count of one of its banks (0 if the
// handle is unknown).
int ctx_device(const bege_ctx* ctx);
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
};
cudaError_t launch_correlate(const PlanDev& p, const CorrelateArgs& a, CorrConfig cfg,
                             cudaStream_t s);

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
  float2* scratch;  // multi_scratch_bytes(): the template spectrum of each CTA
};
size_t multi_scratch_bytes(int sms);
cudaError_t launch_correlate_multi(const PlanDev& p, const MultiArgs& a, cudaStream_t s);

// Per-S launchers (one translation unit each); halfz: Lp <= F.
cudaError_t launch_correlate_s1(const PlanDev& p, const CorrelateArgs& a, CorrConfig c, bool halfz,
                                cudaStream_t s);
cudaError_t launch_correlate_s2(const PlanDev& p, const CorrelateArgs& a, CorrConfig c, bool halfz,
                                cudaStream_t s);
cudaError_t launch_correlate_s4(const PlanDev& p, const CorrelateArgs& a, CorrConfig c, bool halfz,
                                cudaStream_t s);
cudaError_t launch_correlate_s8(const PlanDev& p, const CorrelateArgs& a, CorrConfig c, bool halfz,
                                cudaStream_t s);
cudaError_t launch_correlate_s16(const PlanDev& p, const CorrelateArgs& a, CorrConfig c, bool halfz,
                                 cudaStream_t s);

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
