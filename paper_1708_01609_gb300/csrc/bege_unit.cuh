// The correlation: per-stage functions of one unit (two columns of F points,
// F / 16 threads) shared by the single, block and batch kernels, and the
// single-segment kernels themselves.  N >= 2^14 has S = N / 8192 columns of F =
// 4096 points; shorter segments have S = 2 columns of F = N / 4 = 256 .. 2048.
//
// Stages.  With the column split of bege_corr.cuh, j = S a + b, and R = F /
// 256, write a = k0 + R k1 + 16 R k2 and m = n0 + 16 n1 + 256 n2 (k0, n2 < R,
// the others < 16).  Forward (z -> Z):
//   1  over n2 -> k0   twiddle base b / (R S)
//   2  over n1 -> k1   base (S k0 + b) / (16 R S)
//   3  over n0 -> k2   base (S (k0 + R k1) + b) / H
// inverse (Y -> rho), n = n0 + 16 n1 + 256 n2 + F n3:
//   3' over k2 -> n0   no twiddle
//   2' over k1 -> n1   base n0 / 256
//   1' over k0 -> n2   base (n0 + 16 n1) / F
//   c  over b  -> n3   base (n0 + 16 n1 + 256 n2) / H
// (bases in turns; input r of a stage is turned by r times its base).  Each
// stage is a decimation-in-time DFT whose input twiddles are w^r for one base
// w, so every twiddle, the column's own w_H^(b m) and w_H^(-b n) included,
// enters a radix-2 butterfly a +/- w b as two fused multiply-adds: w b =
// cos (1 -/+ i tan) b, u = (1 -/+ i tan) b and a +/- cos u, six operations
// for a butterfly at any angle, and a 16-point stage needs 8 (cos, tan)
// pairs in place of 15 factors.  The table keeps |cos| >= 2^-30 with tan =
// sin / cos, so cos * tan rounds sin also where the cosine vanishes (the
// leftover 2^-30 is far below an FP32 rounding); each u is rounded once and
// scaled by cos, which costs no more than the rounding of a plain product.
//
// Every stage works in place: a butterfly writes the 16 rows it read, so the
// spectrum sits digit-reversed in shared memory, the product reads its
// coefficients in the same order (segment_unit), and one ordering point between
// stages is enough.  Stages 2, 3, 3', 2' exchange values only between
// threads of the same k0; warp w of a unit holds k0 = w and R - 1 - w (a column
// bin's mirror has every digit complemented), so between them a warp waits
// for itself only and the warps drift: the loads of one overlap the
// arithmetic of another.  Unit 0 (columns 0 and S/2, each its own mirror)
// pairs k0 with R - k0 in column 0 and hands over between warps there.
//
// Rows.  Block k0 (256 rows, 288 16-byte slots) of a unit holds its two
// columns interleaved (float4 {slot 0, slot 1}, row i at slot i) between
// stages 1-2 and from 2' on, and as two arrays of 16 x 18 float2 (column c,
// row n0 + 16 k1 at 288 c + n0 + 18 k1) from 2 to 2': the middle reads and
// writes 16 consecutive values of one column as 8 16-byte accesses, free of
// bank conflicts, and its mirror butterfly in the other column likewise.
//
// Bound: FP32 issue and shared-memory bandwidth (FFT butterflies), not HBM: at
// N = 2^16 a correlation issues 108.6e3 warp instructions (91e3 of them on the
// FMA pipe) and moves 20e3 shared-memory wavefronts, 52% and 37% of what its
// time allows (at N = 2^14 59% and 42%); what is left is latency (barriers, L2
// coefficients) with 16 warps per SM, all that 128 registers a thread allow.
// Per template of 1 s, against Stockham passes with plain twiddle products and
// ten CTA barriers a template (65536 chirps, GB300): N = 2^14 49.6 -> 35.0 ns,
// 2^15 102 -> 78, 2^16 216 -> 165, 2^17 472 -> 354.
// Measured beside it and not kept: packed FP32 pairs (an FFMA2 takes the FMA
// pipe 2.2 to 2.5 cycles, no less than two FFMAs); columns of 2048 points with
// 128-thread units (183 ns at 2^16, 41 at 2^14); stage 1' storing straight
// into the CTA that combines (209 ns against 191 for reading there, with
// clusters of four); one column's butterflies after the other's (level).
#pragma once

#include "bege_corr.cuh"

namespace bege {
namespace unit {

constexpr int kF = 4096;        // column length of N >= 2^14
constexpr int kBlk = 288;       // 16-byte slots of a block of 256 rows
constexpr float kMaxFinite = 3.402823466e38f;
constexpr float kScaleDown = 0x1p-64f, kScaleUp = kLargeSample;  // see "Range"

template <int F>
struct Geo {
  static constexpr int R = F / 256;   // radix of stages 1 and 1', blocks of a unit
  static constexpr int T = F / 16;    // threads of a unit
  static constexpr int W = T < 32 ? 1 : T / 32;
  static constexpr int P = R / 2;     // pairs of an R-point DFT
  static_assert(F == 256 || F == 512 || F == 1024 || F == 2048 || F == 4096, "column length");
};

// Shared memory of a CTA with U units (bytes).  ONE: every unit is the only
// one of a template (S = 2), so they share all tables.
template <int F, int U, bool ONE>
struct Lay {
  using G = Geo<F>;
  static constexpr size_t n3 = 8 * G::T * 8, n2 = 8 * G::R * 16, n1 = (G::P + 1) / 2 * 32;
  static constexpr size_t u1 = 0;                        // [P][256] float2: stage 1'
  static constexpr size_t u2 = u1 + G::P * 256 * 8;      // [8][16] float2: stage 2'
  static constexpr size_t ws = u2 + 8 * 16 * 8;          // [16] float2: w_S^q (folded templates)
  static constexpr size_t rowptr = ws + 16 * 8;          // [8] the units' rows in the cluster
  static constexpr size_t sigall = rowptr + 8 * 8;       // [2][8] units' shares of sum |Y|^2
  static constexpr size_t red = sigall + 2 * 8 * 4;          // [U][W] warp sums
  static constexpr size_t one = align16(red + U * G::W * 4);
  static constexpr size_t units = one + (ONE ? n3 + n2 + n1 : 0);
  // within a unit
  static constexpr size_t rows = 0;                      // R blocks
  static constexpr size_t tab = rows + G::R * kBlk * 16; // its tables (ONE: at `one`)
  static constexpr size_t unit_bytes = tab + (ONE ? 0 : n3 + n2 + n1);
  static constexpr size_t total = units + U * unit_bytes;
  // tables: [8][T] float2: stage 3; [8][R] float4: stage 2, both columns;
  // [P] float4: stage 1, both columns
  static_assert(units % 16 == 0 && unit_bytes % 16 == 0, "16-byte rows");
};

template <int F, int U, bool ONE = false>
struct Sm {
  using L = Lay<F, U, ONE>;
  using G = Geo<F>;
  static __device__ __forceinline__ unsigned char* unit(int ui) {
    return smem_raw + L::units + (U == 1 ? 0 : ui * L::unit_bytes);
  }
  static __device__ __forceinline__ unsigned char* tab(int ui) {
    return ONE ? smem_raw + L::one : unit(ui) + L::tab;
  }
  static __device__ __forceinline__ float4* rows(int ui) { return reinterpret_cast<float4*>(unit(ui) + L::rows); }
  static __device__ __forceinline__ float2* t3(int ui) { return reinterpret_cast<float2*>(tab(ui)); }
  static __device__ __forceinline__ float4* t2(int ui) { return reinterpret_cast<float4*>(tab(ui) + L::n3); }
  static __device__ __forceinline__ float4* t1(int ui) { return reinterpret_cast<float4*>(tab(ui) + L::n3 + L::n2); }
  static __device__ __forceinline__ float* red(int ui) { return reinterpret_cast<float*>(smem_raw + L::red) + ui * G::W; }
  static __device__ __forceinline__ float2* u1() { return reinterpret_cast<float2*>(smem_raw + L::u1); }
  static __device__ __forceinline__ float2* u2() { return reinterpret_cast<float2*>(smem_raw + L::u2); }
  static __device__ __forceinline__ float2* ws() { return reinterpret_cast<float2*>(smem_raw + L::ws); }
  static __device__ __forceinline__ float4** rowptr() { return reinterpret_cast<float4**>(smem_raw + L::rowptr); }
  static __device__ __forceinline__ float* sigall() { return reinterpret_cast<float*>(smem_raw + L::sigall); }
  static __device__ __forceinline__ int tid() { return threadIdx.x & (G::T - 1); }
  // the block k0 that this thread works on in stages 2 and 2', and its n0
  static __device__ __forceinline__ int k0() {
    if constexpr (G::R == 1) return 0;
    const int w = tid() >> 5;
    return (threadIdx.x & 16) ? G::R - 1 - w : w;
  }
  static __device__ __forceinline__ int n0() { return threadIdx.x & 15; }
  // all threads of the unit
  static __device__ __forceinline__ void sync(int ui) {
    if constexpr (G::T <= 32)
      __syncwarp();
    else if constexpr (U == 1)
      __syncthreads();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(ui + 1), "n"(G::T) : "memory");
  }
};

__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// DFTs with merged twiddles
// ---------------------------------------------------------------------------
// (a, b) -> (a + w b, a - w b), w = e^(-/+ i angle) (-/+ i)^K, {c, t} = (cos, tan) of the angle.
template <bool INV, int K>
__device__ __forceinline__ void bfly(float2& a, float2& b, float c, float t) {
  float2 u = rot_a<INV>(b, t);
  if constexpr (K == 1) u = mul_mi<INV>(u);
  b = cfma(a, -c, u);
  a = cfma(a, c, u);
}

// The index that holds output k of an R-point DFT below (bit-reversed).
template <int R>
__host__ __device__ constexpr int rev(int k) {
  int r = 0;
  for (int b = 1; b < R; b <<= 1) r = 2 * r + ((k & b) ? 1 : 0);
  return r;
}

// 16-point DFTs of two columns, twiddle pairs w(q) = {c_a, t_a, c_b, t_b}:
// q = 0: 8 x base, 1: 4 x, 2: 2 x, 3: 2 x + 1/8, 4 + i: base + i/16 (turns).
// HALFZ: inputs 8..15 are zero (and not read).
template <bool INV, bool HALFZ, class W>
__device__ __forceinline__ void dft16x2(float2 (&a)[16], float2 (&b)[16], W w) {
  if constexpr (!HALFZ) {
    const float4 s = w(0);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      bfly<INV, 0>(a[r], a[r + 8], s.x, s.y);
      bfly<INV, 0>(b[r], b[r + 8], s.z, s.w);
    }
  }
  {
    const float4 s = w(1);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if constexpr (HALFZ) {
        a[8 + r] = a[r]; a[12 + r] = a[4 + r];
        b[8 + r] = b[r]; b[12 + r] = b[4 + r];
      }
      bfly<INV, 0>(a[r], a[r + 4], s.x, s.y);
      bfly<INV, 1>(a[8 + r], a[12 + r], s.x, s.y);
      bfly<INV, 0>(b[r], b[r + 4], s.z, s.w);
      bfly<INV, 1>(b[8 + r], b[12 + r], s.z, s.w);
    }
  }
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const float4 s = w(2 + p);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      bfly<INV, 0>(a[8 * p + r], a[8 * p + r + 2], s.x, s.y);
      bfly<INV, 1>(a[8 * p + 4 + r], a[8 * p + 4 + r + 2], s.x, s.y);
      bfly<INV, 0>(b[8 * p + r], b[8 * p + r + 2], s.z, s.w);
      bfly<INV, 1>(b[8 * p + 4 + r], b[8 * p + 4 + r + 2], s.z, s.w);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 s = w(4 + i);
    const int o = 8 * (i & 1) + 4 * (i >> 1);
    bfly<INV, 0>(a[o], a[o + 1], s.x, s.y);
    bfly<INV, 1>(a[o + 2], a[o + 3], s.x, s.y);
    bfly<INV, 0>(b[o], b[o + 1], s.z, s.w);
    bfly<INV, 1>(b[o + 2], b[o + 3], s.z, s.w);
  }
}

// S-point DFT (S = 2 .. 16) of one row.  Level l (of log2 S) of the pairs w(q)
// holds (S / 2^(l+1)) x base + i / 2^(l+1) turns for i < max(1, 2^(l-1)), the
// levels one after the other: S/2 pairs.
template <int S, bool INV, class W>
__device__ __forceinline__ void dft_row(float2 (&x)[S], W w) {
  int q = 0;
#pragma unroll
  for (int half = S / 2; half >= 1; half >>= 1) {
    const int groups = S / 2 / half;           // 2^l groups of 2 half inputs
    const int n = groups > 1 ? groups / 2 : 1; // distinct pairs; the others are turned by 1/4
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float2 s = w(q + i);
      // group index: the bits of i reversed in front, the 1/4-turn bit last
      int g = 0;
#pragma unroll
      for (int b = 1; b < n; b <<= 1) g = 2 * g + ((i & b) ? 1 : 0);
      const int o = groups > 1 ? 4 * half * g : 0;
#pragma unroll
      for (int r = 0; r < half; ++r) {
        bfly<INV, 0>(x[o + r], x[o + r + half], s.x, s.y);
        if (groups > 1) bfly<INV, 1>(x[o + 2 * half + r], x[o + 3 * half + r], s.x, s.y);
      }
    }
    q += n;
  }
}

// ---------------------------------------------------------------------------
// Set-up
// ---------------------------------------------------------------------------
template <class SM, int THREADS>
__device__ __forceinline__ void setup_common(const PlanDev& p) {
  for (int i = threadIdx.x; i < SM::G::P * 256; i += THREADS) SM::u1()[i] = p.u1[i];
  for (int i = threadIdx.x; i < 8 * 16; i += THREADS) SM::u2()[i] = p.u2[i];
}

// Tables of unit ug (columns ug and S - ug; unit 0: 0 and S/2) in slot ui, by
// its threads.
template <class SM>
__device__ __forceinline__ void setup_unit(const PlanDev& p, int S, int ug, int ui) {
  using G = typename SM::G;
  const int t = SM::tid();
  const int ba = ug, bb = ug == 0 ? S / 2 : S - ug;
  for (int i = t; i < 8 * G::T; i += G::T) SM::t3(ui)[i] = p.t3[ug * 8 * G::T + i];
  for (int i = t; i < 8 * G::R; i += G::T) {
    const float2 a = p.t2[ba * 8 * G::R + i], b = p.t2[bb * 8 * G::R + i];
    SM::t2(ui)[i] = make_float4(a.x, a.y, b.x, b.y);
  }
  if (t < G::P) {
    const float2 a = p.t1[ba * G::P + t], b = p.t1[bb * G::P + t];
    SM::t1(ui)[t] = make_float4(a.x, a.y, b.x, b.y);
  }
  if (ui == 0 && t < 16) SM::ws()[t] = t < S ? p.wS[t] : make_float2(1.f, 0.f);
}

// ---------------------------------------------------------------------------
// Stages
// ---------------------------------------------------------------------------
// Writes the outputs of an R-point stage over n2 / k0: butterfly i of a thread
// holds rows tid + T i + 256 r, output k at v[i][rev<R>(k)].
template <class SM>
__device__ __forceinline__ void store_blocks(int ui, const float2 (&va)[16 / SM::G::R][SM::G::R],
                                             const float2 (&vb)[16 / SM::G::R][SM::G::R]) {
  constexpr int R = SM::G::R, T = SM::G::T;
  float4* row = SM::rows(ui) + SM::tid();
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int k = 0; k < R; ++k)
      row[k * kBlk + T * i] = make_float4(va[i][rev<R>(k)].x, va[i][rev<R>(k)].y,
                                          vb[i][rev<R>(k)].x, vb[i][rev<R>(k)].y);
}

// Stage 1 from the template's nz complex samples z.  HALFZ: the upper half of
// the columns is zero (nz <= F / 2).  ONE: two columns (S = 2) and nz <= 2 F.
// Otherwise folded over nfold multiples of F.  WAIT: the cluster's reads of the
// previous contents of the rows are awaited after the loads and the
// arithmetic, before the stores.  arrive: the cluster's barrier is arrived at
// there.  SCALED: z times `scale`.
template <class SM, bool HALFZ, bool ONE, bool WAIT, bool SCALED = false>
__device__ __forceinline__ void stage1(int ui, int S, int ug, const float* __restrict__ src,
                                       int nz, int nfold, bool arrive = false, float scale = 1.f) {
  constexpr int R = SM::G::R, T = SM::G::T, F = 256 * R;
  const float2* z = reinterpret_cast<const float2*>(src);
  const int t = SM::tid();
  auto load = [&](int m) {
    const float2 x = m < nz ? __ldg(z + m) : make_float2(0.f, 0.f);
    return SCALED ? cscale(x, scale) : x;
  };
  float2 va[16 / R][R], vb[16 / R][R];
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int r = 0; r < (HALFZ ? R / 2 : R); ++r) {
      const int m = t + T * i + 256 * r;
      const float2 x = load(m);
      if constexpr (ONE && !HALFZ) {
        const float2 y = load(m + F);
        va[i][r] = cadd(x, y);
        vb[i][r] = csub(x, y);
      } else {
        va[i][r] = vb[i][r] = x;
      }
    }
  if constexpr (!HALFZ && !ONE) {
    const int bb = ug == 0 ? S / 2 : S - ug;
#pragma unroll 1
    for (int f = 1; f < nfold; ++f) {
      const float2 wa = SM::ws()[(ug * f) & (S - 1)], wb = SM::ws()[(bb * f) & (S - 1)];
#pragma unroll
      for (int i = 0; i < 16 / R; ++i)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float2 x = load(t + T * i + 256 * r + F * f);
          va[i][r] = cadd(va[i][r], cmul(x, wa));
          vb[i][r] = cadd(vb[i][r], cmul(x, wb));
        }
    }
  }
  const float4* w = SM::t1(ui);
  if constexpr (R == 16) {
    dft16x2<false, HALFZ>(va[0], vb[0], [&](int q) { return w[q]; });
  } else {
    static_assert(!HALFZ || R == 16, "half-zero columns of 4096 points only");
#pragma unroll
    for (int i = 0; i < 16 / R; ++i) {
      dft_row<R, false>(va[i], [&](int q) { return make_float2(w[q].x, w[q].y); });
      dft_row<R, false>(vb[i], [&](int q) { return make_float2(w[q].z, w[q].w); });
    }
  }
  if constexpr (WAIT) cluster_wait();
  if (arrive) cluster_arrive();
  store_blocks<SM>(ui, va, vb);
}

// Stage 2: rows n0 + 16 n1 of block k0, interleaved in, separate out.
template <class SM>
__device__ __forceinline__ void stage2(int ui) {
  const int k0 = SM::k0(), n0 = SM::n0();
  float4* blk = SM::rows(ui) + k0 * kBlk;
  float2 va[16], vb[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const float4 v = blk[n0 + 16 * r];
    va[r] = make_float2(v.x, v.y);
    vb[r] = make_float2(v.z, v.w);
  }
  const float4* w = SM::t2(ui) + k0;
  dft16x2<false, false>(va, vb, [&](int q) { return w[SM::G::R * q]; });
  __syncwarp();
  float2* c = reinterpret_cast<float2*>(blk) + n0;
#pragma unroll
  for (int k = 0; k < 16; ++k) c[18 * k] = va[rev<16>(k)];
#pragma unroll
  for (int k = 0; k < 16; ++k) c[288 + 18 * k] = vb[rev<16>(k)];
}

// The butterflies of thread t in the middle: (k0, k1) of column slot sa and
// the mirror (k0b, k1b) of slot sb.  self: thread 0 of unit 0, which holds
// butterflies (0, 0) and (0, 8) of column 0, each its own mirror.
struct MidItem {
  int sa, sb, k0, k1, k0b, k1b;
};
template <int R>
__device__ __forceinline__ MidItem mid_item(bool unit0, int t) {
  MidItem m;
  const int l = t & 15, w = t >> 5;
  if (!unit0) {
    m.sa = 0; m.sb = 1;
    m.k0 = (t & 16) ? R - 1 - w : w; m.k1 = l;
    m.k0b = R - 1 - m.k0; m.k1b = 15 - l;
  } else if (R == 1 ? l >= 8 : (t & 16) != 0) {  // column S/2
    m.sa = m.sb = 1;
    m.k0 = w; m.k1 = R == 1 ? l - 8 : l;
    m.k0b = R - 1 - w; m.k1b = 15 - m.k1;
  } else {
    m.sa = m.sb = 0;
    if (w > 0) {
      m.k0 = w; m.k1 = l;
      m.k0b = R - w; m.k1b = 15 - l;
    } else if (l < 8) {
      m.k0 = m.k0b = 0;
      m.k1 = l; m.k1b = l == 0 ? 8 : 16 - l;
    } else {
      m.k0 = m.k0b = R / 2;
      m.k1 = l - 8; m.k1b = 15 - m.k1;
    }
  }
  return m;
}

// A coefficient load that stays where it is written.
__device__ __forceinline__ float4 ld_coef(const float4* p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// Stage 3 of the two butterflies m of thread tid: za[k2] = Z, zb[r] = conj Z of
// the mirror at its row 15 - r, which are the outputs of the same twiddled
// DFT on the conjugated inputs (so both butterflies use one set of twiddles);
// self: zb[r] = Z of its own row r.
template <class SM>
__device__ __forceinline__ const float4* mid_row(int ui, int slot, int k0, int k1) {
  return SM::rows(ui) + k0 * kBlk + (slot * 144 + k1 * 9);
}
// The conjugated inputs of butterfly (0, 8), which has its own base, 1/32 turn,
// and no mirror: conjugated back and turned.
__device__ __forceinline__ void self_turn(float2 (&x)[16]) {
  constexpr float c[16] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f,
                           0.83146961230254523708f, 0.70710678118654752440f,
                           0.55557023301960222474f, 0.38268343236508977173f,
                           0.19509032201612826785f, 0.f, -0.19509032201612826785f,
                           -0.38268343236508977173f, -0.55557023301960222474f,
                           -0.70710678118654752440f, -0.83146961230254523708f,
                           -0.92387953251128675613f, -0.98078528040323044913f};
#pragma unroll
  for (int r = 1; r < 16; ++r) {
    const float s = r < 8 ? c[8 - r] : c[r - 8];  // sin(2 pi r / 32)
    x[r] = cmul(cconj(x[r]), make_float2(c[r], -s));
  }
  x[0] = cconj(x[0]);
}
template <class SM>
__device__ __forceinline__ void stage3(int ui, const MidItem& m, bool self, float2 (&za)[16],
                                       float2 (&zb)[16]) {
  constexpr int kT = SM::G::T;
  const int t = SM::tid();
  const float4* pa = mid_row<SM>(ui, m.sa, m.k0, m.k1);
  const float4* pb = mid_row<SM>(ui, m.sb, m.k0b, m.k1b);
  float2 xa[16], xb[16];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float4 v = pa[r], u = pb[r];
    xa[2 * r] = make_float2(v.x, v.y);
    xa[2 * r + 1] = make_float2(v.z, v.w);
    xb[2 * r] = make_float2(u.x, -u.y);
    xb[2 * r + 1] = make_float2(u.z, -u.w);
  }
  if (self) self_turn(xb);
  const float2* w = SM::t3(ui) + t;
  dft16x2<false, false>(xa, xb, [&](int q) {
    const float2 s = w[kT * q];
    return make_float4(s.x, s.y, s.x, s.y);
  });
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    za[r] = xa[rev<16>(r)];
    zb[r] = xb[rev<16>(r)];
  }
}

// Stage 3, the product with sum |Y|^2, stage 3' of thread t's two
// butterflies, in place.  MULTI: the spectrum is kept in `scratch` (16 float4 a
// thread, stride T) for the block's other segments, or with `reload` read
// from there.  AHEAD: pairs of rows whose coefficients are loaded ahead.
// SCALED: the spectrum times `scale`.
template <class SM, int AHEAD, bool MULTI = false, bool WAIT = false, bool SCALED = false>
__device__ __forceinline__ void middle(int ui, int ug, const float4* __restrict__ coef,
                                       float4* __restrict__ scratch = nullptr,
                                       bool reload = false, float scale = 1.f) {
  constexpr int kT = SM::G::T;
  const int t = SM::tid();
  const bool unit0 = ug == 0, self = unit0 && t == 0;
  const MidItem m = mid_item<SM::G::R>(unit0, t);
  float4* pa = const_cast<float4*>(mid_row<SM>(ui, m.sa, m.k0, m.k1));
  float4* pb = const_cast<float4*>(mid_row<SM>(ui, m.sb, m.k0b, m.k1b));
  const float4* ab = coef + (size_t)ug * (24 * kT) + t;
  float2 za[16], zb[16];
  // the coefficients of the first AHEAD pairs of rows are under way during
  // stage 3, the others AHEAD pairs ahead of their use
  float4 c0[AHEAD], c1[AHEAD], c2[AHEAD];
#pragma unroll
  for (int i = 0; i < AHEAD; ++i) {
    c0[i] = ld_coef(ab + 3 * i * kT);
    c1[i] = ld_coef(ab + (3 * i + 1) * kT);
    c2[i] = ld_coef(ab + (3 * i + 2) * kT);
  }
  if (MULTI && reload) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const float4 v = __ldcg(scratch + r * kT + t);
      za[r] = make_float2(v.x, v.y);
      zb[r] = make_float2(v.z, v.w);
    }
  } else {
    stage3<SM>(ui, m, self, za, zb);
    if constexpr (SCALED) {
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        za[r] = cscale(za[r], scale);
        zb[r] = cscale(zb[r], scale);
      }
    }
    if (MULTI && scratch) {
#pragma unroll
      for (int r = 0; r < 16; ++r)
        __stcg(scratch + r * kT + t, make_float4(za[r].x, za[r].y, zb[r].x, zb[r].y));
    }
  }
  float acc = 0.f;
  float2 yb[16];  // the mirror butterfly's Y by its own k2
  if (!self) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 a0 = c0[i % AHEAD], a1 = c1[i % AHEAD], b = c2[i % AHEAD];
      if (i + AHEAD < 8) {
        c0[i % AHEAD] = ld_coef(ab + 3 * (i + AHEAD) * kT);
        c1[i % AHEAD] = ld_coef(ab + (3 * (i + AHEAD) + 1) * kT);
        c2[i % AHEAD] = ld_coef(ab + (3 * (i + AHEAD) + 2) * kT);
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int r = 2 * i + e;
        const float4 A = e ? a1 : a0;
        const float2 B = e ? make_float2(b.z, b.w) : make_float2(b.x, b.y);
        const float2 x = za[r], g = zb[r];
        za[r] = packed_product(x, cconj(g), make_float2(A.x, A.y), B);
        yb[15 - r] = packed_product(cconj(g), x, make_float2(A.z, A.w), cconj(B));
        acc = fmaf(za[r].x, za[r].x, fmaf(za[r].y, za[r].y, acc));
        acc = fmaf(yb[15 - r].x, yb[15 - r].x, fmaf(yb[15 - r].y, yb[15 - r].y, acc));
      }
    }
  } else {
    // butterfly (0, 0): rows k2 pair with (16 - k2) mod 16; (0, 8): with 15 - k2
    const float2* af = reinterpret_cast<const float2*>(ab);
    auto A = [&](int r, int h) { return __ldcg(af + 2 * (3 * (r >> 1) + (r & 1)) * kT + h); };
    auto B = [&](int r) { return __ldcg(af + 2 * (3 * (r >> 1) + 2) * kT + (r & 1)); };
    const float2 ends = B(0);  // B of rows 0 and 8, both real
    float2 ya[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const float2 b = r == 0 ? make_float2(ends.x, 0.f)
                     : r == 8 ? make_float2(ends.y, 0.f)
                     : r < 8 ? B(r) : cconj(B(16 - r));
      ya[r] = packed_product(za[r], za[(16 - r) & 15], A(r, 0), b);
      acc = fmaf(ya[r].x, ya[r].x, fmaf(ya[r].y, ya[r].y, acc));
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const float2 b = r < 8 ? B(8 + r) : cconj(B(8 + 15 - r));
      yb[r] = packed_product(zb[r], zb[15 - r], A(15 - r, 1), b);
      acc = fmaf(yb[r].x, yb[r].x, fmaf(yb[r].y, yb[r].y, acc));
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) za[r] = ya[r];
  }
  dft<16, true>(za);
  dft<16, true>(yb);
#pragma unroll
  for (int o = kT < 32 ? 8 : 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((t & 31) == 0) SM::red(ui)[t >> 5] = acc;
  if constexpr (WAIT) cluster_wait();
#pragma unroll
  for (int r = 0; r < 8; ++r)
    pa[r] = make_float4(za[2 * r].x, za[2 * r].y, za[2 * r + 1].x, za[2 * r + 1].y);
#pragma unroll
  for (int r = 0; r < 8; ++r)
    pb[r] = make_float4(yb[2 * r].x, yb[2 * r].y, yb[2 * r + 1].x, yb[2 * r + 1].y);
}

// Order the middle after stage 2 (mid_enter) and before stage 2' (mid_leave):
// within the warp.  In unit 0 the middle of warp w also reads and writes block
// 16 - w of column 0, which warp w - 1 holds (warp 0: block 8 of warp 7), so
// each warp hands over to one neighbour through a named barrier of the two
// warps, and all of them still drift; with two units in a CTA there are too
// few named barriers for that, and the unit synchronises.
__device__ __forceinline__ void pair_sync(int id) {
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void pair_arrive(int id) {
  asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}
template <class SM, int U>
__device__ __forceinline__ void mid_enter(int ui, int ug) {
  __syncwarp();
  if (ug != 0 || SM::G::T <= 32) return;
  if constexpr (U > 1 || SM::G::W != 8) {
    SM::sync(ui);
  } else {
    const int w8 = threadIdx.x >> 5;
    if (w8 < 7) pair_arrive(w8 + 1);
    if (w8 == 0 || w8 == 7) pair_sync(15);  // both wait: mid_leave uses 15 the other way
    if (w8 > 0) pair_sync(w8);
  }
}
template <class SM, int U>
__device__ __forceinline__ void mid_leave(int ui, int ug) {
  __syncwarp();
  if (ug != 0 || SM::G::T <= 32) return;
  if constexpr (U > 1 || SM::G::W != 8) {
    SM::sync(ui);
  } else {
    const int w8 = threadIdx.x >> 5;
    pair_arrive(w8 == 0 ? 15 : 7 + w8);
    pair_sync(w8 == 7 ? 15 : 8 + w8);
  }
}

// Stage 2': separate in, interleaved out.
template <class SM>
__device__ __forceinline__ void stage2i(int ui) {
  const int k0 = SM::k0(), n0 = SM::n0();
  float4* blk = SM::rows(ui) + k0 * kBlk;
  const float2* c = reinterpret_cast<const float2*>(blk) + n0;
  float2 va[16], vb[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    va[r] = c[18 * r];
    vb[r] = c[288 + 18 * r];
  }
  const float2* w = SM::u2() + n0;
  dft16x2<true, false>(va, vb, [&](int q) {
    const float2 s = w[16 * q];
    return make_float4(s.x, s.y, s.x, s.y);
  });
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 16; ++k)
    blk[n0 + 16 * k] = make_float4(va[rev<16>(k)].x, va[rev<16>(k)].y, vb[rev<16>(k)].x,
                                   vb[rev<16>(k)].y);
}

// Stage 1': rows of every block, in place; output n2 at v[i][rev<R>(n2)] (see
// store_blocks).
template <class SM>
__device__ __forceinline__ void stage1i(int ui, float2 (&va)[16 / SM::G::R][SM::G::R],
                                        float2 (&vb)[16 / SM::G::R][SM::G::R]) {
  constexpr int R = SM::G::R, T = SM::G::T;
  const int t = SM::tid();
  const float4* row = SM::rows(ui) + t;
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 v = row[r * kBlk + T * i];
      va[i][r] = make_float2(v.x, v.y);
      vb[i][r] = make_float2(v.z, v.w);
    }
#pragma unroll
  for (int i = 0; i < 16 / R; ++i) {
    const float2* w = SM::u1() + t + T * i;
    if constexpr (R == 16) {
      dft16x2<true, false>(va[i], vb[i], [&](int q) {
        const float2 s = w[256 * q];
        return make_float4(s.x, s.y, s.x, s.y);
      });
    } else {
      dft_row<R, true>(va[i], [&](int q) { return w[256 * q]; });
      dft_row<R, true>(vb[i], [&](int q) { return w[256 * q]; });
    }
  }
}

// ---------------------------------------------------------------------------
// S1: segment spectrum D and product coefficients A, B of a unit
// ---------------------------------------------------------------------------
// The strain takes the template's stages 1 to 3 (folded over the S multiples
// of F).  Then D, A and B of a bin and its mirror follow from their two values.
// Bound: latency, of few warps that depend on one another, so the work is
// spread: a thread takes one column's butterfly, not two, and several CTAs run
// the stages of a unit, each to form its share of the pairs.  One launch behind
// the other from device memory (GB300), against one CTA a unit with both
// columns in a thread (and the Stockham kernel before that): N = 2^10 6.4 us
// (7.8, 6.9), 2^12 6.6 (10.5, 7.7), 2^13 8.5 (16.5, 11.0), 2^14 13.0 (23.1,
// 18.0); a load and its wait at 2^15 23 (37, 46), 2^16 25 (41, 71), where loads
// in a row wait for the allocation.
struct BinPair {
  float2 A, B, Am, Bm;  // of bin j and of bin H - j
};
// Bins j and jm = H - j (j = 0: jm = 0 stands for the Nyquist bin's partner)
// with their factors wN^j, wN^jm.
__device__ __forceinline__ BinPair bin_pair(const PlanDev& p, int j, int jm, float2 wj, float2 wm,
                                            float2 zj, float2 zm, float2* __restrict__ D) {
  const int H = p.g.H;
  // D_j = (Zj + conj Zm)/2 - (i/2) wN^j (Zj - conj Zm)
  auto spectrum = [](float2 w, float2 x, float2 y) {
    const float2 s = cadd(x, cconj(y)), d = csub(x, cconj(y));
    const float2 e = cmul(w, d);
    return make_float2(0.5f * (s.x + e.y), 0.5f * (s.y - e.x));
  };
  auto coeffs = [](float2 w, float2 Dx, float2 cH, float2& A, float2& B) {
    // g = (1 + i conj w)/2, d = (1 - i conj w)/2 with i conj(w) = (w.y, w.x)
    const float2 g = make_float2(0.5f * (1.f + w.y), 0.5f * w.x);
    const float2 d = make_float2(0.5f * (1.f - w.y), -0.5f * w.x);
    A = cadd(cmul(cmul(g, g), Dx), cmul(cmul(d, d), cH));
    B = cmul(cmul(g, d), cadd(Dx, cH));
  };
  const float2 Dj = spectrum(wj, zj, zm);
  const float2 Dm = j == jm ? Dj : spectrum(wm, zm, zj);
  const float2 DH = make_float2(zj.x - zj.y, 0.f);  // D_{N/2}, used when j == 0
  BinPair o;
  coeffs(wj, Dj, j == 0 ? DH : cconj(Dm), o.A, o.B);
  coeffs(wm, Dm, j == 0 ? DH : cconj(Dj), o.Am, o.Bm);
  D[j] = Dj;
  if (j != jm) D[jm] = Dm;
  if (j == 0) D[H] = DH;
  return o;
}

// natural: {A, B} of bin j at (j mod S) F + j / S (the tensor-core kernel);
// otherwise where middle reads them.  The first 2 T threads of the CTA run the
// stages and leave the spectrum in shared memory by thread and row (Z of row r
// at 2 r T + t, of its mirror at (2 r + 1) T + t; thread 0 of unit 0: rows r
// of its two butterflies).  Of the 16 T pairs the CTA forms those of its part
// (of parts): a loop keeps the code short (unrolled over the 16 rows of a
// butterfly it took 25 us for N = 2^12, mostly instruction fetches).
template <class SM, bool ONE>
__device__ __forceinline__ void segment_unit(const PlanDev& p, int S, int ug,
                                             const float* __restrict__ y, float2* __restrict__ D,
                                             float4* __restrict__ AB, bool natural, int part = 0,
                                             int parts = 1) {
  constexpr int R = SM::G::R, T = SM::G::T, F = 256 * R;
  auto bin = [&](int b, int k0, int k1, int k2) { return S * (k0 + R * k1 + 16 * R * k2) + b; };
  // thread t of slot h (column h of the unit, in the middle za or zb)
  const int t = SM::tid(), h = ((int)threadIdx.x / T) & 1;
  const bool fft = (int)threadIdx.x < 2 * T;
  const bool self = ug == 0 && t == 0;
  // the tables by the CTA's last T threads, the samples under way meanwhile
  if ((int)(blockDim.x - threadIdx.x) <= T) setup_unit<SM>(p, S, ug, 0);
  // the bins of this thread's next pair and their factors, loaded ahead
  int it = part * blockDim.x + threadIdx.x, j = 0, jm = 0;
  float2 wj, wm;
  auto next_pair = [&] {
    const int u = it & (T - 1), r = it / T;
    const MidItem m = mid_item<R>(ug == 0, u);
    const int ba = ug == 0 ? m.sa * (S / 2) : ug, bb = ug == 0 ? ba : S - ug;
    j = bin(ba, m.k0, m.k1, r);
    jm = bin(bb, m.k0b, m.k1b, 15 - r);
    if (it < 16 * T && (ug != 0 || u != 0)) {
      wj = p.wN[j];
      wm = p.wN[jm];
    }
  };
  next_pair();
  float2* const rows = reinterpret_cast<float2*>(SM::rows(0));
  // once more from y / 2^64 if some value is not finite, see "Range"
  float up = 1.f;
  for (float down = 1.f;; down = kScaleDown, up = kScaleUp) {
    {  // stage 1
      auto load = [&](int m) {
        return cscale(__ldg(reinterpret_cast<const float2*>(y) + m), down);
      };
      float2 v[16 / R][R];
      if (fft) {
#pragma unroll
        for (int i = 0; i < 16 / R; ++i)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int m = t + T * i + 256 * r;
            v[i][r] = load(m);
            if constexpr (ONE) {
              const float2 x = load(m + F);
              v[i][r] = h ? csub(v[i][r], x) : cadd(v[i][r], x);
            }
          }
      }
      __syncthreads();  // the tables
      if (fft) {
        if constexpr (!ONE) {
          const int b = h == 0 ? ug : ug == 0 ? S / 2 : S - ug;
#pragma unroll 1
          for (int f = 1; f < S; ++f) {
            const float2 w = SM::ws()[(b * f) & (S - 1)];
#pragma unroll
            for (int i = 0; i < 16 / R; ++i)
#pragma unroll
              for (int r = 0; r < R; ++r)
                v[i][r] = cadd(v[i][r], cmul(load(t + T * i + 256 * r + F * f), w));
          }
        }
        const float2* const w = reinterpret_cast<const float2*>(SM::t1(0)) + h;
#pragma unroll
        for (int i = 0; i < 16 / R; ++i) {
          dft_row<R, false>(v[i], [&](int q) { return w[2 * q]; });
#pragma unroll
          for (int k = 0; k < R; ++k)
            rows[2 * (k * kBlk + t + T * i) + h] = v[i][rev<R>(k)];
        }
      }
    }
    __syncthreads();
    float2 v[16];
    {  // stage 2
      const int k0 = R == 1 ? 0 : (t & 16) ? R - 1 - (t >> 5) : t >> 5, n0 = t & 15;
      float2* const blk = rows + 2 * k0 * kBlk;
      if (fft) {
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = blk[2 * (n0 + 16 * r) + h];
        const float2* const w = reinterpret_cast<const float2*>(SM::t2(0)) + 2 * k0 + h;
        dft_row<16, false>(v, [&](int q) { return w[2 * R * q]; });
      }
      __syncthreads();
      if (fft) {
#pragma unroll
        for (int k = 0; k < 16; ++k) blk[288 * h + n0 + 18 * k] = v[rev<16>(k)];
      }
    }
    __syncthreads();
    float bad[4] = {0.f, 0.f, 0.f, 0.f};
    if (fft) {  // stage 3: the butterfly, or its mirror conjugated
      const MidItem m = mid_item<R>(ug == 0, t);
      const float4* const x =
          h ? mid_row<SM>(0, m.sb, m.k0b, m.k1b) : mid_row<SM>(0, m.sa, m.k0, m.k1);
      const float sign = h ? -1.f : 1.f;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 u = x[r];
        v[2 * r] = make_float2(u.x, sign * u.y);
        v[2 * r + 1] = make_float2(u.z, sign * u.w);
      }
      if (self && h) self_turn(v);
      const float2* const w = SM::t3(0) + t;
      dft_row<16, false>(v, [&](int q) { return w[T * q]; });
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        bad[r & 1] = fmaf(v[r].x, 0.f, bad[r & 1]);
        bad[2 + (r & 1)] = fmaf(v[r].y, 0.f, bad[2 + (r & 1)]);
      }
    }
    // the rows have been read
    if (__syncthreads_or((bad[0] + bad[1]) + (bad[2] + bad[3]) != 0.f) && down == 1.f) continue;
    if (fft) {
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const float2 z = v[rev<16>(r)];
        rows[(2 * r + h) * T + t] = h && !self ? cconj(z) : z;
      }
    }
    break;
  }
  __syncthreads();
  const float2* const zs = reinterpret_cast<const float2*>(SM::rows(0));
  auto place = [&](int j, float2 A, float2 B) {
    AB[(j % S) * F + j / S] = make_float4(A.x, A.y, B.x, B.y);
  };
  float2* const af = reinterpret_cast<float2*>(AB + (size_t)ug * (24 * T));
  // third q of the pair of rows that holds `row`: {A, A'} of either row, {B, B}
  auto third = [&](int row, int q, int t) { return 2 * ((3 * (row >> 1) + q) * T + t); };
#pragma unroll 2
  while (it < 16 * T) {
    const int t = it & (T - 1), r = it / T, j0 = j, jm0 = jm;
    const float2 wj0 = wj, wm0 = wm;
    it += parts * blockDim.x;
    next_pair();
    if (ug != 0 || t != 0) {
      const int j = j0, jm = jm0;
      const BinPair o = bin_pair(p, j, jm, wj0, wm0, cscale(zs[2 * r * T + t], up),
                                 cscale(zs[(2 * r + 1) * T + t], up), D);
      if (natural) {
        place(j, o.A, o.B);
        place(jm, o.Am, o.Bm);
      } else {
        *reinterpret_cast<float4*>(af + third(r, r & 1, t)) =
            make_float4(o.A.x, o.A.y, o.Am.x, o.Am.y);
        af[third(r, 2, t) + (r & 1)] = o.B;
      }
      continue;
    }
    // rows r and (16 - r) mod 16 of butterfly (0, 0), r and 15 - r of (0, 8);
    // where the product's thread 0 looks for them, see middle
    if (r <= 8) {
      const int rm = (16 - r) & 15, j = bin(0, 0, 0, r), jm = bin(0, 0, 0, rm);
      const BinPair o =
          bin_pair(p, j, jm, p.wN[j], p.wN[jm], cscale(zs[2 * r * T], up), cscale(zs[2 * rm * T], up), D);
      if (natural) {
        place(j, o.A, o.B);
        if (jm != j) place(jm, o.Am, o.Bm);
      } else {
        af[third(r, r & 1, 0)] = o.A;
        if (jm != j) af[third(rm, rm & 1, 0)] = o.Am;
        float2* const b = af + third(r & 7, 2, 0) + (r & 1);
        if (r == 0)
          b->x = o.B.x;
        else if (r == 8)
          b->y = o.B.x;
        else
          *b = o.B;
      }
    }
    if (r < 8) {
      const int j = bin(0, 0, 8, r), jm = bin(0, 0, 8, 15 - r);
      const BinPair o = bin_pair(p, j, jm, p.wN[j], p.wN[jm], cscale(zs[(2 * r + 1) * T], up),
                                 cscale(zs[(2 * (15 - r) + 1) * T], up), D);
      if (natural) {
        place(j, o.A, o.B);
        place(jm, o.Am, o.Bm);
      } else {
        af[third(15 - r, (15 - r) & 1, 0) + 1] = o.A;
        af[third(r, r & 1, 0) + 1] = o.Am;
        af[third(8 + r, 2, 0) + (r & 1)] = o.B;
      }
    }
  }
}

// CTAs per unit: each runs the stages and forms its share of the pairs, one a
// thread.
template <int F>
__host__ __device__ constexpr int segment_threads() {
  return F / 8 < 256 ? 256 : F / 8;
}
template <int F>
__host__ __device__ constexpr int segment_parts() {
  return F / segment_threads<F>();
}
template <int F, bool ONE>
__global__ void __launch_bounds__(segment_threads<F>(), 1)
segment_kernel(PlanDev p, const float* __restrict__ y, float2* __restrict__ D,
               float4* __restrict__ AB, bool natural) {
  constexpr int P = segment_parts<F>();
  segment_unit<Sm<F, 1, ONE>, ONE>(p, unit_geo(p.g).S, blockIdx.x / P, y, D, AB,
                                                  natural, blockIdx.x % P, P);
}

template <int F, bool ONE>
static cudaError_t launch_segment_t(const PlanDev& p, const float* y, float2* D, float4* AB,
                                    bool natural, cudaStream_t s) {
  constexpr size_t smem = Lay<F, 1, ONE>::total;
  auto kern = segment_kernel<F, ONE>;
  cudaError_t e = ensure_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<unit_geo(p.g).S / 2 * segment_parts<F>(), segment_threads<F>(), smem, s>>>(p, y, D, AB, natural);
  return cudaGetLastError();
}

// Sum |Y|^2 of a unit, in warp order (after a barrier that follows the middle).
template <class SM>
__device__ __forceinline__ float unit_power(int ui) {
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < SM::G::W; ++w) s += SM::red(ui)[w];
  return s;
}

// sigma from the units' shares (Eq. PT on the packed spectrum).
__device__ __forceinline__ float sigma_of(const float* shares, int units, int N) {
  float tot = 0.f;
  for (int q = 0; q < units; ++q) tot += shares[q];
  return sqrtf(2.0f * tot) / (float)N;
}

// Stage c and the tails of rows [rank F/C, (rank + 1) F/C) of a group of C
// CTAs (32 / S rows a thread); rowptr: the rows of the group's units.  All
// rows are loaded at once, so their latency (distributed shared memory) is
// paid once; a warp in which some value passes reads them again one by one.
template <int S, int U>
struct Combine {
  static constexpr int C = S / 2 / U;
  static constexpr int per = kF / C;
  static constexpr int kT = Geo<kF>::T;
  static constexpr int R = per / (kT * U);
  float2 w[R][S / 2];

  static __device__ __forceinline__ int row(int rank, int r) {
    return rank * per + r * (kT * U) + (int)threadIdx.x;
  }
  // Rows of unit u in the cluster's shared memory ...
  struct Shared {
    float4* const* rowptr;
    __device__ __forceinline__ float4 operator()(int u, int n1) const {
      return rowptr[u][(n1 >> 8) * kBlk + (n1 & 255)];
    }
  };
  // ... or in the exchange buffer.
  struct Global {
    const float4* x;
    __device__ __forceinline__ float4 operator()(int u, int n1) const {
      return __ldcg(x + u * kF + n1);
    }
  };
  template <class X>
  static __device__ __forceinline__ void load(const X& x, int n1, float2 (&t)[S]) {
#pragma unroll
    for (int u = 0; u < S / 2; ++u) {
      const float4 v = x(u, n1);
      t[u] = make_float2(v.x, v.y);
      t[u == 0 ? S / 2 : S - u] = make_float2(v.z, v.w);
    }
  }
  __device__ __forceinline__ void twiddles(const float2* __restrict__ uc, int rank) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < S / 2; ++q) w[r][q] = __ldg(uc + q * kF + row(rank, r));
  }
  template <bool EXT, class X>
  __device__ __forceinline__ void emit(const X& x, const float2* __restrict__ uc, int rank,
                                       float thr, uint32_t tmpl, int64_t krow,
                                       const TailOut& a, float sigma) {
    float2 t[R][S];
#pragma unroll
    for (int r = 0; r < R; ++r) load(x, row(rank, r), t[r]);
    float big = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      dft_row<S, true>(t[r], [&](int q) { return w[r][q]; });
#pragma unroll
      for (int k = 0; k < S; ++k) big = fmaxf(big, fmaxf(fabsf(t[r][k].x), fabsf(t[r][k].y)));
    }
    if (a.dump || __any_sync(0xffffffffu, big > thr * (float)(S * kF))) {
#pragma unroll 1
      for (int r = 0; r < R; ++r) {
        const int n1 = row(rank, r);
        float2 y[S], o[S];
        load(x, n1, y);
        dft_row<S, true>(y, [&](int q) { return __ldg(uc + q * kF + n1); });
#pragma unroll
        for (int k = 0; k < S; ++k) o[k] = y[rev<S>(k)];
        emit_row<S, kF, EXT>(o, n1, S * kF, thr, tmpl, krow, a, sigma);
      }
    }
  }
};

// S = 2 (the unit holds the whole template): stage 1', stage c and the tails
// in one go.  The rows reach shared memory only where some value of the warp
// passes.
template <class SM, bool EXT>
__device__ __forceinline__ void finish_s2(int ui, const float2* __restrict__ uc, float thr,
                                          uint32_t tmpl, int64_t krow, const TailOut& a,
                                          float sigma) {
  constexpr int S = 2, R = SM::G::R, T = SM::G::T, F = 256 * R;
  const int t = SM::tid();
  float2 va[16 / R][R], vb[16 / R][R];
  stage1i<SM>(ui, va, vb);
  float big = 0.f;
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const float2 s = __ldg(uc + t + T * i + 256 * k);
      float2 &x = va[i][rev<R>(k)], &y = vb[i][rev<R>(k)];
      bfly<true, 0>(x, y, s.x, s.y);
      big = fmaxf(big, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y))));
    }
  if (__any_sync(0xffffffffu, a.dump || big > thr * (float)(S * F))) {
    store_blocks<SM>(ui, va, vb);  // this thread's own rows
    const float4* row = SM::rows(ui) + t;
#pragma unroll 1
    for (int q = 0; q < 16; ++q) {
      const int i = q / R, k = q & (R - 1);
      const float4 v = row[k * kBlk + T * i];
      float2 o[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
      emit_row<S, F, EXT>(o, t + T * i + 256 * k, S * F, thr, tmpl, krow, a, sigma);
    }
  }
}

// ---------------------------------------------------------------------------
// S2-S6 of one segment: C = S / 2 / U CTAs of a cluster share a template
// ---------------------------------------------------------------------------
template <int S, int U, bool HALFZ, bool EXT>
__global__ void __launch_bounds__(256 * U, U == 1 ? 2 : 1) unit_kernel(PlanDev p, CorrelateArgs a) {
  constexpr int C = S / 2 / U;
  using SM = Sm<kF, U>;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cluster.block_rank();
  const int ui = U == 1 ? 0 : (int)threadIdx.x / SM::G::T;
  const int ug = rank * U + ui;
  setup_common<SM, 256 * U>(p);
  setup_unit<SM>(p, S, ug, ui);
  if (threadIdx.x < S / 2) {
    const int c = (int)threadIdx.x / U, u = (int)threadIdx.x % U;
    float4* const rows = C == 1 ? SM::rows(0) : cluster.map_shared_rank(SM::rows(0), (unsigned)c);
    SM::rowptr()[threadIdx.x] = rows + u * (SM::L::unit_bytes / 16);
  }
  if constexpr (C > 1) cluster_arrive();  // paired with the wait of the first stage 1
  __syncthreads();

  const int cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int nz = (int)(a.Lp / 2), nfold = (nz + kF - 1) / kF;
  const TailOut out{a.recs, a.cap, a.counter, a.dump, a.proj, a.kappa_hi, a.lag_end};
  for (int64_t k = a.k0 + cid; k < a.k1; k += ncl) {
    stage1<SM, HALFZ, false, (C > 1)>(ui, S, ug, a.bank + k * a.Lp, nz, nfold);
    SM::sync(ui);
    stage2<SM>(ui);
    mid_enter<SM, U>(ui, ug);
    middle<SM, (S <= 4 ? 2 : 1)>(ui, ug, a.AB);
    mid_leave<SM, U>(ui, ug);
    stage2i<SM>(ui);
    SM::sync(ui);
    const int64_t krow = k - a.k0;
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
    if (rank == 0 && threadIdx.x == 0) a.sigma[krow] = sigma;
    cb.template emit<EXT>(typename Combine<S, U>::Shared{SM::rowptr()}, p.uc, rank, a.kappa * sigma, (uint32_t)k, krow, out, sigma);
    if constexpr (C > 1) {
      __syncwarp();
      cluster_arrive_relaxed();  // every remote value has fed a vote: the reads are done
    } else {
      __syncthreads();
    }
  }
  if constexpr (C > 1) cluster_wait();  // the cluster's last reads of this CTA's rows
}

// The same for S >= 8 with the columns exchanged through the buffer a.exch
// (L2) and the combine one template behind: a CTA writes its units' outputs
// of template k, goes on with template k + 1 and combines k just before it
// writes k + 1, so the cluster's barrier (arrive in stage 1, wait before the
// combine) has most of a template's time to complete and nothing waits for a
// neighbour's pace or for distributed shared memory.  The buffer holds two
// templates of every unit: outputs of template k overwrite those of k - 2,
// which every CTA combined before it arrived for k - 1.  Per template, this /
// unit_kernel: N = 2^16 165 / 171 ns, 2^17 354 / 405 (at N = 2^15, where one CTA
// holds a template, it took 8% longer).
template <int S, int U, bool HALFZ, bool EXT>
__global__ void __launch_bounds__(256 * U, U == 1 ? 2 : 1)
unit_exchange_kernel(PlanDev p, CorrelateArgs a) {
  constexpr int C = S / 2 / U;
  static_assert(C > 1, "a cluster shares the template");
  using SM = Sm<kF, U>;
  using CB = Combine<S, U>;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int ui = U == 1 ? 0 : (int)threadIdx.x / SM::G::T;
  const int ug = rank * U + ui;
  setup_common<SM, 256 * U>(p);
  setup_unit<SM>(p, S, ug, ui);
  // the first template's share goes into the other CTAs' shared memory: all of
  // them have started once the wait that pairs with this (before the first
  // store) returns
  cluster_arrive();
  __syncthreads();

  const int cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int nz = (int)(a.Lp / 2), nfold = (nz + kF - 1) / kF;
  const TailOut out{a.recs, a.cap, a.counter, a.dump, a.proj, a.kappa_hi, a.lag_end};
  float4* const exch = a.exch + (size_t)cid * (S * kF);
  int par = 0;
  auto combine = [&](int64_t k) {  // of the template before, which is in buffer par ^ 1
    CB cb;
    cb.twiddles(p.uc, rank);
    cluster_wait();  // every row and share of the cluster is there
    const float sigma = sigma_of(SM::sigall() + 8 * (par ^ 1), S / 2, S * 2 * kF);
    const int64_t krow = k - a.k0;
    if (rank == 0 && threadIdx.x == 0) a.sigma[krow] = sigma;
    cb.template emit<EXT>(typename CB::Global{exch + (par ^ 1) * (S / 2 * kF)}, p.uc, rank,
                          a.kappa * sigma, (uint32_t)k, krow, out, sigma);
  };
  const int64_t first = a.k0 + cid;
  int64_t k = first;
  for (; k < a.k1; k += ncl) {
    stage1<SM, HALFZ, false, false>(ui, S, ug, a.bank + k * a.Lp, nz, nfold, k != first);
    SM::sync(ui);
    stage2<SM>(ui);
    mid_enter<SM, U>(ui, ug);
    middle<SM, 1>(ui, ug, a.AB);
    mid_leave<SM, U>(ui, ug);
    stage2i<SM>(ui);
    SM::sync(ui);
    if (k != first)
      combine(k - ncl);
    else
      cluster_wait();
    {
      float2 va[1][16], vb[1][16];
      stage1i<SM>(ui, va, vb);
      float4* x = exch + (par * (S / 2) + ug) * kF + SM::tid();
#pragma unroll
      for (int q = 0; q < 16; ++q)
        __stcg(x + 256 * q, make_float4(va[0][rev<16>(q)].x, va[0][rev<16>(q)].y,
                                        vb[0][rev<16>(q)].x, vb[0][rev<16>(q)].y));
    }
    if (SM::tid() == 0) {
      const float share = unit_power<SM>(ui);
#pragma unroll
      for (int q = 0; q < C; ++q)
        *cluster.map_shared_rank(SM::sigall() + 8 * par + ug, (unsigned)q) = share;
    }
    par ^= 1;
  }
  if (k != first) {
    cluster_arrive();
    combine(k - ncl);
  }
}

// S = 2: the units of a CTA (256 threads) take templates of their own and wait
// for nobody else; those beyond the last template repeat the CTA's first and
// write nothing.  Bound as above.  A unit of F / 16 threads keeps every thread
// at work, where one column of N / 2 points per CTA of 256 threads left seven
// eighths of them idle in the passes at N = 2^10; two units of 16 threads share
// a warp there.  Per template (2^18 chirps of N samples at most, GB300),
// against that kernel: N = 2^10 13.5 -> 2.1 ns, 2^11 16.5 -> 4.5, 2^12 23.6 ->
// 9.2, 2^13 29.4 -> 18.7.
template <int F, bool HALFZ, bool EXT>
__global__ void __launch_bounds__(256, 2) short_kernel(PlanDev p, CorrelateArgs a) {
  constexpr int U = 4096 / F;
  using SM = Sm<F, U, true>;
  const int ui = U == 1 ? 0 : (int)threadIdx.x / SM::G::T;
  setup_common<SM, 256>(p);
  if (ui == 0) setup_unit<SM>(p, 2, 0, 0);
  __syncthreads();

  const int nz = (int)(a.Lp / 2);
  for (int64_t base = a.k0 + (int64_t)blockIdx.x * U; base < a.k1; base += (int64_t)gridDim.x * U) {
    const bool active = base + ui < a.k1;
    const int64_t k = active ? base + ui : base;
    stage1<SM, HALFZ, true, false>(ui, 2, 0, a.bank + k * a.Lp, nz, 0);
    SM::sync(ui);
    stage2<SM>(ui);
    mid_enter<SM, U>(ui, 0);
    middle<SM, 2>(ui, 0, a.AB);
    mid_leave<SM, U>(ui, 0);
    stage2i<SM>(ui);
    SM::sync(ui);
    const int64_t krow = k - a.k0;
    const float share = unit_power<SM>(ui);
    const float sigma = sigma_of(&share, 1, 4 * F);
    if (active && SM::tid() == 0) a.sigma[krow] = sigma;
    const TailOut out{a.recs, a.cap, a.counter, active ? a.dump : nullptr, a.proj, a.kappa_hi,
                      a.lag_end};
    finish_s2<SM, EXT>(ui, p.uc, active ? a.kappa * sigma : INFINITY, (uint32_t)k, krow, out, sigma);
  }
}

// ---------------------------------------------------------------------------
// Range
// ---------------------------------------------------------------------------
// At a quarter turn the tangent form holds (1 -/+ 2^30 i) b between its two
// products, so values beyond 2^97 overflow there although the spectrum is
// finite.  Nothing that overflowed leaves a template's sum |Y|^2 finite, and
// one whose sigma is not finite has no tails.  These kernels, launched behind
// a search whose bank holds samples above 2^64 (or is not known), do the
// templates without finite sigma again: from z / 2^64, with the spectrum
// brought back before the product.  Both factors are exact but for values
// 2^126 times smaller than the largest.  A template without a sample above
// 2^64 (its product has overflowed) stays as it is.  With a finite sigma the
// inverse stages stay below 2^81.  They are kernels of their own because any
// of it in the searching kernels, a call behind their loops included, changed
// their registers: 0.97 to 1.03 times their time, batch 1.05.
//
// The factor of unit ui, 1 where it is not (wanted) or of no use.
template <class SM>
__device__ __forceinline__ float range_scale(int* over, int ui, const float* __restrict__ src,
                                             int nz, bool wanted) {
  SM::sync(ui);  // over[ui] has been read
  if (SM::tid() == 0) over[ui] = 0;
  SM::sync(ui);
  bool large = false;
  for (int m = SM::tid(); m < nz; m += SM::G::T) {
    const float2 x = __ldg(reinterpret_cast<const float2*>(src) + m);
    large |= !(fmaxf(fabsf(x.x), fabsf(x.y)) <= kScaleUp);
  }
  if (wanted && large) over[ui] = 1;
  SM::sync(ui);
  return over[ui] ? kScaleDown : 1.f;
}

// Stages 1 to 2' with the factor.
template <class SM, int U, bool HALFZ, bool ONE>
__device__ __forceinline__ void scaled_rows(int ui, int S, int ug, const float* __restrict__ src,
                                            int nz, int nfold, const float4* __restrict__ coef,
                                            float down) {
  stage1<SM, HALFZ, ONE, false, true>(ui, S, ug, src, nz, nfold, false, down);
  SM::sync(ui);
  stage2<SM>(ui);
  mid_enter<SM, U>(ui, ug);
  middle<SM, 1, false, false, true>(ui, ug, coef, nullptr, false, 1.f / down);
  mid_leave<SM, U>(ui, ug);
  stage2i<SM>(ui);
  SM::sync(ui);
}

// The rows [r0, r1) of group g of n groups, and whether one of them has no
// finite sigma (which all CTAs of a group see alike; a barrier of the CTA).
__device__ __forceinline__ bool range_rows(const CorrelateArgs& a, int64_t g, int64_t n,
                                           int64_t* r0, int64_t* r1) {
  const int64_t count = a.k1 - a.k0, per = (count + n - 1) / n;
  *r0 = g * per;
  *r1 = *r0 + per < count ? *r0 + per : count;
  bool bad = false;
  cudaGridDependencySynchronize();  // the search
  for (int64_t r = *r0 + threadIdx.x; r < *r1; r += blockDim.x)
    bad |= !(__ldcg(a.sigma + r) <= kMaxFinite);
  return __syncthreads_or(bad);
}

// N >= 2^15: clusters of S / 4 CTAs of two units, as unit_kernel.
template <int S, bool HALFZ, bool EXT>
__global__ void __launch_bounds__(512, 1) range_kernel(PlanDev p, CorrelateArgs a) {
  constexpr int U = 2, C = S / 2 / U;
  using SM = Sm<kF, U>;
  __shared__ int over[U];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cluster.block_rank();
  const int ui = (int)threadIdx.x / SM::G::T, ug = rank * U + ui;
  int64_t r0, r1;
  if (!range_rows(a, blockIdx.x / C, gridDim.x / C, &r0, &r1)) return;
  setup_common<SM, 256 * U>(p);
  setup_unit<SM>(p, S, ug, ui);
  if (threadIdx.x < S / 2) {
    const int c = (int)threadIdx.x / U, u = (int)threadIdx.x % U;
    float4* const rows = C == 1 ? SM::rows(0) : cluster.map_shared_rank(SM::rows(0), (unsigned)c);
    SM::rowptr()[threadIdx.x] = rows + u * (SM::L::unit_bytes / 16);
  }
  cluster.sync();
  const int nz = (int)(a.Lp / 2), nfold = (nz + kF - 1) / kF;
  const TailOut out{a.recs, a.cap, a.counter, a.dump, a.proj, a.kappa_hi, a.lag_end};
  for (int64_t r = r0; r < r1; ++r) {
    if (__ldcg(a.sigma + r) <= kMaxFinite) continue;
    const int64_t k = a.k0 + r;
    const float* const src = a.bank + k * a.Lp;
    const float down = range_scale<SM>(over, ui, src, nz, true);
    if (down == 1.f) continue;
    scaled_rows<SM, U, HALFZ, false>(ui, S, ug, src, nz, nfold, a.AB, down);
    float2 va[1][16], vb[1][16];
    stage1i<SM>(ui, va, vb);
    store_blocks<SM>(ui, va, vb);
    if (SM::tid() == 0) {
      const float share = unit_power<SM>(ui);
      for (int q = 0; q < C; ++q) *cluster.map_shared_rank(SM::sigall() + ug, (unsigned)q) = share;
    }
    cluster.sync();  // and every CTA has read this sigma
    const float sigma = sigma_of(SM::sigall(), S / 2, S * 2 * kF);
    if (rank == 0 && threadIdx.x == 0) a.sigma[r] = sigma;
    Combine<S, U> cb;
    cb.twiddles(p.uc, rank);
    cb.template emit<EXT>(typename Combine<S, U>::Shared{SM::rowptr()}, p.uc, rank,
                          a.kappa * sigma, (uint32_t)k, r, out, sigma);
    cluster.sync();
  }
}

// N <= 2^14, as short_kernel.
template <int F, bool HALFZ, bool EXT>
__global__ void __launch_bounds__(256, 2) range_short_kernel(PlanDev p, CorrelateArgs a) {
  constexpr int U = 4096 / F;
  using SM = Sm<F, U, true>;
  __shared__ int over[U];
  const int ui = U == 1 ? 0 : (int)threadIdx.x / SM::G::T;
  int64_t r0, r1;
  if (!range_rows(a, blockIdx.x, gridDim.x, &r0, &r1)) return;
  setup_common<SM, 256>(p);
  if (ui == 0) setup_unit<SM>(p, 2, 0, 0);
  __syncthreads();
  const int nz = (int)(a.Lp / 2);
  for (; r0 < r1; r0 += U) {  // a unit's barriers are its own; units of a warp go together
    const int64_t r = r0 + ui < r1 ? r0 + ui : r0, k = a.k0 + r;
    const bool wanted = r0 + ui < r1 && !(__ldcg(a.sigma + r) <= kMaxFinite);
    if (!__any_sync(0xffffffffu, wanted)) continue;
    const float* const src = a.bank + k * a.Lp;
    const float down = range_scale<SM>(over, ui, src, nz, wanted);
    const bool active = down != 1.f;
    if (!__any_sync(0xffffffffu, active)) continue;
    scaled_rows<SM, U, HALFZ, true>(ui, 2, 0, src, nz, 0, a.AB, down);
    const float share = unit_power<SM>(ui);
    const float sigma = sigma_of(&share, 1, 4 * F);
    if (active && SM::tid() == 0) a.sigma[r] = sigma;
    const TailOut out{a.recs, a.cap, a.counter, active ? a.dump : nullptr, a.proj, a.kappa_hi,
                      a.lag_end};
    finish_s2<SM, EXT>(ui, p.uc, active ? a.kappa * sigma : INFINITY, (uint32_t)k, r, out, sigma);
  }
}

template <int S, int U, bool HALFZ, bool EXT>
static cudaError_t launch_unit_t(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  constexpr int C = S / 2 / U;
  if constexpr (S >= 8 && U == 2) {
    if (a.exch)
      return launch_clusters<unit_exchange_kernel<S, U, HALFZ, EXT>>(
          C, 256 * U, Lay<kF, U, false>::total, 1, 1, p, a, s);
  }
  return launch_clusters<unit_kernel<S, U, HALFZ, EXT>>(C, 256 * U, Lay<kF, U, false>::total,
                                                        U == 1 ? 2 : 1, 1, p, a, s);
}

// The extended epilogue (bege_correlate_max, bege_correlate_band,
// bege_correlate_ex) runs in its own instantiation.
static bool extended(const PlanDev& p, const CorrelateArgs& a) {
  return a.proj || a.kappa_hi > 0.f || a.lag_end < (uint32_t)p.g.N;
}

template <int S, int U>
static cudaError_t launch_unit(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  if (a.Lp <= kF)
    return extended(p, a) ? launch_unit_t<S, U, true, true>(p, a, s)
                          : launch_unit_t<S, U, true, false>(p, a, s);
  return extended(p, a) ? launch_unit_t<S, U, false, true>(p, a, s)
                        : launch_unit_t<S, U, false, false>(p, a, s);
}

template <int F, bool HALFZ>
static cudaError_t launch_short(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  constexpr int U = 4096 / F;
  constexpr size_t smem = Lay<F, U, true>::total;
  return extended(p, a)
             ? launch_clusters<short_kernel<F, HALFZ, true>>(1, 256, smem, 2, U, p, a, s)
             : launch_clusters<short_kernel<F, HALFZ, false>>(1, 256, smem, 2, U, p, a, s);
}

template <int S>
static cudaError_t launch_range(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  constexpr int C = S / 4;
  constexpr size_t smem = Lay<kF, 2, false>::total;
  const bool ext = extended(p, a);
  if (a.Lp <= kF)
    return ext ? launch_clusters<range_kernel<S, true, true>, true>(C, 512, smem, 1, 1, p, a, s)
               : launch_clusters<range_kernel<S, true, false>, true>(C, 512, smem, 1, 1, p, a, s);
  return ext ? launch_clusters<range_kernel<S, false, true>, true>(C, 512, smem, 1, 1, p, a, s)
             : launch_clusters<range_kernel<S, false, false>, true>(C, 512, smem, 1, 1, p, a, s);
}

template <int F, bool HALFZ>
static cudaError_t launch_range_short(const PlanDev& p, const CorrelateArgs& a, cudaStream_t s) {
  constexpr int U = 4096 / F;
  constexpr size_t smem = Lay<F, U, true>::total;
  return extended(p, a)
             ? launch_clusters<range_short_kernel<F, HALFZ, true>, true>(1, 256, smem, 2, U, p, a, s)
             : launch_clusters<range_short_kernel<F, HALFZ, false>, true>(1, 256, smem, 2, U, p, a, s);
}

}  // namespace unit
}  // namespace bege
