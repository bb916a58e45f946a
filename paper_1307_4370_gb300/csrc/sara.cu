// SARA dictionary (§3.3): Psi = (1/sqrt q) [Dirac, db1, ..., db8], Psi^H its adjoint.
//
// Each Daubechies plane is a periodic, separable, orthonormal 2-D DWT in
// Mallat layout.  One launch per level processes every wavelet basis at once
// (grid.z = basis): a CTA loads the input region its coefficient tile needs
// (with periodic wrap, also when the filter is longer than the signal),
// filters rows then columns in shared memory, and writes the four sub-bands.
// The synthesis runs the transpose level by level; its finest level sums all
// bases and the Dirac plane in the same CTA, so x is written once.  In prox
// mode the analysis epilogue applies the weighted soft threshold of §4.4
// eq. prox1 and the dual update of Algorithm 1 steps 7-9 to each final
// coefficient as it is produced, so alpha itself is never stored; each
// block leaves one FP64 partial of f1, and the first synthesis launch that
// follows sums them into f1 and the halting quantity zeta (§4.4).
#include <cmath>
#include <complex>
#include <vector>

#include "common.cuh"
#include "reduce.cuh"

namespace purify {

constexpr int kTile = 16;     // coefficient tile (analysis) / half output tile (synthesis)

struct LevelGeom {
  int tile;     // coefficient tile side (analysis) / half output tile (synthesis); divides L/2
  int n;        // image side (plane row stride)
  int L;        // input side of this analysis level / output side of this synthesis level
  int nb;       // wavelet planes in the launch
  int plane0;   // index of the first wavelet plane in the coefficient array
  int last;     // analysis: last level (LL goes to the plane); synthesis: finest level
  float scale;  // 1 / sqrt(q)
  int first;    // analysis: first level
  int dirac;    // analysis, first level: plane of the Dirac basis handled by the CTAs with z = nb, or -1
  int f1_off;   // analysis, prox mode: index of this launch's first f1 partial
};

// Daubechies orders of the wavelet planes, four bits each (an array indexed by
// the plane would be copied to local memory by every thread).
struct BasisList {
  unsigned packed;  // at most eight planes
  __host__ __device__ int p(int k) const { return (int)(packed >> (4 * k)) & 15; }
};

// The filters as kernel parameters: each tap as the (w, w) pair of a packed
// FP32x2 multiply-add, db_p from p (p - 1).
struct WaveletTaps {
  float2 h[72], g[72];
};

// Soft threshold + dual update for one final coefficient alpha at index j;
// returns w |alpha| (its term of f1), summed per thread in FP32 (a few terms)
// and across threads in FP64.
// The same with z1_j and w_j already loaded.
__device__ __forceinline__ float sara_prox_v(float2 al, float2 z, float w, int j, float2* z1, float2* u1,
                                             float gamma) {
  const float2 a = cadd(al, z);
  // shrink factor (|a| - lam)^+ / |a| = max(1 - lam / |a|, 0), with 1 / |a|
  // from the hardware reciprocal square root (0 where a = 0)
  const float m2 = fmaf(a.x, a.x, a.y * a.y);
  const float s = m2 > 0.0f ? fmaxf(fmaf(-gamma * w, rsqrtf(m2), 1.0f), 0.0f) : 0.0f;
  const float2 r1 = cscale(a, s);
  const float2 z1n = csub(a, r1);
  z1[j] = z1n;
  u1[j] = csub(r1, z1n);
  const float al2 = fmaf(al.x, al.x, al.y * al.y);
  return w * (al2 > 0.0f ? al2 * rsqrtf(al2) : 0.0f);
}

__device__ __forceinline__ float sara_prox(float2 al, size_t j, const SaraProxArgs& pa, float gamma) {
  const float w = pa.w ? pa.w[j] : 1.0f;
  return sara_prox_v(al, pa.z1[j], w, 0, pa.z1 + j, pa.u1 + j, gamma);
}

// ---------------------------------------------------------------------------
// Dirac plane: alpha_0 = x / sqrt(q) (plain), or its prox update.
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void k_dirac(const float2* __restrict__ x, float2* __restrict__ alpha, int64_t N, float scale,
                        SaraProxArgs pa, double* partials, DevScalars* sc) {
  pdl_sync(x, alpha, partials, sc);
  float f1 = 0.f;
  const float gamma = (MODE == kSaraProx) ? (float)sc->gamma : 0.f;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const float2 al = cscale(x[j], scale);
    if (MODE == kSaraPlain) alpha[j] = al;
    else f1 += sara_prox(al, (size_t)j, pa, gamma);
  }
  if (MODE == kSaraProx) {
    const FPair f1p{f1, 0.f};
    double tot;
    if (reduce_last_block<1>(&f1p, partials + kCntF1 * 2 * kMaxPartials, &sc->counter[kCntF1], &tot))
      sc->f1 = tot;  // first contribution of this analysis
  }
}

// One wavelet plane of one analysis level, for the Daubechies order P fixed at
// compile time (filters in registers, tap loops unrolled).  Returns this
// thread's terms of f1 (prox mode).
//
// FAST (tiles of a multiple of four): a thread filters four adjacent outputs
// of a row, then two of a column, from one window of inputs, (2P + 6) / 8 and
// (2P + 2) / 4 shared-memory loads per output instead of P (one output pair
// per thread: all four levels at 1024^2 83 us; 74 us so, issue-bound), and
// lanes take consecutive rows of an odd stride, so neither pass has bank
// conflicts.
template <int P, int MODE, bool FAST>
__device__ __forceinline__ float dwt_plane(const float2* __restrict__ in, int in_shared, float2* __restrict__ ll_out,
                                           float2* __restrict__ coef, const LevelGeom& G, const WaveletTaps& wf,
                                           const SaraProxArgs& pa, int k, float gamma) {
  extern __shared__ float2 sm[];
  constexpr int taps = 2 * P;
  constexpr int hoff = P * (P - 1);  // db_p starts after db_1 .. db_(p-1): sum of 2q, q < p
  const float2 *h = wf.h + hoff, *g = wf.g + hoff;
  float f1 = 0.f;
  const int L = G.L, H = L / 2;
  const int TI = G.tile;
  const int I1 = blockIdx.y * TI, I2 = blockIdx.x * TI;
  const int RH = 2 * TI + taps - 2;  // input rows/cols the tile needs
  const int RHS = RH | 1, RS = 2 * TI + 1;  // row strides (odd)
  float2* inb = sm;                  // RH x RH
  float2* rowp = sm + RH * RHS;      // RH x 2TI  ([a | d] per input row)
  const float2* src = in_shared ? in : in + (size_t)k * (G.n / 2) * (G.n / 2);
  const Div dTI = make_div(TI), d2TI = make_div(2 * TI);
  // input tile with its halo (periodic): warps take rows, lanes columns (RH <=
  // 2 * 16 + 14 = 46, two column rounds); the halo wraps past L at most once
  // when L >= RH, and index by index (a remainder) otherwise
  {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    auto wrapped = [&](int i) { return L >= RH ? (i >= L ? i - L : i) : i % L; };
    const int cA = wrapped(2 * I2 + lane), cB = wrapped(2 * I2 + lane + 32);
    const bool hasB = lane + 32 < RH, hasA = lane < RH;
    for (int rr0 = (threadIdx.x >> 5); rr0 < RH; rr0 += 4 * nw) {
      float2 v[4][2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int rr = rr0 + q * nw;
        if (rr < RH) {
          const float2* row = src + wrapped(2 * I1 + rr) * L;
          if (hasA) v[q][0] = row[cA];
          if (hasB) v[q][1] = row[cB];
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int rr = rr0 + q * nw;
        if (rr < RH) {
          if (hasA) inb[rr * RHS + lane] = v[q][0];
          if (hasB) inb[rr * RHS + lane + 32] = v[q][1];
        }
      }
    }
  }
  __syncthreads();
  // rows: a[i2] = sum_m h[m] s[2 i2 + m], d[i2] = sum_m g[m] s[2 i2 + m]
  if constexpr (FAST) {
    const float inv_rh = 1.0f / (float)RH;
    for (int idx = threadIdx.x; idx < RH * (TI / 4); idx += blockDim.x) {
      const int qq = quot_small(idx, inv_rh), rr = idx - qq * RH;
      const float2* sp = inb + rr * RHS + 8 * qq;
      float2 a[4], d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = d[j] = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < taps + 6; ++m) {
        const float2 v = sp[m];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (m - 2 * j >= 0 && m - 2 * j < taps) {
            a[j] = __ffma2_rn(h[m - 2 * j], v, a[j]);
            d[j] = __ffma2_rn(g[m - 2 * j], v, d[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        rowp[rr * RS + 4 * qq + j] = a[j];
        rowp[rr * RS + TI + 4 * qq + j] = d[j];
      }
    }
  } else {
    for (int idx = threadIdx.x; idx < RH * TI; idx += blockDim.x) {
      const int rr = udiv(idx, dTI), i2 = idx - rr * TI;
      const float2* sp = inb + rr * RHS + 2 * i2;
      float2 a = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < taps; ++m) {
        const float2 v = sp[m];
        a = __ffma2_rn(h[m], v, a);
        d = __ffma2_rn(g[m], v, d);
      }
      rowp[rr * RS + i2] = a;
      rowp[rr * RS + TI + i2] = d;
    }
  }
  __syncthreads();
  // columns, and the write-out of the four sub-bands
  float2* plane = coef + (size_t)(G.plane0 + k) * G.n * G.n;
  float2* llk = ll_out + (size_t)k * (G.n / 2) * (G.n / 2);
  // columns of this thread's (at most two, TI <= 16) outputs, then every
  // output with its prox operands loaded together
  constexpr int kMaxIdx = 2;  // TI * 2TI / 256
  float2 lov[kMaxIdx], hiv[kMaxIdx];
  int i1v[kMaxIdx], kcv[kMaxIdx];  // coefficient row and column of [a | d], i1 = -1: none
#pragma unroll
  for (int t = 0; t < kMaxIdx; ++t) {
    const int idx = threadIdx.x + t * blockDim.x;
    if (FAST) {  // rows 2 j and 2 j + 1
      const int j = udiv(threadIdx.x, d2TI);
      i1v[t] = 2 * j < TI ? 2 * j + t : -1;
      kcv[t] = threadIdx.x - j * (2 * TI);
    } else {
      const int i1 = udiv(idx, d2TI);
      i1v[t] = idx < TI * 2 * TI ? i1 : -1;
      kcv[t] = idx - i1 * (2 * TI);
    }
    lov[t] = hiv[t] = make_float2(0.f, 0.f);
  }
  if constexpr (FAST) {
    if (i1v[0] >= 0) {
      const float2* cp = rowp + (2 * i1v[0]) * RS + kcv[0];
#pragma unroll
      for (int m = 0; m < taps + 2; ++m) {
        const float2 v = cp[m * RS];
        if (m < taps) {
          lov[0] = __ffma2_rn(h[m], v, lov[0]);
          hiv[0] = __ffma2_rn(g[m], v, hiv[0]);
        }
        if (m >= 2) {
          lov[1] = __ffma2_rn(h[m - 2], v, lov[1]);
          hiv[1] = __ffma2_rn(g[m - 2], v, hiv[1]);
        }
      }
    }
  } else {
#pragma unroll
    for (int t = 0; t < kMaxIdx; ++t) {
      if (i1v[t] < 0) continue;
      const float2* cp = rowp + (2 * i1v[t]) * RS + kcv[t];
#pragma unroll
      for (int m = 0; m < taps; ++m) {
        const float2 v = cp[m * RS];
        lov[t] = __ffma2_rn(h[m], v, lov[t]);
        hiv[t] = __ffma2_rn(g[m], v, hiv[t]);
      }
    }
  }
  // destinations (offsets in the plane, at most 2048^2): LL = lo of a
  // (top-left), LH = lo of d (top-right), HL = hi of a (H rows below), HH = hi
  // of d; on levels before the last LL goes to llk
  const int Hn = H * G.n;
  float2* z1 = MODE == kSaraProx ? pa.z1 + (size_t)(G.plane0 + k) * G.n * G.n : nullptr;
  const float* w = MODE == kSaraProx && pa.w ? pa.w + (size_t)(G.plane0 + k) * G.n * G.n : nullptr;
  float2* u1 = MODE == kSaraProx ? pa.u1 + (size_t)(G.plane0 + k) * G.n * G.n : nullptr;
  float2 zv[2 * kMaxIdx];
  float wv[2 * kMaxIdx];
  int off[kMaxIdx];
  bool lo_out[kMaxIdx];
#pragma unroll
  for (int t = 0; t < kMaxIdx; ++t) {
    off[t] = 0;
    lo_out[t] = false;
    if (i1v[t] < 0) continue;
    const bool rowlow = kcv[t] < TI;
    const int gi1 = I1 + i1v[t], gi2 = I2 + (rowlow ? kcv[t] : kcv[t] - TI);
    off[t] = gi1 * G.n + (rowlow ? gi2 : H + gi2);
    lo_out[t] = !rowlow || G.last;
    if (!lo_out[t]) llk[gi1 * H + gi2] = lov[t];
    if (MODE == kSaraProx) {  // the prox operands of every output, loaded together
      if (lo_out[t]) {
        zv[2 * t] = z1[off[t]];
        wv[2 * t] = w ? w[off[t]] : 1.0f;
      }
      zv[2 * t + 1] = z1[off[t] + Hn];
      wv[2 * t + 1] = w ? w[off[t] + Hn] : 1.0f;
    }
  }
#pragma unroll
  for (int t = 0; t < kMaxIdx; ++t) {
    if (i1v[t] < 0) continue;
    const float2 lo = cscale(lov[t], G.scale), hi = cscale(hiv[t], G.scale);
    if (MODE == kSaraPlain) {
      if (lo_out[t]) plane[off[t]] = lo;
      plane[off[t] + Hn] = hi;
    } else {
      if (lo_out[t]) f1 += sara_prox_v(lo, zv[2 * t], wv[2 * t], off[t], z1, u1, gamma);
      f1 += sara_prox_v(hi, zv[2 * t + 1], wv[2 * t + 1], off[t] + Hn, z1, u1, gamma);
    }
  }
  return f1;
}

// ---------------------------------------------------------------------------
// One analysis level for every wavelet plane.
//   input  : level 0: x (shared by all planes); else ll_in + k * (n/2)^2, L x L
//   output : LH, HL, HH at their Mallat positions of plane k; LL to
//            ll_out + k * (n/2)^2, or to the plane on the last level.
// CTA: coefficient tile [I1, I1 + TI) x [I2, I2 + TI) of the L/2 x L/2 sub-bands.
// ---------------------------------------------------------------------------
template <int MODE, bool FAST>
__global__ void __launch_bounds__(256) k_dwt_level(const float2* __restrict__ in, int in_shared,
                                                   float2* __restrict__ ll_out, float2* __restrict__ coef,
                                                   LevelGeom G, BasisList bl, const __grid_constant__ WaveletTaps wf,
                                                   SaraProxArgs pa, double* partials, DevScalars* sc) {
  pdl_sync(in, ll_out, coef, partials, sc);
  extern __shared__ float2 sm[];
  const int k = blockIdx.z;
  const float gamma = (MODE == kSaraProx) ? (float)sc->gamma : 0.f;
  float f1 = 0.f;
  if (k == G.nb) {
    // the Dirac plane (first level only): alpha_0 = x / sqrt(q) on this CTA's
    // 2TI x 2TI block of pixels, with its prox update
    const int TI = G.tile, r0 = 2 * blockIdx.y * TI, c0 = 2 * blockIdx.x * TI;
    const Div d2TI = make_div(2 * TI);
    const size_t base = (size_t)G.dirac * G.n * G.n;
    for (int e = threadIdx.x; e < 4 * TI * TI; e += blockDim.x) {
      const int rr = udiv(e, d2TI), cc = e - rr * (2 * TI);
      const size_t j = (size_t)(r0 + rr) * G.n + c0 + cc;
      const float2 al = cscale(in[j], G.scale);
      if (MODE == kSaraPlain) coef[base + j] = al;
      else f1 += sara_prox(al, base + j, pa, gamma);
    }
  } else {
    switch (bl.p(k)) {
      case 1: f1 += dwt_plane<1, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 2: f1 += dwt_plane<2, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 3: f1 += dwt_plane<3, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 4: f1 += dwt_plane<4, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 5: f1 += dwt_plane<5, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 6: f1 += dwt_plane<6, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      case 7: f1 += dwt_plane<7, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
      default: f1 += dwt_plane<8, MODE, FAST>(in, in_shared, ll_out, coef, G, wf, pa, k, gamma); break;
    }
  }
  if (MODE == kSaraProx) {
    // this block's f1 partial; the first synthesis launch adds them all up
    const FPair f1p{f1, 0.f};
    double f1d;
    block_reduce<1>(&f1p, &f1d);
    if (threadIdx.x == 0)
      partials[kCntF1 * 2 * kMaxPartials + G.f1_off + blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] =
          f1d;
  }
}

// ---------------------------------------------------------------------------
// The coarse levels of small planes in one launch per direction: once a
// level's side is at most kTailAnalysis (kTailSynthesis), one CTA per plane
// runs all the levels that remain, the plane's low-low band in shared memory
// between them.  A level of 8 to 64 pixels a side is bound by its launch and a
// CTA's dependent loads (4 to 6 us), not by arithmetic: at 64^2 four analysis
// levels with the prox 26 -> 13 us and three synthesis levels 17 -> 8 us (the
// iteration 188 -> 176 us, 128^2, M = 20000, 214 -> 209 us).  The sides are
// where it stops paying: three levels from 96 take 13 us so and 12 us in three
// launches (analysis), 23 and 13 us (synthesis); two from 64 the same.
// The filters wrap (also when longer than the signal), so the analysis extends
// each row, then each column, periodically by the filter's length before it
// filters; the synthesis reads its few wrapped coefficients by index.
// ---------------------------------------------------------------------------
constexpr int kTailAnalysis = 64, kTailSynthesis = 48;
constexpr int kTailThreads = 512;
constexpr int kTailExt = 14;  // 2 p - 2 for p = 8

struct TailGeom {
  int n, L, levels;  // image side; side of the tail's first (analysis) or last (synthesis) level; levels in it
  int nb, plane0;
  float scale;
  int dirac;   // analysis from level 0: plane of the Dirac basis, handled by CTA nb, or -1
  int f1_off;  // analysis, prox mode
};

template <int P, int MODE>
__device__ __forceinline__ void dwt_tail_plane(const float2* __restrict__ src, int src_stride, float2* __restrict__ pl,
                                               const TailGeom& G, const WaveletTaps& wf, float2* z1, float2* u1,
                                               const float* w, float gamma, FPair& f1) {
  extern __shared__ float2 sm[];
  constexpr int taps = 2 * P;
  const float2 *h = wf.h + P * (P - 1), *g = wf.g + P * (P - 1);
  const int ST = (G.L + kTailExt) | 1;  // row stride (odd)
  float2 *A = sm, *B = sm + (G.L + kTailExt) * ST;
  int L = G.L;
  Div dL = make_div(L);
  for (int e = threadIdx.x; e < L * L; e += kTailThreads) {
    const int r = udiv(e, dL), c = e - r * L;
    A[r * ST + c] = src[r * src_stride + c];
  }
  __syncthreads();
  for (int lev = 0; lev < G.levels; ++lev, L /= 2) {
    const int H = L / 2;
    const bool last = lev == G.levels - 1;
    dL = make_div(L);
    // rows, extended by taps - 2 (an extension longer than the signal repeats it)
    for (int e = threadIdx.x; e < L * (taps - 2); e += kTailThreads) {
      const int c = udiv(e, dL), r = e - c * L;
      A[r * ST + L + c] = A[r * ST + c - udiv(c, dL) * L];
    }
    __syncthreads();
    const int bq = H % 4 == 0 ? 4 : 1;
    for (int e = threadIdx.x; e < L * (H / bq); e += kTailThreads) {  // lanes take consecutive rows
      const int q = udiv(e, dL), r = e - q * L;
      const float2* sp = A + r * ST + 2 * bq * q;
      float2 a[4], d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = d[j] = make_float2(0.f, 0.f);
      if (bq == 4) {
#pragma unroll
        for (int m = 0; m < taps + 6; ++m) {
          const float2 v = sp[m];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (m - 2 * j >= 0 && m - 2 * j < taps) {
              a[j] = __ffma2_rn(h[m - 2 * j], v, a[j]);
              d[j] = __ffma2_rn(g[m - 2 * j], v, d[j]);
            }
          }
        }
      } else {
#pragma unroll
        for (int m = 0; m < taps; ++m) {
          const float2 v = sp[m];
          a[0] = __ffma2_rn(h[m], v, a[0]);
          d[0] = __ffma2_rn(g[m], v, d[0]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j >= bq) continue;
        B[r * ST + bq * q + j] = a[j];
        B[r * ST + H + bq * q + j] = d[j];
      }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < L * (taps - 2); e += kTailThreads) {
      const int r = udiv(e, dL), c = e - r * L;
      B[(L + r) * ST + c] = B[(r - udiv(r, dL) * L) * ST + c];
    }
    __syncthreads();
    // columns: low-low to A (or the plane, on the last level), the rest to the
    // plane; the prox operands of an output are loaded before its filter loop
    struct Operands {
      float2 zl, zh;
      float wl, wh;
    };
    const int Hn = H * G.n;
    auto operands = [&](int i1, int kc) {
      Operands p{};
      if (MODE == kSaraProx) {
        const int o = i1 * G.n + kc;
        if (kc >= H || last) {
          p.zl = z1[o];
          p.wl = w ? w[o] : 1.0f;
        }
        p.zh = z1[o + Hn];
        p.wh = w ? w[o + Hn] : 1.0f;
      }
      return p;
    };
    auto emit = [&](int i1, int kc, float2 lo, float2 hi, const Operands& p) {
      const int o = i1 * G.n + kc;  // Mallat position: columns [0, H) of a, [H, L) of d
      const bool ll = kc < H && !last;
      if (ll) A[i1 * ST + kc] = lo;
      const float2 ls = cscale(lo, G.scale), hs = cscale(hi, G.scale);
      if (MODE == kSaraPlain) {
        if (!ll) pl[o] = ls;
        pl[o + Hn] = hs;
      } else {
        if (!ll) f1.add(sara_prox_v(ls, p.zl, p.wl, o, z1, u1, gamma), 0.f);
        f1.add(sara_prox_v(hs, p.zh, p.wh, o + Hn, z1, u1, gamma), 0.f);
      }
    };
    if (H % 2 == 0) {
      for (int e = threadIdx.x; e < L * (H / 2); e += kTailThreads) {
        const int j = udiv(e, dL), kc = e - j * L;
        const float2* cp = B + 4 * j * ST + kc;
        const Operands p0 = operands(2 * j, kc), p1 = operands(2 * j + 1, kc);
        float2 lo[2], hi[2];
        lo[0] = lo[1] = hi[0] = hi[1] = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < taps + 2; ++m) {
          const float2 v = cp[m * ST];
          if (m < taps) {
            lo[0] = __ffma2_rn(h[m], v, lo[0]);
            hi[0] = __ffma2_rn(g[m], v, hi[0]);
          }
          if (m >= 2) {
            lo[1] = __ffma2_rn(h[m - 2], v, lo[1]);
            hi[1] = __ffma2_rn(g[m - 2], v, hi[1]);
          }
        }
        emit(2 * j, kc, lo[0], hi[0], p0);
        emit(2 * j + 1, kc, lo[1], hi[1], p1);
      }
    } else {
      for (int e = threadIdx.x; e < L * H; e += kTailThreads) {
        const int i1 = udiv(e, dL), kc = e - i1 * L;
        const float2* cp = B + 2 * i1 * ST + kc;
        const Operands p0 = operands(i1, kc);
        float2 lo = make_float2(0.f, 0.f), hi = lo;
#pragma unroll
        for (int m = 0; m < taps; ++m) {
          const float2 v = cp[m * ST];
          lo = __ffma2_rn(h[m], v, lo);
          hi = __ffma2_rn(g[m], v, hi);
        }
        emit(i1, kc, lo, hi, p0);
      }
    }
    __syncthreads();
  }
}

template <int MODE>
__global__ void __launch_bounds__(kTailThreads) k_dwt_tail(const float2* __restrict__ in, int in_shared,
                                                           float2* __restrict__ coef, TailGeom G, BasisList bl,
                                                           const __grid_constant__ WaveletTaps wf, SaraProxArgs pa,
                                                           double* partials, DevScalars* sc) {
  pdl_sync(in, coef, partials, sc);
  const int k = blockIdx.x;
  const float gamma = (MODE == kSaraProx) ? (float)sc->gamma : 0.f;
  FPair f1;  // (a thread has a dozen terms, summed exactly; one to four a level in k_dwt_level)
  if (k == G.nb) {  // the Dirac plane
    const size_t base = (size_t)G.dirac * G.n * G.n;
    for (int e = threadIdx.x; e < G.n * G.n; e += kTailThreads) {
      const float2 al = cscale(in[e], G.scale);
      if (MODE == kSaraPlain) coef[base + e] = al;
      else f1.add(sara_prox(al, base + e, pa, gamma), 0.f);
    }
  } else {
    const size_t base = (size_t)(G.plane0 + k) * G.n * G.n;
    const float2* src = in_shared ? in : in + (size_t)k * (G.n / 2) * (G.n / 2);
    float2 *z1 = MODE == kSaraProx ? pa.z1 + base : nullptr, *u1 = MODE == kSaraProx ? pa.u1 + base : nullptr;
    const float* w = MODE == kSaraProx && pa.w ? pa.w + base : nullptr;
    float2* pl = coef + base;
    switch (bl.p(k)) {
      case 1: dwt_tail_plane<1, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 2: dwt_tail_plane<2, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 3: dwt_tail_plane<3, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 4: dwt_tail_plane<4, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 5: dwt_tail_plane<5, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 6: dwt_tail_plane<6, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      case 7: dwt_tail_plane<7, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
      default: dwt_tail_plane<8, MODE>(src, G.L, pl, G, wf, z1, u1, w, gamma, f1); break;
    }
  }
  if (MODE == kSaraProx) {
    double f1d;
    block_reduce<1>(&f1, &f1d);
    if (threadIdx.x == 0) partials[kCntF1 * 2 * kMaxPartials + G.f1_off + blockIdx.x] = f1d;
  }
}

// f1 of §4.4 as the sum of the analysis levels' block partials (in index
// order), and the halting quantity zeta = |f1 - f1_prev| / f1_prev.
__device__ __forceinline__ void sara_f1_finish(const double* __restrict__ part, int n, DevScalars* sc) {
  // eight independent sums per thread (loads in flight together), in a fixed order
  constexpr int U = 8;
  const int nt = blockDim.x;
  double a[U];
#pragma unroll
  for (int u = 0; u < U; ++u) a[u] = 0.0;
  int i = threadIdx.x;
  for (; i + (U - 1) * nt < n; i += U * nt) {
    double t[U];
#pragma unroll
    for (int u = 0; u < U; ++u) t[u] = __ldcg(&part[i + u * nt]);
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] += t[u];
  }
  for (; i < n; i += nt) a[0] += __ldcg(&part[i]);
  const double mine = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
  double v;
  block_reduce<1>(&mine, &v);
  if (threadIdx.x == 0) {
    sc->f1 = v;
    const double prev = sc->f1_prev;
    sc->zeta = (prev != 0.0) ? fabs(v - prev) / fabs(prev) : INFINITY;
    sc->f1_prev = v;
  }
}

// Column then row synthesis of one plane's coefficient windows (in shared
// memory) for the Daubechies order P fixed at compile time; the finest level
// accumulates into accum, coarser levels write their low-low output.
//
// FAST (even tiles): a thread forms four adjacent outputs (two of each parity)
// of a column, then of a row, from one window of P + 1 coefficients, a quarter
// of the shared-memory loads of one output per thread, which bound this kernel
// (the four levels at 1024^2: 134 us with one output per
// thread, 95 us so).
constexpr int kIdwtMaxOut = 4;  // (2TO)^2 / blockDim outputs per thread: 1024 / 256
template <int P, bool FAST>
__device__ __forceinline__ void idwt_filter(const float2* LLs, const float2* HLs, const float2* LHs,
                                            const float2* HHs, float2* As, float2* Ds, const LevelGeom& G,
                                            const WaveletTaps& wf, int k, int K1, int K2,
                                            float2* __restrict__ ll_out, float2 (&accum)[kIdwtMaxOut]) {
  constexpr int hoff = P * (P - 1);
  const float2 *h = wf.h + hoff, *g = wf.g + hoff;
  const int L = G.L;
  const int TO = G.tile;
  const int CW = TO + P - 1, CWS = CW | 1;  // As, Ds: odd row stride
  const Div d2TO = make_div(2 * TO);
  // column synthesis: output row k1 in [0, 2TO), window column t2; taps of one
  // parity: m = par + 2u, t1 = (k1 - par) / 2 - u + P - 1
  if constexpr (FAST) {
    const float inv_cw = 1.0f / (float)CW;
    for (int idx = threadIdx.x; idx < (TO / 2) * CW; idx += blockDim.x) {
      const int qq = quot_small(idx, inv_cw), t2 = idx - qq * CW;
      float2 av[2][2], dv[2][2];  // [pair][parity]: output row 4 qq + 2 pair + parity
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int par = 0; par < 2; ++par) av[e][par] = dv[e][par] = make_float2(0.f, 0.f);
      const int w0 = 2 * qq * CW + t2;
#pragma unroll
      for (int w = P; w >= 0; --w) {  // window row 2 qq + w
        const float2 ll = LLs[w0 + w * CW], hl = HLs[w0 + w * CW], lh = LHs[w0 + w * CW], hh = HHs[w0 + w * CW];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int u = e + P - 1 - w;
          if (u < 0 || u >= P) continue;
#pragma unroll
          for (int par = 0; par < 2; ++par) {
            av[e][par] = __ffma2_rn(h[2 * u + par], ll, __ffma2_rn(g[2 * u + par], hl, av[e][par]));
            dv[e][par] = __ffma2_rn(h[2 * u + par], lh, __ffma2_rn(g[2 * u + par], hh, dv[e][par]));
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int par = 0; par < 2; ++par) {
          As[(4 * qq + 2 * e + par) * CWS + t2] = av[e][par];
          Ds[(4 * qq + 2 * e + par) * CWS + t2] = dv[e][par];
        }
    }
  } else {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int t2 = threadIdx.x >> 5; t2 < CW; t2 += nw)
      for (int k1 = lane; k1 < 2 * TO; k1 += 32) {
        const int par = k1 & 1;
        const int tb = (k1 - par) / 2 + P - 1;
        float2 av = make_float2(0.f, 0.f), dv = make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < P; ++u) {
          const int t1 = tb - u;
          const float2 hm = par ? h[2 * u + 1] : h[2 * u], gm = par ? g[2 * u + 1] : g[2 * u];
          const float2 ll = LLs[t1 * CW + t2], hl = HLs[t1 * CW + t2];
          const float2 lh = LHs[t1 * CW + t2], hh = HHs[t1 * CW + t2];
          av = __ffma2_rn(hm, ll, __ffma2_rn(gm, hl, av));
          dv = __ffma2_rn(hm, lh, __ffma2_rn(gm, hh, dv));
        }
        As[k1 * CWS + t2] = av;
        Ds[k1 * CWS + t2] = dv;
      }
  }
  __syncthreads();
  // row synthesis
  float2* llk = ll_out + (size_t)k * (G.n / 2) * (G.n / 2);
  if constexpr (FAST) {
    const int qq = udiv(threadIdx.x, d2TO), k1 = threadIdx.x - qq * (2 * TO);
    if (2 * qq < TO) {  // at most one group of four outputs per thread
      float2 sv[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int par = 0; par < 2; ++par) sv[e][par] = make_float2(0.f, 0.f);
      const int w0 = k1 * CWS + 2 * qq;
#pragma unroll
      for (int w = P; w >= 0; --w) {
        const float2 av = As[w0 + w], dv = Ds[w0 + w];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int u = e + P - 1 - w;
          if (u < 0 || u >= P) continue;
#pragma unroll
          for (int par = 0; par < 2; ++par)
            sv[e][par] = __ffma2_rn(h[2 * u + par], av, __ffma2_rn(g[2 * u + par], dv, sv[e][par]));
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int par = 0; par < 2; ++par) {
          if (G.last) accum[2 * e + par] = cadd(accum[2 * e + par], sv[e][par]);
          else llk[(size_t)(K1 + k1) * L + K2 + 4 * qq + 2 * e + par] = sv[e][par];
        }
    }
  } else {
#pragma unroll
    for (int t = 0; t < kIdwtMaxOut; ++t) {
      const int idx = threadIdx.x + t * blockDim.x;
      if (idx >= 4 * TO * TO) continue;
      const int k1 = udiv(idx, d2TO), k2 = idx - k1 * (2 * TO);
      const int par = k2 & 1;
      const int tb = (k2 - par) / 2 + P - 1;
      float2 sacc = make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < P; ++u) {
        const int t2 = tb - u;
        const float2 hm = par ? h[2 * u + 1] : h[2 * u], gm = par ? g[2 * u + 1] : g[2 * u];
        const float2 av = As[k1 * CWS + t2], dv = Ds[k1 * CWS + t2];
        sacc = __ffma2_rn(hm, av, __ffma2_rn(gm, dv, sacc));
      }
      if (G.last) accum[t] = cadd(accum[t], sacc);
      else llk[(size_t)(K1 + k1) * L + K2 + k2] = sacc;
    }
  }
}

// ---------------------------------------------------------------------------
// One synthesis level for every wavelet plane (transpose of k_dwt_level):
//   A  = colsyn(LL, HL), Dr = colsyn(LH, HH), s = rowsyn(A, Dr),
//   s[k] = sum_{m = k mod 2} h[m] a[((k - m)/2) mod H] + g[m] d[((k - m)/2) mod H].
// Output: L x L; to ll_out + k (n/2)^2, or, on the finest level, summed over
// planes (plus the Dirac plane) into x, scaled by 1/sqrt(q).
// CTA: output tile [K1, K1 + 2TO) x [K2, K2 + 2TO).
// ---------------------------------------------------------------------------
template <bool FAST>
__global__ void __launch_bounds__(256, 3) k_idwt_level(const float2* __restrict__ ll_in, int ll_from_plane,
                                                    float2* __restrict__ ll_out, const float2* __restrict__ coef,
                                                    float2* __restrict__ x, int dirac_plane, LevelGeom G,
                                                    BasisList bl, const __grid_constant__ WaveletTaps wf,
                                                    const double* f1_part, int f1_n,
                                                    DevScalars* sc) {
  pdl_sync(ll_in, ll_out, coef, x, f1_part, sc);
  extern __shared__ float2 sm[];
  // with f1 partials to sum, the first z slice is extra (dispatched first, so
  // that its block (0, 0), which forms f1 and zeta, overlaps the tiles)
  if (f1_n > 0 && blockIdx.z == 0) {
    if (blockIdx.x == 0 && blockIdx.y == 0) sara_f1_finish(f1_part, f1_n, sc);
    return;
  }
  const int bz = (int)blockIdx.z - (f1_n > 0 ? 1 : 0);  // the plane slice of this block
  const int L = G.L, H = L / 2;
  const int TO = G.tile;
  const int K1 = blockIdx.y * 2 * TO, K2 = blockIdx.x * 2 * TO;
  // the finest level loops over all planes in one CTA; otherwise one plane per z
  const int kbeg = G.last ? 0 : bz;
  const int kend = G.last ? G.nb : bz + 1;
  constexpr int kMaxOut = kIdwtMaxOut;
  float2 accum[kMaxOut];
  const int nout = (2 * TO) * (2 * TO);
  const Div dH = make_div(H), d2TO = make_div(2 * TO);
#pragma unroll
  for (int t = 0; t < kMaxOut; ++t) accum[t] = make_float2(0.f, 0.f);
  // the four coefficient windows of plane kk, loaded into registers (CW^2 <=
  // 23^2 <= 3 blockDim for TO <= 16, p <= 8): plane k + 1's loads are in flight while
  // plane k is synthesised
  float2 v[3][4];
  auto issue = [&](int kk) {
    const int pk = bl.p(kk);
    const int CWk = TO + pk - 1;
    const float2* plk = coef + (size_t)(G.plane0 + kk) * G.n * G.n;
    const float2* llk = ll_from_plane ? plk : ll_in + (size_t)kk * (G.n / 2) * (G.n / 2);
    const int lls = ll_from_plane ? G.n : H;
    // window origin: coefficient K/2 - p + 1 (mod H); the window wraps at most
    // once when H >= CW, and index by index (shifted to stay >= 0) otherwise
    const int o1 = K1 / 2 - pk + 1, o2 = K2 / 2 - pk + 1;
    const bool once = H >= CWk;
    const float rcw = 1.0f / (float)CWk;
    auto wrapped = [&](int i) {
      if (once) return i < 0 ? i + H : (i >= H ? i - H : i);
      i += 8 * H;
      return i - udiv(i, dH) * H;
    };
    const int Hn = H * G.n;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int e = threadIdx.x + q * blockDim.x;
      if (e < CWk * CWk) {
        const int t1 = quot_small(e, rcw), t2 = e - t1 * CWk;
        const int c1 = wrapped(o1 + t1), c2 = wrapped(o2 + t2);
        const float2* pl = plk + c1 * G.n + c2;
        v[q][0] = llk[c1 * lls + c2];
        v[q][1] = pl[Hn];
        v[q][2] = pl[H];
        v[q][3] = pl[Hn + H];
      }
    }
  };
  issue(kbeg);
  for (int k = kbeg; k < kend; ++k) {
    const int p = bl.p(k);
    const int CW = TO + p - 1;                 // coefficient window per axis
    float2* LLs = sm;                          // CW x CW each
    float2* HLs = LLs + CW * CW;
    float2* LHs = HLs + CW * CW;
    float2* HHs = LHs + CW * CW;
    float2* As = HHs + CW * CW;
    float2* Ds = As + 2 * TO * (CW | 1);       // 2TO x CW each, rows CW | 1 apart
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int e = threadIdx.x + q * blockDim.x;
      if (e < CW * CW) {
        LLs[e] = v[q][0];
        HLs[e] = v[q][1];
        LHs[e] = v[q][2];
        HHs[e] = v[q][3];
      }
    }
    __syncthreads();
    if (k + 1 < kend) issue(k + 1);
    switch (p) {
      case 1: idwt_filter<1, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 2: idwt_filter<2, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 3: idwt_filter<3, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 4: idwt_filter<4, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 5: idwt_filter<5, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 6: idwt_filter<6, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      case 7: idwt_filter<7, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
      default: idwt_filter<8, FAST>(LLs, HLs, LHs, HHs, As, Ds, G, wf, k, K1, K2, ll_out, accum); break;
    }
  }
  if (G.last) {
#pragma unroll
    for (int t = 0; t < kMaxOut; ++t) {
      int k1, k2;
      if (FAST) {
        const int qq = udiv(threadIdx.x, d2TO);
        k1 = threadIdx.x - qq * (2 * TO);
        k2 = 4 * qq + t;
        if (k2 >= 2 * TO) continue;
      } else {
        const int idx = threadIdx.x + t * blockDim.x;
        if (idx >= nout) continue;
        k1 = udiv(idx, d2TO);
        k2 = idx - k1 * (2 * TO);
      }
      float2 s = accum[t];
      const size_t j = (size_t)(K1 + k1) * G.n + K2 + k2;
      if (dirac_plane >= 0) s = cadd(s, coef[(size_t)dirac_plane * G.n * G.n + j]);
      x[j] = cscale(s, G.scale);
    }
  }
}

// The synthesis of the coarse levels, one CTA per plane (see k_dwt_tail): from
// the coarsest level up to the one whose output side is G.L, written to
// ll_out.  With f1 partials to sum, CTA nb forms f1 and zeta.
template <int P>
__device__ __forceinline__ void idwt_tail_plane(const float2* __restrict__ pl, float2* __restrict__ out,
                                                const TailGeom& G, const WaveletTaps& wf) {
  extern __shared__ float2 sm[];
  const float2 *h = wf.h + P * (P - 1), *g = wf.g + P * (P - 1);
  const int ST = G.L | 1;
  float2 *A = sm, *B = sm + G.L * ST;
  int L = G.L >> (G.levels - 1);
  for (int lev = 0; lev < G.levels; ++lev, L *= 2) {
    const int H = L / 2;
    const Div dL = make_div(L), dH = make_div(H);
    // A: [LL LH; HL HH]; LL of the levels after the first is there already
    for (int e = threadIdx.x; e < L * L; e += kTailThreads) {
      const int r = udiv(e, dL), c = e - r * L;
      if (lev == 0 || r >= H || c >= H) A[r * ST + c] = pl[r * G.n + c];
    }
    __syncthreads();
    auto wrapped = [&](int i) {  // i in (-P, H)
      if (H >= P) return i < 0 ? i + H : i;
      i += 8 * H;
      return i - udiv(i, dH) * H;
    };
    // columns, then rows: outputs 2 i and 2 i + 1 from coefficients i - u
    for (int e = threadIdx.x; e < H * L; e += kTailThreads) {
      const int i = udiv(e, dL), c = e - i * L;
      float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
      for (int u = 0; u < P; ++u) {
        const int t = wrapped(i - u);
        const float2 lo = A[t * ST + c], hi = A[(H + t) * ST + c];
        s0 = __ffma2_rn(h[2 * u], lo, __ffma2_rn(g[2 * u], hi, s0));
        s1 = __ffma2_rn(h[2 * u + 1], lo, __ffma2_rn(g[2 * u + 1], hi, s1));
      }
      B[2 * i * ST + c] = s0;
      B[(2 * i + 1) * ST + c] = s1;
    }
    __syncthreads();
    const bool last = lev == G.levels - 1;
    for (int e = threadIdx.x; e < H * L; e += kTailThreads) {
      const int j = udiv(e, dL), r = e - j * L;
      float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
      for (int u = 0; u < P; ++u) {
        const int t = wrapped(j - u);
        const float2 av = B[r * ST + t], dv = B[r * ST + H + t];
        s0 = __ffma2_rn(h[2 * u], av, __ffma2_rn(g[2 * u], dv, s0));
        s1 = __ffma2_rn(h[2 * u + 1], av, __ffma2_rn(g[2 * u + 1], dv, s1));
      }
      if (last) {
        out[r * L + 2 * j] = s0;
        out[r * L + 2 * j + 1] = s1;
      } else {
        A[r * ST + 2 * j] = s0;
        A[r * ST + 2 * j + 1] = s1;
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kTailThreads) k_idwt_tail(const float2* __restrict__ coef,
                                                            float2* __restrict__ ll_out, TailGeom G, BasisList bl,
                                                            const __grid_constant__ WaveletTaps wf,
                                                            const double* f1_part, int f1_n, DevScalars* sc) {
  pdl_sync(coef, ll_out, f1_part, sc);
  const int k = blockIdx.x;
  if (k == G.nb) {
    sara_f1_finish(f1_part, f1_n, sc);
    return;
  }
  const float2* pl = coef + (size_t)(G.plane0 + k) * G.n * G.n;
  float2* out = ll_out + (size_t)k * (G.n / 2) * (G.n / 2);
  switch (bl.p(k)) {
    case 1: idwt_tail_plane<1>(pl, out, G, wf); break;
    case 2: idwt_tail_plane<2>(pl, out, G, wf); break;
    case 3: idwt_tail_plane<3>(pl, out, G, wf); break;
    case 4: idwt_tail_plane<4>(pl, out, G, wf); break;
    case 5: idwt_tail_plane<5>(pl, out, G, wf); break;
    case 6: idwt_tail_plane<6>(pl, out, G, wf); break;
    case 7: idwt_tail_plane<7>(pl, out, G, wf); break;
    default: idwt_tail_plane<8>(pl, out, G, wf); break;
  }
}

__global__ void __launch_bounds__(256) k_f1_finish(const double* __restrict__ part, int n, DevScalars* sc) {
  pdl_sync(part, sc);
  sara_f1_finish(part, n, sc);
}

// Dirac-only synthesis: x = alpha_0 / sqrt(q).
__global__ void k_dirac_syn(const float2* __restrict__ a, float2* __restrict__ x, int64_t N, float scale) {
  pdl_sync(a, x);
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x)
    x[j] = cscale(a[j], scale);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static void basis_layout(const purify_ctx* c, int& dirac_plane, int& plane0, BasisList& bl, int& nb) {
  dirac_plane = -1;
  nb = 0;
  plane0 = 0;
  for (int k = 0; k < c->q; ++k) {
    if (c->bases[k] == 0) dirac_plane = k;
    else {
      if (nb == 0) plane0 = k;
      bl.packed |= (unsigned)c->bases[k] << (4 * nb++);
    }
  }
}

// Tile of one level: the largest divisor t <= kTile of H whose grid of
// (H / t)^2 tiles per plane times `planes` gives every SM a CTA; failing
// that, the largest divisor <= kMinTile (deep levels are small, and a CTA per
// tile of a few coefficients only wastes its halo).  Every divisor of
// H = 2^a or 3 * 2^a has the same form, as the index splits need.
constexpr int kMinTile = 4;
static int tile_for(int H, int64_t planes, int sms) {
  int fallback = 1;
  for (int t = std::min(kTile, H); t >= 1; --t) {
    if (H % t != 0) continue;
    if ((int64_t)(H / t) * (H / t) * planes >= (int64_t)sms) return t;
    if (t <= kMinTile) {
      fallback = t;
      break;
    }
  }
  return fallback;
}

// Finish zeta when the dictionary has no wavelet plane (Dirac only).
__global__ void k_finish_zeta(DevScalars* sc) {
  pdl_sync(sc);
  const double prev = sc->f1_prev;
  sc->zeta = (prev != 0.0) ? fabs(sc->f1 - prev) / fabs(prev) : INFINITY;
  sc->f1_prev = sc->f1;
}

static WaveletTaps wavelet_taps(const WaveletFilters& wf) {
  WaveletTaps t;
  for (int p = 1; p <= 8; ++p) {
    const float* h = wf.h + wf.off[p];
    for (int m = 0; m < 2 * p; ++m) {
      const float gm = (m & 1) ? -h[2 * p - 1 - m] : h[2 * p - 1 - m];
      t.h[wf.off[p] + m] = make_float2(h[m], h[m]);
      t.g[wf.off[p] + m] = make_float2(gm, gm);
    }
  }
  return t;
}

static size_t dwt_smem(int TI, int taps) {
  const int RH = 2 * TI + taps - 2;
  return (size_t)(RH * (RH | 1) + RH * (2 * TI + 1)) * sizeof(float2);
}

static size_t idwt_smem(int TO, int p) {
  const int CW = TO + p - 1;
  return (size_t)(4 * CW * CW + 2 * 2 * TO * (CW | 1)) * sizeof(float2);
}

int sara_analysis(purify_ctx* c, const float2* x, float2* alpha, SaraMode mode, const SaraProxArgs& pa,
                  cudaStream_t s, int* f1_parts) {
  if (f1_parts) *f1_parts = 0;
  int dirac_plane, plane0, nb;
  BasisList bl{};
  basis_layout(c, dirac_plane, plane0, bl, nb);
  const int64_t N = (int64_t)c->n * c->n;
  const float scale = 1.0f / sqrtf((float)c->q);
  if (dirac_plane >= 0 && nb == 0) {
    int blocks = (int)std::min<int64_t>((N + 255) / 256, 1024);
    if (mode == kSaraPlain)
      PURIFY_LAUNCH(c, "dirac", s,
                    (pdl_launch(k_dirac<kSaraPlain>, LaunchCfg{blocks, 256, 0, s, false}, x,
                        alpha + (size_t)dirac_plane * N, N, scale, pa,
                                                                c->d_partials, c->d_sc)));
    else
      PURIFY_LAUNCH(c, "dirac", s,
                    (pdl_launch(k_dirac<kSaraProx>, LaunchCfg{blocks, 256, 0, s, false}, x, nullptr, N, scale, pa,
                        c->d_partials, c->d_sc)));
  }
  if (nb == 0) {
    if (mode == kSaraProx) PURIFY_LAUNCH(c, "finish_zeta", s, (pdl_launch(k_finish_zeta, LaunchCfg{1, 1, 0, s},
        c->d_sc)));
    return check_cuda(cudaGetLastError());
  }
  int maxp = 1;
  for (int k = 0; k < nb; ++k) maxp = std::max(maxp, bl.p(k));
  const WaveletTaps taps = wavelet_taps(c->wf);
  int f1_off = 0;
  for (int lev = 0; lev < c->levels; ++lev) {
    const int L = c->n >> lev;
    const int H = L / 2;
    if (L <= kTailAnalysis && lev < c->levels - 1) {  // the levels that remain in one launch
      TailGeom G{c->n, L, c->levels - lev, nb, plane0, scale, lev == 0 ? dirac_plane : -1, f1_off};
      const float2* in = (lev == 0) ? x : c->d_ll[(lev - 1) & 1];
      const int ctas = nb + (G.dirac >= 0 ? 1 : 0);
      const size_t sm = (size_t)2 * (L + kTailExt) * ((L + kTailExt) | 1) * sizeof(float2);
      const LaunchCfg lc{ctas, kTailThreads, sm, s, lev > 0};
      f1_off += ctas;
      if (mode == kSaraPlain) {
        allow_smem(k_dwt_tail<kSaraPlain>, sm);
        PURIFY_LAUNCH(c, "dwt_level", s,
                      (pdl_launch(k_dwt_tail<kSaraPlain>, lc, in, lev == 0, alpha, G, bl, taps, pa, c->d_partials,
                          c->d_sc)));
      } else {
        allow_smem(k_dwt_tail<kSaraProx>, sm);
        PURIFY_LAUNCH(c, "dwt_level", s,
                      (pdl_launch(k_dwt_tail<kSaraProx>, lc, in, lev == 0, pa.z1, G, bl, taps, pa, c->d_partials,
                          c->d_sc)));
      }
      break;
    }
    const int TI = tile_for(H, nb + (lev == 0 && dirac_plane >= 0 ? 1 : 0), c->sms);
    LevelGeom G{TI, c->n, L, nb, plane0, lev == c->levels - 1, scale, lev == 0, lev == 0 ? dirac_plane : -1, f1_off};
    const float2* in = (lev == 0) ? x : c->d_ll[(lev - 1) & 1];
    float2* llo = c->d_ll[lev & 1];
    dim3 grid(H / TI, H / TI, nb + (G.dirac >= 0 ? 1 : 0));
    f1_off += (int)(grid.x * grid.y * grid.z);
    if (mode == kSaraProx && f1_off > 2 * kMaxPartials) return PURIFY_E_SIZE;  // the kCntF1 slot holds 2 kMaxPartials
    const size_t sm = dwt_smem(TI, 2 * maxp);
    const LaunchCfg lc{grid, 256, sm, s, lev > 0};
#define DWT(MD, FAST, COEF)                                                                                  \
  PURIFY_LAUNCH(c, "dwt_level", s,                                                                           \
                (pdl_launch(k_dwt_level<MD, FAST>, lc, in, lev == 0, llo, COEF, G, bl, taps, pa, c->d_partials, \
                            c->d_sc)))
    if (mode == kSaraPlain) {
      if (TI % 4 == 0) DWT(kSaraPlain, true, alpha);
      else DWT(kSaraPlain, false, alpha);
    } else {
      if (TI % 4 == 0) DWT(kSaraProx, true, pa.z1);
      else DWT(kSaraProx, false, pa.z1);
    }
#undef DWT
  }
  if (mode == kSaraProx) {
    if (f1_parts) {
      *f1_parts = f1_off;
    } else {  // no synthesis follows to finish f1: one block does
      PURIFY_LAUNCH(c, "f1_finish", s,
                    (pdl_launch(k_f1_finish, LaunchCfg{1, 256, 0, s}, c->d_partials + kCntF1 * 2 * kMaxPartials,
                        f1_off, c->d_sc)));
    }
  }
  return check_cuda(cudaGetLastError());
}

int sara_synthesis(purify_ctx* c, const float2* alpha, float2* x, cudaStream_t s, int f1_parts) {
  int dirac_plane, plane0, nb;
  BasisList bl{};
  basis_layout(c, dirac_plane, plane0, bl, nb);
  const int64_t N = (int64_t)c->n * c->n;
  const float scale = 1.0f / sqrtf((float)c->q);
  if (nb == 0) {
    int blocks = (int)std::min<int64_t>((N + 255) / 256, 1024);
    PURIFY_LAUNCH(c, "dirac", s, (pdl_launch(k_dirac_syn, LaunchCfg{blocks, 256, 0, s},
        alpha + (size_t)dirac_plane * N, x, N, scale)));
    return check_cuda(cudaGetLastError());
  }
  int maxp = 1;
  for (int k = 0; k < nb; ++k) maxp = std::max(maxp, bl.p(k));
  const WaveletTaps taps = wavelet_taps(c->wf);
  // the coarse levels (never the finest, which sums the planes) in one launch
  int top = c->levels - 1;  // coarsest level left to the per-level launches
  for (int lev = 1; lev < c->levels; ++lev) {
    const int L = c->n >> lev;
    if (L > kTailSynthesis || lev == c->levels - 1) continue;
    TailGeom G{c->n, L, c->levels - lev, nb, plane0, scale, -1, 0};
    const size_t sm = (size_t)2 * L * (L | 1) * sizeof(float2);
    allow_smem(k_idwt_tail, sm);
    PURIFY_LAUNCH(c, "idwt_level", s,
                  (pdl_launch(k_idwt_tail, LaunchCfg{nb + (f1_parts > 0 ? 1 : 0), kTailThreads, sm, s}, alpha,
                              c->d_ll[lev & 1], G, bl, taps, c->d_partials + kCntF1 * 2 * kMaxPartials, f1_parts,
                              c->d_sc)));
    top = lev - 1;
    break;
  }
  for (int lev = top; lev >= 0; --lev) {
    const int L = c->n >> lev;  // output side
    const int H = L / 2;
    const int TO = tile_for(H, lev == 0 ? 1 : nb, c->sms);
    LevelGeom G{TO, c->n, L, nb, plane0, lev == 0, scale, 0, -1};
    const bool from_plane = (lev == c->levels - 1);
    const float2* llin = from_plane ? nullptr : c->d_ll[(lev + 1) & 1];
    float2* llo = c->d_ll[lev & 1];
    // the first launch (coarsest level) carries one more z slice (the first)
    // whose first block forms f1 and zeta from the analysis partials
    const int f1n = (lev == c->levels - 1) ? f1_parts : 0;
    dim3 grid(L / (2 * TO), L / (2 * TO), (lev == 0 ? 1 : nb) + (f1n > 0 ? 1 : 0));
    const size_t sm = idwt_smem(TO, maxp);
    const LaunchCfg lc{grid, 256, sm, s};
#define IDWT(FAST)                                                                                             \
  PURIFY_LAUNCH(c, "idwt_level", s,                                                                            \
                (pdl_launch(k_idwt_level<FAST>, lc, llin, from_plane, llo, alpha, x, dirac_plane, G, bl, taps, \
                            c->d_partials + kCntF1 * 2 * kMaxPartials, f1n, c->d_sc)))
    if (TO % 2 == 0) IDWT(true);
    else IDWT(false);
#undef IDWT
  }
  return check_cuda(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Daubechies filters by spectral factorisation (Daubechies 1988): the roots y_k
// of P(y) = sum_{k<p} C(p-1+k, k) y^k (Durand-Kerner iteration), each mapped to
// the zero inside the unit circle of z^2 - (2 - 4y) z + 1; h is the coefficient
// list of (z + 1)^p prod (z - z_k) in descending powers, scaled to sum sqrt(2).
// ---------------------------------------------------------------------------
static std::vector<double> daubechies(int p) {
  using cd = std::complex<double>;
  const int d = p - 1;
  std::vector<double> P(p);
  double binom = 1.0;  // C(p-1+k, k)
  for (int k = 0; k < p; ++k) {
    if (k > 0) binom = binom * (double)(p - 1 + k) / (double)k;
    P[k] = binom;
  }
  std::vector<cd> roots(d);
  if (d > 0) {
    // monic in y: divide by the leading coefficient P[d]
    std::vector<cd> r(d);
    const cd seed(0.4, 0.9);
    cd pw(1.0, 0.0);
    for (int k = 0; k < d; ++k) { r[k] = pw; pw *= seed; }
    auto evalP = [&](cd y) {
      cd acc = P[d];
      for (int k = d - 1; k >= 0; --k) acc = acc * y + P[k];
      return acc / P[d];
    };
    for (int it = 0; it < 2000; ++it) {
      double delta = 0.0;
      for (int k = 0; k < d; ++k) {
        cd den(1.0, 0.0);
        for (int j = 0; j < d; ++j)
          if (j != k) den *= (r[k] - r[j]);
        const cd step = evalP(r[k]) / den;
        r[k] -= step;
        delta = std::max(delta, std::abs(step));
      }
      if (delta < 1e-17) break;
    }
    roots = r;
  }
  // polynomial coefficients in ascending powers of z
  std::vector<cd> poly(1, cd(1.0, 0.0));
  auto mul_root = [&](cd z0) {  // poly *= (z - z0)
    std::vector<cd> out(poly.size() + 1, cd(0.0, 0.0));
    for (size_t i = 0; i < poly.size(); ++i) {
      out[i + 1] += poly[i];
      out[i] -= z0 * poly[i];
    }
    poly.swap(out);
  };
  for (int k = 0; k < p; ++k) mul_root(cd(-1.0, 0.0));
  for (int k = 0; k < d; ++k) {
    const cd c = 2.0 - 4.0 * roots[k];
    const cd disc = std::sqrt(c * c - 4.0);
    cd z1 = (c + disc) / 2.0, z2 = (c - disc) / 2.0;
    mul_root(std::abs(z1) < 1.0 ? z1 : z2);
  }
  // descending powers: h[m] = coefficient of z^(2p-1-m)
  std::vector<double> h(2 * p);
  double sum = 0.0;
  for (int m = 0; m < 2 * p; ++m) {
    h[m] = poly[2 * p - 1 - m].real();
    sum += h[m];
  }
  for (auto& v : h) v *= std::sqrt(2.0) / sum;
  return h;
}

void make_daubechies(WaveletFilters& wf) {
  int off = 0;
  wf.off[0] = 0;
  for (int p = 1; p <= 8; ++p) {
    wf.off[p] = off;
    std::vector<double> h = daubechies(p);
    for (int m = 0; m < 2 * p; ++m) wf.h[off + m] = (float)h[m];
    off += 2 * p;
  }
}

}  // namespace purify
