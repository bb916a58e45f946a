// Deterministic FP64 block reductions with a "last block finishes" epilogue.
//
// Every block writes its partial sums to a slot of a partial buffer, then
// takes a ticket on a counter; the block that takes the last ticket sums the
// partials in a fixed order and runs the finishing code.  The result does not
// depend on block scheduling, and no extra kernel launch is needed.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace purify {

// ---------------------------------------------------------------------------
// Per-thread accumulation without FP64 arithmetic (GB300 has little FP64
// throughput): terms are formed exactly with error-free transformations
// (TwoSum for a difference, an FMA for a product's rounding error) and summed
// into a float pair (hi, lo); the pairs of a warp are added as triples (below),
// and the sums across warps and blocks are FP64.  With the few terms each thread
// holds, the per-thread error is far below FP64 rounding of the total.
// ---------------------------------------------------------------------------
struct FPair {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float p, float pe) {  // += p + pe
    const float s = hi + p;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (p - bb);
    hi = s;
    lo += e + pe;
  }
  // += x * y (exact product)
  __device__ __forceinline__ void add_prod(float x, float y) {
    const float p = x * y;
    add(p, fmaf(x, y, -p));
  }
  // += (a - b)^2 with a - b formed exactly
  __device__ __forceinline__ void add_sq_diff(float a, float b) {
    const float d = a - b;
    const float bb = d - a;
    const float de = (a - (d - bb)) + (-b - bb);
    const float p = d * d;
    add(p, fmaf(d, d, -p) + 2.f * d * de);
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// FP64 adds are the scarce resource of these reductions: GB300 starts about
// two per clock and SM, so one warp-wide add occupies the SM's FP64 unit for
// 16 clocks, and the ten of a warp's shuffle tree over two values, for every
// warp of a block, cost more than the kernel's own work (degridding with the
// norms of the l2 branch at 1024^2, M = 2^21: 98 us against 63 us without).
// So the lanes of a warp are summed in FP32 as well, in triples whose three
// components hold what every addition rounds off (the terms dropped are below
// 2^-68 of the largest partial sum, so the one rounding to FP64 at the end is
// the only error that FP64 can show; a pair, 2^-47, would lose bits that an
// FP64 tree keeps), and only the sums across warps and blocks are FP64.  A
// warp that holds a value which could overflow the triple (or is not finite)
// takes the FP64 tree instead.
constexpr float kPairMax = 1.2676506e30f;  // 2^100: 32 such values stay far below FP32's maximum

// a + b = two_sum + e, exactly (Knuth's TwoSum)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
  return s;
}

struct FTriple {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float ta, float tb, float tc) {
    float e1, e2, e3;
    a = two_sum(a, ta, e1);
    b = two_sum(b, tb, e2);
    b = two_sum(b, e1, e3);
    c += tc + (e2 + e3);
  }
  __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

// Tree over the first `valid` lanes of a warp whose first `present` lanes
// exist (any block size, including a partial last warp); every present lane
// calls it, and the result is valid in lane 0.
__device__ __forceinline__ double warp_tree(double v, int lane, int present, int valid) {
  const unsigned mask = present >= 32 ? 0xffffffffu : ((1u << present) - 1u);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (o >= valid) continue;  // (uniform) nothing to add at this distance
    const double t = __shfl_down_sync(mask, v, o);
    if (lane + o < valid) v += t;
  }
  return v;
}

__device__ __forceinline__ double warp_tree(FTriple v, int lane, int present, int valid) {
  const unsigned mask = present >= 32 ? 0xffffffffu : ((1u << present) - 1u);
  if (__any_sync(mask, !(fabsf(v.a) < kPairMax))) return warp_tree(v.value(), lane, present, valid);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (o >= valid) continue;
    const float a = __shfl_down_sync(mask, v.a, o), b = __shfl_down_sync(mask, v.b, o);
    const float c = __shfl_down_sync(mask, v.c, o);
    if (lane + o < valid) v.add(a, b, c);
  }
  return v.value();
}

__device__ __forceinline__ double warp_tree(FPair v, int lane, int present, int valid) {
  return warp_tree(FTriple{v.hi, v.lo, 0.f}, lane, present, valid);
}

// Two sums over a full warp at once: the halves of the warp first exchange what
// the other one takes, then the lower half adds the first value and the upper
// half the second: five triple additions instead of ten.  With one warp per
// scheduler, as in the row passes of the CG, the time goes by instructions
// (256^2, CG of ten steps: two trees of pairs 275.6 us, two trees of triples
// 2.3 % more, this one 272.8 us).  The first sum is valid in lane 0, the second in lane 16.
__device__ __forceinline__ double warp_tree2(FTriple v0, FTriple v1, int lane) {
  const unsigned mask = 0xffffffffu;
  const bool up = (lane & 16) != 0;
  if (__any_sync(mask, !(fabsf(v0.a) < kPairMax && fabsf(v1.a) < kPairMax))) {
    const double s0 = warp_tree(v0, lane, 32, 32), s1 = warp_tree(v1, lane, 32, 32);
    const double s1b = __shfl_sync(mask, s1, 0);
    return up ? s1b : s0;
  }
  FTriple v = up ? v1 : v0;
  const FTriple w = up ? v0 : v1;
  v.add(__shfl_xor_sync(mask, w.a, 16), __shfl_xor_sync(mask, w.b, 16), __shfl_xor_sync(mask, w.c, 16));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)  // (lanes past a half's first o are not used any more)
    v.add(__shfl_down_sync(mask, v.a, o), __shfl_down_sync(mask, v.b, o), __shfl_down_sync(mask, v.c, o));
  return v.value();
}

__device__ __forceinline__ FTriple to_triple(FPair v) { return FTriple{v.hi, v.lo, 0.f}; }
__device__ __forceinline__ FTriple to_triple(FTriple v) { return v; }

// Sum of NV values (FPair, FTriple or double) over the block; out is valid in thread 0.
template <int NV, class V>
__device__ __forceinline__ void block_reduce(const V* v, double* out) {
  __shared__ double sh[NV][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  const int mylanes = min(32, (int)blockDim.x - wid * 32);
  bool two = false;  // (uniform per warp) out[0] holds the first sum in lane 0, the second in lane 16
  if constexpr (NV == 2 && !std::is_same<V, double>::value) two = mylanes == 32;
  if constexpr (NV == 2 && !std::is_same<V, double>::value) {
    if (two) out[0] = warp_tree2(to_triple(v[0]), to_triple(v[1]), lane);
  }
  if (!two) {
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = warp_tree(v[k], lane, mylanes, mylanes);
  }
  __syncthreads();
  if (two) {
    if ((lane & 15) == 0) sh[NV == 2 ? lane >> 4 : 0][wid] = out[0];
  } else if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k][wid] = out[k];
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = warp_tree(lane < nw ? sh[k][lane] : 0.0, lane, mylanes, nw);
  }
}

// Largest of one float per thread, over the block (valid in thread 0; any
// block size).
__device__ __forceinline__ float block_max(float v) {
  __shared__ float sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  const int mylanes = min(32, (int)blockDim.x - wid * 32);
  const unsigned mask = mylanes >= 32 ? 0xffffffffu : ((1u << mylanes) - 1u);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float t = __shfl_down_sync(mask, v, o);
    if (lane + o < mylanes) v = fmaxf(v, t);
  }
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (wid == 0)
    for (int k = 0; k < nw; ++k) v = fmaxf(v, sh[k]);
  return v;
}

// Takes a ticket after this block's thread 0 has written its partials; true
// (in every thread) in the block that takes the last one.
__device__ __forceinline__ bool last_block_ticket(unsigned int* counter, unsigned int nblk) {
  __shared__ bool am_last;
  if (threadIdx.x == 0) {
    __threadfence();
    am_last = (atomicAdd(counter, 1u) == nblk - 1);
  }
  __syncthreads();
  if (!am_last) return false;
  __threadfence();
  return true;
}

// Writes the block's NV partials, and in the last block to finish sums all
// partials (fixed order) into total[0..NV).  Returns true in thread 0 of that
// last block only.  partials holds NV x kMaxPartials doubles; the grid must
// have at most kMaxPartials blocks.  The counter is reset for the next use.
template <int NV, class V>
__device__ __forceinline__ bool reduce_last_block(const V* v, double* partials, unsigned int* counter, double* total) {
  const unsigned int nblk = gridDim.x * gridDim.y * gridDim.z;
  const unsigned int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  double acc[NV];
  block_reduce<NV>(v, acc);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) partials[k * kMaxPartials + bid] = acc[k];
  }
  if (!last_block_ticket(counter, nblk)) return false;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    double s = 0.0;
    for (unsigned int i = threadIdx.x; i < nblk; i += blockDim.x) s += __ldcg(&partials[k * kMaxPartials + i]);
    acc[k] = s;
  }
  block_reduce<NV>(acc, total);
  if (threadIdx.x == 0) *counter = 0u;
  return threadIdx.x == 0;
}

// ---------------------------------------------------------------------------
// Step sizes of single-reduction CG (Chronopoulos & Gear 1989), formed by the
// kernel that applies the update rather than by a last block of the kernel
// that produced the inner products.  CG step j's Q-epilogue left per-block
// partials of gamma_j = <r, r> and delta_j = <Qr, r>; every block of the
// consumer adds them in the same fixed order (so all blocks agree bit for
// bit) and forms
//   beta_j  = gamma_j / gamma_{j-1}         (0 for the first step)
//   alpha_j = gamma_j / (delta_j - beta_j gamma_j / alpha_{j-1}),
// reading step j-1's (gamma, alpha) from slot (j-1) & 1; block 0 stores step
// j's in slot j & 1, which no block of this kernel reads.  Every thread of
// the block calls it; the results are returned to all of them.  With many
// partials (large images) a one-block kernel forms them once instead
// (k_cg_scalars) and the consumers pass nblk = 0 to read its result.
// ---------------------------------------------------------------------------
struct CgStep {
  float alpha, beta;
  bool first;
};

__device__ __forceinline__ CgStep cg_consume(const double* __restrict__ part, int nblk, int j, DevScalars* sc) {
  __shared__ float s_al, s_be;
  __shared__ int s_first;
  if (nblk == 0) {  // formed by k_cg_scalars for this step (many partials)
    return CgStep{(float)sc->alpha, (float)sc->beta, sc->cg_step_first != 0};
  }
  // the first warp adds the partials (fixed order) and forms the step sizes:
  // gamma's quotients by step j - 1's gamma and alpha on lanes 0 and 1 together
  // (an FP64 division takes 560 clocks), then alpha.  Reciprocals formed while
  // the partials arrive would save one division, at a rounding more per quotient.
  if (threadIdx.x < 32) {  // (blocks have at least two threads)
    const int lane = threadIdx.x, present = min(32, (int)blockDim.x);
    const unsigned mask = present >= 32 ? 0xffffffffu : ((1u << present) - 1u);
    double v[2] = {0.0, 0.0};
    const int prev = (j - 1) & 1;
    double old = 0.0;  // gamma (even lanes) and alpha (odd lanes) of step j - 1
    if (j > 0) old = (lane & 1) ? sc->cg_alpha[prev] : sc->cg_rho[prev];
    for (int i = lane; i < nblk; i += present) {
      v[0] += __ldcg(&part[i]);
      v[1] += __ldcg(&part[kMaxPartials + i]);
    }
    const unsigned zero = __ballot_sync(mask, old == 0.0);
    v[0] = warp_tree(v[0], lane, present, min(present, nblk));
    const double gamma = __shfl_sync(mask, v[0], 0);
    const double quot = gamma / old;
    const double quot_al = __shfl_sync(mask, quot, 1);
    v[1] = warp_tree(v[1], lane, present, min(present, nblk));
    if (lane == 0) {
      const double delta = v[1];
      const bool first = j == 0 || (zero & 3u) != 0u;
      const double beta = first ? 0.0 : quot;
      const double den = first ? delta : delta - beta * quot_al;
      const double alpha = den > 0.0 ? gamma / den : 0.0;
      s_al = (float)alpha;
      s_be = (float)beta;
      s_first = first ? 1 : 0;
      if (blockIdx.x == 0) {
        sc->cg_rho[j & 1] = gamma;
        sc->cg_alpha[j & 1] = alpha;
        sc->alpha = alpha;
        sc->beta = beta;
        sc->rho = gamma;
        sc->pqp = den;
        sc->cg_res = sqrt(gamma);
        sc->cg_step_first = first ? 1 : 0;
      }
    }
  }
  __syncthreads();
  return CgStep{s_al, s_be, s_first != 0};
}

}  // namespace purify
