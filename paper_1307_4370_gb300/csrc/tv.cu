// Weighted total variation prior (§3.3 eq. tvproblem, §5 weighted TV).
//
// f1(x) = ||W grad x||_1 with the isotropic gradient magnitude of forward
// differences (zero on the last row and column), complex pixels counted by
// modulus.  Its prox, prox_{lam f1}(b) = argmin 1/2||x - b||^2 + lam f1(x),
// is computed as §5 states SOPT does, with the fast gradient projection of
// Beck & Teboulle (2009) on the dual pair (p, q):
//   L(p, q)_{i,j} = p_{i,j} + q_{i,j} - p_{i-1,j} - q_{i,j-1}      (-div)
//   L^T(z)        = (z_{i,j} - z_{i+1,j}, z_{i,j} - z_{i,j+1})      (-grad)
//   (p, q)_k = Proj_{|.| <= w}[(r, s) + L^T(b - lam L(r, s)) / (8 lam)]
//   (r, s)   = (p, q)_k + c_k ((p, q)_k - (p, q)_{k-1}),  c_k = (t_k - 1) / t_{k+1}
//   x        = b - lam L(p_K, q_K)
// A launch advances several FGP iterations on tiles with a halo (the iterations
// are coupled through the neighbours only).  The momentum coefficients are
// host constants.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "reduce.cuh"

#define TV_TRY(expr)                  \
  do {                                \
    const int _st = (expr);           \
    if (_st != PURIFY_OK) return _st; \
  } while (0)

namespace purify {

namespace {

// L(r, s) at (i, j) of an m x n image (row-major, m = n here).
__device__ __forceinline__ float2 op_L(const float2* __restrict__ r, const float2* __restrict__ s, int i, int j,
                                       int n) {
  float2 v = make_float2(0.f, 0.f);
  const int k = i * n + j;
  if (i < n - 1) v = cadd(v, r[k]);
  if (j < n - 1) v = cadd(v, s[k]);
  if (i > 0) v = csub(v, r[k - n]);
  if (j > 0) v = csub(v, s[k - 1]);
  return v;
}

__device__ __forceinline__ float tv_lambda(const DevScalars* sc, float lam) {
  return sc ? (float)sc->gamma : lam;
}

// Up to K FGP iterations per launch.  An iteration couples a pixel with its
// neighbours only, so a CTA advances its TB x TB tile K iterations on a region
// K pixels larger on each side: (r, s) and z = b - lam L(r, s) in shared
// memory, (p, q) and b of each pixel in registers, the outermost ring of the
// region becoming invalid with every iteration.  The pixels of the rings are
// computed again by the neighbouring CTAs, with the same operations, so the
// result does not depend on the split.  One iteration per launch read and
// wrote 9 image vectors each time (512^2: 20 launches, 191 us; 68 us
// for 4); a region of 42 x 42 for K = 5 does 1.7 times the arithmetic instead.
// first: the dual variables are zero and b = xa (+ xb), stored for the next
// launches; otherwise they are read from (r, s, p, q) and written to the other
// set (CTAs read their neighbours' pixels).
constexpr int kTvK = 5;
struct TvMomentum {
  float c[kTvK];
};
struct TvDual {
  float2 *r, *s, *p, *q;
};

template <int TB>
__global__ void __launch_bounds__(256, 2) k_tv_fgp(int n, int tiles, const float2* xa, const float2* xb, float2* b_io,
                                                TvDual in, TvDual out, const float* w, int count, TvMomentum mom,
                                                int first, int last, const DevScalars* sc, float lam_host) {
  pdl_sync(xa, xb, b_io, w, sc);
  constexpr int LW = TB + 2 * kTvK, NP = LW * LW, NQ = (NP + 255) / 256;
  extern __shared__ float2 tv_sm[];
  float2 *R = tv_sm, *S = tv_sm + NP, *Z = tv_sm + 2 * NP;
  const float lam = tv_lambda(sc, lam_host);
  const int ti = blockIdx.x / tiles, tj = blockIdx.x - ti * tiles;
  const int i0 = ti * TB - kTvK, j0 = tj * TB - kTvK;  // the region's first pixel
  float2 bb[NQ], pp[NQ], qq[NQ];
  float rad[NQ];
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    const int e = threadIdx.x + u * 256, li = e / LW, lj = e - li * LW;
    const int i = i0 + li, j = j0 + lj;
    bb[u] = pp[u] = qq[u] = make_float2(0.f, 0.f);
    rad[u] = 1.0f;
    float2 r = bb[u], s = bb[u];
    if (e < NP && i >= 0 && i < n && j >= 0 && j < n) {
      const int k = i * n + j;
      if (first) {
        bb[u] = xb ? cadd(xa[k], xb[k]) : xa[k];
      } else {
        bb[u] = b_io[k];
        pp[u] = in.p[k];
        qq[u] = in.q[k];
        r = in.r[k];
        s = in.s[k];
      }
      if (w) rad[u] = w[k];
    }
    if (e < NP) {
      R[e] = r;
      S[e] = s;
    }
  }
  const bool active = lam > 0.f;  // otherwise the prox is the identity
  const float step = 1.0f / (8.0f * lam);
  for (int it = 0; it < count && active; ++it) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NQ; ++u) {
      const int e = threadIdx.x + u * 256, li = e / LW, lj = e - li * LW;
      if (e >= NP) continue;
      const int i = i0 + li, j = j0 + lj;
      // L(r, s); what lies outside the region belongs to invalid rings
      float2 v = make_float2(0.f, 0.f);
      if (i < n - 1) v = cadd(v, R[e]);
      if (j < n - 1) v = cadd(v, S[e]);
      if (i > 0 && li > 0) v = csub(v, R[e - LW]);
      if (j > 0 && lj > 0) v = csub(v, S[e - 1]);
      Z[e] = csub(bb[u], cscale(v, lam));
    }
    __syncthreads();
    const float cmom = mom.c[it];
#pragma unroll
    for (int u = 0; u < NQ; ++u) {
      const int e = threadIdx.x + u * 256, li = e / LW, lj = e - li * LW;
      if (e >= NP) continue;
      const int i = i0 + li, j = j0 + lj;
      const float2 z0 = Z[e], r = R[e], s = S[e];
      float2 g1 = make_float2(0.f, 0.f), g2 = g1;
      if (i < n - 1 && li < LW - 1) g1 = csub(z0, Z[e + LW]);
      if (j < n - 1 && lj < LW - 1) g2 = csub(z0, Z[e + 1]);
      float2 pn = make_float2(fmaf(step, g1.x, r.x), fmaf(step, g1.y, r.y));
      float2 qn = make_float2(fmaf(step, g2.x, s.x), fmaf(step, g2.y, s.y));
      if (i == n - 1) pn = make_float2(0.f, 0.f);
      if (j == n - 1) qn = make_float2(0.f, 0.f);
      // projection of the pair onto the disc of radius w
      const float mag = sqrtf(pn.x * pn.x + pn.y * pn.y + qn.x * qn.x + qn.y * qn.y);
      if (mag > rad[u]) {
        const float f = rad[u] / mag;
        pn = cscale(pn, f);
        qn = cscale(qn, f);
      }
      const float2 po = pp[u], qo = qq[u];
      pp[u] = pn;
      qq[u] = qn;
      R[e] = make_float2(fmaf(cmom, pn.x - po.x, pn.x), fmaf(cmom, pn.y - po.y, pn.y));
      S[e] = make_float2(fmaf(cmom, qn.x - qo.x, qn.x), fmaf(cmom, qn.y - qo.y, qn.y));
    }
  }
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    const int e = threadIdx.x + u * 256, li = e / LW, lj = e - li * LW;
    const int i = i0 + li, j = j0 + lj;
    if (li < kTvK || li >= kTvK + TB || lj < kTvK || lj >= kTvK + TB || i >= n || j >= n) continue;
    const int k = i * n + j;
    if (first) b_io[k] = bb[u];
    out.p[k] = pp[u];
    out.q[k] = qq[u];
    if (!last) {  // (this thread's own pixels)
      out.r[k] = R[e];
      out.s[k] = S[e];
    }
  }
}

// No iteration at all: b alone, with zero dual variables.
__global__ void k_tv_init(int64_t N, const float2* __restrict__ xa, const float2* __restrict__ xb,
                          float2* __restrict__ b, float2* __restrict__ p, float2* __restrict__ q) {
  pdl_sync(xa, xb, b, p, q);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
    b[k] = xb ? cadd(xa[k], xb[k]) : xa[k];
    p[k] = q[k] = make_float2(0.f, 0.f);
  }
}

// x = b - lam L(p, q).  SDMM mode (z1 non-null): r1 = x, z1 <- b - r1 (= z1 +
// x_hat - r1), x1 = r1 - z1, and f1 = ||W grad x_hat||_1 with zeta (FP64
// across threads, exact FP32 products per thread).  Plain mode: out = x.
__global__ void k_tv_finish(int n, const float2* __restrict__ b, const float2* __restrict__ p,
                            const float2* __restrict__ q, float2* __restrict__ out, float2* __restrict__ z1,
                            const float2* __restrict__ xhat, const float* __restrict__ w, double* partials,
                            DevScalars* sc, float lam_host) {
  pdl_sync(b, p, q, out, z1, xhat, w, partials, sc);
  const float lam = tv_lambda(z1 ? sc : nullptr, lam_host);
  const int64_t N = (int64_t)n * n;
  FPair f1;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)k / n, j = (int)k - i * n;
    const float2 bk = b[k];
    const float2 x = (lam > 0.f) ? csub(bk, cscale(op_L(p, q, i, j, n), lam)) : bk;
    if (!z1) {
      out[k] = x;
      continue;
    }
    const float2 zn = csub(bk, x);  // z1 + x_hat - r1
    z1[k] = zn;
    out[k] = csub(x, zn);           // x1 = r1 - z1
    // f1 term of this pixel: w |grad x_hat|
    const float2 xc = xhat[k];
    float2 d1 = make_float2(0.f, 0.f), d2 = d1;
    if (i < n - 1) d1 = csub(xhat[k + n], xc);
    if (j < n - 1) d2 = csub(xhat[k + 1], xc);
    const float mag = sqrtf(d1.x * d1.x + d1.y * d1.y + d2.x * d2.x + d2.y * d2.y);
    f1.add_prod(w ? w[k] : 1.0f, mag);
  }
  if (!z1) return;
  double tot;
  if (reduce_last_block<1>(&f1, partials + kCntF1 * 2 * kMaxPartials, &sc->counter[kCntF1], &tot)) {
    sc->f1 = tot;
    const double prev = sc->f1_prev;
    sc->zeta = (prev != 0.0) ? fabs(tot - prev) / fabs(prev) : INFINITY;
    sc->f1_prev = tot;
  }
}

// |grad x| per pixel, as complex (|grad x|, 0) so the complex max and
// reweighting kernels apply.
__global__ void k_tv_gradmag(int n, const float2* __restrict__ x, float2* __restrict__ g) {
  pdl_sync(x, g);
  const int64_t N = (int64_t)n * n;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)k / n, j = (int)k - i * n;
    const float2 xc = x[k];
    float2 d1 = make_float2(0.f, 0.f), d2 = d1;
    if (i < n - 1) d1 = csub(x[k + n], xc);
    if (j < n - 1) d2 = csub(x[k + 1], xc);
    g[k] = make_float2(sqrtf(d1.x * d1.x + d1.y * d1.y + d2.x * d2.x + d2.y * d2.y), 0.f);
  }
}

unsigned tv_blocks(int64_t N) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, 4096)); }

}  // namespace

// `iters` FGP iterations for b = xa (+ xb): b into scratch, the dual pair into
// *p, *q.  `sc` non-null takes lam = gamma from the device scalars (SDMM),
// otherwise lam_host.  Scratch: b and two sets of (r, s, p, q), 9 N complex.
// chained: the first launch may be a programmatic dependent of the kernel
// before it (not after the stream has waited on another one).
static int tv_fgp(purify_ctx* c, float2* scratch, const float2* xa, const float2* xb, const float* w, int iters,
                  const DevScalars* sc, float lam_host, bool chained, float2** p, float2** q, cudaStream_t s) {
  const int64_t N = ((int64_t)c->n * c->n);
  float2* b = scratch;
  TvDual set[2];
  for (int k = 0; k < 2; ++k) {
    float2* d = scratch + (1 + 4 * k) * N;
    set[k] = TvDual{d, d + N, d + 2 * N, d + 3 * N};
  }
  int a = 0;  // the set that holds the current dual variables
  if (iters == 0)
    PURIFY_LAUNCH(c, "tv_init", s,
                  (pdl_launch(k_tv_init, LaunchCfg{tv_blocks(N), 256, 0, s, chained}, N, xa, xb, b, set[0].p,
                      set[0].q)));
  // tiles of 32 once they give every SM one, of 16 (a region of 26 x 26, 2.6
  // times the arithmetic) on smaller images
  const int t32 = (c->n + 31) / 32, t16 = (c->n + 15) / 16;
  const bool big = t32 * t32 >= c->sms;
  const int tiles = big ? t32 : t16, lw = (big ? 32 : 16) + 2 * kTvK;
  const size_t sm = (size_t)3 * lw * lw * sizeof(float2);
  allow_smem(k_tv_fgp<32>, sm);
  double t = 1.0;
  for (int k = 0; k < iters; k += kTvK) {
    const int count = std::min(kTvK, iters - k);
    TvMomentum mom{};
    for (int u = 0; u < count; ++u) {
      const double tn = 0.5 * (1.0 + std::sqrt(1.0 + 4.0 * t * t));
      mom.c[u] = (float)((t - 1.0) / tn);
      t = tn;
    }
    const LaunchCfg lc{tiles * tiles, 256, sm, s, k > 0 || chained};
    const int last = k + count >= iters ? 1 : 0;
    PURIFY_LAUNCH(c, "tv_fgp", s,
                  (pdl_launch(big ? k_tv_fgp<32> : k_tv_fgp<16>, lc, c->n, tiles, xa, xb, b, set[a], set[a ^ 1], w,
                              count, mom, k == 0 ? 1 : 0, last, sc, lam_host)));
    a ^= 1;
  }
  *p = set[a].p;
  *q = set[a].q;
  return check_cuda(cudaGetLastError());
}

int tv_scratch_ready(purify_ctx* c, float2** out) {
  if (!c->d_tv) {
    const int64_t N = ((int64_t)c->n * c->n);
    if (cudaMalloc(&c->d_tv, 9 * N * sizeof(float2)) != cudaSuccess) {
      c->d_tv = nullptr;
      cudaGetLastError();
      return PURIFY_E_ALLOC;
    }
  }
  *out = c->d_tv;
  return PURIFY_OK;
}

// SDMM branch i = 1 for the TV prior: r1 = prox_{gamma f1}(x_hat + z1),
// z1 <- z1 + x_hat - r1, x1 = r1 - z1, and f1, zeta.
int tv_sdmm_branch(purify_ctx* c, purify_sdmm_state* st, cudaStream_t s) {
  const int64_t N = ((int64_t)c->n * c->n);
  float2* sc_buf = nullptr;
  TV_TRY(tv_scratch_ready(c, &sc_buf));
  float2 *p, *q;
  TV_TRY(tv_fgp(c, sc_buf, st->xhat, st->z1, st->w, st->fgp_iters, c->d_sc, 0.f, false, &p, &q, s));
  PURIFY_LAUNCH(c, "tv_finish", s,
                (pdl_launch(k_tv_finish, LaunchCfg{tv_blocks(N), 256, 0, s}, c->n, sc_buf, p, q, st->x1, st->z1,
                            st->xhat, st->w, c->d_partials, c->d_sc, 0.f)));
  return check_cuda(cudaGetLastError());
}

// |grad x| into the TV scratch (complex), for gamma and reweighting.
int tv_gradmag(purify_ctx* c, const float2* x, float2** g, cudaStream_t s) {
  float2* sc_buf = nullptr;
  TV_TRY(tv_scratch_ready(c, &sc_buf));
  PURIFY_LAUNCH(c, "tv_gradmag", s, (pdl_launch(k_tv_gradmag, LaunchCfg{tv_blocks(((int64_t)c->n * c->n)), 256, 0,
      s}, c->n, x, sc_buf)));
  *g = sc_buf;
  return check_cuda(cudaGetLastError());
}

// Standalone prox of lam ||W grad .||_1.
int tv_prox(purify_ctx* c, const float2* in, const float* w, float lam, int iters, float2* out, cudaStream_t s) {
  const int64_t N = ((int64_t)c->n * c->n);
  float2* sc_buf = nullptr;
  TV_TRY(tv_scratch_ready(c, &sc_buf));
  float2 *p, *q;
  TV_TRY(tv_fgp(c, sc_buf, in, nullptr, w, iters, nullptr, lam, true, &p, &q, s));
  PURIFY_LAUNCH(c, "tv_finish", s,
                (pdl_launch(k_tv_finish, LaunchCfg{tv_blocks(N), 256, 0, s}, c->n, sc_buf, p, q, out, nullptr, nullptr,
                            nullptr, nullptr, nullptr, lam)));
  return check_cuda(cudaGetLastError());
}

}  // namespace purify
