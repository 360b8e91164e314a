// fbs_kernels.cu -- CUDA kernels of one Gibbs sweep (Algorithm 1 of Landau &
// Niemi, arXiv 1606.06659) for sm_103a, plus initialisation and trace kernels.
//
// A sweep is three launches:
//   eps kernel    one thread per eps_gn: its slice update (Algorithm 1 step 1);
//   gb kernel     one thread per gene g: the conjugate gamma_g draw (step 2), slice
//                 updates of beta_g1..beta_gL in order (step 5), and the per-block
//                 FP64 partial sums that feed steps 3, 4, 6, 7;
//                 both with width tuning (Algorithm 2 step 7) and Welford moments
//                 (Section 3.1);
//   hyper kernel  one block: fixed-order reduction of the partials beside all that
//                 needs no sums, then nu (slice, step 3) and tau (step 4) on warp 0
//                 while warp 1 draws theta_l (step 6) and sigma_l^2 (step 7) on
//                 lane l (fbs_hyper.cuh).
// Drawing beta before nu and tau is exact: the beta_gl conditional involves
// neither, and theirs involve no beta (Figure 3); the counter-based generator
// gives every variable the same uniforms in either order.
// With ModelConst::all_slice the gamma_g draw (gb kernel), tau (warp 0 of the
// hyper kernel, after nu) and sigma_l (a warp each) are slice updates of the same
// full conditionals instead, each variable with its own tuned width, as
// Section 4.2 slice-samples every non-normal conditional.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fbs_common.cuh"
#include "fbs_kernels.h"
#include "fbs_rng.cuh"
#include "fbs_hyper.cuh"

namespace fbs {

namespace cg = cooperative_groups;

// ---------------------------------------------------------------- densities

// log f(eps_gn = x | ...) = y x - exp(A + x) - x^2 hg, with A = h_n + X_n beta_g and
// hg = 1/(2 gamma_g).  aux = exp(A + x), the Poisson mean at x.
struct EpsDensity {
  int32_t y;
  double A, hg;
  __device__ __forceinline__ double operator()(double x, double* aux) const {
    const double e = exp(A + x);
    *aux = e;
    return (double)y * x - e - x * x * hg;
  }
};

// log f(beta_gl = b | ...) = b T_gl - sum_j Q_j exp(v_j (b - b0)) - (b - theta_l)^2 hs,
// where Q_j sums exp(h_n + eps_gn + X_n beta_g) (current beta, beta_gl = b0) over
// the samples n whose X_nl equals the j-th distinct non-zero value v_j of
// column l.  Samples with X_nl = 0 only add a constant.  hs = 1/(2 sigma_l^2).  The
// class count NC is fixed at compile time (NC = kMaxCls keeps the runtime bound
// `ncls`).
template <int NC>
struct BetaDensityT {
  double T, b0, theta, hs;
  int ncls;
  double Q[NC];
  double v[NC];
  int8_t kind[NC];
  __device__ __forceinline__ double operator()(double b, double* aux) const {
    const double dlt = b - b0;
    const double z = exp(dlt);
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      if (NC < kMaxCls || j < ncls) {
        double e;
        if (kind[j] == kClsPlus) e = z;
        else if (kind[j] == kClsMinus) e = 1.0 / z;
        else e = exp(v[j] * dlt);
        s += Q[j] * e;
      }
    }
    *aux = z;
    const double dv = b - theta;
    return b * T - s - dv * dv * hs;
  }
};

// FP32 filters of the FP64 slice updates (slice_update_filtered).  Each returns
// Delta = log f(x0 + d) - log f(x0) in the relative form of the FP32 sweep, which
// needs no evaluation at x0, and a bound on |Delta32 - Delta| + |the FP64
// evaluation's error|, with e = 2^-24 the FP32 unit roundoff:
//   - 2^-20 (16 e) times the magnitudes of the terms.  A term is a product of at
//     most six rounded factors, the series for e^z - 1 - z below |z| = 1/2 is within
//     8 e of itself, and the terms are added with two more roundings;
//   - the FP32 inputs' roundings times the sensitivities of Delta to them, where
//     these are not multiples of a term, with twice to four times the roundoff;
//   - for |z| >= 1/2, where e^z - 1 - z is a difference of rounded numbers (expf is
//     within 4 e of itself), 2^-21 (8 e) times their magnitudes;
//   - derr, the error of d, times 5/4 of a bound on |Delta'| there (a derr that
//     could change the exponential by more than a tenth is refused: infinite
//     bound, the comparison is made in FP64);
//   - 2^-46 (64 times the FP64 unit roundoff) times the magnitudes of the terms of
//     log f(p), log f(x0) and the level.
// What matters is that no part grows with the counts alone: near the decision the
// terms are of order one whatever the count, while a bound of a fixed fraction of
// the rate sent every evaluation of a gene with 10^5 counts to FP64 (0.35% of all
// at N=16 G=40000, most warps had some).

// eps: Delta = d (y - mu0) - mu0 (e^d - 1 - d) - d (d + 2 x0) hg.  mu0 carries the
// rounding of the log-rate at x0 (|log-rate| e) and of expf: amag = |log-rate| + 8.
struct EpsFilter {
  float y, mu0, x0f, hg, amag, c64;  // c64: log f(x0) magnitude
  __device__ __forceinline__ float operator()(float d, float derr, float* eb) const {
    const float ad = fabsf(d), ax = fabsf(x0f);
    const float e = em1mx(d);
    const float ed1 = d + e;             // e^d - 1
    const float mued = mu0 + mu0 * ed1;  // mu0 e^d, the rate at the point
    const float t1 = d * (y - mu0);
    const float t2 = mu0 * e;
    const float t3 = d * (d + 2.0f * x0f) * hg;
    const float b20 = fabsf(t1) + fabsf(t2) + ad * (ad + 2.0f * ax) * hg;
    const float b22 = ad * y + amag * mu0 * fabsf(ed1);
    const float slope = y + mued + 2.0f * (ad + ax) * hg;
    const float px = ax + ad;
    const float b64 = c64 + y * px + mued * (amag + ad) + px * px * hg;
    float b = 0x1p-20f * b20 + 0x1p-22f * b22 + 1.25f * derr * slope + 0x1p-46f * b64;
    if (ad >= 0.5f) b += 0x1p-21f * mu0 * (2.0f + fabsf(ed1) + ad);
    *eb = derr < 0.1f ? b : INFINITY;
    return t1 - t2 - t3;
  }
};

// beta_gl: Delta = d D - sum_j Q_j (e^{z_j} - 1 - z_j) - d (d + 2 (b0 - theta)) hs with
// z_j = v_j d and D = T - sum_j v_j Q_j, taken in FP64 before the loop.
template <int NC>
struct BetaFilterT {
  float D, bt, hs, b0f, Tm, c64;  // bt = b0 - theta; Tm >= |T|; c64: log f(b0) magnitude
  int ncls;
  float Q[NC], v[NC];
  __device__ __forceinline__ float operator()(float d, float derr, float* eb) const {
    const float ad = fabsf(d), abt = fabsf(bt);
    float s = 0.0f, sz = 0.0f, sl = 0.0f, se = 0.0f, sx = 0.0f, big = 0.0f;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      if (NC < kMaxCls || j < ncls) {
        const float z = v[j] * d, az = fabsf(z), av = fabsf(v[j]);
        const float em = em1mx(z);
        const float ej1 = fabsf(z + em);  // |e^z - 1|
        const float vd = av * derr;
        s += Q[j] * em;
        sz += Q[j] * ej1 * az;
        sl += Q[j] * av * (ej1 + 2.0f * vd * (1.0f + ej1));
        se += Q[j] * (2.0f + ej1);
        if (az >= 0.5f) sx += Q[j] * (2.0f + ej1 + az);
        big = fmaxf(big, vd);
      }
    }
    const float t1 = d * D;
    const float t3 = d * (d + 2.0f * bt) * hs;
    const float b20 = fabsf(t1) + s + ad * (ad + 2.0f * abt) * hs;
    const float slope = fabsf(D) + sl + 2.0f * (ad + abt) * hs;
    const float pb = fabsf(b0f) + ad, pt = abt + ad;
    const float b64 = c64 + pb * Tm + se + pt * pt * hs;
    const float b = 0x1p-20f * b20 + 0x1p-21f * (sz + sx) + 1.25f * derr * slope + 0x1p-46f * b64;
    *eb = big < 0.1f ? b : INFINITY;
    return t1 - s - t3;
  }
};

// log f(gamma_g = x | ...) = -shape1 log x - B / x on x > 0, with shape1 = (N + nu)/2 + 1
// and B = (sum_n eps_gn^2 + nu tau)/2: the Inverse-Gamma full conditional of step 2,
// slice-sampled in the all-slice variant (Section 4.2).
struct GamDensity {
  double shape1, B;
  __device__ __forceinline__ double operator()(double x, double* aux) const {
    *aux = 0.0;
    if (!(x > 0.0)) return -INFINITY;
    return -shape1 * log(x) - B / x;
  }
};

// gamma_g: Delta = -s1 log(1 + r) + bx r / (1 + r) with r = d / x0 and bx = B / x0; a
// point below zero (1 + r below zero by more than its error) is never inside the
// slice, and one within a few errors of zero is left to FP64.
struct GamFilter {
  float s1, bx, ix, c64;  // ix = 1 / x0
  __device__ __forceinline__ float operator()(float d, float derr, float* eb) const {
    const float r = d * ix, q = 1.0f + r;
    const float dr = fmaf(0x1p-22f, 1.0f + fabsf(r), derr * ix);  // error of r and of q
    if (q < -2.0f * dr) {
      *eb = 0.0f;
      return -INFINITY;
    }
    const float iq = 1.0f / q;
    const float lr = log1pf(r);
    const float t1 = s1 * lr, t2 = bx * (r * iq);
    const float slope = (s1 + bx * iq) * iq;
    const float b = 0x1p-20f * (fabsf(t1) + fabsf(t2)) + 1.5f * dr * slope +
                    0x1p-46f * (c64 + fabsf(t1) + bx * iq);
    *eb = dr < 0.1f * q ? b : INFINITY;
    return t2 - t1;
  }
};

// ---------------------------------------------------------------- block reduction

template <int NV>
__device__ __forceinline__ void block_sum_to(double (&v)[NV], double* out, double* smem) {
  // warp-shuffle tree, then one value per warp through shared memory
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    double x = v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) smem[warp * NV + i] = x;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
    for (int w = 0; w < nwarp; ++w) s += smem[w * NV + threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// ---------------------------------------------------------------- sweep kernels (FP64)
//
// Step 1 and steps 2 and 5 are two launches, so that every SM gets work at any G
// and the hyperparameter kernel of sweep m can run concurrently with the eps
// kernel of sweep m+1 (the eps conditionals involve no hyperparameter).
// fbs_sweep_noalloc, which has no room for the rates between the two, runs the
// same device functions in one kernel (k_sweep_f64).

__device__ __forceinline__ void add_counters_u(unsigned long long* base, unsigned evals_e,
                                               unsigned evals_b, unsigned caps, unsigned gcaps,
                                               unsigned nonfin, unsigned* flags,
                                               unsigned evals_g = 0) {
  unsigned v[6] = {evals_e, evals_b, caps, gcaps, nonfin, evals_g};
#pragma unroll
  for (int i = 0; i < 6; ++i) v[i] = __reduce_add_sync(0xffffffffu, v[i]);  // warp sum
  if ((threadIdx.x & 31) == 0) {
    if (v[0]) atomicAdd(&base[FBS_CNT_EVALS_EPS], (unsigned long long)v[0]);
    if (v[1]) atomicAdd(&base[FBS_CNT_EVALS_BETA], (unsigned long long)v[1]);
    if (v[2]) atomicAdd(&base[FBS_CNT_SLICE_CAPS], (unsigned long long)v[2]);
    if (v[3]) atomicAdd(&base[FBS_CNT_GAMMA_CAPS], (unsigned long long)v[3]);
    if (v[4]) {
      atomicAdd(&base[FBS_CNT_NONFINITE], (unsigned long long)v[4]);
      atomicOr(flags, kFlagNonfinite);
    }
    if (v[5]) atomicAdd(&base[FBS_CNT_EVALS_GAMMA], (unsigned long long)v[5]);
  }
}

// The FP64 comparisons throughout, for starts that the FP32 filter does not cover
// (out of line: rare, and its exponentials would double the kernels' code).
template <class F>
static __device__ __noinline__ SliceResult slice_update_ol(double x0, double w, const F& f, Rng& r,
                                                           int K, int shrink_max) {
  return slice_update(x0, w, f, r, K, shrink_max);
}

// Whether FP32 holds a slice width with room for its multiples.
__device__ __forceinline__ bool width_fits(double w) {
  const float wf = (float)w;
  return wf > 1e-30f && wf < 1e30f;
}

// The iteration a launch runs and the weight 1/k of its draw in the running
// moments (0: none), from the segment snapshot.
__device__ __forceinline__ double eps_moment_weight(const Hyper* hy, long long it) {
  long long before = (it - 1) - (hy->seg_it > hy->burnin ? hy->seg_it : hy->burnin);
  if (before < 0) before = 0;
  return 1.0 / (double)(hy->seg_nmom + before + 1);
}

// s + x^2 with one rounding, or (kRounded) with that of x^2 too.  The sweep on
// caller-owned arrays rounds the squares of the eps and the other forms do not, each
// as it always has: which of them the compiler fuses must not change with the code
// around them.
template <bool kRounded>
__device__ __forceinline__ double add_square(double s, double x) {
  return kRounded ? __dadd_rn(__dmul_rn(x, x), s) : __fma_rn(x, x, s);
}

// Step 1 for one eps_gn: the update, the width, the moments and the rate at the
// new value (returned in aux).  hg = 1/(2 gamma_g) and inv_k (the weight of the
// draw in the moments) are the same for many elements and come from the caller.
template <bool kRounded = false>
__device__ __forceinline__ SliceResult eps_update_f64(const ModelConst& mc, const DevPtrs& p, int n,
                                                      int g, double hg, float hgf, long long it,
                                                      double inv_k) {
  const int G = mc.G, N = mc.N, L = mc.L;
  const long long burnin = p.hyp->burnin, tune_start = p.hyp->tune_start;
  const size_t e = (size_t)n * G + g;
  double A = mc.h[n];
#pragma unroll
  for (int l = 0; l < kMaxL; ++l)
    if (l < L) A += mc.X[n * kMaxL + l] * p.beta[(size_t)l * G + g];
  EpsDensity f{p.y[e], A, hg};
  Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamEps, (uint32_t)((size_t)g * N + n), (uint32_t)it);
  const double x0 = p.eps[e];
  double w = p.w_eps[e];
  // comparisons decided in FP32 where an error bound allows (the same result);
  // a start whose rate does not fit FP32 takes the FP64 comparisons throughout
  const float af = (float)(A + x0), yf = (float)f.y, x0f = (float)x0;
  const float mu0f = expf(af);
  SliceResult s;
  if (isfinite(mu0f) && isfinite(hgf) && isfinite(x0f) && af < 80.0f && width_fits(w)) {
    const float amag = fabsf(af) + 8.0f;
    EpsFilter ff{yf, mu0f, x0f, hgf, amag, yf * fabsf(x0f) + mu0f * amag + x0f * x0f * hgf + 64.0f};
    s = slice_update_filtered(x0, w, f, ff, r, mc.K, mc.shrink_max);
    s.aux = exp(A + s.x);  // the rate at the result, as the density computes it
  } else {
    s = slice_update_ol(x0, w, f, r, mc.K, mc.shrink_max);
  }
  p.eps[e] = s.x;
  if (it <= burnin) {
    double waux = p.waux_eps[e];
    tune_width(w, waux, it, s.x, x0, burnin, tune_start);
    p.w_eps[e] = w;
    p.waux_eps[e] = waux;
  } else if (mc.moments_eps) {
    const double m = p.m_eps[e], q = p.q_eps[e];
    p.m_eps[e] = m + (s.x - m) * inv_k;
    p.q_eps[e] = q + add_square<kRounded>(-q, s.x) * inv_k;
  }
  return s;
}

// Step 1: one thread per eps_gn, a block 32 genes and blockDim.x / 32 samples (one
// warp each), so that 1/(2 gamma_g) and the moments' weight, an FP64 division of a
// dozen instructions each, are taken once per block instead of by every warp.
// Bound by the FP64 pipe (16 cycles per warp instruction; 78% busy).  N=16 G=40000
// L=5: 88 us; 258 us with the offsets taken in FP64 per evaluation, bounds that
// grow with the counts, the divisions per thread and the level's density and log
// in every update.
__global__ void __launch_bounds__(256, 3) k_eps_f64(ModelConst mc, DevPtrs p, int seg_i) {
  __shared__ double s_hg[32], s_inv_k;
  __shared__ float s_hgf[32];
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i);
  const Hyper* hy = p.hyp;
  const long long it = hy->seg_it + seg_i + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rows = blockDim.x >> 5;
  const int n = blockIdx.y * rows + warp;
  const int g = blockIdx.x * 32 + lane;
  if (warp == 0) {
    const double hg = g < mc.G ? 0.5 / p.gam[g] : 0.0;
    s_hg[lane] = hg;
    s_hgf[lane] = (float)hg;
  }
  if (warp == rows - 1 && lane == 0) s_inv_k = it > hy->burnin ? eps_moment_weight(hy, it) : 0.0;
  __syncthreads();
  unsigned evals = 0, caps = 0, nonfin = 0;
  if (g < mc.G && n < mc.N) {
    const SliceResult s = eps_update_f64(mc, p, n, g, s_hg[lane], s_hgf[lane], it, s_inv_k);
    evals = s.evals;
    caps = s.capped;
    nonfin = s.nonfinite;
    p.mu[(size_t)n * mc.G + g] = s.aux;
  }
  add_counters_u(p.counters + ((blockIdx.x + blockIdx.y) % kCounterCopies) * FBS_NUM_COUNTERS, evals,
                 0, caps, 0, nonfin, &p.hyp->flags);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i);
}

// What a gamma/beta launch reads and counts, per thread.
struct GbF64 {
  const Hyper* hy;
  long long it, burnin, tune_start, trace_row;
  bool mom, trace_now;
  double inv_k;
  unsigned evals_b, evals_g, caps, gcaps, nonfin;
};

// One slice update of beta_gl (step 5) for a column with NC value classes, with
// the class sums of the rates in shared memory, the moments, trace and partials.
// hs = 1/(2 sigma_l^2).
template <int NC>
__device__ __forceinline__ void beta_column_f64(const ModelConst& mc, const DevPtrs& p, int l,
                                                int g, double* mu, double* bs, double* ps, int B,
                                                int tid, double theta, double hs, GbF64& c) {
  const int G = mc.G, N = mc.N, L = mc.L;
  const size_t e = (size_t)l * G + g;
  BetaDensityT<NC> f;
  f.T = p.T[e];
  const double b_cur = bs[l * B + tid];
  f.b0 = b_cur;
  f.theta = theta;
  f.hs = hs;
  f.ncls = mc.ncls[l];
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    f.Q[j] = 0.0;
    f.v[j] = mc.cval[l][j];
    f.kind[j] = mc.ckind[l][j];
  }
  for (int n = 0; n < N; ++n) {
    const int k = mc.cls[l][n];
    const double m = mu[n * B + tid];
#pragma unroll
    for (int j = 0; j < NC; ++j)
      if (j == k) f.Q[j] += m;
  }
  Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamBeta, (uint32_t)((size_t)g * L + l),
        (uint32_t)c.it);
  const double x0 = b_cur;
  double w = p.w_beta[e];
  // comparisons decided in FP32 where an error bound allows (the same result)
  BetaFilterT<NC> ff;
  ff.b0f = (float)x0;
  ff.bt = (float)(x0 - theta);
  ff.hs = (float)hs;
  ff.ncls = f.ncls;
  float qs = 0.0f, vq = 0.0f;
  double D = f.T;
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    ff.Q[j] = (float)f.Q[j];
    ff.v[j] = mc.cvalf[l][j];
    if (NC < kMaxCls || j < f.ncls) {
      D -= f.v[j] * f.Q[j];
      qs += ff.Q[j];
      vq += fabsf(ff.v[j]) * ff.Q[j];
    }
  }
  ff.D = (float)D;
  ff.Tm = 1.01f * (fabsf(ff.D) + vq);
  ff.c64 = fabsf(ff.b0f) * ff.Tm + qs + ff.bt * ff.bt * ff.hs + 64.0f;
  SliceResult s = isfinite(ff.c64) && isfinite(ff.Tm) && width_fits(w)
                      ? slice_update_filtered(x0, w, f, ff, r, mc.K, mc.shrink_max)
                      : slice_update_ol(x0, w, f, r, mc.K, mc.shrink_max);
  c.evals_b += s.evals;
  c.caps += s.capped;
  c.nonfin += s.nonfinite;
  if (s.x != x0) {
    const double dlt = s.x - x0;
    double ej[NC];
    const double z = exp(dlt);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      ej[j] = 1.0;
      if (NC < kMaxCls || j < f.ncls) {
        if (f.kind[j] == kClsPlus) ej[j] = z;
        else if (f.kind[j] == kClsMinus) ej[j] = 1.0 / z;
        else ej[j] = exp(f.v[j] * dlt);
      }
    }
    for (int n = 0; n < N; ++n) {
      const int k = mc.cls[l][n];
      double fac = 1.0;
#pragma unroll
      for (int j = 0; j < NC; ++j)
        if (j == k) fac = ej[j];
      if (k >= 0) mu[n * B + tid] *= fac;
    }
  }
  bs[l * B + tid] = s.x;
  p.beta[e] = s.x;
  if (c.it <= c.burnin) {
    double waux = p.waux_beta[e];
    tune_width(w, waux, c.it, s.x, x0, c.burnin, c.tune_start);
    p.w_beta[e] = w;
    p.waux_beta[e] = waux;
  }
  if (c.mom) {
    const double m = p.m_beta[e], q = p.q_beta[e];
    p.m_beta[e] = m + (s.x - m) * c.inv_k;
    p.q_beta[e] = q + (s.x * s.x - q) * c.inv_k;
  }
  if (c.trace_now) p.trace_beta[(size_t)c.trace_row * L * G + e] = s.x;
  const double dv = s.x - theta;
  ps[(2 + l) * B + tid] = dv;
  ps[(2 + kMaxL + l) * B + tid] = dv * dv;
}

// Columns of three and more classes, out of line: their register needs (up to
// eight class sums in FP64) would otherwise be the kernel's.
template <int NC>
static __device__ __noinline__ void beta_column_f64_ol(const ModelConst& mc, const DevPtrs& p, int l,
                                                       int g, double* mu, double* bs, double* ps,
                                                       int B, int tid, double theta, double hs,
                                                       GbF64& c) {
  beta_column_f64<NC>(mc, p, l, g, mu, bs, ps, B, tid, theta, hs, c);
}

// The values that are the same for every gene of a launch: lane l < L of a warp
// takes 1/(2 sigma_l^2), lane L the moments' weight (one division for all).
struct GbUniform {
  double hs[kMaxL], inv_k;
};

__device__ __forceinline__ void gb_uniform(const ModelConst& mc, const Hyper* hy, bool mom,
                                           int lane, GbUniform* u) {
  if (lane <= mc.L) {
    const double num = lane < mc.L ? 0.5 : 1.0;
    const double den = lane < mc.L ? hy->phi[2 + mc.L + lane] : (double)(hy->n_mom + 1);
    const double q = num / den;
    if (lane < mc.L) u->hs[lane] = q;
    else u->inv_k = mom ? q : 0.0;
  }
}

__device__ __forceinline__ GbF64 gb_begin_f64(const ModelConst& mc, const DevPtrs& p, int seg_i) {
  const Hyper* hy = p.hyp;
  GbF64 c;
  c.hy = hy;
  c.it = hy->seg_it + seg_i + 1;
  c.burnin = hy->burnin;
  c.tune_start = hy->tune_start;
  c.mom = c.it > c.burnin;
  c.trace_now = c.mom && mc.trace_beta && p.trace_beta != nullptr &&
                ((c.it - c.burnin) % hy->thin == 0) && hy->trace_rows < hy->trace_cap;
  c.trace_row = hy->trace_rows;
  c.inv_k = 0.0;
  c.evals_b = c.evals_g = c.caps = c.gcaps = c.nonfin = 0;
  return c;
}

// Step 2 for gene g (column tid of the B genes of ps [kNumPart][B], the terms of
// the sums for steps 3, 4, 6, 7): the gamma_g draw and its moments.  It and the beta
// updates need the sweep's eps and the hyperparameters but not each other, so they
// may run on different warps.
template <bool kRounded = false>
__device__ __forceinline__ void gb_gamma_f64(const ModelConst& mc, const DevPtrs& p, int g, int B,
                                             int tid, double* ps, GbF64& c) {
  const int G = mc.G, N = mc.N;
  const Hyper* hy = c.hy;
  const double nu = hy->phi[0], tau = hy->phi[1];
  double ss = 0.0;
#pragma unroll 8
  for (int n = 0; n < N; ++n) {
    ss = add_square<kRounded>(ss, p.eps[(size_t)n * G + g]);
  }
  // ---- step 2: gamma_g ~ IG((N + nu)/2, (sum eps^2 + nu tau)/2), exactly or
  // (all_slice) by a slice update of that density with the gene's own width
  {
    Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamGamma, (uint32_t)g, (uint32_t)c.it);
    const double shape = 0.5 * ((double)N + nu);
    const double scale = 0.5 * (ss + nu * tau);
    double gam;
    if (mc.all_slice) {
      const double x0 = p.gam[g];
      double w = p.w_gam[g], waux = p.waux_gam[g];
      const GamDensity f{shape + 1.0, scale};
      GamFilter ff;
      const float x0f = (float)x0;
      ff.s1 = (float)f.shape1;
      ff.ix = 1.0f / x0f;
      ff.bx = (float)scale * ff.ix;
      ff.c64 = ff.s1 * (fabsf(__logf(x0f)) + 1.0f) + ff.bx + 64.0f;
      const bool filt = x0f > 1e-30f && ff.ix > 0.0f && isfinite(ff.c64) && width_fits(w);
      SliceResult s = filt ? slice_update_filtered(x0, w, f, ff, r, mc.K, mc.shrink_max)
                           : slice_update_ol(x0, w, f, r, mc.K, mc.shrink_max);
      c.evals_g += s.evals;
      c.caps += s.capped;
      c.nonfin += s.nonfinite;
      gam = s.x;
      if (c.it <= c.burnin) {
        tune_width(w, waux, c.it, s.x, x0, c.burnin, c.tune_start);
        p.w_gam[g] = w;
        p.waux_gam[g] = waux;
      }
    } else {
      bool gcap = false;
      gam = scale / gamma_mt(shape, r, 0, &gcap);
      c.gcaps += gcap;
    }
    p.gam[g] = gam;
    if (c.mom) {
      const double m = p.m_gam[g], q = p.q_gam[g];
      p.m_gam[g] = m + (gam - m) * c.inv_k;
      p.q_gam[g] = q + (gam * gam - q) * c.inv_k;
    }
    ps[0 * B + tid] = log(gam);
    ps[1 * B + tid] = 1.0 / gam;
  }
}

// Step 5 for gene g, whose rates mu [N][B] are in shared memory: the beta_gl, l =
// 1..L in order, with their moments, trace and terms of the sums.
__device__ __forceinline__ void gb_beta_f64(const ModelConst& mc, const DevPtrs& p, int g, int B,
                                            int tid, double* mu, double* bs, double* ps,
                                            const GbUniform& u, GbF64& c) {
  const int G = mc.G, L = mc.L;
  for (int l = 0; l < L; ++l) bs[l * B + tid] = p.beta[(size_t)l * G + g];
  for (int l = 0; l < L; ++l) {
    const double theta = c.hy->phi[2 + l], hs = u.hs[l];
    switch (mc.ncls[l]) {
      case 1: beta_column_f64<1>(mc, p, l, g, mu, bs, ps, B, tid, theta, hs, c); break;
      case 2: beta_column_f64<2>(mc, p, l, g, mu, bs, ps, B, tid, theta, hs, c); break;
      case 3: beta_column_f64_ol<3>(mc, p, l, g, mu, bs, ps, B, tid, theta, hs, c); break;
      default: beta_column_f64_ol<kMaxCls>(mc, p, l, g, mu, bs, ps, B, tid, theta, hs, c);
    }
  }
  // contrast probabilities (§3.1): count the iterations whose beta_g satisfies
  // each proposition
  if (c.mom && p.con != nullptr) {
    const Contrasts* cs = p.con;
    for (int q = 0; q < cs->n; ++q) {
      bool ok = true;
      for (int k = 0; k < cs->terms[q] && ok; ++k) {
        double sv = 0.0;
        for (int l = 0; l < L; ++l) sv = __dadd_rn(sv, __dmul_rn(cs->v[q][k][l], bs[l * B + tid]));
        ok = sv > cs->b[q][k];
      }
      if (ok) p.con_count[(size_t)q * G + g] += 1u;
    }
  }
}

// The sum over a warp's 32 genes of every row of ps, on lane 0.
template <class Store>
__device__ __forceinline__ void warp_sums(const double* ps, int lane, Store store) {
#pragma unroll
  for (int i = 0; i < kNumPart; ++i) {
    double x = ps[i * 32 + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) store(i, x);
  }
}

// Steps 2 and 5: one thread per gene, after the eps kernel of this sweep and the
// hyperparameter kernel of the previous one.  At most 168 registers, so that all
// 1250 one-warp blocks of G=40000 are resident at once (at 248 eight fit an SM,
// 1216 in all, and 34 ran alone).  N=16 G=40000 L=5: 92 us; 301 us before the filter's
// bounds were freed of the counts and the level taken only when needed.
__global__ void __launch_bounds__(128, 3) k_gb_f64(ModelConst mc, DevPtrs p, int seg_i) {
  // shared: mu[N][B], beta[L][B], partials[kNumPart][B] (values indexed by a runtime
  // l live here rather than in local memory), then the reduction scratch
  extern __shared__ double smem_dyn[];
  __shared__ GbUniform u;
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i + 1);
  const int G = mc.G, N = mc.N;
  GbF64 c = gb_begin_f64(mc, p, seg_i);
  const int B = blockDim.x;
  double* mu = smem_dyn;
  double* bs = mu + (size_t)N * B;
  double* ps = bs + (size_t)kMaxL * B;
  const int tid = threadIdx.x;
  const int g = blockIdx.x * B + tid;
  const bool active = g < G;
  if (active) {
#pragma unroll 8
    for (int n = 0; n < N; ++n) mu[n * B + tid] = p.mu[(size_t)n * G + g];
  }
#pragma unroll
  for (int i = 0; i < kNumPart; ++i) ps[i * B + tid] = 0.0;
  if (tid < 32) gb_uniform(mc, c.hy, c.mom, tid, &u);
  __syncthreads();
  c.inv_k = u.inv_k;
  if (active) {
    gb_gamma_f64(mc, p, g, B, tid, ps, c);
    gb_beta_f64(mc, p, g, B, tid, mu, bs, ps, u, c);
  }

  double part[kNumPart];
#pragma unroll
  for (int i = 0; i < kNumPart; ++i) part[i] = ps[i * B + tid];
  double* red = ps + (size_t)kNumPart * B;
  block_sum_to<kNumPart>(part, p.partial + (size_t)blockIdx.x * kNumPart, red);
  add_counters_u(p.counters, 0, c.evals_b, c.caps, c.gcaps, c.nonfin, &p.hyp->flags, c.evals_g);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i + 1);
}

// k_gb_f64 for blocks of 32 genes with the beta updates on one warp and the gamma
// draws on another, for datasets whose blocks leave parts of the SMs idle: a
// warp's FP64 instructions take 64 cycles each, on its quarter of the SM alone, so
// the kernel lasts as long as its longest warp.  N=4 G=1000 L=2: 33.4 -> 22.6 us; N=16
// L=5: 58.6 -> 49.3 at G=5000, 71.5 -> 69.6 at 29000, where its two warps per block
// still all fit (beyond that the one-warp blocks have twice the genes resident).
constexpr int kSplitBlocks = 6;  // resident blocks per SM

__global__ void __launch_bounds__(64, kSplitBlocks) k_gb_split_f64(ModelConst mc, DevPtrs p,
                                                                  int seg_i) {
  extern __shared__ double smem_dyn[];  // mu[N][32], beta[kMaxL][32], partials[kNumPart][32]
  __shared__ GbUniform u;
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i + 1);
  const int G = mc.G, N = mc.N;
  GbF64 c = gb_begin_f64(mc, p, seg_i);
  double* mu = smem_dyn;
  double* bs = mu + (size_t)N * 32;
  double* ps = bs + (size_t)kMaxL * 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = blockIdx.x * 32 + lane;
  if (warp == 0) {
    if (g < G) {
#pragma unroll 8
      for (int n = 0; n < N; ++n) mu[n * 32 + lane] = p.mu[(size_t)n * G + g];
    }
#pragma unroll
    for (int i = 0; i < kNumPart; ++i) ps[i * 32 + lane] = 0.0;
  } else {
    gb_uniform(mc, c.hy, c.mom, lane, &u);
  }
  __syncthreads();
  c.inv_k = u.inv_k;
  if (g < G) {
    if (warp == 0) gb_beta_f64(mc, p, g, 32, lane, mu, bs, ps, u, c);
    else gb_gamma_f64(mc, p, g, 32, lane, ps, c);
  }
  __syncthreads();
  if (warp == 0)
    warp_sums(ps, lane,
              [&](int i, double x) { p.partial[(size_t)blockIdx.x * kNumPart + i] = 0.0 + x; });
  add_counters_u(p.counters, 0, c.evals_b, c.caps, c.gcaps, c.nonfin, &p.hyp->flags, c.evals_g);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i + 1);
}

// Steps 1, 2 and 5 in one launch for fbs_sweep_noalloc: a block takes 32 genes, its
// four warps the samples' eps updates in turn with the rates kept in shared
// memory, then the first warp the genes' beta updates beside the second's gamma
// draws.  The four blocks
// of a cluster are the 128 genes of one row of partial sums (what the fixed
// scratch has rows for) and add their sums in order through distributed shared
// memory.  32 genes per block, not 128: N=16 G=20011 is 626 blocks for 152 SMs
// instead of 157, and a few blocks share an SM, so that the one's serial gene
// phase runs beside the other's eps phase.  Bound by the FP64 pipe.  One sweep of
// N=16 G=20011 L=5: 659 us with one thread per gene making its 16 eps updates in a
// row in FP64, 182 us so.
constexpr int kSweepWarps = 4, kSweepCluster = 4;

__global__ void __cluster_dims__(kSweepCluster, 1, 1) __launch_bounds__(32 * kSweepWarps, 3)
    k_sweep_f64(ModelConst mc, DevPtrs p) {
  extern __shared__ double smem_dyn[];  // mu[N][32], beta[kMaxL][32], partials[kNumPart][32]
  __shared__ GbUniform u;
  __shared__ double s_hg[32], s_inv_k, s_sum[kNumPart];
  __shared__ float s_hgf[32];
  const int G = mc.G, N = mc.N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = blockIdx.x * 32 + lane;
  double* mu = smem_dyn;
  double* bs = mu + (size_t)N * 32;
  double* ps = bs + (size_t)kMaxL * 32;
  GbF64 c = gb_begin_f64(mc, p, 0);
  if (warp == 0) {
    const double hg = g < G ? 0.5 / p.gam[g] : 0.0;
    s_hg[lane] = hg;
    s_hgf[lane] = (float)hg;
  } else if (warp == 1) {
    gb_uniform(mc, c.hy, c.mom, lane, &u);
  } else if (warp == 2) {
    if (lane == 0) s_inv_k = c.mom ? eps_moment_weight(c.hy, c.it) : 0.0;
#pragma unroll
    for (int i = 0; i < kNumPart; ++i) ps[i * 32 + lane] = 0.0;
  }
  __syncthreads();
  unsigned evals_e = 0;
  if (g < G) {
    for (int n = warp; n < N; n += kSweepWarps) {
      const SliceResult s =
          eps_update_f64<true>(mc, p, n, g, s_hg[lane], s_hgf[lane], c.it, s_inv_k);
      evals_e += s.evals;
      c.caps += s.capped;
      c.nonfin += s.nonfinite;
      mu[n * 32 + lane] = s.aux;
    }
  }
  __syncthreads();
  c.inv_k = u.inv_k;
  if (g < G) {
    if (warp == 0) gb_beta_f64(mc, p, g, 32, lane, mu, bs, ps, u, c);
    else if (warp == 1) gb_gamma_f64<true>(mc, p, g, 32, lane, ps, c);
  }
  __syncthreads();
  if (warp == 0) warp_sums(ps, lane, [&](int i, double x) { s_sum[i] = x; });
  add_counters_u(p.counters, evals_e, c.evals_b, c.caps, c.gcaps, c.nonfin, &p.hyp->flags, c.evals_g);
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x < kNumPart) {
    double sum = 0.0;
    for (unsigned r = 0; r < kSweepCluster; ++r) sum += cl.map_shared_rank(s_sum, r)[threadIdx.x];
    p.partial[(size_t)(blockIdx.x / kSweepCluster) * kNumPart + threadIdx.x] = sum;
  }
  cl.sync();  // the other blocks' sums stay until they are read
}

__global__ void __launch_bounds__(kHyperThreads) k_hyper(ModelConst mc, DevPtrs p, int nblk) {
  // the sweep of the segment this launch completes (probe slot only)
  const int slot = p.ktime ? 3 * (int)(p.hyp->it - p.hyp->seg_it) + 2 : 0;
  ktime_begin(p.ktime, p.ktime_n, slot);
  hyper_body<kHyperThreads>(mc, p.partial, p.hyp, p.trace_phi, p.counters, nblk);
  ktime_end(p.ktime, p.ktime_n, slot);
}

// ---------------------------------------------------------------- reading back
//
// These kernels write in the gene-major order [G][R] of the caller's arrays from
// planes [R][G]: thread e takes output e, so a warp's stores are contiguous, and
// the 256 threads of a block read R planes at 256 / R neighbouring genes each,
// whole 32-byte sectors of which stay in L1 for the block.  The transposed
// results then need no pass on the host, which took 1.7 ms for the summaries at
// N=16 G=40000 L=5 and 8.7 ms at N=32 G=200000 (0.36 and 0.55 ms without).

// Index into planes [R][G] of element e of the gene-major order from gene g0 on.
__device__ __forceinline__ long long plane_index(long long e, int R, long long G, long long g0) {
  return (e % R) * G + g0 + e / R;
}

__global__ void __launch_bounds__(256) k_gather(GatherArgs a, double* __restrict__ out) {
  const GatherJob& j = a.job[blockIdx.y];
  const long long n = j.ng * j.R, comp = (long long)j.R * a.G;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = plane_index(e, j.R, a.G, j.g0);
    double v;
    if (j.kind == GatherKind::f64) {
      v = static_cast<const double*>(j.src)[i];
    } else {
      const float* f = static_cast<const float*>(j.src);
      v = (double)f[i];
      if (j.kind == GatherKind::kahan) v -= (double)f[comp + i];
    }
    out[j.off + e] = v;
  }
}

cudaError_t launch_gather(const GatherArgs& a, double* out, cudaStream_t s) {
  long long most = 0;
  for (int i = 0; i < a.n; ++i) {
    const long long n = a.job[i].ng * a.job[i].R;
    if (n > most) most = n;
  }
  if (most == 0) return cudaSuccess;
  const long long blocks = (most + 255) / 256;
  const dim3 grid((unsigned)(blocks < 8 * 152 ? blocks : 8 * 152), (unsigned)a.n);
  k_gather<<<grid, 256, 0, s>>>(a, out);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_mh_stats(const unsigned* __restrict__ acc,
                                                  const unsigned* __restrict__ tried,
                                                  const uint8_t* __restrict__ use, int G,
                                                  unsigned long long* out) {
  unsigned long long v[4] = {0, 0, 0, 0};
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    v[0] += (unsigned long long)acc[g] + acc[(size_t)G + g];
    v[1] += (unsigned long long)tried[g] + tried[(size_t)G + g];
    v[2] += use[g] != 0;
    v[3] += use[g] == kMovePrior;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if ((threadIdx.x & 31) == 0 && v[i]) atomicAdd(out + i, v[i]);
  }
}

cudaError_t launch_mh_stats(const unsigned* acc, const unsigned* tried, const uint8_t* use, int G,
                            unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, 4 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int blocks = (G + 255) / 256;
  k_mh_stats<<<blocks < 152 ? blocks : 152, 256, 0, s>>>(acc, tried, use, G, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- convergence

// Gelman-Rubin potential scale reduction of parameter i (§3.1) from the chains'
// running means and mean squares over M draws each.
__global__ void k_rhat(RhatInput in, double* __restrict__ out) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= in.n) return;
  const long long i = plane_index(e, in.R, in.G, in.g0), comp = in.R * in.G;
  const int C = in.C;
  const double M = (double)in.M;
  double mean[FBS_MAX_RHAT_CHAINS], msq[FBS_MAX_RHAT_CHAINS];
  double tot = 0.0;
  for (int c = 0; c < C; ++c) {
    if (in.f32) {
      const float* b = in.mf[c];
      mean[c] = (double)b[i] - (double)b[comp + i];
      msq[c] = (double)b[2 * comp + i] - (double)b[3 * comp + i];
    } else {
      mean[c] = in.m[c][i];
      msq[c] = in.q[c][i];
    }
    tot += mean[c];
  }
  const double grand = tot / C;
  double bsum = 0.0, wsum = 0.0;
  for (int c = 0; c < C; ++c) {
    const double dm = mean[c] - grand;
    bsum += dm * dm;
    wsum += M / (M - 1.0) * (msq[c] - mean[c] * mean[c]);
  }
  const double B = M / (C - 1) * bsum;
  const double W = wsum / C;
  out[e] = W > 0.0 ? sqrt(1.0 + (B / W - 1.0) / M) : NAN;
}

// Posterior summaries of parameter i (§3.1) from C chains' running means and
// mean squares, pooled over the chains: mean = (1/C) sum_c mean_c, msq = (1/C)
// sum_c msq_c, sd = sqrt(msq - mean^2) (0 where rounding makes it negative), and
// the normal-approximation interval mean -/+ z sd.  out: [4][n] = mean, sd, lo, hi.
__global__ void k_estimates(RhatInput in, double z, double* __restrict__ out) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= in.n) return;
  const long long i = plane_index(e, in.R, in.G, in.g0), comp = in.R * in.G;
  double mean = 0.0, msq = 0.0;
  for (int c = 0; c < in.C; ++c) {
    if (in.f32) {
      const float* b = in.mf[c];
      mean += (double)b[i] - (double)b[comp + i];
      msq += (double)b[2 * comp + i] - (double)b[3 * comp + i];
    } else {
      mean += in.m[c][i];
      msq += in.q[c][i];
    }
  }
  mean /= in.C;
  msq /= in.C;
  const double var = msq - mean * mean;
  const double sd = var > 0.0 ? sqrt(var) : 0.0;
  out[e] = mean;
  out[in.n + e] = sd;
  out[2 * in.n + e] = mean - z * sd;
  out[3 * in.n + e] = mean + z * sd;
}

cudaError_t launch_estimates(const RhatInput& in, double z, double* out, cudaStream_t s) {
  if (in.n <= 0) return cudaSuccess;
  const int blk = 128;
  k_estimates<<<(unsigned)((in.n + blk - 1) / blk), blk, 0, s>>>(in, z, out);
  return cudaGetLastError();
}

cudaError_t launch_rhat(const RhatInput& in, double* out, cudaStream_t s) {
  if (in.n <= 0) return cudaSuccess;
  const int blk = 128;
  k_rhat<<<(unsigned)((in.n + blk - 1) / blk), blk, 0, s>>>(in, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- set-up kernels

__global__ void k_set_run(Hyper* hy, long long burnin, long long tune_start, long long thin) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    hy->burnin = burnin;
    hy->tune_start = tune_start;
    hy->thin = thin;
  }
}

__global__ void k_init_run(Hyper* hy, long long trace_cap) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    hy->burnin = 0;
    hy->tune_start = 0;
    hy->thin = 1;
    hy->trace_cap = trace_cap;
  }
}

// y to [N][G]; T[l][g] = sum_n y X_nl; default beta_g = P (log(y+1) - h); eps = 0;
// gamma = 1; widths w0; tuning sums and moments 0.
__global__ void k_init_genes(ModelConst mc, DevPtrs p, const int32_t* y_in, int gene_major,
                             const double* __restrict__ pinv, double w0, int set_state) {
  const int G = mc.G, N = mc.N, L = mc.L;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    double r[kMaxN];
    double T[kMaxL];
#pragma unroll
    for (int l = 0; l < kMaxL; ++l) T[l] = 0.0;
    for (int n = 0; n < N; ++n) {
      const int32_t yv = gene_major ? y_in[(size_t)g * N + n] : y_in[(size_t)n * G + g];
      const_cast<int32_t*>(p.y)[(size_t)n * G + g] = yv;
      r[n] = log((double)yv + 1.0) - mc.h[n];
#pragma unroll
      for (int l = 0; l < kMaxL; ++l)
        if (l < L) T[l] += (double)yv * mc.X[n * kMaxL + l];
    }
    for (int l = 0; l < L; ++l) {
      const_cast<double*>(p.T)[(size_t)l * G + g] = T[l];
      if (set_state) {
        double s = 0.0;
        for (int n = 0; n < N; ++n) s += pinv[l * kMaxN + n] * r[n];
        p.beta[(size_t)l * G + g] = s;
        p.w_beta[(size_t)l * G + g] = w0;
        p.waux_beta[(size_t)l * G + g] = 0.0;
      }
    }
    if (set_state) {
      for (int n = 0; n < N; ++n) {
        p.eps[(size_t)n * G + g] = 0.0;
        p.w_eps[(size_t)n * G + g] = w0;
        p.waux_eps[(size_t)n * G + g] = 0.0;
      }
      p.gam[g] = 1.0;
      if (p.w_gam) {
        p.w_gam[g] = w0;
        p.waux_gam[g] = 0.0;
      }
    }
  }
}

// Zero the running moments and the chain bookkeeping.
__global__ void k_zero_moments(ModelConst mc, DevPtrs p) {
  const int G = mc.G, N = mc.N, L = mc.L;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    if (p.m_eps)
      for (int n = 0; n < N; ++n) {
        p.m_eps[(size_t)n * G + g] = 0.0;
        p.q_eps[(size_t)n * G + g] = 0.0;
      }
    for (int l = 0; l < L; ++l) {
      p.m_beta[(size_t)l * G + g] = 0.0;
      p.q_beta[(size_t)l * G + g] = 0.0;
    }
    p.m_gam[g] = 0.0;
    p.q_gam[g] = 0.0;
  }
}

// Default hyperparameters from the starting beta: theta_l the mean, sigma_l^2 the
// variance clamped to [1e-6, s_l^2/4] (two passes, one block), nu = min(3, d/2),
// tau = 1.
__global__ void k_init_hyper(ModelConst mc, Hyper* hy, const double* beta_d,
                             const float* beta_f, double w0, int set_state) {
  __shared__ double red[1024 / 32][kMaxL];
  __shared__ double mean_s[kMaxL];
  const int G = mc.G, L = mc.L;
  if (set_state) {
    for (int pass = 0; pass < 2; ++pass) {
      double acc[kMaxL];
#pragma unroll
      for (int l = 0; l < kMaxL; ++l) acc[l] = 0.0;
      for (int g = threadIdx.x; g < G; g += blockDim.x) {
#pragma unroll
        for (int l = 0; l < kMaxL; ++l) {
          if (l < L) {
            const size_t e = (size_t)l * G + g;
            const double b = beta_d ? beta_d[e] : (double)beta_f[e];
            if (pass == 0) acc[l] += b;
            else {
              const double dv = b - mean_s[l];
              acc[l] += dv * dv;
            }
          }
        }
      }
#pragma unroll
      for (int l = 0; l < kMaxL; ++l) {
        double x = acc[l];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][l] = x;
      }
      __syncthreads();
      if (threadIdx.x < L) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
        if (pass == 0) mean_s[threadIdx.x] = s / (double)G;
        else {
          const double var = s / (double)G;
          const double upper = 0.25 * mc.s2[threadIdx.x];
          hy->phi[2 + threadIdx.x] = mean_s[threadIdx.x];
          hy->phi[2 + L + threadIdx.x] = fmin(fmax(var, 1e-6), upper);
        }
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    if (set_state) {
      hy->phi[0] = fmin(3.0, 0.5 * mc.d);
      hy->phi[1] = 1.0;
      hy->w_nu = w0;
      hy->waux_nu = 0.0;
      for (int i = 0; i <= kMaxL; ++i) {
        hy->w_hyp[i] = w0;
        hy->waux_hyp[i] = 0.0;
      }
      hy->it = 0;
    }
    for (int i = 0; i < kMaxP; ++i) {
      hy->m_phi[i] = 0.0;
      hy->q_phi[i] = 0.0;
    }
    hy->n_mom = 0;
    hy->trace_rows = 0;
    hy->flags = 0;
  }
}

// ---------------------------------------------------------------- uniforms

__global__ void k_uniforms(uint32_t seed_lo, uint32_t seed_hi, uint32_t chain, uint32_t stream,
                           uint32_t index0, int n_index, uint32_t iter, uint32_t k0, int n_k,
                           double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_index) return;
  Rng r(seed_lo, seed_hi, chain, stream, index0 + (uint32_t)i, iter);
  for (int k = 0; k < n_k; ++k) out[(size_t)i * n_k + k] = r.u(k0 + (uint32_t)k);
}

// ---------------------------------------------------------------- launchers

cudaError_t launch_sweep_f64(const ModelConst& mc, const DevPtrs& p, cudaStream_t s) {
  const int nblk = (mc.G + 127) / 128 * kSweepCluster;
  const size_t smem = ((size_t)mc.N + kMaxL + kNumPart) * 32 * sizeof(double);
  k_sweep_f64<<<nblk, 32 * kSweepWarps, smem, s>>>(mc, p);
  return cudaGetLastError();
}

cudaError_t launch_hyper(const ModelConst& mc, const DevPtrs& p, int nblk, cudaStream_t s) {
  k_hyper<<<1, kHyperThreads, 0, s>>>(mc, p, nblk);
  return cudaGetLastError();
}

constexpr size_t gb_smem_bytes_f64(int N, int block) {
  return ((size_t)N + kMaxL + kNumPart) * block * sizeof(double) +
         (size_t)(block / 32) * kNumPart * sizeof(double);
}

cudaError_t prepare_gene_kernel() {
  return set_smem_limit(k_gb_f64, gb_smem_bytes_f64(kMaxN, 128));
}

cudaError_t launch_eps_f64(const ModelConst& mc, const DevPtrs& p, int seg_i, cudaStream_t s) {
  // as few idle warps as blocks of up to eight samples leave
  const int groups = (mc.N + 7) / 8, rows = (mc.N + groups - 1) / groups;
  const dim3 grid((unsigned)((mc.G + 31) / 32), (unsigned)groups);
  k_eps_f64<<<grid, 32 * rows, 0, s>>>(mc, p, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_gb_f64(const ModelConst& mc, const DevPtrs& p, int block, int seg_i,
                          cudaStream_t s) {
  const int nblk = (mc.G + block - 1) / block;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // split while all its blocks are resident (both measured at k_gb_split_f64)
  if (block == 32 && nblk <= kSplitBlocks * sms) {
    k_gb_split_f64<<<nblk, 64, gb_smem_bytes_f64(mc.N, 32), s>>>(mc, p, seg_i);
    return cudaGetLastError();
  }
  k_gb_f64<<<nblk, block, gb_smem_bytes_f64(mc.N, block), s>>>(mc, p, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_set_run(Hyper* hy, long long burnin, long long tune_start, long long thin,
                           cudaStream_t s) {
  k_set_run<<<1, 32, 0, s>>>(hy, burnin, tune_start, thin);
  return cudaGetLastError();
}

cudaError_t launch_init(const ModelConst& mc, const DevPtrs& p, const int32_t* y_in,
                        int gene_major, const double* pinv, double w0, int set_state,
                        long long trace_cap, cudaStream_t s) {
  const int blk = 256;
  const int grid = (mc.G + blk - 1) / blk;
  k_init_run<<<1, 32, 0, s>>>(p.hyp, trace_cap);
  k_init_genes<<<grid, blk, 0, s>>>(mc, p, y_in, gene_major, pinv, w0, set_state);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_zero_moments<<<grid, blk, 0, s>>>(mc, p);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_init_hyper<<<1, 1024, 0, s>>>(mc, p.hyp, p.beta, nullptr, w0, set_state);
  return cudaGetLastError();
}

cudaError_t launch_zero_moments(const ModelConst& mc, const DevPtrs& p, cudaStream_t s) {
  const int blk = 256;
  const int grid = (mc.G + blk - 1) / blk;
  k_zero_moments<<<grid, blk, 0, s>>>(mc, p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_init_hyper<<<1, 1024, 0, s>>>(mc, p.hyp, p.beta, nullptr, 0.0, 0);
  return cudaGetLastError();
}

cudaError_t launch_init_hyper(const ModelConst& mc, Hyper* hy, const double* beta_d,
                              const float* beta_f, double w0, int set_state, cudaStream_t s) {
  k_init_hyper<<<1, 1024, 0, s>>>(mc, hy, beta_d, beta_f, w0, set_state);
  return cudaGetLastError();
}

cudaError_t launch_init_run(Hyper* hy, long long trace_cap, cudaStream_t s) {
  k_init_run<<<1, 32, 0, s>>>(hy, trace_cap);
  return cudaGetLastError();
}

cudaError_t launch_uniforms(uint64_t seed, uint32_t chain, uint32_t stream, uint32_t index0,
                            int n_index, uint32_t iter, uint32_t k0, int n_k, double* out,
                            cudaStream_t s) {
  const int blk = 128;
  k_uniforms<<<(n_index + blk - 1) / blk, blk, 0, s>>>((uint32_t)seed, (uint32_t)(seed >> 32),
                                                        chain, stream, index0, n_index, iter, k0,
                                                        n_k, out);
  return cudaGetLastError();
}

}  // namespace fbs
