// fbs_gene_f32.cu -- the per-gene kernel of the Gibbs sweep in its FP32 form
// (Landau & Niemi, arXiv 1606.06659, Algorithm 1 steps 1, 2, 5 with Algorithm
// 2), plus its set-up kernels.
//
// Slice evaluations run in FP32 on the log density relative to the start
// point x0, Delta(x) = log f(x) - log f(x0), written so that no two large terms
// cancel:
//   eps:  Delta(x) = d (y - mu0) - mu0 (e^d - 1 - d) - d (d + 2 x0) / (2 gamma)
//   beta: Delta(b) = sum_j [v_j d (Y_j - Q_j) - Q_j (e^{v_j d} - 1 - v_j d)]
//                    - d (d + 2 (b0 - theta)) / (2 sigma^2)
// with d = x - x0, mu0 = exp(h + x0 + X beta) the Poisson mean at x0, Y_j and
// Q_j the counts and Poisson means summed over the samples whose X_nl is the
// j-th distinct value v_j of column l.  Since Delta(x0) = 0, the slice level is
// log U and no evaluation at x0 is needed.  Uniforms are 23-bit FP32 numbers,
// four per Philox block.  The partial sums for the hyperparameter steps are
// reduced exactly to FP64 (error-free FP32 pair sums within a warp, FP64
// across warps and blocks), and the running moments are Kahan-compensated
// FP32 pairs.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "fbs_common.cuh"
#include "fbs_kernels.h"
#include "fbs_rng.cuh"
#include "fbs_hyper.cuh"
#include "fbs_tc.cuh"

namespace fbs {

// ---------------------------------------------------------------- FP32 random numbers

// The uniforms of one random variable in the FP32 form: uniform k is word k%4 of
// Philox block k/4, as ((w >> 9) + 1/2) / 2^23 (exact in FP32, inside (0,1)).
//
// OL: the Philox rounds as a call.  The gamma/beta kernels draw at a dozen places,
// and with two warps per scheduler they wait for instructions a quarter of the
// time: one copy of the rounds stays in the instruction cache.  The eps kernel,
// which issues in most cycles, has them inline.
static __device__ __noinline__ uint4 philox_ol(uint4 c, uint32_t k0, uint32_t k1) {
  return philox4x32_10(c, k0, k1);
}

template <bool OL>
struct Rng4T {
  uint32_t key0, key1, index, sblk, iter, chain;
  uint32_t cached;
  uint4 w;

  __device__ __forceinline__ Rng4T(uint32_t seed_lo, uint32_t seed_hi, uint32_t chain_,
                                  uint32_t stream, uint32_t index_, uint32_t iter_)
      : key0(seed_lo), key1(seed_hi), index(index_), sblk(stream << 24), iter(iter_),
        chain(chain_), cached(0xFFFFFFFFu), w(make_uint4(0, 0, 0, 0)) {}

  __device__ __forceinline__ float u(uint32_t k) {
    block(k >> 2);
    const uint32_t j = k & 3u;
    const uint32_t x = j == 0 ? w.x : (j == 1 ? w.y : (j == 2 ? w.z : w.w));
    return word(x);
  }

  // The uniform of Philox word x.
  static __device__ __forceinline__ float word(uint32_t x) {
    return __fmul_rn(__fadd_rn(__uint2float_rn(x >> 9), 0.5f), 0x1p-23f);
  }

  // Philox block blk (uniforms 4 blk .. 4 blk + 3), cached.
  __device__ __forceinline__ uint4 block(uint32_t blk) {
    if (blk != cached) {
      const uint4 c = make_uint4(index, sblk | blk, iter, chain);
      w = OL ? philox_ol(c, key0, key1) : philox4x32_10(c, key0, key1);
      cached = blk;
    }
    return w;
  }
};
using Rng4 = Rng4T<false>;
using Rng4OL = Rng4T<true>;

__device__ __forceinline__ float normal_bm_f(float u1, float u2) {
  return sqrtf(-2.0f * __logf(u1)) * __cosf(6.2831853071795865f * u2);
}

// Gamma(shape, 1), Marsaglia & Tsang (2000), uniform layout as in the FP64 form.
template <class R>
__device__ __forceinline__ float gamma_mt_f(float shape, R& r, uint32_t k0, bool* capped) {
  const float alpha = shape < 1.0f ? shape + 1.0f : shape;
  const float dd = alpha - (1.0f / 3.0f);
  const float cc = rsqrtf(9.0f * dd);
  float boost = 1.0f;
  if (shape < 1.0f) boost = __powf(r.u(k0 + 3), 1.0f / shape);
  for (uint32_t j = 0; j < (uint32_t)kGammaAttempts; ++j) {
    const float u1 = r.u(k0 + 4 * j), u2 = r.u(k0 + 4 * j + 1);
    const float x = normal_bm_f(u1, u2);
    float v = 1.0f + cc * x;
    if (v <= 0.0f) continue;
    v = v * v * v;
    const float u = r.u(k0 + 4 * j + 2);
    const float x2 = x * x;
    if (u < 1.0f - 0.0331f * x2 * x2) return dd * v * boost;
    if (__logf(u) < 0.5f * x2 + dd * (1.0f - v + __logf(v))) return dd * v * boost;
  }
  *capped = true;
  return shape;
}

// ---------------------------------------------------------------- densities

struct EpsDensityF {
  float D, mu0, x0, hg;  // D = y - mu0, hg = 1 / (2 gamma)
  __device__ __forceinline__ float operator()(float x, float* aux) const {
    const float d = x - x0;
    const float e = em1mx(d);
    *aux = mu0 + mu0 * (d + e);
    return d * D - mu0 * e - d * (d + 2.0f * x0) * hg;
  }
};

// Relative log density of beta_gl: with d = b - b0 and the column's value
// classes j (value v_j, rate sum Q_j and count sum Y_j at b0, D_j = Y_j - Q_j),
// Delta(b) = sum_j [v_j d D_j - Q_j em1mx(v_j d)] - d (d + 2 (b0 - theta)) / (2 sigma^2).
// The class count NC is fixed at compile time, so that the loops run over the
// classes a column has (NC = kMaxCls keeps the runtime bound `ncls`).
template <int NC>
struct BetaDensityFT {
  float bt, hs, b0;
  int ncls;
  float Q[NC], D[NC], v[NC];
  __device__ __forceinline__ float operator()(float b, float* aux) const {
    const float d = b - b0;
    float s = 0.0f;
    if constexpr (NC <= 3) {
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float z = v[j] * d;
        s += z * D[j] - Q[j] * em1mx(z);
      }
    } else {
      // with many classes the exponentials are worth a branch (N=22 G=9973 with an
      // eight-level covariate: gamma/beta 21.2 -> 19.0 us; with two they are not)
      float e[NC];
      bool big = false;
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        e[j] = em1mx_series(v[j] * d);
        big |= !(fabsf(v[j] * d) < 0.5f);
      }
      if (big) {
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          const float z = v[j] * d, t = em1mx_direct(z);
          e[j] = fabsf(z) < 0.5f ? e[j] : t;
        }
      }
#pragma unroll
      for (int j = 0; j < NC; ++j)
        if (j < ncls) {
          const float z = v[j] * d;
          s += z * D[j] - Q[j] * e[j];
        }
    }
    *aux = d;
    return s - d * (d + 2.0f * bt) * hs;
  }
};

struct SliceResultF {
  float x, aux;
  unsigned evals;
  bool capped, nonfinite;
};

// Algorithm 2, steps 1-6, on Delta (Delta(x0) = 0): level log U_0, interval from
// U_1, K_L from U_2, the j-th shrinkage proposal from U_{3+j}.
template <class F, class R>
__device__ __forceinline__ SliceResultF slice_update_f(float x0, float aux0, float w, const F& f,
                                                       R& r, int K, int shrink_max) {
  SliceResultF res;
  res.evals = 0;
  res.nonfinite = !(isfinite(x0) && isfinite(aux0));
  const float logu = __logf(r.u(0));
  const float v = __fmul_rn(w, r.u(1));
  float lo = __fsub_rn(x0, v);
  float hi = __fadd_rn(lo, w);
  int KL = (int)__fmul_rn((float)(K + 1), r.u(2));
  if (KL > K) KL = K;
  const int KR = K - KL;
  float aux;
  for (int k = 0; k < KL; ++k) {
    ++res.evals;
    if (logu < f(lo, &aux)) lo = __fsub_rn(lo, w); else break;
  }
  for (int k = 0; k < KR; ++k) {
    ++res.evals;
    if (logu < f(hi, &aux)) hi = __fadd_rn(hi, w); else break;
  }
  // shrinkage: proposal j takes uniform 3 + j (word 3 of block 0, then the four
  // words of block 1, 2, ..), so that the word is a compile-time choice
  auto propose = [&](float u) -> bool {
    const float xs = __fadd_rn(lo, __fmul_rn(__fsub_rn(hi, lo), u));
    ++res.evals;
    if (logu < f(xs, &aux)) {
      res.x = xs;
      res.aux = aux;
      res.capped = false;
      return true;
    }
    if (xs > x0) hi = xs; else lo = xs;
    return false;
  };
  if (shrink_max > 0 && propose(Rng4::word(r.block(0u).w))) return res;
  for (int j = 1, b = 1; j < shrink_max; ++b) {
    const uint4 q = r.block((uint32_t)b);
    if (propose(Rng4::word(q.x))) return res;
    if (++j >= shrink_max) break;
    if (propose(Rng4::word(q.y))) return res;
    if (++j >= shrink_max) break;
    if (propose(Rng4::word(q.z))) return res;
    if (++j >= shrink_max) break;
    if (propose(Rng4::word(q.w))) return res;
    ++j;
  }
  res.x = x0;
  res.aux = aux0;
  res.capped = true;
  return res;
}

__device__ __forceinline__ void tune_width_f(float& w, float& waux, long long it, float x_new,
                                             float x_old, long long burnin, long long tune_start) {
  if (it > burnin) return;
  waux += (float)it * fabsf(x_new - x_old);
  if (it > tune_start) {
    const float wn = waux / (0.5f * (float)it * (float)(it + 1));
    if (wn > 0.0f && isfinite(wn)) w = wn;
  }
}

// Welford update of a Kahan-compensated FP32 pair (m, c) representing m - c, of the
// mean and the mean square: the four planes' values v of one element.
struct KahanMoments {
  float v[4];
  __device__ __forceinline__ void load(const float* base, size_t plane, size_t e) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = base[i * plane + e];
  }
  __device__ __forceinline__ void store(float* base, size_t plane, size_t e) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) base[i * plane + e] = v[i];
  }
  __device__ __forceinline__ void update(float x, float inv_k);
};

__device__ __forceinline__ void KahanMoments::update(float x, float inv_k) {
  float &m = v[0], &c = v[1], &q = v[2], &cq = v[3];
  {
    const float inc = (x - (m - c)) * inv_k;
    const float y = inc - c;
    const float t = m + y;
    c = __fsub_rn(__fsub_rn(t, m), y);
    m = t;
  }
  {
    const float inc = (x * x - (q - cq)) * inv_k;
    const float y = inc - cq;
    const float t = q + y;
    cq = __fsub_rn(__fsub_rn(t, q), y);
    q = t;
  }
}

__device__ __forceinline__ void welford_kahan(float* base, size_t plane, size_t e, float x,
                                              float inv_k) {
  KahanMoments m;
  m.load(base, plane, e);
  m.update(x, inv_k);
  m.store(base, plane, e);
}

// Error-free FP32 pair addition (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// ---------------------------------------------------------------- sweep kernels (FP32)


// Warp sums of the counters, one atomic per warp into one of several copies.
__device__ __forceinline__ void add_counters(unsigned long long* base, unsigned evals_e,
                                             unsigned evals_b, unsigned caps, unsigned gcaps,
                                             unsigned nonfin, unsigned* flags) {
  unsigned v[5] = {evals_e, evals_b, caps, gcaps, nonfin};
#pragma unroll
  for (int i = 0; i < 5; ++i) v[i] = __reduce_add_sync(0xffffffffu, v[i]);  // warp sum
  if ((threadIdx.x & 31) == 0) {
    if (v[0]) atomicAdd(&base[FBS_CNT_EVALS_EPS], (unsigned long long)v[0]);
    if (v[1]) atomicAdd(&base[FBS_CNT_EVALS_BETA], (unsigned long long)v[1]);
    if (v[2]) atomicAdd(&base[FBS_CNT_SLICE_CAPS], (unsigned long long)v[2]);
    if (v[3]) atomicAdd(&base[FBS_CNT_GAMMA_CAPS], (unsigned long long)v[3]);
    if (v[4]) {
      atomicAdd(&base[FBS_CNT_NONFINITE], (unsigned long long)v[4]);
      atomicOr(flags, kFlagNonfinite);
    }
  }
}

// Step 1 of Algorithm 1 in the FP32 form: one thread per eps_gn (element e of
// the [N][G] planes).  It reads beta_g and gamma_g of the previous iteration and
// writes the new eps_gn and mu_gn = exp(h_n + eps_gn + X_n beta_g) for the
// gamma/beta kernel.  It involves no hyperparameter, so within a captured
// segment it runs concurrently with the hyperparameter kernel of the previous
// iteration; its iteration number comes from the segment snapshot.
__device__ __forceinline__ void eps_f32_body(const ModelConst& mc, const DevPtrsF32& p, int seg_i,
                                             int n, int g, int copy) {
  const int G = mc.G, N = mc.N, L = mc.L;
  const Hyper* hy = p.hyp;
  const long long it = hy->seg_it + seg_i + 1;
  const long long burnin = hy->burnin, tune_start = hy->tune_start;
  const bool mom = it > burnin;
  long long before = (it - 1) - (hy->seg_it > burnin ? hy->seg_it : burnin);
  if (before < 0) before = 0;
  const float inv_k = mom ? 1.0f / (float)(hy->seg_nmom + before + 1) : 0.0f;
  const size_t NG = (size_t)N * G;
  const size_t e = (size_t)n * G + g;
  unsigned evals = 0, caps = 0, nonfin = 0;
  if (g < G) {
    float A = mc.hf[n];
#pragma unroll
    for (int l = 0; l < kMaxL; ++l)
      if (l < L) A += mc.Xf[n * kMaxL + l] * p.beta[(size_t)l * G + g];
    const float hg = 0.5f / p.gam[g];
    const float x0 = p.eps[e];
    const float mu0 = expf(A + x0);
    EpsDensityF f{(float)p.y[e] - mu0, mu0, x0, hg};
    Rng4 r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamEps, (uint32_t)((size_t)g * N + n),
           (uint32_t)it);
    float w = p.w_eps[e];
    SliceResultF s = slice_update_f(x0, mu0, w, f, r, mc.K, mc.shrink_max);
    evals = s.evals;
    caps = s.capped;
    nonfin = s.nonfinite;
    p.mu[e] = s.aux;
    p.eps[e] = s.x;
    if (it <= burnin) {
      float waux = p.waux_eps[e];
      tune_width_f(w, waux, it, s.x, x0, burnin, tune_start);
      p.w_eps[e] = w;
      p.waux_eps[e] = waux;
    }
    if (mom && mc.moments_eps) welford_kahan(p.mom_eps, NG, e, s.x, inv_k);
  }
  add_counters(p.counters + copy * FBS_NUM_COUNTERS, evals, 0, caps, 0, nonfin, &p.hyp->flags);
}

// At least 5 blocks of 256 per SM (at most 51 registers, no spills): 5 rather
// than 4 resident blocks took the kernel from 24.1 to 22.9 us at N=16 G=40000
// (6 blocks: 23.2 us).
__global__ void __launch_bounds__(256, 5) k_eps_f32(ModelConst mc, DevPtrsF32 p, int seg_i) {
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i);
  eps_f32_body(mc, p, seg_i, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x,
               (blockIdx.x + blockIdx.y) % kCounterCopies);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i);
}

// Which proposal gene g uses at iteration it: 0 none, kMoveNet the network's,
// kMovePrior the prior-centred one.  p.mh_all = 0: the calibrated per-gene
// choice; 1 or 2: that kind for every gene; 3 (calibration): every gene, the
// network on even and the prior on odd iterations.
__device__ __forceinline__ int move_kind(const DevPtrsF32& p, int g, long long it) {
  if (p.mh_all == 3) return (it & 1) ? kMovePrior : kMoveNet;
  if (p.mh_all) return p.mh_all;
  return (int)p.use_mh[g];
}

// The learned-proposal move of gene g (FP32): beta* from the multivariate t
// distribution with kTDof degrees of freedom, centre mu and scale C C^T given by
// the proposal network (beta* = mu + s C xi, s = sqrt(kTDof / chi2)), and
// eps* = eps - X (beta* - beta), so that every log-rate h_n + eps_n + X_n beta is
// unchanged and the Poisson likelihood cancels; accepted with probability
// min(1, pi(eps*, beta*) q(beta) / (pi(eps, beta) q(beta*))), where pi holds the
// Normal(0, gamma) priors of eps and the Normal(theta, sigma^2) priors of beta.
// The proposal depends only on quantities the move leaves unchanged, so this is
// an exact Metropolis-Hastings step; the t tails dominate the target's Gaussian
// tails, which keeps the ratio target / proposal bounded (uniform ergodicity).
// Uniforms 0..2L-1 give the normals, uniform 2L the acceptance and uniforms
// 2L+1..2L+4 the chi-square variate chi2 = -2 log(U1 U2 U3 U4) (kTDof = 8).
// kind kMoveNet takes the centre and scale from the network; kind kMovePrior
// from the hyperparameters alone (centre theta, scale diag(sigma)), which suits
// genes whose conditional is close to the prior (very large gamma_g), where the
// network, trained mostly on typical genes, extrapolates poorly.  Either way
// the proposal depends only on quantities the move keeps.
// The network's outputs are read from prop[k pstride + pidx]; es holds the gene's
// eps ([N][B], changed in place when accepted).  Returns true when accepted.
constexpr int kTDof = 8;
constexpr int kGbBatch = 16;  // samples whose rate, count and eps are in flight at a time

// The hyperparameters of a gamma/beta launch in FP32, once per block: the
// conversions run on the FP64 pipe and every thread used to make them per column.
struct GbHyper {
  float th[kMaxL], s2[kMaxL], hs[kMaxL];  // theta_l, sigma_l^2, 1/(2 sigma_l^2)
  float nu, tau, inv_k;                   // inv_k: weight of the draw in the moments
};

__device__ __forceinline__ void gb_hyper_load(const ModelConst& mc, const Hyper* hy, bool mom,
                                              int tid, GbHyper* u) {
  if (tid < mc.L) {
    const float s2 = (float)hy->phi[2 + mc.L + tid];
    u->th[tid] = (float)hy->phi[2 + tid];
    u->s2[tid] = s2;
    u->hs[tid] = 0.5f / s2;
  } else if (tid == kMaxL) {
    u->nu = (float)hy->phi[0];
    u->tau = (float)hy->phi[1];
    u->inv_k = mom ? 1.0f / (float)(hy->n_mom + 1) : 0.0f;
  }
}

template <int L>
__device__ __forceinline__ bool mh_move_l(const ModelConst& mc, int g, uint32_t it32, float* bs,
                                          float* es, int B, int tid,
                                          const GbHyper& u_, float hg, int kind,
                                          const float* prop, size_t pstride, int pidx) {
  const int N = mc.N;
  float mu[L], C[L][L], xi[L], bn[L], d[L];
#pragma unroll
  for (int i = 0; i < L; ++i) {
    mu[i] = u_.th[i];  // the prior's centre and scales
#pragma unroll
    for (int j = 0; j < L; ++j) C[i][j] = 0.0f;
    C[i][i] = sqrtf(u_.s2[i]);
  }
  if (kind == kMoveNet) {
    int k = 2 * L;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      mu[i] = prop[(size_t)i * pstride + pidx];
      C[i][i] = expf(prop[(size_t)(L + i) * pstride + pidx]);
#pragma unroll
      for (int j = 0; j < i; ++j) C[i][j] = prop[(size_t)(k++) * pstride + pidx];
    }
  }
  // the 2L + 5 uniforms, block by block
  constexpr int kU = 2 * L + 5, kBlk = (kU + 3) / 4;
  float un[4 * kBlk];
  Rng4OL r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamMH, (uint32_t)g, it32);
#pragma unroll
  for (int b = 0; b < kBlk; ++b) {
    const uint4 q = r.block((uint32_t)b);
    un[4 * b] = Rng4OL::word(q.x);
    un[4 * b + 1] = Rng4OL::word(q.y);
    un[4 * b + 2] = Rng4OL::word(q.z);
    un[4 * b + 3] = Rng4OL::word(q.w);
  }
  float lp = 0.0f;  // log prior ratio of beta
  float xx = 0.0f;  // |xi|^2
#pragma unroll
  for (int i = 0; i < L; ++i) {
    xi[i] = normal_bm_f(un[2 * i], un[2 * i + 1]);
    xx += xi[i] * xi[i];
  }
  const float log_u = __logf(un[2 * L]);
  const float chi2 = -2.0f * (logf(un[2 * L + 1]) + logf(un[2 * L + 2]) + logf(un[2 * L + 3]) +
                              logf(un[2 * L + 4]));
  const float st = sqrtf((float)kTDof / chi2);
#pragma unroll
  for (int i = 0; i < L; ++i) {
    float v = 0.0f;
#pragma unroll
    for (int j = 0; j <= i; ++j) v += C[i][j] * xi[j];
    v = mu[i] + st * v;
    bn[i] = v;
    d[i] = v - bs[i * B + tid];
  }
  float u[L];
  float uu = 0.0f;  // |C^-1 (beta - mu)|^2
#pragma unroll
  for (int i = 0; i < L; ++i) {
    float v = bs[i * B + tid] - mu[i];
#pragma unroll
    for (int j = 0; j < i; ++j) v -= C[i][j] * u[j];
    u[i] = v / C[i][i];
    uu += u[i] * u[i];
    const float bt = bs[i * B + tid] - u_.th[i];
    lp -= d[i] * (d[i] + 2.0f * bt) * u_.hs[i];
  }
  // log q(beta) - log q(beta*), with C^-1 (beta* - mu) = st xi
  const float inv_dof = 1.0f / (float)kTDof;
  const float lq = -0.5f * (float)(kTDof + L) *
                   (log1pf(uu * inv_dof) - log1pf(st * st * xx * inv_dof));
  // eps prior ratio: sum_n [eps_n^2 - (eps_n - X_n d)^2] / (2 gamma)
  auto shift = [&](int n) {  // X_n d
    float xd = 0.0f;
#pragma unroll
    for (int l = 0; l < L; ++l) xd += mc.Xf[n * kMaxL + l] * d[l];
    return xd;
  };
  float se = 0.0f;
#pragma unroll 4
  for (int n = 0; n < N; ++n) {
    const float xd = shift(n);
    se += xd * (2.0f * es[n * B + tid] - xd);
  }
  const float la = se * hg + lp + lq;
  const bool acc = log_u < la;
  if (acc) {
#pragma unroll 4
    for (int n = 0; n < N; ++n) es[n * B + tid] -= shift(n);
#pragma unroll
    for (int i = 0; i < L; ++i) bs[i * B + tid] = bn[i];
  }
  return acc;
}

// One copy of the move per number of columns: with L a constant its matrices are
// registers and its 2L + 5 uniforms are drawn block by block (with L a variable
// every uniform had its own copy of the generator behind a test: 17 000 cycles
// per move at L = 5).
__device__ __forceinline__ bool mh_move_f32(const ModelConst& mc, int g, uint32_t it32, float* bs,
                                            float* es, int B, int tid,
                                            const GbHyper& u, float hg, int kind,
                                            const float* prop, size_t pstride, int pidx) {
  static_assert(kMaxL == 8, "one case per number of columns");
  switch (mc.L) {
    case 1: return mh_move_l<1>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 2: return mh_move_l<2>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 3: return mh_move_l<3>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 4: return mh_move_l<4>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 5: return mh_move_l<5>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 6: return mh_move_l<6>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    case 7: return mh_move_l<7>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
    default: return mh_move_l<8>(mc, g, it32, bs, es, B, tid, u, hg, kind, prop, pstride, pidx);
  }
}

// One slice update of beta_gl (step 5) for a column with NC value classes: class
// sums Q_j (rates) and Y_j (counts), the update, and the rates carried to the new
// value.  With use_pat the sums run over the row patterns' sums E and Yp, picked
// by the classes' pattern masks (one constant each; a class number per pattern
// made every addition wait for a constant load and a branch: 1500 cycles per
// column); else over the class's samples in the per-thread rows in shared memory,
// the samples in the order of their classes, each class's sums left in the
// scratch rows qs [kMaxCls] and qs + kMaxCls rows as it ends.
template <int NC>
__device__ __forceinline__ void beta_column_f32(const ModelConst& mc, const DevPtrsF32& p, int l,
                                                int g, float* mu, const float* ys, float* qs,
                                                float* bs, const float* ws, int B, int tid,
                                                const GbHyper& u, long long it, uint32_t it32,
                                                long long burnin, long long tune_start,
                                                unsigned& evals_b, unsigned& caps,
                                                unsigned& nonfin, bool use_pat, float* E,
                                                const float* Yp) {
  const int G = mc.G, L = mc.L;
  BetaDensityFT<NC> f;
  const float b_cur = bs[l * B + tid];
  f.b0 = b_cur;
  f.bt = b_cur - u.th[l];
  f.hs = u.hs[l];
  f.ncls = mc.ncls[l];
  float Y[NC];
  unsigned mask[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    f.Q[j] = 0.0f;
    Y[j] = 0.0f;
    f.v[j] = mc.cvalf[l][j];
    mask[j] = mc.pmask[l][j];
  }
  const int nk = mc.ncl[l];
  if (use_pat) {
#pragma unroll
    for (int j = 0; j < NC; ++j)
#pragma unroll
      for (int r = 0; r < kMaxPat; ++r)
        if (mask[j] & (1u << r)) {
          f.Q[j] += E[r];
          Y[j] += Yp[r];
        }
  } else {
    float am = 0.0f, ay = 0.0f;
#pragma unroll 4
    for (int k = 0; k < nk; ++k) {
      const unsigned c = mc.cinfo[l][k];
      const int n = mc.cord[l][k];
      if (c & kRunFirst) am = ay = 0.0f;
      am += mu[n * B + tid];
      ay += ys[n * B + tid];
      if (c & kRunLast) {
        qs[(c >> kRunShift) * B + tid] = am;
        qs[((c >> kRunShift) + kMaxCls) * B + tid] = ay;
      }
    }
#pragma unroll
    for (int j = 0; j < NC; ++j)
      if (j < f.ncls) {
        f.Q[j] = qs[j * B + tid];
        Y[j] = qs[(j + kMaxCls) * B + tid];
      }
  }
#pragma unroll
  for (int j = 0; j < NC; ++j) f.D[j] = Y[j] - f.Q[j];
  Rng4OL r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamBeta, (uint32_t)((size_t)g * L + l), it32);
  const float x0 = b_cur;
  float w = ws[l * B + tid];
  SliceResultF s = slice_update_f(x0, 0.0f, w, f, r, mc.K, mc.shrink_max);
  evals_b += s.evals;
  caps += s.capped;
  nonfin += s.nonfinite;
  if (s.x != x0) {
    const float d = s.x - x0;
    float fac[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      const float z = f.v[j] * d;
      fac[j] = 1.0f + (z + em1mx(z));
    }
    if (use_pat) {
#pragma unroll
      for (int j = 0; j < NC; ++j)
#pragma unroll
        for (int r = 0; r < kMaxPat; ++r)
          if (mask[j] & (1u << r)) E[r] *= fac[j];
    } else {
#pragma unroll
      for (int j = 0; j < NC; ++j) qs[j * B + tid] = fac[j];
#pragma unroll 4
      for (int k = 0; k < nk; ++k)
        mu[mc.cord[l][k] * B + tid] *= qs[(mc.cinfo[l][k] >> kRunShift) * B + tid];
    }
  }
  bs[l * B + tid] = s.x;
  if (it <= burnin) {
    const size_t e = (size_t)l * G + g;
    float waux = p.waux_beta[e];
    tune_width_f(w, waux, it, s.x, x0, burnin, tune_start);
    p.w_beta[e] = w;
    p.waux_beta[e] = waux;
  }
}

// Shared memory of the gamma/beta updates for blocks of B threads, in rows of B
// floats: the partials ps [kNumPart] (until they are written, the row patterns'
// sums, or a column's class sums), beta and its widths [2 kMaxL], the running
// moments of beta and gamma [4 (L + 1)], with the learned move eps [N], without
// row patterns the rates mu and counts y [2 N]; then FP64 warp sums.  Threads only
// touch their own column of the rows, but for the partials at the end.
struct GbLayout {
  int bs, ws, mom, es, mu, rows;
};

__host__ __device__ constexpr GbLayout gb_layout_f32(int N, int L, bool pat, bool move) {
  GbLayout o{};
  o.bs = kNumPart;
  o.ws = o.bs + kMaxL;
  o.mom = o.ws + kMaxL;
  o.es = o.mom + 4 * (L + 1);
  o.mu = o.es + (move ? N : 0);
  o.rows = o.mu + (pat ? 0 : 2 * N);
  return o;
}

__host__ __device__ constexpr size_t gb_smem_bytes_f32(int N, int L, int B, bool pat, bool move) {
  return ((size_t)gb_layout_f32(N, L, pat, move).rows * B + 2) * sizeof(float) +
         (size_t)(B / 32) * kNumPart * sizeof(double);
}

// What the largest dataset in the largest block needs (the kernels' limits).
constexpr size_t kGbMostSmem = gb_smem_bytes_f32(kMaxN, kMaxL, 128, false, false);
constexpr size_t kGbMoveMostSmem = gb_smem_bytes_f32(kMaxN, kMaxL, 128, false, true);
static_assert(kGbMoveMostSmem <= 227 * 1024, "a block's shared memory");

// A thread's own copy of one word into its shared memory, without a register and
// without waiting (cp_wait).
__device__ __forceinline__ void cp_word(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Steps 2 and 5 of Algorithm 1 in the FP32 form: one thread per gene.  The
// hyperparameter kernel of the previous iteration has finished when it runs.
// Genes marked for the learned proposal first make its move (which keeps every
// log-rate, so the rates mu stay valid); the slice updates of beta_g follow the
// gamma draw, for every gene unless the move replaces them (p.mh_replace).
// net_ok: false when this block's network pass gave up (its genes then skip the
// network's move); prop_s: the network's outputs of the block's genes in shared
// memory ([K][B]), or nullptr (the move reads p.prop, [K][G]).
//
// Bound by latency (2 warps per scheduler at G = 40000), so everything a thread
// reads is under way before it waits for any of it: the state and the moments as
// asynchronous copies, the rates and counts 16 samples at a time, in the order of
// the row patterns, whose sums they are added into on arrival.  N=16 G=40000 L=5:
// 19.5 us (21.9 with a column's loads behind its stores, one wait each, and a
// constant load and branch per addition).
template <bool kMove>
__device__ __forceinline__ void gb_f32_body(const ModelConst& mc, const DevPtrsF32& p, int seg_i,
                                            int blk, bool net_ok = true,
                                            const float* prop_s = nullptr) {
  extern __shared__ float smem_f[];
  __shared__ GbHyper u;
  const int G = mc.G, N = mc.N, L = mc.L;
  const Hyper* hy = p.hyp;
  const long long it = hy->seg_it + seg_i + 1;
  const uint32_t it32 = (uint32_t)it;
  const long long burnin = hy->burnin, tune_start = hy->tune_start;
  const bool mom = it > burnin;
  const bool trace_now = mom && mc.trace_beta && p.trace_beta != nullptr &&
                         ((it - burnin) % hy->thin == 0) && hy->trace_rows < hy->trace_cap;
  const long long trace_row = hy->trace_rows;
  const size_t LG = (size_t)L * G;

  const int B = blockDim.x;
  const bool use_pat = mc.npat <= kMaxPat;
  const GbLayout lay = gb_layout_f32(N, L, use_pat, kMove);
  float* ps = smem_f;
  float* bs = smem_f + (size_t)lay.bs * B;
  float* ws = smem_f + (size_t)lay.ws * B;
  float* ms = smem_f + (size_t)lay.mom * B;
  float* es = smem_f + (size_t)lay.es * B;
  float* mu = smem_f + (size_t)lay.mu * B;
  float* ys = mu + (size_t)N * B;
  const int tid = threadIdx.x;
  const int g = blk * B + tid;
  const bool active = g < G;
  unsigned evals_b = 0, caps = 0, gcaps = 0, nonfin = 0;
  float ss = 0.0f;
  float E[kMaxPat], Yp[kMaxPat];

  if (active) {
    for (int l = 0; l < L; ++l) {
      cp_word(bs + l * B + tid, p.beta + (size_t)l * G + g);
      cp_word(ws + l * B + tid, p.w_beta + (size_t)l * G + g);
    }
    if (kMove)
      for (int n = 0; n < N; ++n) cp_word(es + n * B + tid, p.eps + (size_t)n * G + g);
    cp_commit();
    float am = 0.0f, ay = 0.0f;  // sums of the pattern being read
    for (int k0 = 0; k0 < N; k0 += kGbBatch) {
      float m[kGbBatch], x[kGbBatch];
      int32_t y[kGbBatch];
#pragma unroll
      for (int i = 0; i < kGbBatch; ++i)
        if (k0 + i < N) {
          // the samples in the patterns' order, the eps (whose squares are added
          // in the samples' order) in theirs
          const size_t e = (size_t)(use_pat ? mc.pord[k0 + i] : k0 + i) * G + g;
          m[i] = p.mu[e];
          y[i] = p.y[e];
          if (!kMove) x[i] = p.eps[(size_t)(k0 + i) * G + g];
        }
      if (k0 == 0 && mom) {
        for (int l = 0; l < L; ++l)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            cp_word(ms + (4 * l + i) * B + tid, p.mom_beta + i * LG + (size_t)l * G + g);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          cp_word(ms + (4 * L + i) * B + tid, p.mom_gam + (size_t)i * G + g);
      }
#pragma unroll
      for (int i = 0; i < kGbBatch; ++i)
        if (k0 + i < N) {
          const float yf = (float)y[i];
          if (!kMove) ss += x[i] * x[i];
          if (use_pat) {
            const unsigned c = mc.pinfo[k0 + i];
            if (c & kRunFirst) am = ay = 0.0f;
            am += m[i];
            ay += yf;
            if (c & kRunLast) {
              ps[(c >> kRunShift) * B + tid] = am;
              ps[((c >> kRunShift) + kMaxPat) * B + tid] = ay;
            }
          } else {
            mu[(k0 + i) * B + tid] = m[i];
            ys[(k0 + i) * B + tid] = yf;
          }
        }
    }
    cp_commit();
  }
  gb_hyper_load(mc, hy, mom, tid, &u);
  cp_wait<1>();     // beta, its widths and eps; the moments are still on their way
  __syncthreads();  // the block's hyperparameters
  const float inv_k = u.inv_k;
  // the per-pattern sums of the rates and counts, in registers, when X has at most
  // kMaxPat distinct rows (the move keeps every rate)
#pragma unroll
  for (int r = 0; r < kMaxPat; ++r) {
    const bool on = active && use_pat && r < mc.npat;
    E[r] = on ? ps[r * B + tid] : 0.0f;
    Yp[r] = on ? ps[(r + kMaxPat) * B + tid] : 0.0f;
  }

  if (active) {
    // ---- learned-proposal move (keeps every log-rate, so mu stays valid)
    bool mh_gene = false;
    if constexpr (kMove) {
      int kind = move_kind(p, g, it);
      if (kind == kMoveNet && !net_ok) kind = 0;
      mh_gene = kind != 0;
      if (mh_gene) {
        const float hg = 0.5f / p.gam[g];
        const size_t ci = (size_t)(kind - 1) * G + g;
        const unsigned tried = p.mh_try[ci], accepted = p.mh_acc[ci];
        const bool in_smem = prop_s != nullptr;
        const bool acc = mh_move_f32(mc, g, it32, bs, es, B, tid, u, hg, kind,
                                     in_smem ? prop_s : p.prop, in_smem ? (size_t)B : (size_t)G,
                                     in_smem ? tid : g);
        p.mh_try[ci] = tried + 1u;
        if (acc) {
          p.mh_acc[ci] = accepted + 1u;
          for (int n = 0; n < N; ++n) p.eps[(size_t)n * G + g] = es[n * B + tid];
        }
      }
#pragma unroll 8
      for (int n = 0; n < N; ++n) {
        const float x = es[n * B + tid];
        ss += x * x;
      }
    }

    // ---- step 2: gamma_g ~ IG((N + nu)/2, (sum eps^2 + nu tau)/2)
    float gam;
    {
      Rng4OL r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamGamma, (uint32_t)g, it32);
      bool gcap = false;
      const float shape = 0.5f * ((float)N + u.nu);
      const float scale = 0.5f * (ss + u.nu * u.tau);
      gam = scale / gamma_mt_f(shape, r, 0, &gcap);
      gcaps += gcap;
      p.gam[g] = gam;
      ps[0 * B + tid] = __logf(gam);
      ps[1 * B + tid] = 1.0f / gam;
    }

    // ---- step 5: beta_gl, l = 1..L in order (genes without the learned move)
    const bool skip_slices = mh_gene && p.mh_replace;
    for (int l = 0; l < L && !skip_slices; ++l) {
      switch (mc.ncls[l]) {
        case 1:
          beta_column_f32<1>(mc, p, l, g, mu, ys, ps + 2 * B, bs, ws, B, tid, u, it, it32, burnin,
                             tune_start, evals_b, caps, nonfin, use_pat, E, Yp);
          break;
        case 2:
          beta_column_f32<2>(mc, p, l, g, mu, ys, ps + 2 * B, bs, ws, B, tid, u, it, it32, burnin,
                             tune_start, evals_b, caps, nonfin, use_pat, E, Yp);
          break;
        case 3:
          beta_column_f32<3>(mc, p, l, g, mu, ys, ps + 2 * B, bs, ws, B, tid, u, it, it32, burnin,
                             tune_start, evals_b, caps, nonfin, use_pat, E, Yp);
          break;
        default:
          beta_column_f32<kMaxCls>(mc, p, l, g, mu, ys, ps + 2 * B, bs, ws, B, tid, u, it, it32,
                                   burnin, tune_start, evals_b, caps, nonfin, use_pat, E, Yp);
      }
    }

    // ---- the new beta_g: state, moments, trace, partial sums for steps 6-7
    cp_wait<0>();
    if (mom) {
      for (int l = 0; l <= L; ++l) {  // the columns, then gamma
        KahanMoments m;
        m.load(ms + (size_t)4 * l * B, (size_t)B, (size_t)tid);
        m.update(l < L ? bs[l * B + tid] : gam, inv_k);
        if (l < L) m.store(p.mom_beta, LG, (size_t)l * G + g);
        else m.store(p.mom_gam, (size_t)G, (size_t)g);
      }
    }
    for (int l = 0; l < L; ++l) {
      const size_t e = (size_t)l * G + g;
      const float b = bs[l * B + tid];
      p.beta[e] = b;
      if (trace_now) p.trace_beta[(size_t)trace_row * LG + e] = (double)b;
      const float dv = b - u.th[l];
      ps[(2 + l) * B + tid] = dv;
      ps[(2 + kMaxL + l) * B + tid] = dv * dv;
    }
    for (int l = L; l < kMaxL; ++l) ps[(2 + l) * B + tid] = ps[(2 + kMaxL + l) * B + tid] = 0.0f;
    // contrast probabilities (§3.1), evaluated in FP32
    if (mom && p.con != nullptr) {
      const Contrasts* cs = p.con;
      for (int q = 0; q < cs->n; ++q) {
        bool ok = true;
        for (int k = 0; k < cs->terms[q] && ok; ++k) {
          float sv = 0.0f;
          for (int l = 0; l < L; ++l) sv = __fadd_rn(sv, __fmul_rn(cs->vf[q][k][l], bs[l * B + tid]));
          ok = sv > cs->bf[q][k];
        }
        if (ok) p.con_count[(size_t)q * G + g] += 1u;
      }
    }
  }

  if (!active) {
#pragma unroll
    for (int i = 0; i < kNumPart; ++i) ps[i * B + tid] = 0.0f;
  }

  // ---- partial sums: error-free FP32 pair sums within the warp, FP64 beyond.
  // Lane i < kNumPart sums row i of the warp's 32 values (read in an order
  // rotated by i, so that the lanes hit distinct shared-memory banks).
  const int lane = tid & 31, warp = tid >> 5, nwarp = B >> 5;
  double* red = reinterpret_cast<double*>(smem_f + (((size_t)lay.rows * B + 1) & ~(size_t)1));
  __syncwarp();
  if (lane < kNumPart) {
    const float* row = ps + (size_t)lane * B + warp * 32;
    float sm = 0.0f, c = 0.0f;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
      float t, e;
      two_sum(sm, row[(j + lane) & 31], t, e);
      sm = t;
      c += e;
    }
    red[warp * kNumPart + lane] = (double)sm + (double)c;
  }
  __syncthreads();
  if (tid < kNumPart) {
    double acc = 0.0;
    for (int w = 0; w < nwarp; ++w) acc += red[w * kNumPart + tid];
    p.partial[(size_t)blk * kNumPart + tid] = acc;
  }
  add_counters(p.counters, 0, evals_b, caps, gcaps, nonfin, &p.hyp->flags);
}

// At most 128 registers: four blocks per SM, which G = 200000 needs (80 against 90 us
// at N = 32 with three).
__global__ void __launch_bounds__(128, 4) k_gb_f32(ModelConst mc, DevPtrsF32 p, int seg_i) {
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i + 1);
  gb_f32_body<false>(mc, p, seg_i, blockIdx.x);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i + 1);
}

// With the learned move, the network's outputs read from global memory (block
// sizes other than 128, or the network in a kernel of its own).
__global__ void __launch_bounds__(128) k_gb_move_f32(ModelConst mc, DevPtrsF32 p, int seg_i) {
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i + 1);
  gb_f32_body<true>(mc, p, seg_i, blockIdx.x);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i + 1);
}

// Shared memory of the fused kernel: the network pass (its weight image; the A
// operands are in tensor memory) from offset 0, then the gamma/beta updates'
// arrays from offset 0, and
// the network's outputs of the block's genes ([K][128] floats) at
// gb_net_stash_offset, past both the weight image and those arrays.
__host__ __device__ inline size_t gb_net_stash_offset(int N, int L, bool pat) {
  size_t off_a;
  tc_smem_layout(L, &off_a);
  const size_t gb = gb_smem_bytes_f32(N, L, 128, pat, true);
  return ((off_a > gb ? off_a : gb) + 15) & ~(size_t)15;
}

static size_t gb_net_smem_bytes(int N, int L, bool pat) {
  const size_t tc = tc_smem_layout(L, nullptr);
  const size_t st = gb_net_stash_offset(N, L, pat) + (size_t)tc_shape(L).K * 128 * sizeof(float);
  return tc > st ? tc : st;
}

// Every part grows with N and L, and without row patterns.
static size_t gb_net_most_smem() { return gb_net_smem_bytes(kMaxN, kMaxL, false); }

// With the learned proposal (128 threads): the block first evaluates the network
// for its 128 genes on the tensor cores (outputs to shared memory, read by the
// same threads in the move: a round trip through global memory less), then frees
// the tensor memory and reuses the shared memory below the outputs for the
// gamma/beta updates.  A kernel of its own, so that the plain gamma/beta kernel
// keeps its own register allocation.  kBlocks: resident blocks per SM it is
// compiled for: 3 (154 registers) while the genes fit them, else 4 (128, a few
// spilled).  N=16 L=5: 34.6 against 35.7 us at G = 40000 (33.4 since the network's
// columns are loops), 61.9 against 41.7 at 59500 (one block more than 3 per SM hold),
// 99 against 79 at 120000.
template <int kBlocks>
__global__ void __launch_bounds__(128, kBlocks) k_gb_net_f32(ModelConst mc, DevPtrsF32 p, int seg_i,
                                                    const uint8_t* __restrict__ img) {
  ktime_begin(p.ktime, p.ktime_n, 3 * seg_i + 1);
  bool net_ok;
  float* prop_s;
  {
    extern __shared__ __align__(1024) uint8_t sm_tc[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    const TcShape t = tc_shape(mc.L);
    __shared__ NetHyper nh;
    if (threadIdx.x == 0) s_abort = 0;
    net_hyper_load(mc, p.hyp, (int)threadIdx.x, &nh);
    TcBlock c;
    tc_begin(c, bars, &tmem_slot, img, sm_tc, t.bytes, p.tc_polls);
    if (!c.w_ok) s_abort = 1;
    __syncthreads();
    const int g = blockIdx.x * 128 + (int)threadIdx.x;
    prop_s = reinterpret_cast<float*>(sm_tc + gb_net_stash_offset(mc.N, mc.L, mc.npat <= kMaxPat));
    if (!s_abort)
      tc_tile(c, mc, p, nh, t, sm_tc, g, net_gene(p, g, mc.G), prop_s, 128, (int)threadIdx.x,
              &s_abort);
    __syncthreads();
    net_ok = s_abort == 0;
    tc_end(c, !net_ok, &p.hyp->flags);
    fence_async_smem();
    __syncthreads();  // below the outputs, the shared memory is the gamma/beta updates' from here on
  }
  gb_f32_body<true>(mc, p, seg_i, blockIdx.x, net_ok, prop_s);
  ktime_end(p.ktime, p.ktime_n, 3 * seg_i + 1);
}

// The learned move alone, at the current state, for the genes that use it (every
// gene when p.mh_all), with the random numbers of iteration `it`.
__global__ void __launch_bounds__(128) k_mh_step_f32(ModelConst mc, DevPtrsF32 p, long long it) {
  extern __shared__ float es[];  // [N][128]
  __shared__ float bs[kMaxL * 128];
  __shared__ GbHyper u;
  const int B = blockDim.x, tid = threadIdx.x;
  const int g = blockIdx.x * B + tid;
  gb_hyper_load(mc, p.hyp, false, tid, &u);
  __syncthreads();
  if (g >= mc.G) return;
  const int kind = move_kind(p, g, it);
  if (kind == 0) return;
  const int G = mc.G, N = mc.N, L = mc.L;
  for (int l = 0; l < L; ++l) bs[l * B + tid] = p.beta[(size_t)l * G + g];
  for (int n = 0; n < N; ++n) es[n * B + tid] = p.eps[(size_t)n * G + g];
  const bool acc = mh_move_f32(mc, g, (uint32_t)it, bs, es, B, tid, u,
                               0.5f / p.gam[g], kind, p.prop, (size_t)G, g);
  const size_t ci = (size_t)(kind - 1) * G + g;
  p.mh_try[ci] += 1u;
  if (acc) {
    p.mh_acc[ci] += 1u;
    for (int l = 0; l < L; ++l) p.beta[(size_t)l * G + g] = bs[l * B + tid];
    for (int n = 0; n < N; ++n) p.eps[(size_t)n * G + g] = es[n * B + tid];
  }
}

__global__ void k_seg_begin(Hyper* hy) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    hy->seg_it = hy->it;
    hy->seg_nmom = hy->n_mom;
  }
}

// ---------------------------------------------------------------- persistent sweeps (FP32)
//
// A whole segment of sweeps of one chain (Algorithm 1, every step) in one
// cooperative launch whose blocks are all resident: per sweep, every block takes
// tiles of 128 eps_gn updates (step 1), a grid barrier, every block takes
// 128-gene blocks of gamma/beta updates (steps 2, 5), a grid barrier, then block 0
// runs the hyperparameter steps (3, 4, 6, 7) while the other blocks go on to the
// next sweep's eps updates, which involve no hyperparameter; the next barrier
// also waits for block 0.  The per-element, per-gene and hyperparameter device
// functions are those of k_eps_f32, k_gb_f32 and k_hyper, with the same Philox
// counters and the same per-gene-block partial sums, so the chain is
// bit-identical to the graph of separate launches.

// Sense-reversing grid barrier in device memory (zeroed before each launch).
struct GridSync {
  unsigned int count, gen;
};

// Polls of a barrier wait (each followed by a 64 ns sleep, about 4 s in all)
// before the wait gives up, sets kFlagTimeout and ends the launch.
constexpr unsigned kGridWaitLimit = 1u << 26;

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_gpu(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Every block of the grid arrives; the last one to arrive resets the count and
// opens the next generation.  Writes of every block before the barrier are
// visible to every block after it.  Returns false in every thread of a block
// whose wait gave up.
__device__ __forceinline__ bool grid_sync(GridSync* gs, unsigned* flags, volatile int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned gen = ld_acquire_gpu(&gs->gen);
    __threadfence();
    const unsigned arrived = atomicAdd(&gs->count, 1u) + 1u;
    int ok = 1;
    if (arrived == gridDim.x) {
      atomicExch(&gs->count, 0u);
      __threadfence();
      st_release_gpu(&gs->gen, gen + 1u);
    } else {
      unsigned polls = 0;
      while (ld_acquire_gpu(&gs->gen) == gen) {
        if (++polls >= kGridWaitLimit) {
          ok = 0;
          atomicOr(flags, kFlagTimeout);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__global__ void __launch_bounds__(128, 4) k_sweeps_f32(ModelConst mc, DevPtrsF32 p, DevPtrs hp,
                                                   int n_sweeps, int nblk, GridSync* gs) {
  __shared__ int s_ok;
  const int tiles_g = (mc.G + 127) / 128;
  const int n_tiles = tiles_g * mc.N;
  for (int i = 0; i < n_sweeps; ++i) {
    // block 0 is still at the previous sweep's hyperparameters: the others take its
    // eps tiles too (N=16 G=40000 L=5: 83 -> 66 us per sweep, N=22 G=9973 71 ->
    // 62)
    const int busy = i > 0 && gridDim.x > 1 ? 1 : 0;
    for (int t = (int)blockIdx.x - busy; t < n_tiles && t >= 0; t += (int)gridDim.x - busy) {
      const int n = t / tiles_g;
      eps_f32_body(mc, p, i, n, (t - n * tiles_g) * 128 + (int)threadIdx.x, t % kCounterCopies);
    }
    if (!grid_sync(gs, &p.hyp->flags, &s_ok)) return;
    for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
      gb_f32_body<false>(mc, p, i, b);
      __syncthreads();  // the next gene block reuses the shared memory
    }
    if (!grid_sync(gs, &p.hyp->flags, &s_ok)) return;
    if (blockIdx.x == 0) hyper_body<128>(mc, hp.partial, hp.hyp, hp.trace_phi, hp.counters, nblk);
  }
}

cudaError_t launch_sweeps_f32(const ModelConst& mc, const DevPtrsF32& p, const DevPtrs& hp,
                              int n_sweeps, void* gsync, cudaStream_t s, int* grid_out) {
  const int block = 128;
  const int nblk = (mc.G + block - 1) / block;
  const size_t smem = gb_smem_f32(mc, block, false);
  cudaError_t e = set_smem_limit(k_sweeps_f32, kGbMostSmem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweeps_f32, block, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int grid = per_sm * sms;
  const int most = nblk > ((mc.G + 127) / 128) * mc.N ? nblk : ((mc.G + 127) / 128) * mc.N;
  if (grid > most) grid = most;
  if ((e = cudaMemsetAsync(gsync, 0, sizeof(GridSync), s)) != cudaSuccess) return e;
  ModelConst mc_ = mc;
  DevPtrsF32 p_ = p;
  DevPtrs hp_ = hp;
  int n_ = n_sweeps, nb_ = nblk;
  GridSync* gs_ = (GridSync*)gsync;
  void* args[] = {&mc_, &p_, &hp_, &n_, &nb_, &gs_};
  if (grid_out) *grid_out = grid;
  return cudaLaunchCooperativeKernel((const void*)k_sweeps_f32, dim3(grid), dim3(block), args, smem,
                                     s);
}

// ---------------------------------------------------------------- batched kernels (FP32)
//
// Many independent datasets / chains in one launch.  Each dataset keeps its own
// model constants and device pointers in global memory; a block table maps every
// block of a launch to one dataset (and to a sample row and gene block for the
// eps kernel), so a block never straddles two datasets and uneven N and G need no
// padding beyond the last block of each dataset.

// At most 51 registers (at least 5 blocks of 256 per SM, as k_eps_f32): 454 -> 511
// batch sweeps/s on the 64-dataset batch.
__global__ void __launch_bounds__(256, 5) k_eps_f32_batch(const ModelConst* __restrict__ mcs,
                                                       const DevPtrsF32* __restrict__ ps,
                                                       const int4* __restrict__ tab, int seg_i) {
  const int4 t = tab[blockIdx.x];  // dataset, sample row n, gene block, counter copy
  eps_f32_body(mcs[t.x], ps[t.x], seg_i, t.y, t.z * blockDim.x + threadIdx.x, t.w);
}

__global__ void __launch_bounds__(128, 4) k_gb_f32_batch(const ModelConst* __restrict__ mcs,
                                                      const DevPtrsF32* __restrict__ ps,
                                                      const int2* __restrict__ tab, int seg_i) {
  const int2 t = tab[blockIdx.x];  // dataset, gene block within the dataset
  gb_f32_body<false>(mcs[t.x], ps[t.x], seg_i, t.y);
}

// One block per dataset.
__global__ void __launch_bounds__(kHyperThreads) k_hyper_batch(const ModelConst* __restrict__ mcs,
                                                               const DevPtrsF32* __restrict__ ps,
                                                               const int* __restrict__ nblk) {
  const int c = blockIdx.x;
  const DevPtrsF32& p = ps[c];
  hyper_body<kHyperThreads>(mcs[c], p.partial, p.hyp, p.trace_phi, p.counters, nblk[c], p.psi);
}

// Top level of the three-level model, one warp, after the datasets' hyper
// steps of the same sweep: lane 0 draws b ~ Gamma(a_b + sum_k a_k, rate b_b +
// sum_k tau_k), lane 1+l draws m_l ~ N(w sum_k theta_kl / c_kl^2, w) with
// w = 1 / (sum_k 1/c_kl^2 + 1/e_l^2); the sums over k run in dataset order.
// Moments and trace follow dataset 0's iteration, burn-in and thinning.
__global__ void __launch_bounds__(32) k_top_level(const ModelConst* __restrict__ mcs,
                                                  const DevPtrsF32* __restrict__ ps, int C,
                                                  TopLevel* __restrict__ top,
                                                  double* __restrict__ trace) {
  const int lane = threadIdx.x;
  const int L = top->L;
  const Hyper* h0 = ps[0].hyp;
  const long long it = h0->it;
  const uint32_t it32 = (uint32_t)it;
  double x = 0.0;
  if (lane == 0) {
    double sa = 0.0, st = 0.0;
    for (int k = 0; k < C; ++k) {
      sa += mcs[k].a;
      st += ps[k].hyp->phi[1];
    }
    Rng r(top->seed_lo, top->seed_hi, 0u, kStreamPsi, 0u, it32);
    bool cap = false;
    x = gamma_mt(top->a_b + sa, r, 0, &cap) / (top->b_b + st);
    if (cap) atomicAdd(&top->gamma_caps, 1ull);
  } else if (lane <= L) {
    const int l = lane - 1;
    double prec = 0.0, s = 0.0;
    for (int k = 0; k < C; ++k) {
      const double c2 = mcs[k].c2[l];
      prec += 1.0 / c2;
      s += ps[k].hyp->phi[2 + l] / c2;
    }
    const double w = 1.0 / (prec + 1.0 / top->e2[l]);
    Rng r(top->seed_lo, top->seed_hi, 0u, kStreamPsi, (uint32_t)lane, it32);
    x = __dadd_rn(__dmul_rn(w, s), __dmul_rn(sqrt(w), normal_bm(r, 0)));
  }
  const bool mom = it > h0->burnin;
  const bool tr = mom && ((it - h0->burnin) % h0->thin == 0) && top->trace_rows < top->trace_cap &&
                  trace != nullptr;
  if (lane <= L) {
    top->psi[lane] = x;
    if (mom) {
      const double inv_k = 1.0 / (double)(top->n_mom + 1);
      const double m = top->m_psi[lane], q = top->q_psi[lane];
      top->m_psi[lane] = m + (x - m) * inv_k;
      top->q_psi[lane] = q + (x * x - q) * inv_k;
    }
    if (tr) trace[(size_t)top->trace_rows * (L + 1) + lane] = x;
  }
  __syncwarp();
  if (lane == 0) {
    if (mom) top->n_mom += 1;
    if (tr) top->trace_rows += 1;
  }
}

__global__ void k_seg_begin_batch(const DevPtrsF32* __restrict__ ps, int C) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < C) {
    Hyper* hy = ps[c].hyp;
    hy->seg_it = hy->it;
    hy->seg_nmom = hy->n_mom;
  }
}

__global__ void k_set_run_batch(const DevPtrsF32* __restrict__ ps, int C, long long burnin,
                                long long tune_start, long long thin) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < C) {
    Hyper* hy = ps[c].hyp;
    hy->burnin = burnin;
    hy->tune_start = tune_start;
    hy->thin = thin;
  }
}

cudaError_t prepare_batch_kernels() { return set_smem_limit(k_gb_f32_batch, kGbMostSmem); }

cudaError_t launch_eps_f32_batch(const ModelConst* mcs, const DevPtrsF32* ps, const int4* tab,
                                 int n_blocks, int block, int seg_i, cudaStream_t s) {
  k_eps_f32_batch<<<n_blocks, block, 0, s>>>(mcs, ps, tab, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_gb_f32_batch(const ModelConst* mcs, const DevPtrsF32* ps, const int2* tab,
                                int n_blocks, int block, size_t smem, int seg_i, cudaStream_t s) {
  k_gb_f32_batch<<<n_blocks, block, smem, s>>>(mcs, ps, tab, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_hyper_batch(const ModelConst* mcs, const DevPtrsF32* ps, const int* nblk,
                               int C, cudaStream_t s) {
  k_hyper_batch<<<C, kHyperThreads, 0, s>>>(mcs, ps, nblk);
  return cudaGetLastError();
}

cudaError_t launch_top_level(const ModelConst* mcs, const DevPtrsF32* ps, int C, TopLevel* top,
                             double* trace, cudaStream_t s) {
  k_top_level<<<1, 32, 0, s>>>(mcs, ps, C, top, trace);
  return cudaGetLastError();
}

cudaError_t launch_seg_begin_batch(const DevPtrsF32* ps, int C, cudaStream_t s) {
  k_seg_begin_batch<<<(C + 127) / 128, 128, 0, s>>>(ps, C);
  return cudaGetLastError();
}

cudaError_t launch_set_run_batch(const DevPtrsF32* ps, int C, long long burnin,
                                 long long tune_start, long long thin, cudaStream_t s) {
  k_set_run_batch<<<(C + 127) / 128, 128, 0, s>>>(ps, C, burnin, tune_start, thin);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- set-up kernels (FP32)

// Same starting values as the FP64 form, computed in FP64 and stored in FP32.
__global__ void k_init_genes_f32(ModelConst mc, DevPtrsF32 p, const int32_t* y_in,
                                 int gene_major, const double* __restrict__ pinv, double w0,
                                 int set_state) {
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
      p.asinh_T[(size_t)l * G + g] = asinhf((float)T[l]);
      if (set_state) {
        double s = 0.0;
        for (int n = 0; n < N; ++n) s += pinv[l * kMaxN + n] * r[n];
        p.beta[(size_t)l * G + g] = (float)s;
        p.w_beta[(size_t)l * G + g] = (float)w0;
        p.waux_beta[(size_t)l * G + g] = 0.0f;
      }
    }
    if (set_state) {
      for (int n = 0; n < N; ++n) {
        p.eps[(size_t)n * G + g] = 0.0f;
        p.w_eps[(size_t)n * G + g] = (float)w0;
        p.waux_eps[(size_t)n * G + g] = 0.0f;
      }
      p.gam[g] = 1.0f;
    }
  }
}

__global__ void k_zero_moments_f32(ModelConst mc, DevPtrsF32 p) {
  const size_t NG = (size_t)mc.N * mc.G, LG = (size_t)mc.L * mc.G, G = mc.G;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < 4 * NG;
       i += (size_t)gridDim.x * blockDim.x) {
    p.mom_eps[i] = 0.0f;
    if (i < 4 * LG) p.mom_beta[i] = 0.0f;
    if (i < 4 * G) p.mom_gam[i] = 0.0f;
  }
}

size_t gb_smem_f32(const ModelConst& mc, int block, bool move) {
  return gb_smem_bytes_f32(mc.N, mc.L, block, mc.npat <= kMaxPat, move);
}

cudaError_t prepare_gene_kernel_f32() {
  cudaError_t e = set_smem_limit(k_gb_f32, kGbMostSmem);
  return e == cudaSuccess ? set_smem_limit(k_gb_move_f32, kGbMoveMostSmem) : e;
}

cudaError_t launch_eps_f32(const ModelConst& mc, const DevPtrsF32& p, int seg_i,
                           cudaStream_t s) {
  const int blk = 256;
  const dim3 grid((unsigned)((mc.G + blk - 1) / blk), (unsigned)mc.N);
  k_eps_f32<<<grid, blk, 0, s>>>(mc, p, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_gb_f32(const ModelConst& mc, const DevPtrsF32& p, int block, int seg_i,
                          cudaStream_t s, const void* img) {
  const int nblk = (mc.G + block - 1) / block;
  if (img != nullptr) {
    if (block != 128) return cudaErrorInvalidValue;  // one thread per gene of a 128-gene tile
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const size_t smem = gb_net_smem_bytes(mc.N, mc.L, mc.npat <= kMaxPat);
    const auto kernel = nblk <= 3 * sms ? k_gb_net_f32<3> : k_gb_net_f32<4>;
    e = set_smem_limit(kernel, gb_net_most_smem());
    if (e != cudaSuccess) return e;
    kernel<<<nblk, block, smem, s>>>(mc, p, seg_i, (const uint8_t*)img);
    return cudaGetLastError();
  }
  const size_t smem = gb_smem_f32(mc, block, p.prop != nullptr);
  if (p.prop != nullptr) k_gb_move_f32<<<nblk, block, smem, s>>>(mc, p, seg_i);
  else k_gb_f32<<<nblk, block, smem, s>>>(mc, p, seg_i);
  return cudaGetLastError();
}

cudaError_t launch_mh_step_f32(const ModelConst& mc, const DevPtrsF32& p, long long it,
                              cudaStream_t s) {
  const int block = 128;
  k_mh_step_f32<<<(mc.G + block - 1) / block, block, (size_t)mc.N * block * sizeof(float), s>>>(
      mc, p, it);
  return cudaGetLastError();
}

cudaError_t launch_seg_begin(Hyper* hy, cudaStream_t s) {
  k_seg_begin<<<1, 32, 0, s>>>(hy);
  return cudaGetLastError();
}

cudaError_t launch_init_f32(const ModelConst& mc, const DevPtrsF32& p, const int32_t* y_in,
                            int gene_major, const double* pinv, double w0, int set_state,
                            cudaStream_t s) {
  const int blk = 256;
  const int grid = (mc.G + blk - 1) / blk;
  k_init_genes_f32<<<grid, blk, 0, s>>>(mc, p, y_in, gene_major, pinv, w0, set_state);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_zero_moments_f32(mc, p, s);
}

cudaError_t launch_zero_moments_f32(const ModelConst& mc, const DevPtrsF32& p, cudaStream_t s) {
  const size_t n = 4 * (size_t)mc.N * mc.G;
  const int blk = 256;
  const unsigned grid = (unsigned)((n + blk - 1) / blk);
  k_zero_moments_f32<<<grid, blk, 0, s>>>(mc, p);
  return cudaGetLastError();
}

}  // namespace fbs
