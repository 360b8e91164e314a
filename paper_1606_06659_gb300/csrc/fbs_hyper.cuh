// fbs_hyper.cuh -- the hyperparameter steps of one Gibbs sweep (Algorithm 1
// steps 3, 4, 6, 7 of Landau & Niemi, arXiv 1606.06659) as a block-level device
// function, shared by the single-chain and the batched hyperparameter kernels.
// tau and sigma_l^2 are drawn exactly, or (ModelConst::all_slice) by slice
// updates of their conditionals, each spread over a warp.
#pragma once

#include <math.h>
#include <stdint.h>

#include "fbs_common.cuh"
#include "fbs_rng.cuh"

namespace fbs {

// ---------------------------------------------------------------- hyper kernel

// log f(nu | ...) = -G lgamma(nu/2) + (G nu/2) log(nu tau/2) - (nu/2)(S1 + tau S2) on
// (0, d), S1 = sum_g log gamma_g, S2 = sum_g 1/gamma_g (Algorithm 1 step 3, the
// sum read as log gamma_g + tau/gamma_g, which the Inverse-Gamma(nu/2, nu tau/2)
// prior of the gamma_g gives).
// lgamma(nu/2) and log(nu tau/2) need no sums, so other warps evaluate them while
// the sums are added up.
static __device__ __noinline__ double lgamma_ol(double x) { return lgamma(x); }

struct NuDensity {
  double G, d, tau, S1, S2;
  __device__ __forceinline__ bool inside(double nu) const { return nu > 0.0 && nu < d; }
  // from lg = lgamma(nu/2) and lt = log(nu tau/2)
  __device__ __forceinline__ double combine(double nu, double lg, double lt) const {
    if (!inside(nu)) return -INFINITY;
    return -G * lg + 0.5 * G * nu * lt - 0.5 * nu * (S1 + tau * S2);
  }
  __device__ __forceinline__ double operator()(double nu) const {
    if (!inside(nu)) return -INFINITY;
    return combine(nu, lgamma_ol(0.5 * nu), log_ol(0.5 * nu * tau));
  }
};

// log f(tau | ...) = (shape - 1) log tau - rate tau on tau > 0, shape = a + G nu/2,
// rate = b + (nu/2) S2: the Gamma full conditional of step 4, slice-sampled in the
// all-slice variant (Section 4.2).
struct TauDensity {
  double shape, rate;
  __device__ __forceinline__ double operator()(double x, double* aux) const {
    *aux = 0.0;
    if (!(x > 0.0)) return -INFINITY;
    return (shape - 1.0) * log(x) - rate * x;
  }
};

// log f(sigma_l | ...) = -G log sigma_l - hS / sigma_l^2 on 0 < sigma_l < s_l, hS =
// sum_g (beta_gl - theta_l)^2 / 2: G Normal(theta_l, sigma_l^2) terms times the flat
// Uniform(0, s_l) prior, the step 7 conditional of sigma_l itself (all-slice variant).
struct SigDensity {
  double G, hS, s;
  __device__ __forceinline__ double operator()(double x, double* aux) const {
    *aux = 0.0;
    if (!(x > 0.0 && x < s)) return -INFINITY;
    return -G * log(x) - hS / (x * x);
  }
};

// Out-of-line copies of the transcendental-heavy steps (one copy each in the
// kernel's code instead of one per call site).
static __device__ __noinline__ double hyper_gamma(double shape, Rng& r, uint32_t k0, bool* capped) {
  return gamma_mt(shape, r, k0, capped);
}

// The first attempts of a Marsaglia-Tsang draw whose shape is not known yet:
// the normal x_j = normal_bm(r, k0 + 4j) and the uniform u_j = r.u(k0 + 4j + 2)
// of attempts j < kPreAttempts, with log u_j.  They depend only on the random
// numbers, so another warp computes them while the shape is being found.
constexpr int kPreAttempts = 2;  // lanes 0..1 and 2..3 of warp 3
struct GammaPre {
  double x[kPreAttempts], u[kPreAttempts], logu[kPreAttempts];
};

// gamma_mt(shape, r, k0, capped) with the first attempts' random quantities
// taken from *g: the same operations on the same numbers, so the same result.
// A shape below 1 needs the boost uniform and takes gamma_mt itself.
static __device__ __noinline__ double gamma_mt_pre(double shape, const GammaPre* g, Rng& r,
                                                  uint32_t k0, bool* capped) {
  if (shape < 1.0) return gamma_mt(shape, r, k0, capped);
  const double dd = __dsub_rn(shape, 1.0 / 3.0);
  const double cc = 1.0 / sqrt(__dmul_rn(9.0, dd));
  for (uint32_t j = 0; j < (uint32_t)kGammaAttempts; ++j) {
    const bool pre = j < (uint32_t)kPreAttempts;
    const double x = pre ? g->x[j] : normal_bm(r, k0 + 4 * j);
    double v = __dadd_rn(1.0, __dmul_rn(cc, x));
    if (v <= 0.0) continue;
    v = __dmul_rn(__dmul_rn(v, v), v);
    const double u = pre ? g->u[j] : r.u(k0 + 4 * j + 2);
    const double x2 = __dmul_rn(x, x);
    if (u < __dsub_rn(1.0, __dmul_rn(__dmul_rn(0.0331, x2), x2)))
      return __dmul_rn(__dmul_rn(dd, v), 1.0);
    const double rhs = __dadd_rn(__dmul_rn(0.5, x2),
                                 __dmul_rn(dd, __dadd_rn(__dsub_rn(1.0, v), log(v))));
    if ((pre ? g->logu[j] : log(u)) < rhs) return __dmul_rn(__dmul_rn(dd, v), 1.0);
  }
  *capped = true;
  return shape;
}

// trunc_invgamma of fbs_rng.cuh whose first attempt's gamma draw gv0 (with its
// cap flag) was made beforehand; later attempts draw their own.
static __device__ __noinline__ double hyper_trunc_invgamma(double shape, double scale,
                                                           double upper, double keep, double gv0,
                                                           bool gcap0, Rng& r, bool* gcap,
                                                           bool* tcap) {
  *gcap = *gcap || gcap0;
  const double x0 = scale / gv0;
  if (x0 < upper) return x0;
  for (uint32_t t = 1; t < (uint32_t)kTruncAttempts; ++t) {
    const double gv = hyper_gamma(shape, r, kTruncStride * t, gcap);
    const double x = scale / gv;
    if (x < upper) return x;
  }
  *tcap = true;
  return keep;
}

// The block's warps.  An FP64 instruction keeps a warp's quarter of the SM busy for
// 64 cycles, dependent or not, so what counts is how many of them one warp makes
// in a row (the nu update's lgamma alone about 80), and the warps of different
// quarters make theirs at the same time.  Everything that needs no sums is under
// way while the sums are added up:
//   warp 0  lgamma at the nu update's first 31 points, then (with the sums) the
//           update, then tau
//   warp 1  the logs at the same points, then theta_l and sigma_l^2 (lane l)
//   warp 2  the first gamma draw of every sigma_l^2 (its shape (G-1)/2 is known)
//   warp 3  what needs random numbers alone: the log of the nu update's level, the
//           random quantities of tau's first attempts, the normals of the theta_l
//   warps 4-7  the sums; then warps 4, 5 lgamma and log at the first two
//           proposals that follow each outcome of the nu update's stepping out with
//           at most three steps per side (four sweeps in five need no other)
// A block of 128 threads (the persistent sweep's) adds the sums with all its warps
// first and evaluates the proposals when they are known.
// N=16 G=40000 L=5: 15.6 us (22.1 with the sums first and the update's two
// rounds of densities one after the other).
constexpr int kHyperThreads = 256;
// the partial sums are read by 7 threads per column (126 threads): thread t takes
// column t mod kNumPart and every 7th row from row t / kNumPart
constexpr int kRedThreads = 128;
constexpr int kRedRows = kRedThreads / kNumPart;

__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// The nu update's interval and stepping-out bounds from its first uniforms.
struct NuStart {
  double lo0, hi0;
  int KL, KR;
};

__device__ __forceinline__ NuStart nu_start(double x0, double w, Rng& r, int K) {
  NuStart s;
  const double v = __dmul_rn(w, r.u(1));
  s.lo0 = __dsub_rn(x0, v);
  s.hi0 = __dadd_rn(s.lo0, w);
  s.KL = step_split(K, r.bits(2));
  s.KR = K - s.KL;
  return s;
}

// x moved k times by w (each step rounded, as the slice update's loop moves it).
__device__ __forceinline__ double step_by(double x, double w, int k) {
  for (int i = 0; i < k; ++i) x = __dadd_rn(x, w);
  return x;
}

// Lane's point of the nu update's first round: lane 0 x0, lanes 1..15 the first
// left points, 16..31 the first right ones.
__device__ __forceinline__ double nu_point(const NuStart& s, double x0, double w, int lane) {
  const bool left = lane < 16;
  const double pt = step_by(left ? s.lo0 : s.hi0, left ? -w : w,
                            lane == 0 ? 0 : (left ? lane - 1 : lane - 16));
  return lane == 0 ? x0 : pt;
}

// What the warps hand to the nu update: the logs at the first round's points, the
// log of the level's uniform, and per lane (jl << 3 | jr << 1 | i) the i-th proposal
// after jl steps to the left and jr to the right, with its lgamma and log.
struct NuShared {
  double lt[32], logu;
  double px[32], plg[32], plt[32];
};

// slice_update_warp for nu, with the first round's lgamma in lg (this lane's) and
// logs in nus->lt and, when spec, the first two proposals of the common outcomes in
// nus.  The same points in the same order, so the same result.
__device__ __forceinline__ SliceResult nu_update_warp(double x0, double w, const NuStart& st,
                                                      double pt, double lg, const NuDensity& f,
                                                      const NuShared* nus, bool spec, Rng& r,
                                                      int shrink_max) {
  const int lane = threadIdx.x & 31;
  SliceResult res;
  res.aux = 0.0;
  const bool need = lane == 0 || (lane < 16 ? lane - 1 < st.KL : lane - 16 < st.KR);
  double fv = need ? f.combine(pt, lg, nus->lt[lane]) : 0.0;
  const double f0 = __shfl_sync(0xffffffffu, fv, 0);
  res.nonfinite = !isfinite(f0);
  const double logu = __dadd_rn(f0, nus->logu);
  res.evals = 1;

  // stepping out: a side stops at its first failing point or after K_side points
  double lo = st.lo0, hi = st.hi0;
  bool open_l = st.KL > 0, open_r = st.KR > 0;
  int base_l = 0, base_r = 0;  // index of this round's first point per side
  int steps_l = 0, steps_r = 0;
  for (int round = 0; open_l || open_r; ++round) {
    // points of the round per side, from lanes off_l and 16
    const int nl = round == 0 ? 15 : 16, off_l = round == 0 ? 1 : 0;
    if (round > 0) {
      const bool left = lane < 16;
      const int k = lane & 15;
      const bool act = left ? (open_l && base_l + k < st.KL) : (open_r && base_r + k < st.KR);
      const double q = step_by(left ? lo : hi, left ? -w : w, k);
      fv = act ? f(q) : 0.0;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, logu < fv);
    if (open_l) {
      const int m = min(nl, st.KL - base_l);  // points of this round the loop would reach
      const unsigned fails = ~(bal >> off_l) & ((1u << m) - 1u);
      const int j = fails ? __ffs(fails) - 1 : m;  // passes before the first failure
      res.evals += (unsigned)(j < m ? j + 1 : m);
      lo = step_by(lo, -w, j);
      steps_l += j;
      base_l += m;
      if (j < m || base_l >= st.KL) open_l = false;
    }
    if (open_r) {
      const int m = min(16, st.KR - base_r);
      const unsigned fails = ~(bal >> 16) & ((1u << m) - 1u);
      const int j = fails ? __ffs(fails) - 1 : m;
      res.evals += (unsigned)(j < m ? j + 1 : m);
      hi = step_by(hi, w, j);
      steps_r += j;
      base_r += m;
      if (j < m || base_r >= st.KR) open_r = false;
    }
  }

  // shrinkage: lane j proposes the (base + j)-th point of the rejection chain, first
  // the two proposals known beforehand, then 8, later 32 at a time.  Lane j draws
  // only the uniform of its proposal; every lane walks the chain with the uniforms
  // broadcast from their lanes, keeping its own point, and ends with the bracket
  // left after rejecting all m points.
  if (spec) named_sync(4, 96);  // the proposals of warps 4 and 5
  const int slot = (steps_l << 3) | (steps_r << 1);
  bool pre = spec && steps_l < 4 && steps_r < 4;
  for (int base = 0, width = pre ? 2 : 8; base < shrink_max;) {
    const int m = min(width, shrink_max - base);
    const double u_mine = !pre && lane < m ? r.u(3u + (uint32_t)(base + lane)) : 0.0;
    double xs = pre ? nus->px[slot | (lane & 1)] : 0.0;
    for (int i = 0; i < m; ++i) {
      double xi;
      if (pre) {
        xi = nus->px[slot | i];
      } else {
        const double ui = __shfl_sync(0xffffffffu, u_mine, i);
        xi = __dadd_rn(lo, __dmul_rn(__dsub_rn(hi, lo), ui));
        if (i == lane) xs = xi;
      }
      // the bracket walks on; it is only used when all m are rejected
      if (xi > x0) hi = xi;
      else lo = xi;
    }
    const bool act = lane < m;
    if (!act) fv = -INFINITY;
    else if (pre) fv = f.combine(xs, nus->plg[slot | (lane & 1)], nus->plt[slot | (lane & 1)]);
    else fv = f(xs);
    const unsigned bal = __ballot_sync(0xffffffffu, act && logu < fv);
    if (bal) {
      const int j = __ffs(bal) - 1;
      res.evals += (unsigned)(j + 1);
      res.x = __shfl_sync(0xffffffffu, xs, j);
      res.capped = false;
      return res;
    }
    res.evals += (unsigned)m;
    base += width;
    width = pre ? 8 : 32;
    pre = false;
  }
  res.x = x0;
  res.capped = true;
  return res;
}

// The sums of the partials: thread t < kRedThreads sums column t mod kNumPart over
// rows t / kNumPart + kRedRows k, alternately into two accumulators that are added
// at the end (a fixed order), 16 rows in flight; consecutive threads read
// consecutive words.
__device__ __forceinline__ void hyper_red(const double* partial, int nblk, int t,
                                          double (*red)[kNumPart]) {
  if (t >= kRedRows * kNumPart) return;
  const int col = t % kNumPart, r0 = t / kNumPart;
  constexpr int kPairs = 8;
  double a0 = 0.0, a1 = 0.0;
  for (int b = r0; b < nblk; b += 2 * kPairs * kRedRows) {
    double v0[kPairs], v1[kPairs];
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
      const int row = b + 2 * i * kRedRows;
      if (row < nblk) v0[i] = partial[(size_t)row * kNumPart + col];
      if (row + kRedRows < nblk) v1[i] = partial[(size_t)(row + kRedRows) * kNumPart + col];
    }
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
      const int row = b + 2 * i * kRedRows;
      if (row < nblk) a0 += v0[i];
      if (row + kRedRows < nblk) a1 += v1[i];
    }
  }
  red[r0][col] = a0 + a1;
}

// Steps 3, 4, 6, 7 for one chain, executed by one block of NT threads: the chain's
// `nblk` per-block partial sums are folded in a fixed order.  psi: null, or the top
// level (b, m_1..m_L) of the three-level model, which replaces the rate b of the
// tau prior and the zero mean of the theta_l priors.
template <int NT>
__device__ __forceinline__ void hyper_body(const ModelConst& mc, const double* partial, Hyper* hy,
                                           double* trace_phi, unsigned long long* counters,
                                           int nblk, const double* psi = nullptr) {
  static_assert(NT == kHyperThreads || NT == kRedThreads, "warp roles");
  constexpr bool kWide = NT == kHyperThreads;  // warps 4-7 add the sums meanwhile
  __shared__ double red[kRedRows][kNumPart];
  __shared__ double tot[kNumPart];
  __shared__ double phi_new[kMaxP];
  __shared__ Hyper sh;  // a copy of the chain's Hyper block: one load instead of a
                        // chain of dependent global reads on the serial path
  __shared__ NuShared nus;               // from warps 1, 3, 4, 5 for warp 0
  __shared__ GammaPre tau_pre;           // from warp 3, for warp 0
  __shared__ double theta_z[kMaxL];      // from warp 3, for warp 1
  __shared__ double sig_g[kMaxL];        // from warp 2, for warp 1
  __shared__ int sig_gcap[kMaxL];
  __shared__ double sig_S[kMaxL];        // all_slice: sum (beta - theta_new)^2
  __shared__ double inv_k;               // weight of the draw in the moments
  static_assert(sizeof(Hyper) % 8 == 0, "Hyper is copied as 8-byte words");
  const int L = mc.L, P = mc.P;
  const double G = (double)mc.G;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < (int)(sizeof(Hyper) / 8); i += NT)
    reinterpret_cast<unsigned long long*>(&sh)[i] = reinterpret_cast<const unsigned long long*>(hy)[i];
  const long long it = hy->it + 1;
  const uint32_t it32 = (uint32_t)it;
  if (!kWide) hyper_red(partial, nblk, tid, red);
  __syncthreads();
  auto total = [&](int i) {
    double s = 0.0;
    for (int r = 0; r < kRedRows; ++r) s += red[r][i];
    tot[i] = s;
  };
  if (!kWide) {
    if (tid < kNumPart) total(tid);
    __syncthreads();
  }
  // barriers: 1 sig_g, 2 warp 3's numbers, 3 the sums and the logs at the nu points,
  // 4 the proposals, 5 warps 4-7 among themselves, 6 (all_slice) sig_S
  constexpr int kSumsCount = kWide ? 96 : 64;

  if (warp == 0) {
    // step 3: nu, the slice update spread over warp 0
    const double tau_old = sh.phi[1];
    Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamNu, 0u, it32);
    const double x0 = sh.phi[0], w_nu = sh.w_nu;
    const NuStart start = nu_start(x0, w_nu, r, mc.K);
    const double pt = nu_point(start, x0, w_nu, lane);
    const double lg = lgamma_ol(0.5 * (pt > 0.0 && pt < mc.d ? pt : x0));
    named_sync(2, 96);          // warp 3's numbers
    named_sync(3, kSumsCount);  // the sums, the logs
    const double S1 = tot[0], S2 = tot[1];
    const NuDensity f{G, mc.d, tau_old, S1, S2};
    const SliceResult s = nu_update_warp(x0, w_nu, start, pt, lg, f, &nus, kWide, r, mc.shrink_max);
    const double nu = s.x;
    Rng rt(mc.seed_lo, mc.seed_hi, mc.chain, kStreamTau, 0u, it32);
    const double shape = mc.a + 0.5 * G * nu;
    const double rate = (psi ? psi[0] : mc.b) + 0.5 * nu * S2;
    SliceResult st;
    if (mc.all_slice)  // step 4 by a slice update of the Gamma conditional, on warp 0
      st = slice_update_warp(sh.phi[1], sh.w_hyp[0], TauDensity{shape, rate}, rt, mc.K,
                             mc.shrink_max);
    if (tid == 0) {
      if (it <= sh.burnin) {
        double w = sh.w_nu, waux = sh.waux_nu;
        tune_width(w, waux, it, nu, x0, sh.burnin, sh.tune_start);
        hy->w_nu = w;
        hy->waux_nu = waux;
      }
      atomicAdd(&counters[FBS_CNT_EVALS_NU], (unsigned long long)s.evals);
      if (s.capped) atomicAdd(&counters[FBS_CNT_SLICE_CAPS], 1ull);
      if (s.nonfinite) {
        atomicAdd(&counters[FBS_CNT_NONFINITE], 1ull);
        atomicOr(&hy->flags, kFlagNonfinite);
      }
      // step 4: tau ~ Gamma(a + G nu/2, rate b + nu S2 / 2)
      double tau;
      if (mc.all_slice) {
        tau = st.x;
        if (it <= sh.burnin) {
          double w = sh.w_hyp[0], waux = sh.waux_hyp[0];
          tune_width(w, waux, it, tau, sh.phi[1], sh.burnin, sh.tune_start);
          hy->w_hyp[0] = w;
          hy->waux_hyp[0] = waux;
        }
        atomicAdd(&counters[FBS_CNT_EVALS_HYPER], (unsigned long long)st.evals);
        if (st.capped) atomicAdd(&counters[FBS_CNT_SLICE_CAPS], 1ull);
        if (st.nonfinite) {
          atomicAdd(&counters[FBS_CNT_NONFINITE], 1ull);
          atomicOr(&hy->flags, kFlagNonfinite);
        }
      } else {
        bool gcap = false;
        tau = gamma_mt_pre(shape, &tau_pre, rt, 0, &gcap) / rate;
        if (gcap) atomicAdd(&counters[FBS_CNT_GAMMA_CAPS], 1ull);
      }
      phi_new[0] = nu;
      phi_new[1] = tau;
    }
  } else if (warp == 1) {
    // the logs at the nu update's first points
    {
      Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamNu, 0u, it32);
      const double x0 = sh.phi[0];
      const NuStart st = nu_start(x0, sh.w_nu, r, mc.K);
      const double pt = nu_point(st, x0, sh.w_nu, lane);
      nus.lt[lane] = log_ol(0.5 * (pt > 0.0 && pt < mc.d ? pt : x0) * sh.phi[1]);
    }
    named_sync(2, 96);
    named_sync(3, kSumsCount);
    const int l = lane;
    const bool on = l < L;
    // step 6: theta_l ~ N(v B1 / sigma^2, v), v = 1/(G/sigma^2 + 1/c^2);
    // the partials hold B1' = sum (beta - theta_old), B2' = sum (beta - theta_old)^2
    double th = 0.0, th_old = 0.0, sig2 = 0.0, S = 0.0;
    if (on) {
      th_old = sh.phi[2 + l];
      sig2 = sh.phi[2 + L + l];
      const double B1s = tot[2 + l], B2s = tot[2 + kMaxL + l];
      const double B1 = B1s + G * th_old;
      const double v = 1.0 / (G / sig2 + 1.0 / mc.c2[l]);
      const double mean = psi ? v * (B1 / sig2 + psi[1 + l] / mc.c2[l]) : v * B1 / sig2;
      th = mean + sqrt(v) * theta_z[l];
      const double dl = th - th_old;
      S = B2s - 2.0 * dl * B1s + G * dl * dl;
    }
    if (!mc.all_slice) named_sync(1, 64);  // sig_g from warp 2
    if (on) {
      // step 7: sigma_l^2 ~ IG((G-1)/2, S/2) on (0, s_l^2), S = sum (beta - theta_new)^2
      Rng rs(mc.seed_lo, mc.seed_hi, mc.chain, kStreamSigma, (uint32_t)l, it32);
      if (mc.all_slice) {
        sig_S[l] = S;  // sigma_l by a slice update, on a warp of its own below
      } else {
        double s2n;
        bool gcap = false, tcap = false;
        s2n = hyper_trunc_invgamma(0.5 * (G - 1.0), 0.5 * S, mc.s2[l], sig2, sig_g[l],
                                   sig_gcap[l] != 0, rs, &gcap, &tcap);
        if (gcap) atomicAdd(&counters[FBS_CNT_GAMMA_CAPS], 1ull);
        if (tcap) atomicAdd(&counters[FBS_CNT_TRUNC_CAPS], 1ull);
        phi_new[2 + L + l] = s2n;
      }
      phi_new[2 + l] = th;
    }
  } else if (warp == 2) {
    // the first truncated-draw attempt of every sigma_l^2: a Gamma((G-1)/2) draw
    if (!mc.all_slice) {
      const int l = lane;
      if (l < L) {
        Rng rs(mc.seed_lo, mc.seed_hi, mc.chain, kStreamSigma, (uint32_t)l, it32);
        bool gcap = false;
        sig_g[l] = hyper_gamma(0.5 * (G - 1.0), rs, 0, &gcap);
        sig_gcap[l] = gcap ? 1 : 0;
      }
      named_arrive(1, 64);
    }
  } else if (warp == 3) {
    // lanes 0..1 tau's normals, 8..8+L-1 the theta_l's, lanes 2..3 the logs of tau's
    // acceptance uniforms, lane 4 that of the nu update's level: one log for all,
    // then the normals' square roots and cosines (normal_bm's operations)
    const bool theta = lane >= 8 && lane < 8 + L, tau_n = lane < 2, tau_u = lane == 2 || lane == 3;
    Rng r(mc.seed_lo, mc.seed_hi, mc.chain,
          theta ? kStreamTheta : (lane < 4 ? kStreamTau : kStreamNu), theta ? (uint32_t)(lane - 8) : 0u,
          it32);
    const uint32_t k = tau_n ? 4u * (uint32_t)lane : (tau_u ? 4u * (uint32_t)(lane - 2) + 2u : 0u);
    const double u1 = r.u(k), lu = log_ol(u1);
    if (tau_n || theta) {
      const double u2 = r.u(k + 1u);
      const double z = __dmul_rn(sqrt(__dmul_rn(-2.0, lu)), cos(__dmul_rn(kTwoPi, u2)));
      if (theta) theta_z[lane - 8] = z;
      else tau_pre.x[lane] = z;
    } else if (tau_u) {
      tau_pre.u[lane - 2] = u1;
      tau_pre.logu[lane - 2] = lu;
    } else if (lane == 4) {
      nus.logu = lu;
    }
    __syncwarp();
    named_arrive(2, 96);
  }
  if (kWide && warp >= 4) {
    hyper_red(partial, nblk, tid - kRedThreads, red);
    named_sync(5, 128);
    if (warp == 6) {
      if (lane < kNumPart) total(lane);
      __syncwarp();
      named_arrive(3, kSumsCount);
    } else if (warp < 6) {
      // lane (jl << 3 | jr << 1 | i): proposal i after jl left and jr right steps
      Rng r(mc.seed_lo, mc.seed_hi, mc.chain, kStreamNu, 0u, it32);
      const double x0 = sh.phi[0], w = sh.w_nu;
      const NuStart st = nu_start(x0, w, r, mc.K);
      double lo = step_by(st.lo0, -w, lane >> 3), hi = step_by(st.hi0, w, (lane >> 1) & 3);
      double xs = __dadd_rn(lo, __dmul_rn(__dsub_rn(hi, lo), r.u(3)));
      if (lane & 1) {
        if (xs > x0) hi = xs;
        else lo = xs;
        xs = __dadd_rn(lo, __dmul_rn(__dsub_rn(hi, lo), r.u(4)));
      }
      const double x = 0.5 * (xs > 0.0 && xs < mc.d ? xs : x0);
      if (warp == 4) {
        nus.px[lane] = xs;
        nus.plg[lane] = lgamma_ol(x);
      } else {
        nus.plt[lane] = log_ol(x * sh.phi[1]);
      }
      __syncwarp();
      named_arrive(4, 96);
    }
  }
  if (tid == NT - 1) inv_k = 1.0 / (double)(sh.n_mom + 1);
  if (kWide && mc.all_slice && warp != 0 && warp != 3) {
    // all_slice (never in the 128-thread block of the FP32 form): slice updates of the
    // sigma_l themselves on (0, s_l), each spread over a warp; the state keeps
    // sigma_l^2.  One after the other on a lane each they were the kernel's longest
    // part.
    named_sync(6, 192);  // sig_S
    const int slot = warp < 3 ? warp - 1 : warp - 2;
    for (int l = slot; l < L; l += 6) {
      Rng rs(mc.seed_lo, mc.seed_hi, mc.chain, kStreamSigma, (uint32_t)l, it32);
      const double x0 = sqrt(sh.phi[2 + L + l]);
      const SliceResult ss = slice_update_warp(x0, sh.w_hyp[1 + l],
                                               SigDensity{G, 0.5 * sig_S[l], mc.s[l]}, rs, mc.K,
                                               mc.shrink_max);
      if (lane == 0) {
        phi_new[2 + L + l] = ss.x * ss.x;
        if (it <= sh.burnin) {
          double w = sh.w_hyp[1 + l], waux = sh.waux_hyp[1 + l];
          tune_width(w, waux, it, ss.x, x0, sh.burnin, sh.tune_start);
          hy->w_hyp[1 + l] = w;
          hy->waux_hyp[1 + l] = waux;
        }
        atomicAdd(&counters[FBS_CNT_EVALS_HYPER], (unsigned long long)ss.evals);
        if (ss.capped) atomicAdd(&counters[FBS_CNT_SLICE_CAPS], 1ull);
        if (ss.nonfinite) {
          atomicAdd(&counters[FBS_CNT_NONFINITE], 1ull);
          atomicOr(&hy->flags, kFlagNonfinite);
        }
      }
    }
  }
  __syncthreads();

  const bool mom = it > sh.burnin;
  if (tid < P) {
    const double x = phi_new[tid];
    hy->phi[tid] = x;
    if (mom) {
      const double m = sh.m_phi[tid], q = sh.q_phi[tid];
      hy->m_phi[tid] = m + (x - m) * inv_k;
      hy->q_phi[tid] = q + (x * x - q) * inv_k;
    }
    if (mom && ((it - sh.burnin) % sh.thin == 0) && sh.trace_rows < sh.trace_cap &&
        trace_phi != nullptr)
      trace_phi[(size_t)sh.trace_rows * P + tid] = x;
  }
  __syncthreads();
  if (tid == 0) {
    if (mom && ((it - sh.burnin) % sh.thin == 0) && sh.trace_rows < sh.trace_cap)
      hy->trace_rows = sh.trace_rows + 1;
    if (mom) hy->n_mom = sh.n_mom + 1;
    hy->it = it;
    atomicAdd(&counters[FBS_CNT_SWEEPS], 1ull);
  }
}

}  // namespace fbs
