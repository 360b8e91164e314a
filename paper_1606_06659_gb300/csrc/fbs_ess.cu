// fbs_ess.cu -- effective sample size (Geyer's initial monotone sequence) of
// every series of a [rows][S] trace.
//
// The work is the autocovariances sum_t a_t a_{t+k} of the centred series a at
// the lags k = 0, 1, .. up to the first pair of lags whose sum is not positive.
// In FP64 that is one fused multiply-add per (t, k) at best, 1/64 of the FP32
// rate here, so the sums are made in integers: a is rounded to a fixed-point
// number of 50 bits below the power of two above max |a| (the rounding is at
// most 2^-51 of that power, against the 2^-53 |partial sum| which every FP64
// addition of the sum makes), split into a signed high part and a 26-bit low
// part, and the four partial products are accumulated exactly in 64 bits.  The
// sums being exact, any split over threads gives the same result.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fbs_common.cuh"
#include "fbs_kernels.h"

namespace fbs {

namespace {

// One series in FP64, row by row: any number of rows, any range of values.
__device__ double ess_series(const double* __restrict__ tr, long long n, long long S,
                             long long s) {
  double mean = 0.0;
  for (long long t = 0; t < n; ++t) mean += tr[t * S + s];
  mean /= (double)n;
  double c0 = 0.0;
  for (long long t = 0; t < n; ++t) {
    const double dv = tr[t * S + s] - mean;
    c0 += dv * dv;
  }
  c0 /= (double)n;
  if (!(c0 > 0.0)) return (double)n;
  double sum = 0.0, prev = INFINITY;
  for (long long j = 0; 2 * j + 1 < n; ++j) {
    double pair = 0.0;
    for (long long k = 2 * j; k <= 2 * j + 1; ++k) {
      double ck = 0.0;
      for (long long t = 0; t + k < n; ++t)
        ck += (tr[t * S + s] - mean) * (tr[(t + k) * S + s] - mean);
      pair += ck / (double)n / c0;
    }
    if (!(pair > 0.0)) break;
    if (pair > prev) pair = prev;
    sum += pair;
    prev = pair;
  }
  double tau = -1.0 + 2.0 * sum;
  if (tau < 1.0 / (double)n) tau = 1.0 / (double)n;
  return (double)n / tau;
}

// Series s = l G + g of the trace goes to ess[g L + l] (gene-major).
__device__ __forceinline__ long long ess_slot(long long s, int L, int G) {
  return (s % G) * L + s / G;
}

// One thread per series, for traces of more rows than a block holds.
__global__ void k_ess(const double* __restrict__ tr, long long rows, long long S, int L, int G,
                      double* ess) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < S) ess[ess_slot(s, L, G)] = ess_series(tr, rows, S, s);
}

// The mean of every series, rows added in order (a constant series then has the
// same residuals, zero or not, as in ess_series).
__global__ void k_ess_mean(const double* __restrict__ tr, long long rows, long long S,
                           double* __restrict__ mean) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  double m = 0.0;
#pragma unroll 8
  for (long long t = 0; t < rows; ++t) m += tr[t * S + s];
  mean[s] = m / (double)rows;
}

constexpr int kEssThreads = 512, kEssWarps = kEssThreads / 32;
constexpr int kEssLags = 16;   // lags per round
constexpr int kEssHalf = 8;    // lags per thread: 3 x 8 64-bit sums and a window of 8 values
constexpr int kEssPad = 48;    // zero rows behind the series (a window reads up to 31 past the end)
constexpr int kEssMaxRows = 5000;  // 2^50 rows < 2^63 needs rows < 8192; shared memory less

struct Wide {  // a 128-bit integer sum
  long long hi;
  unsigned long long lo;
};

__host__ __device__ constexpr size_t ess_smem_bytes(long long rows, int spb) {
  return (((size_t)(rows + kEssPad) * (spb + 1) * 8 + 15) & ~(size_t)15) +
         (size_t)(kEssWarps / 2) * kEssLags * spb * sizeof(Wide) + (size_t)kEssLags * spb * 8 +
         (size_t)spb * 8 + (size_t)spb * 4 + 16;
}

// SPB series per block.  The block keeps its series in shared memory (one read of
// the trace; row stride SPB + 1, so that threads on different rows hit different
// banks) and goes through the lags 16 at a time: a thread takes one series, 8 of
// the lags and a range of rows, holds the 8 values ahead of its row in
// registers, and per row reads two words and issues 32 multiply-adds.  Before
// each round the block's threads are dealt out over the series that are not
// finished yet (the lag at which a series ends varies from a few to hundreds),
// so that the long ones get more threads and no lane waits.  Bound by the
// 32 x 32 -> 64 multiply-add rate.  fbs_beta_ess of 30035 series of 1000 rows:
// 145 ms with one thread per series in FP64, 8.0 ms with the threads fixed to
// their series, 5.8 ms so.
template <int SPB>
__global__ void __launch_bounds__(kEssThreads) k_ess_block(const double* __restrict__ tr, int rows,
                                                           long long S, int L, int G,
                                                           const double* __restrict__ mean,
                                                           double* __restrict__ ess) {
  extern __shared__ __align__(16) unsigned char sm_ess[];
  constexpr int ST = SPB + 1;
  int2* A = reinterpret_cast<int2*>(sm_ess);  // [rows + kEssPad][ST]
  double* Ad = reinterpret_cast<double*>(sm_ess);
  Wide* red = reinterpret_cast<Wide*>(sm_ess + (((size_t)(rows + kEssPad) * ST * 8 + 15) & ~(size_t)15));
  double* ckd = reinterpret_cast<double*>(red + kEssWarps / 2 * kEssLags * SPB);  // [kEssLags][SPB]
  double* mx = ckd + kEssLags * SPB;               // [SPB]
  int* list = reinterpret_cast<int*>(mx + SPB);    // [SPB] unfinished series
  int* n_list = list + SPB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // centred values and their largest magnitude
  {
    constexpr int NSEG = kEssThreads / SPB;
    const int sl = tid % SPB, seg = tid / SPB;
    const long long s = (long long)blockIdx.x * SPB + sl;
    const bool on = s < S;
    const double m = on ? mean[s] : 0.0;
    double big = 0.0;
    int bad = 0;
#pragma unroll 4
    for (int t = seg; t < rows; t += NSEG) {
      const double a = on ? tr[(long long)t * S + s] - m : 0.0;
      bad |= !isfinite(a);
      big = fmax(big, fabs(a));
      Ad[t * ST + sl] = a;
    }
    for (int t = rows + seg; t < rows + kEssPad; t += NSEG) A[t * ST + sl] = make_int2(0, 0);
#pragma unroll
    for (int o = SPB; o < 32; o <<= 1) {
      big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if (bad) big = INFINITY;
    if (lane < SPB) reinterpret_cast<double*>(red)[warp * SPB + lane] = big;
  }
  __syncthreads();

  // lane i of warp 0 holds series i of the block from here on
  const long long s_mine = (long long)blockIdx.x * SPB + lane;
  const bool mine = warp == 0 && lane < SPB && s_mine < S;
  bool act = false;
  auto deal = [&]() {  // warp 0: the unfinished series, in order
    const unsigned todo = __ballot_sync(0xffffffffu, act);
    if (act) list[__popc(todo & ((1u << lane) - 1u))] = lane;
    if (lane == 0) *n_list = __popc(todo);
  };
  if (warp == 0) {
    if (lane < SPB) {
      double b = 0.0;
      for (int w = 0; w < kEssWarps; ++w) b = fmax(b, reinterpret_cast<double*>(red)[w * SPB + lane]);
      mx[lane] = b;
      // a constant series (every residual zero) has ess = rows; a range of values
      // that fixed point or its squares do not hold is left to ess_series
      act = mine && b > 0x1p-400 && b < 0x1p400;
      if (mine && !act)
        ess[ess_slot(s_mine, L, G)] = b == 0.0 ? (double)rows : ess_series(tr, rows, S, s_mine);
    }
    __syncwarp();
    deal();
  }
  __syncthreads();
  int n_act = *n_list;

  // fixed point: |a| 2^(49 - e) <= 2^50 with 2^e <= max |a|
  for (int i = tid; i < rows * n_act; i += kEssThreads) {
    const int sl = list[i % n_act], at = (i / n_act) * ST + sl;
    const long long v = __double2ll_rn(Ad[at] * scalbn(1.0, 49 - ilogb(mx[sl])));
    const int hi = (int)((v + (1ll << 25)) >> 26);
    A[at] = make_int2(hi, (int)(v - ((long long)hi << 26)));
  }
  __syncthreads();

  const double n = (double)rows;
  double c0 = 0.0, sum = 0.0, prev = INFINITY;  // of this lane's series (warp 0)
  for (int k0 = 0; n_act > 0; k0 += kEssLags) {
    // thread: entry q of the list, lags k0 + 8 half .. + 7, rows t0 .. t1 - 1
    const int lw = 32 - __clz(n_act - 1);  // log2 of the list's length, rounded up
    const int q = tid & ((1 << lw) - 1), half = (tid >> lw) & 1, seg = tid >> (lw + 1);
    const int m = rows - k0;  // terms of lag k0 (the rows past the end are zero)
    const int nseg = kEssThreads >> (lw + 1);
    const int per = ((m + nseg - 1) / nseg) | 1;  // odd: threads on different banks
    const int t0 = seg * per, t1 = min(m, t0 + per);
    long long hh[kEssHalf], md[kEssHalf], ll[kEssHalf];
#pragma unroll
    for (int j = 0; j < kEssHalf; ++j) hh[j] = md[j] = ll[j] = 0;
    if (q < n_act && t0 < t1) {
      const int2* a = A + list[q];
      const int k = k0 + half * kEssHalf;
      int2 w[kEssHalf];
#pragma unroll
      for (int j = 0; j < kEssHalf; ++j) w[j] = a[(t0 + k + j) * ST];
      for (int tb = t0; tb < t1; tb += kEssHalf) {
#pragma unroll
        for (int i = 0; i < kEssHalf; ++i) {
          int2 x = a[(tb + i) * ST];
          if (tb + i >= t1) x = make_int2(0, 0);
#pragma unroll
          for (int j = 0; j < kEssHalf; ++j) {
            const int2 v = w[(i + j) % kEssHalf];
            hh[j] += (long long)x.x * v.x;
            ll[j] += (long long)x.y * v.y;
          }
#pragma unroll
          for (int j = 0; j < kEssHalf; ++j) md[j] += (long long)x.x * w[(i + j) % kEssHalf].y;
#pragma unroll
          for (int j = 0; j < kEssHalf; ++j) md[j] += (long long)x.y * w[(i + j) % kEssHalf].x;
          w[i] = a[(tb + i + k + kEssHalf) * ST];
        }
      }
    }
    for (int o = 2 << lw; o < 32; o <<= 1) {
#pragma unroll
      for (int j = 0; j < kEssHalf; ++j) {
        hh[j] += __shfl_xor_sync(0xffffffffu, hh[j], o);
        md[j] += __shfl_xor_sync(0xffffffffu, md[j], o);
        ll[j] += __shfl_xor_sync(0xffffffffu, ll[j], o);
      }
    }
    // the warps' sums: the upper half of the warps first, the lower half adds its own
    Wide* slot = red + ((size_t)(warp % (kEssWarps / 2)) * kEssLags + half * kEssHalf) * SPB + q;
    const bool writes = lane < (2 << lw) && q < n_act;
#pragma unroll
    for (int step = 0; step < 2; ++step) {
      if (writes && (warp >= kEssWarps / 2) == (step == 0)) {
#pragma unroll
        for (int j = 0; j < kEssHalf; ++j) {
          __int128 v = ((__int128)hh[j] << 52) + ((__int128)md[j] << 26) + ll[j];
          if (step == 1) v += ((__int128)slot[j * SPB].hi << 64) + slot[j * SPB].lo;
          slot[j * SPB] = Wide{(long long)(v >> 64), (unsigned long long)v};
        }
      }
      __syncthreads();
    }
    for (int i = tid; i < kEssLags * SPB; i += kEssThreads) {
      if (i % SPB >= n_act) continue;
      __int128 v = 0;
#pragma unroll
      for (int w = 0; w < kEssWarps / 2; ++w) {
        const Wide x = red[w * kEssLags * SPB + i];
        v += ((__int128)x.hi << 64) + x.lo;
      }
      ckd[i] = (double)(long long)(v >> 64) * 0x1p64 + (double)(unsigned long long)v;
    }
    __syncthreads();
    if (warp == 0) {
      const unsigned todo = __ballot_sync(0xffffffffu, act);
      if (act) {
        const double* ck = ckd + __popc(todo & ((1u << lane) - 1u));
        if (k0 == 0) c0 = ck[0] / n;
        bool go = true;
        for (int j = 0; j < kEssLags && go; j += 2) {
          go = false;
          if (k0 + j + 1 >= rows) break;
          double pair = ck[j * SPB] / n / c0 + ck[(j + 1) * SPB] / n / c0;
          if (!(pair > 0.0)) break;
          if (pair > prev) pair = prev;
          sum += pair;
          prev = pair;
          go = true;
        }
        if (!go || k0 + kEssLags >= rows) {
          double tau = -1.0 + 2.0 * sum;
          if (tau < 1.0 / n) tau = 1.0 / n;
          ess[ess_slot(s_mine, L, G)] = n / tau;
          act = false;
        }
      }
      __syncwarp();
      deal();
    }
    __syncthreads();
    n_act = *n_list;
  }
}

template <int SPB>
cudaError_t launch_block(const double* tr, int rows, long long S, int L, int G,
                         const double* mean, double* ess, cudaStream_t s) {
  const size_t smem = ess_smem_bytes(rows, SPB);
  cudaError_t e = cudaFuncSetAttribute(k_ess_block<SPB>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_ess_block<SPB><<<(unsigned)((S + SPB - 1) / SPB), kEssThreads, smem, s>>>(tr, rows, S, L, G,
                                                                             mean, ess);
  return cudaGetLastError();
}

}  // namespace

// mean: S doubles of scratch.  16 series per block where their rows fit its
// shared memory (about 1400) and the blocks then fill the chip, else 8 (2900) or
// 4 (5000); longer traces take one thread per series.
cudaError_t launch_ess(const double* tr, long long rows, int L, int G, double* mean, double* ess,
                       cudaStream_t s) {
  constexpr size_t kSmem = 227 * 1024;
  constexpr long long kBlocks = 152;
  const long long S = (long long)L * G;
  const int blk = 128;
  const unsigned grid = (unsigned)((S + blk - 1) / blk);
  if (rows > kEssMaxRows) {
    k_ess<<<grid, blk, 0, s>>>(tr, rows, S, L, G, ess);
    return cudaGetLastError();
  }
  k_ess_mean<<<grid, blk, 0, s>>>(tr, rows, S, mean);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (ess_smem_bytes(rows, 16) <= kSmem && S >= 16 * kBlocks)
    return launch_block<16>(tr, (int)rows, S, L, G, mean, ess, s);
  if (ess_smem_bytes(rows, 8) <= kSmem && S >= 8 * kBlocks)
    return launch_block<8>(tr, (int)rows, S, L, G, mean, ess, s);
  return launch_block<4>(tr, (int)rows, S, L, G, mean, ess, s);
}

}  // namespace fbs
