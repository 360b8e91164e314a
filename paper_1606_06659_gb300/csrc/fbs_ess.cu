// fbs_ess.cu -- effective sample size (Geyer's initial monotone sequence) of
// every series of a [rows][S] trace.
//
// The work is the autocovariances sum_t a_t a_{t+k} of the centred series a at
// the lags k = 0, 1, .. up to the first pair of lags whose sum is not positive.
// In FP64 that is one fused multiply-add per (t, k) at best, 1/64 of the FP32
// rate here, so the sums are made in integers: a is rounded to a fixed-point
// number of 55 bits below the power of two above max |a| (two bits more than the
// largest values have; the rounding, at most 2^-55 max |a|, is what a series with
// outliers loses in its small values), split into a signed high part and a 28-bit
// low part, and the partial products are accumulated exactly in 64 bits: high x high,
// low x low and (high + low) x (high + low) modulo 2^64 (Karatsuba: the third
// less the first two is the sum of the cross products).  The sums being exact, any
// split over threads gives the same result.
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
// same residuals, zero or not, as in ess_series).  A few warps per SM and one chain
// of additions per series: bound by the latency of the reads, so the next 32 rows
// are on their way while 32 are added (30035 series of 1000 rows: fbs_beta_ess 2.0 ms
// with 16 rows unrolled in 32 registers, 1.85 ms so).
__global__ void __launch_bounds__(64) k_ess_mean(const double* __restrict__ tr, long long rows,
                                                 long long S, double* __restrict__ mean) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  constexpr int R = 32;
  const double* x = tr + s;
  const long long full = rows / R * R;
  double m = 0.0, v[R];
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = i < rows ? x[i * S] : 0.0;
  for (long long t = 0; t < full; t += R) {
    double w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) w[i] = t + R + i < rows ? x[(t + R + i) * S] : 0.0;
#pragma unroll
    for (int i = 0; i < R; ++i) m += v[i];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = w[i];
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
    if (full + i < rows) m += v[i];
  mean[s] = m / (double)rows;
}

constexpr int kEssThreads = 128, kEssWarps = kEssThreads / 32;
constexpr int kEssBlocks = 4;  // per SM, where their shared memory fits
constexpr int kEssLags = 16;   // lags per round while all series of a block go on
constexpr int kEssPart = 8;    // lags per thread: 3 x 8 64-bit sums and a window of 8 values
constexpr int kEssPad = 72;    // zero rows behind the series (a window reads up to 64 past the end)
constexpr int kEssMaxRows = 8000;  // shared memory holds 9000
constexpr int kEssBits = 55, kEssLow = 28;  // of a fixed-point value, of its low part

constexpr int kEssFourRows = 1295;  // most rows at which four blocks of 4 series fit an SM

struct Wide {  // a 128-bit integer sum
  long long hi;
  unsigned long long lo;
};

__host__ __device__ constexpr size_t ess_smem_bytes(long long rows, int spb) {
  return (((size_t)(rows + kEssPad) * (spb + 1) * 8 + 15) & ~(size_t)15) +
         (size_t)(kEssWarps / 2) * kEssLags * spb * sizeof(Wide) + (size_t)kEssLags * spb * 8 +
         2 * (size_t)spb * 8 + (size_t)spb * 4 + 16;
}

// an SM's shared memory, 1 KB per block its own
static_assert(kEssBlocks * (ess_smem_bytes(kEssFourRows, 4) + 1024) <= 228 * 1024 &&
                  kEssBlocks * (ess_smem_bytes(kEssFourRows + 1, 4) + 1024) > 228 * 1024,
              "four blocks of 4 series");
static_assert(ess_smem_bytes(kEssMaxRows, 2) <= 227 * 1024, "a block of 2 series");

// Rows that one thread sums at most, of m rows with SPB series per block (odd, so
// that threads on different rows hit different banks).
__host__ __device__ constexpr int ess_thread_rows(int m, int spb) {
  return ((m + kEssThreads / (2 * spb) - 1) / (kEssThreads / (2 * spb))) | 1;
}

// A thread's sums must fit 63 bits (its warp and block add them in 128): with high and
// low parts up to 2^27, of products up to 2^54, and of 2^55 for the cross products.
static_assert(kEssBits - kEssLow == 27 && kEssLow - 1 == 27, "parts up to 2^27");
static_assert(2ll * ess_thread_rows(kEssMaxRows, 2) < 1ll << (63 - 54), "sums of 63 bits");
static_assert(2ll * ess_thread_rows(kEssFourRows, 4) < 1ll << (63 - 54), "sums of 63 bits");

// SPB (4 or 2) series per block.  The block keeps its series in shared memory (one
// read of the trace; row stride SPB + 1, so that threads on different rows hit
// different banks) and goes through the lags in rounds: a thread takes one series,
// 8 lags and a range of rows, holds the 8 values ahead of its row in registers, and
// per row reads two words and issues 24 multiply-adds.  A round takes 16 lags of
// SPB series; before each one the block's threads are dealt out over the series
// that are not finished yet (the lag at which a series ends varies from a few to
// hundreds): half the series, twice the lags, so that every round has the same
// work and no lane waits.  Bound by the 32 x 32 -> 64 multiply-add rate and, at a
// round's end, by barriers, which is why four small blocks share an SM (one works
// while another waits).  fbs_beta_ess of 30035 series of 1000 rows: 145 ms with one
// thread per series in FP64; with 16 series on 512 threads 8.0 ms with the threads
// fixed to their series, 5.8 ms dealt out with 16 lags per round and four
// multiply-adds per lag, 3.3 ms with three, up to 64 lags and the divisions off the
// serial part; 2.7 ms with 8 series on 256 threads, 2.3 ms with 4 on 128,
// 2.0 ms with the largest magnitude found in integers and one scale per series; 1.85
// ms with the means read ahead; 1.81 ms with a thread's three sums per lag joined to
// one of 128 bits before the warp adds them.
template <int SPB>
__global__ void __launch_bounds__(kEssThreads, kEssBlocks)
    k_ess_block(const double* __restrict__ tr, int rows, long long S, int L, int G,
                const double* __restrict__ mean, double* __restrict__ ess) {
  extern __shared__ __align__(16) unsigned char sm_ess[];
  constexpr int ST = SPB + 1, LW = SPB == 4 ? 2 : 1;  // log2 SPB
  int2* A = reinterpret_cast<int2*>(sm_ess);  // [rows + kEssPad][ST]
  double* Ad = reinterpret_cast<double*>(sm_ess);
  Wide* red = reinterpret_cast<Wide*>(sm_ess + (((size_t)(rows + kEssPad) * ST * 8 + 15) & ~(size_t)15));
  double* ckd = reinterpret_cast<double*>(red + kEssWarps / 2 * kEssLags * SPB);  // [kEssLags][SPB]
  double* scale = ckd + kEssLags * SPB;            // [SPB]
  double* c0 = scale + SPB;                        // [SPB] variances
  int* list = reinterpret_cast<int*>(c0 + SPB);    // [SPB] unfinished series
  int* n_list = list + SPB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // centred values and their largest magnitude (compared as integers: the order of
  // the magnitudes, with infinity and NaN above all)
  {
    constexpr int NSEG = kEssThreads / SPB;
    const int sl = tid % SPB, seg = tid / SPB;
    const long long s = (long long)blockIdx.x * SPB + sl;
    const bool on = s < S;
    const double m = on ? mean[s] : 0.0;
    unsigned long long big = 0;
#pragma unroll 4
    for (int t = seg; t < rows; t += NSEG) {
      const double a = on ? tr[(long long)t * S + s] - m : 0.0;
      big = max(big, (unsigned long long)__double_as_longlong(a) & ~(1ull << 63));
      Ad[t * ST + sl] = a;
    }
    for (int t = rows + seg; t < rows + kEssPad; t += NSEG) A[t * ST + sl] = make_int2(0, 0);
#pragma unroll
    for (int o = SPB; o < 32; o <<= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
    if (lane < SPB) reinterpret_cast<unsigned long long*>(red)[warp * SPB + lane] = big;
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
      unsigned long long big = 0;
      for (int w = 0; w < kEssWarps; ++w)
        big = max(big, reinterpret_cast<unsigned long long*>(red)[w * SPB + lane]);
      const double b = __longlong_as_double((long long)big);
      // a constant series (every residual zero) has ess = rows; a range of values
      // that fixed point or its squares do not hold is left to ess_series
      act = mine && b > 0x1p-400 && b < 0x1p400;
      scale[lane] = act ? scalbn(1.0, kEssBits - 1 - ilogb(b)) : 0.0;
      if (mine && !act)
        ess[ess_slot(s_mine, L, G)] = b == 0.0 ? (double)rows : ess_series(tr, rows, S, s_mine);
    }
    __syncwarp();
    deal();
  }
  __syncthreads();
  int n_act = *n_list;

  // fixed point: |a| 2^(kEssBits - 1 - e) <= 2^kEssBits with 2^e <= max |a|
  for (int i = tid; i < rows * SPB; i += kEssThreads) {
    const int at = i / SPB * ST + i % SPB;
    const long long v = __double2ll_rn(Ad[at] * scale[i % SPB]);
    const int hi = (int)((v + (1ll << (kEssLow - 1))) >> kEssLow);
    A[at] = make_int2(hi, (int)(v - ((long long)hi << kEssLow)));
  }
  __syncthreads();

  const double n = (double)rows;
  double sum = 0.0, prev = INFINITY;  // of this lane's series (warp 0)
  for (int k0 = 0, lags; n_act > 0; k0 += lags) {
    // thread: entry q of the list, lags k0 + 8 part .. + 7, rows t0 .. t1 - 1
    const int lw = 32 - __clz(n_act - 1);  // log2 of the list's length, rounded up
    lags = kEssLags << (LW - lw);
    const int q = tid & ((1 << lw) - 1), part = (tid & (2 * SPB - 1)) >> lw;
    const int seg = tid / (2 * SPB);
    const int m = rows - k0;  // terms of lag k0 (the rows past the end are zero)
    const int per = ess_thread_rows(m, SPB);
    const int t0 = seg * per, t1 = min(m, t0 + per);
    long long hh[kEssPart], ll[kEssPart];
    unsigned long long ss[kEssPart];
#pragma unroll
    for (int j = 0; j < kEssPart; ++j) {
      hh[j] = ll[j] = 0;
      ss[j] = 0;
    }
    if (q < n_act && t0 < t1) {
      const int2* a = A + list[q] + t0 * ST;
      const int2* b = a + (k0 + part * kEssPart) * ST;
      int2 w[kEssPart];
      int ws[kEssPart];
#pragma unroll
      for (int j = 0; j < kEssPart; ++j) {
        w[j] = b[j * ST];
        ws[j] = w[j].x + w[j].y;
      }
      auto row = [&](int i) {  // row i of eight: the window starts at w[i]
        const int2 x = a[i * ST];
        const int xs = x.x + x.y;
#pragma unroll
        for (int j = 0; j < kEssPart; ++j) {
          const int2 v = w[(i + j) % kEssPart];
          hh[j] += (long long)x.x * v.x;
          ll[j] += (long long)x.y * v.y;
          ss[j] += (unsigned long long)((long long)xs * ws[(i + j) % kEssPart]);
        }
        w[i] = b[(i + kEssPart) * ST];
        ws[i] = w[i].x + w[i].y;
      };
      int left = t1 - t0;
      for (; left >= kEssPart; left -= kEssPart, a += kEssPart * ST, b += kEssPart * ST) {
#pragma unroll
        for (int i = 0; i < kEssPart; ++i) row(i);
      }
#pragma unroll
      for (int i = 0; i < kEssPart - 1; ++i) {
        if (i >= left) break;
        row(i);
      }
    }
    __int128 sums[kEssPart];
#pragma unroll
    for (int j = 0; j < kEssPart; ++j) {
      const long long cross = (long long)(ss[j] - (unsigned long long)hh[j] - (unsigned long long)ll[j]);
      __int128 v = ((__int128)hh[j] << (2 * kEssLow)) + ((__int128)cross << kEssLow) + ll[j];
#pragma unroll
      for (int o = 2 * SPB; o < 32; o <<= 1) {
        const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
        const long long hi = __shfl_xor_sync(0xffffffffu, (long long)(v >> 64), o);
        v += (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo);
      }
      sums[j] = v;
    }
    // the warps' sums, [lag][series of the list]: the upper half of the warps first,
    // the lower half adds its own
    Wide* slot = red + (size_t)(warp % (kEssWarps / 2)) * kEssLags * SPB + (part * kEssPart << lw) + q;
    const bool writes = lane < 2 * SPB && q < n_act;
#pragma unroll
    for (int step = 0; step < 2; ++step) {
      if (writes && (warp >= kEssWarps / 2) == (step == 0)) {
#pragma unroll
        for (int j = 0; j < kEssPart; ++j) {
          __int128 v = sums[j];
          if (step == 1) v += ((__int128)slot[j << lw].hi << 64) + slot[j << lw].lo;
          slot[j << lw] = Wide{(long long)(v >> 64), (unsigned long long)v};
        }
      }
      __syncthreads();
    }
    {
      // a thread per lag and series: the autocorrelation (the divisions here, not in
      // warp 0's loop below)
      const bool on = tid < kEssLags * SPB && q < n_act;
      const int sl = on ? list[q] : 0;
      double ck = 0.0;
      if (on) {
        __int128 v = 0;
#pragma unroll
        for (int w = 0; w < kEssWarps / 2; ++w) {
          const Wide x = red[w * kEssLags * SPB + tid];
          v += ((__int128)x.hi << 64) + x.lo;
        }
        ck = ((double)(long long)(v >> 64) * 0x1p64 + (double)(unsigned long long)v) / n;
      }
      if (k0 == 0) {
        if (on && tid < 1 << lw) c0[sl] = ck;
        __syncthreads();
      }
      if (on) ckd[tid] = ck / c0[sl];
    }
    __syncthreads();
    if (warp == 0) {
      const unsigned todo = __ballot_sync(0xffffffffu, act);
      if (act) {
        const double* ck = ckd + __popc(todo & ((1u << lane) - 1u));
        bool go = true;
        for (int j = 0; j < lags && go; j += 2) {
          go = false;
          if (k0 + j + 1 >= rows) break;
          double pair = ck[j << lw] + ck[(j + 1) << lw];
          if (!(pair > 0.0)) break;
          if (pair > prev) pair = prev;
          sum += pair;
          prev = pair;
          go = true;
        }
        if (!go || k0 + lags >= rows) {
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

// most: the most rows that come here with SPB series per block
template <int SPB>
cudaError_t launch_block(const double* tr, int rows, int most, long long S, int L, int G,
                         const double* mean, double* ess, cudaStream_t s) {
  cudaError_t e = set_smem_limit(k_ess_block<SPB>, ess_smem_bytes(most, SPB));
  if (e != cudaSuccess) return e;
  k_ess_block<SPB><<<(unsigned)((S + SPB - 1) / SPB), kEssThreads, ess_smem_bytes(rows, SPB), s>>>(
      tr, rows, S, L, G, mean, ess);
  return cudaGetLastError();
}

}  // namespace

// mean: S doubles of scratch.  4 series per block where four such blocks fit an SM
// (1295 rows), else 2 (2000 rows of 15000 series: 2.9 ms against 3.6 ms
// with 4; 4000 rows of 10000: 5.6 against 8.0); longer traces take one thread per
// series.
cudaError_t launch_ess(const double* tr, long long rows, int L, int G, double* mean, double* ess,
                       cudaStream_t s) {
  const long long S = (long long)L * G;
  const int blk = 128;
  const unsigned grid = (unsigned)((S + blk - 1) / blk);
  if (rows > kEssMaxRows) {
    k_ess<<<grid, blk, 0, s>>>(tr, rows, S, L, G, ess);
    return cudaGetLastError();
  }
  k_ess_mean<<<(unsigned)((S + 63) / 64), 64, 0, s>>>(tr, rows, S, mean);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (rows <= kEssFourRows)
    return launch_block<4>(tr, (int)rows, kEssFourRows, S, L, G, mean, ess, s);
  return launch_block<2>(tr, (int)rows, kEssMaxRows, S, L, G, mean, ess, s);
}

}  // namespace fbs
