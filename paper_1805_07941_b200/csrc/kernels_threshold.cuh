// Algorithm 1 (Section 3): search of the clamping threshold gamma over the bin edges of a
// histogram of abs(x), as ONE kernel: two warps per candidate i clip the cdf at i, resample it onto the (n, p) grid and
// back and measure the distance to the cdf; the CTA that finishes last takes the smallest measure (the lowest i among
// equal ones).  float64 throughout, every reduction a fixed tree, so that results do not depend on scheduling.
//
// A search is ~4 M evaluations of the resampled cdf, microseconds of arithmetic: what it costs is latency.  Hence
//  - a candidate belongs to two warps: with a CTA per candidate the warps spent most of their time at the barriers
//    around its short serial parts (the grid samples, the reduction);
//  - a CTA's four candidates share the cdf, which every CTA makes itself (exact integer prefix sums) instead of waiting
//    for a kernel that makes it once;
//  - the grid interval a bin falls into comes from the type's own encoding (one float conversion, corrected by two
//    comparisons) instead of a seven-step binary search in shared memory;
//  - on a grid interval the resampled cdf is a line over the bins, two float64 operations per bin, where interpolating
//    twice took two float64 divisions (a kept division, by the total, goes over its reciprocal: div_by);
//  - the arg-min needs no launch and the result no copy of its own.
// 2048 bins: 65 -> 35 us host to host (kernels 31 -> 18 us).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace qc {

constexpr int kThrMaxBins = 4096;
constexpr int kThrMaxLevels = 128;
constexpr int kThrThreads = 256;
constexpr int kThrWarps = kThrThreads / 32;
constexpr int kThrSplit = 2;                             // warps that share a candidate's bins
constexpr int kThrCandidates = kThrWarps / kThrSplit;    // candidates of a CTA

enum : int { kMeasureL1 = 0, kMeasureKS = 1, kMeasureCvM = 2, kMeasureKL = 3 };

struct ThresholdBest {               // (in pinned host memory: the last CTA writes it there itself)
  double delta;
  int index, pad;
};

struct ThresholdShared {
  double fp[kThrMaxLevels], inv_gap[kThrMaxLevels];        // fpspace(0, 1, n, p), reciprocals of its spacings
  // per candidate: where fp[k] lies on the bin axis, the clipped cdf there (r_interp) and its slope per bin up to fp[k+1]
  double pos[kThrCandidates][kThrMaxLevels];
  double2 line[kThrCandidates][kThrMaxLevels];
  int start[kThrCandidates][kThrMaxLevels];                // first bin at or past fp[k]
  double red[kThrThreads];
  unsigned long long part[(kThrMaxBins / kThrThreads) * kThrWarps];       // sums of 32 consecutive bins
  int at[kThrThreads];
  int last;
};

inline size_t threshold_smem(int nbins) { return sizeof(ThresholdShared) + sizeof(double) * static_cast<size_t>(nbins); }

// What a bin's grid interval is found from.
struct ThresholdGrid {
  int levels, p, uniform;            // uniform: p = n - 1, equal spacing
};

// a / b given r = 1 / b rounded to nearest: the remainder of a first quotient corrects it (Markstein: correctly rounded
// whenever r is).
__device__ __forceinline__ double div_by(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-q, b, a), r, q);
}

// q[j] for U bins j, j + 32 kThrSplit, ...: r_interp interpolated back onto linspace(0, 1, i), for -1 <= j < i (at -1 the
// value is of no use, but nothing is read out of bounds).  per_bin: beta_max / (i - 1).  Straight-line code on U bins
// side by side, step by step: a bin is a chain of some ten dependent operations.
template <int U>
__device__ __forceinline__ void resampled(const ThresholdShared& sh, int mine, const ThresholdGrid& g, int j, int last_bin, float per_bin,
                                          double (&q)[U]) {
  int lo[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const float v = static_cast<float>(j + kThrSplit * 32 * u) * per_bin;
    // the pattern of the largest grid value <= v: v itself below 2^(p+1), else exponent and leading significand bits
    const int whole = static_cast<int>(v), coded = static_cast<int>((__float_as_uint(v) - (static_cast<uint32_t>(126 + g.p) << 23)) >> (23 - g.p));
    lo[u] = max(min((g.uniform || v < static_cast<float>(2 << g.p)) ? whole : coded, g.levels - 2), 0);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    // start[lo] <= j < start[lo + 1] (the last interval also holds the last bin); the float may be off by one grid point
    const int jj = j + kThrSplit * 32 * u;
    const int down = sh.start[mine][lo[u]] > jj ? 1 : 0, up = sh.start[mine][lo[u] + 1] <= jj ? 1 : 0;
    lo[u] = max(min(lo[u] - down + up, g.levels - 2), 0);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const double2 l = sh.line[mine][lo[u]];
    const int jj = j + kThrSplit * 32 * u;
    const double v = fma(l.y, static_cast<double>(jj) - sh.pos[mine][lo[u]], l.x);
    // the last kept bin is the last grid point: exactly 1 (the KL measure divides by the step to the clipped bins)
    q[u] = jj == last_bin ? 1.0 : v;
  }
}

template <int MEASURE>
__global__ void __launch_bounds__(kThrThreads)
threshold_search_kernel(const unsigned long long* __restrict__ hist, const double* __restrict__ fp_g, int nbins, int levels, int p,
                        int uniform, float top, int first, double kl_floor, double* __restrict__ deltas,
                        unsigned int* __restrict__ ticket, ThresholdBest* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char thr_smem[];
  ThresholdShared& sh = *reinterpret_cast<ThresholdShared*>(thr_smem);
  double* cdf = reinterpret_cast<double*>(thr_smem + sizeof(ThresholdShared));
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const ThresholdGrid grid{levels, p, uniform};
  for (int k = t; k < levels; k += kThrThreads) {
    const double f = fp_g[k];
    sh.fp[k] = f;
    sh.inv_gap[k] = 1.0 / (k + 1 < levels ? fp_g[k + 1] - f : 1.0);
  }
  // cdf[j] = (h[0] + ... + h[j]) / total: sums inside 32 bins by shuffles, then over the groups of 32
  constexpr int kRows = kThrMaxBins / kThrThreads, kWarps = kThrWarps;
  const int rows = (nbins + kThrThreads - 1) / kThrThreads;
  unsigned long long run[kRows];
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    if (u < rows) {
      const int j = u * kThrThreads + t;
      unsigned long long v = j < nbins ? __ldg(hist + j) : 0ull;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long up = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += up;
      }
      run[u] = v;
      if (lane == 31) sh.part[u * kWarps + warp] = v;
    }
  }
  __syncthreads();
  if (warp == 0) {                                    // exclusive sums over up to 128 groups, 4 per lane
    unsigned long long g4[4], s = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) { const int at = lane * 4 + k; g4[k] = at < rows * kWarps ? sh.part[at] : 0ull; s += g4[k]; }
    unsigned long long before = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long up = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += up;
    }
    before -= s;
#pragma unroll
    for (int k = 0; k < 4; ++k) { const int at = lane * 4 + k; if (at < rows * kWarps) sh.part[at] = before; before += g4[k]; }
    if (lane == 31) sh.red[0] = static_cast<double>(before);
  }
  __syncthreads();
  const double total = sh.red[0], inv_total = 1.0 / total;
#pragma unroll
  for (int u = 0; u < kRows; ++u) {
    const int j = u * kThrThreads + t;
    if (u < rows && j < nbins) cdf[j] = div_by(static_cast<double>(run[u] + sh.part[u * kWarps + warp]), total, inv_total);
  }
  __syncthreads();
  const int mine = warp / kThrSplit, part = warp % kThrSplit;
  const int i = first + blockIdx.x * kThrCandidates + mine;   // candidate: bins [0, i) are kept, gamma = edge i
  if (i <= nbins) {
    const double last = static_cast<double>(i - 1), inv_last = 1.0 / last;
    const float per_bin = top * static_cast<float>(inv_last);
    // r = cdf with r[i-1:] = 1;  r_interp = r[:i] on linspace(0, 1, i), read at the representable points
    // (both warps of a candidate write the same values)
    for (int k = lane; k < levels; k += 32) {
      const double pos = sh.fp[k] * last;
      int j0 = static_cast<int>(pos);
      sh.start[mine][k] = j0 + (pos > static_cast<double>(j0) ? 1 : 0);
      if (j0 > i - 2) j0 = i - 2;
      const double a = cdf[j0];                         // j0 <= i-2: never clipped
      const double b = (j0 + 1 >= i - 1) ? 1.0 : cdf[j0 + 1];
      sh.pos[mine][k] = pos;
      sh.line[mine][k].x = a + (b - a) * (pos - static_cast<double>(j0));
    }
    __syncwarp();
    for (int k = lane; k + 1 < levels; k += 32)
      sh.line[mine][k].y = (sh.line[mine][k + 1].x - sh.line[mine][k].x) * sh.inv_gap[k] * inv_last;
    __syncwarp();
    auto join = [&](double a, double b) { return MEASURE == kMeasureKS ? fmax(a, b) : a + b; };
    // the measure's term at bin j, q and q_before the resampled cdf there and one bin before
    auto term = [&](int j, double q, double q_before) {
      const double c = cdf[j];
      if (MEASURE == kMeasureKL) {
        const double P = c - (j > 0 ? cdf[j - 1] : 0.0);
        return P > 0.0 ? P * log(P / fmax(q - q_before, kl_floor)) : 0.0;
      }
      const double d = fabs(c - q);
      return MEASURE == kMeasureCvM ? d * d : d;
    };
    constexpr int U = 4;
    double acc = 0.0;
    constexpr int kStep = 32 * kThrSplit;
    int j = 32 * part + lane;
    for (; j + kStep * (U - 1) < i; j += kStep * U) {
      double q[U], q_before[U] = {};
      resampled<U>(sh, mine, grid, j, i - 1, per_bin, q);
      if (MEASURE == kMeasureKL) resampled<U>(sh, mine, grid, j - 1, i - 1, per_bin, q_before);
      if (MEASURE == kMeasureKL && j == 0) q_before[0] = 0.0;
#pragma unroll
      for (int u = 0; u < U; ++u) acc = join(acc, term(j + kStep * u, q[u], q_before[u]));
    }
    for (; j < nbins; j += kStep) {                     // the last kept bins one by one, then the clipped ones, where q is 1
      double q[1] = {1.0}, q_before[1] = {1.0};
      if (j < i) resampled<1>(sh, mine, grid, j, i - 1, per_bin, q);
      if (MEASURE == kMeasureKL && j == 0) q_before[0] = 0.0;
      else if (MEASURE == kMeasureKL && j - 1 < i) resampled<1>(sh, mine, grid, j - 1, i - 1, per_bin, q_before);
      acc = join(acc, term(j, q[0], q_before[0]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = join(acc, __shfl_down_sync(0xffffffffu, acc, o));
    if (lane == 0) sh.red[warp] = acc;
  }
  __syncthreads();
  if (t < kThrCandidates && first + static_cast<int>(blockIdx.x) * kThrCandidates + t <= nbins) {
    double v = sh.red[t * kThrSplit];
    for (int k = 1; k < kThrSplit; ++k) v = MEASURE == kMeasureKS ? fmax(v, sh.red[t * kThrSplit + k]) : v + sh.red[t * kThrSplit + k];
    if (MEASURE == kMeasureL1 || MEASURE == kMeasureCvM) v /= static_cast<double>(nbins);
    deltas[first + blockIdx.x * kThrCandidates + t] = v;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) {
    __threadfence();
    sh.last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!sh.last) return;
  // delta starts at infinity and gamma at the last edge; a candidate replaces them only when strictly
  // better, so among equal measures the lowest i wins and a NaN never wins.
  __threadfence();
  double v = INFINITY;
  int at = nbins;
  for (int c = first + t; c <= nbins; c += kThrThreads) {
    const double d = __ldcg(deltas + c);
    if (d < v) { v = d; at = c; }                     // ascending per thread: first minimum kept
  }
  sh.red[t] = v; sh.at[t] = at;
  __syncthreads();
  for (int off = kThrThreads / 2; off > 0; off >>= 1) {
    if (t < off) {
      const double ov = sh.red[t + off];
      const int oi = sh.at[t + off];
      if (ov < sh.red[t] || (ov == sh.red[t] && oi < sh.at[t])) { sh.red[t] = ov; sh.at[t] = oi; }
    }
    __syncthreads();
  }
  if (t == 0) { out->delta = sh.red[0]; out->index = sh.at[0]; *ticket = 0u; }
}

}  // namespace qc
