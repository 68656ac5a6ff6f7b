// Calibration statistics over one batch of float activations: max |x|, finite / non-finite
// counts, fp64 sum and sum of squares (pass 1) and the histogram of |x| (pass 2) -- the
// hist(abs(x)) that opens Algorithm 1 and the maximum Section 3 uses as default threshold.
//
// Both passes are streams of 4 bytes per value and bound by memory.  Every thread keeps four 16-byte loads in flight
// (one load per iteration left them at 3.9 and 3.2 TB/s), every block of a pass is resident at once, and the second
// walks the tensor from its end, where what the first pass read last is still in the 126 MB L2.  The second pass runs two blocks of 1024 threads per SM
// rather than eight of 256: every block adds its whole histogram to the global one at the end.  Whole call on 25.7 M
// values: 104 -> 61 us, on 1000 values 36 -> 25 us.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include "kernels_simple.cuh"

namespace qc {

constexpr int kCalibMaxBins = 4096;
constexpr int kCalibMaxBlocks = 2048;
constexpr int kCalibBlocksPerSm = 5;  // pass 1: every block resident at once
constexpr int kCalibHistThreads = 1024;

struct CalibHead {
  unsigned int maxabs_bits;          // float bits of max |x| (non-negative floats order as uints)
  unsigned int pad;
  unsigned long long finite;
  unsigned long long nonfinite;
  double sum, sumsq;
};

// What the host reads: the last block of the second pass writes it to pinned host memory itself (a copy of its own would
// cost a launch and a gap, 7 us of a small tensor's 31).
struct CalibResult {
  CalibHead head;
  unsigned long long hist[kCalibMaxBins];
};

// Device scratch shared by the two passes.  The accumulators are zero between calls: the block that finishes a pass
// puts them back, so no call has to clear them first.
struct CalibScratch {
  CalibResult res;
  unsigned int acc_max, ticket;
  unsigned long long acc_nonfinite;
  double part_sum[kCalibMaxBlocks];
  double part_sumsq[kCalibMaxBlocks];
};

// f(float) on every value of x, four 16-byte loads at a time; BACKWARD: from the end of the tensor.
template <bool BACKWARD, class F>
__device__ __forceinline__ void for_each_value(const float* __restrict__ x, size_t count, int vec_ok, F&& f) {
  const size_t tid = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const size_t nthreads = static_cast<size_t>(gridDim.x) * blockDim.x;
  const size_t nvec = vec_ok ? count / 4 : 0;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  auto at = [&](size_t i) { return __ldg(x4 + (BACKWARD ? nvec - 1 - i : i)); };
  auto four = [&](const float4& v) { f(v.x); f(v.y); f(v.z); f(v.w); };
  size_t i = tid;
  for (; i + 3 * nthreads < nvec; i += 4 * nthreads) {
    const float4 a = at(i), b = at(i + nthreads), c = at(i + 2 * nthreads), d = at(i + 3 * nthreads);
    four(a); four(b); four(c); four(d);
  }
  for (; i < nvec; i += nthreads) four(at(i));
  for (size_t j = nvec * 4 + tid; j < count; j += nthreads) f(x[j]);
}

__global__ void __launch_bounds__(256, kCalibBlocksPerSm)
calib_pass1_kernel(const float* __restrict__ x, size_t count, CalibScratch* sc, int nbins, int vec_ok) {
  chain_sync();
  float mx = 0.0f;
  unsigned int nf = 0;
  double s = 0.0, ss = 0.0;
  // the second pass, which starts after this kernel, adds to a clear histogram
  for (int b = blockIdx.x * 256 + threadIdx.x; b < nbins; b += gridDim.x * 256) sc->res.hist[b] = 0ull;
  for_each_value<false>(x, count, vec_ok, [&](float v) {
    const float a = fabsf(v);
    if (a <= 3.402823466e+38f) {     // finite (false for NaN and Inf)
      mx = fmaxf(mx, a);
      const double d = static_cast<double>(v);
      s += d;
      ss = fma(d, d, ss);
    } else {
      nf += 1u;
    }
  });

  // block reduction: warp shuffles, then one partial per warp through shared memory
  __shared__ float s_mx[8];
  __shared__ unsigned int s_nf[8];
  __shared__ double s_s[8], s_ss[8];
  __shared__ bool s_last;
  for (int o = 16; o > 0; o >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    nf += __shfl_xor_sync(0xffffffffu, nf, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { s_mx[warp] = mx; s_nf[warp] = nf; s_s[warp] = s; s_ss[warp] = ss; }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long nft = 0;
    for (int w = 1; w < 8; ++w) { mx = fmaxf(mx, s_mx[w]); s += s_s[w]; ss += s_ss[w]; }
    for (int w = 0; w < 8; ++w) nft += s_nf[w];
    atomicMax(&sc->acc_max, __float_as_uint(mx));
    if (nft) atomicAdd(&sc->acc_nonfinite, nft);
    sc->part_sum[blockIdx.x] = s;
    sc->part_sumsq[blockIdx.x] = ss;
    __threadfence();
    s_last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // The last block sums the blocks' partials with a fixed tree (deterministic for a given grid) and writes the head.
  __threadfence();
  s = 0.0; ss = 0.0;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += 256) { s += __ldcg(&sc->part_sum[b]); ss += __ldcg(&sc->part_sumsq[b]); }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
  if (lane == 0) { s_s[warp] = s; s_ss[warp] = ss; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) { s += s_s[w]; ss += s_ss[w]; }
    const unsigned long long bad = __ldcg(&sc->acc_nonfinite);
    sc->res.head = CalibHead{__ldcg(&sc->acc_max), 0u, static_cast<unsigned long long>(count) - bad, bad, s, ss};
    sc->acc_max = 0u; sc->ticket = 0u; sc->acc_nonfinite = 0ull;
  }
}

// Pass 2: bin = min(nbins-1, (int)(|x| * inv_w)), inv_w = (float)nbins / hi in fp32, one
// multiply.  hi <= 0 on the host side means "use the maximum found by pass 1".  Zeros (half
// of a post-ReLU tensor) are counted in a register instead of hammering one shared counter.
__global__ void __launch_bounds__(kCalibHistThreads, 2)
calib_hist_kernel(const float* __restrict__ x, size_t count, CalibScratch* sc, int nbins,
                  float range_hi, int vec_ok, CalibResult* __restrict__ landing) {
  extern __shared__ unsigned int s_hist[];
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) s_hist[b] = 0u;
  __syncthreads();
  chain_sync();
  const float hi = range_hi > 0.0f ? range_hi : __uint_as_float(__ldcg(&sc->res.head.maxabs_bits));
  const float inv_w = hi > 0.0f ? __fdiv_rn(static_cast<float>(nbins), hi) : 0.0f;
  const float fb = static_cast<float>(nbins);
  unsigned int zeros = 0;
  for_each_value<true>(x, count, vec_ok, [&](float v) {
    const float a = fabsf(v);
    if (!(a <= 3.402823466e+38f)) return;
    const float t = __fmul_rn(a, inv_w);
    const int b = t >= fb ? nbins - 1 : static_cast<int>(t);
    if (b == 0) zeros += 1u; else atomicAdd(&s_hist[b], 1u);
  });
  for (int o = 16; o > 0; o >>= 1) zeros += __shfl_xor_sync(0xffffffffu, zeros, o);
  if ((threadIdx.x & 31) == 0 && zeros) atomicAdd(&s_hist[0], zeros);
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    unsigned int c = s_hist[b];
    if (c) atomicAdd(&sc->res.hist[b], static_cast<unsigned long long>(c));
  }
  if (!landing) return;
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) landing->hist[b] = __ldcg(&sc->res.hist[b]);
  if (threadIdx.x == 0) {
    landing->head = sc->res.head;
    sc->ticket = 0u;
  }
}

}  // namespace qc
