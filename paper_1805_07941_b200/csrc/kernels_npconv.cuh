// Convolution on dynamic floating-point operands (Section 2.1 type, Eq. 6): the pieces around the
// tensor-core GEMM.  The betas of an (n, p) type are integers up to beta_max (Eq. 5: 1984 for (8, 4),
// 245760 for (8, 3)), so the sum of Eq. 6 is an exact integer sum -- but its terms do not fit the int8
// operands of the MMA.  Each beta is therefore written in base 128 with balanced digits,
//   beta = d_0 + 128 d_1 + 128^2 d_2,   d_0, d_1 in [-64, 63], the last digit whatever is left (up to 127 of a one-digit type; of the
// types with two and three digits at most 16, so that a sum of any two digits fits an int8),
// and the product of two betas is taken from products of single digits and of sums of two digits (Karatsuba; see
// np_products in qconv_api.cu).  The kernel below writes the digit combinations of the input that these products need
// as planes side by side along the channel axis.  One tensor-core layer (igemm_i8_kernel<EPI_NP>) then accumulates every
// product in columns of its own (int32, exact), adds them up in 64 bits with their weights, adds the bias, applies ReLU
// and converts to the output type in its epilogue.
// 32 x 28 x 28 x 128 -> 128, 3x3, (8, 4): 115 -> 32 us against one GEMM over all digit pairs with its int32 sums
// written out and combined by a third kernel.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include "epilogue.cuh"
#include "kernels_simple.cuh"

namespace qc {

// Digit combinations of the input: bit i of a mask takes digit i into the plane's sum.
struct NpPlanes {
  int count = 0;
  int mask[6] = {0, 0, 0, 0, 0, 0};
};

// Pattern (without sign) -> beta (Eq. 2 with the exponent field of Eq. 4).
__device__ __forceinline__ int np_decode_mag(int c, int n, int p) {
  if (p == n - 1) return c;
  const int E = c >> p, m = c & ((1 << p) - 1);
  return E == 0 ? m : ((1 << p) + m) << (E - 1);
}

// codes [pixels][C] -> planes [pixels][planes][c_pad], 16 codes per thread.  Decoding, splitting and summing digits take
// some forty instructions per code, so every block first makes a table of what each of the 256 patterns contributes to
// the planes (a byte per plane), and a code costs a lookup and its share of a byte transpose.
__global__ void __launch_bounds__(256)
np_split_kernel(const uint8_t* __restrict__ codes, int8_t* __restrict__ planes, size_t pixels, int C, int c_pad, int n, int p,
                int digits, NpPlanes pl) {
  __shared__ uint32_t table[2][256];                       // planes 0-3, planes 4-5
  {
    const int c = threadIdx.x;
    int beta = np_decode_mag(c & ((1 << (n - 1)) - 1), n, p);
    if ((c >> (n - 1)) & 1) beta = -beta;
    int dig[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (i < digits) {
        // balanced digit in [-64, 63]; the last one keeps what is left
        dig[i] = i + 1 < digits ? ((beta + 64) & 127) - 64 : beta;
        beta = (beta - dig[i]) >> 7;
      }
    }
    uint32_t w[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      // a sum of at most two digits, which stays inside an int8
      const int sum = ((pl.mask[k] & 1) ? dig[0] : 0) + ((pl.mask[k] & 2) ? dig[1] : 0) + ((pl.mask[k] & 4) ? dig[2] : 0);
      w[k >> 2] |= static_cast<uint32_t>(sum & 0xFF) << (8 * (k & 3));
    }
    table[0][c] = w[0];
    table[1][c] = w[1];
  }
  __syncthreads();
  chain_sync();
  const int cv = C / 16;
  const size_t total = pixels * cv;
  for (size_t idx = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; idx < total;
       idx += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t pix = idx / cv;
    const int c0 = static_cast<int>(idx - pix * cv) * 16;
    if (!QC_IN(pix * C + c0 + 15, pixels * C)) continue;
    const uint4 raw = __ldg(reinterpret_cast<const uint4*>(codes + pix * C + c0));
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
    int8_t* dst = planes + pix * static_cast<size_t>(pl.count) * c_pad + c0;
    for (int half = 0; half * 4 < pl.count; ++half) {
      uint32_t o[4][4];                                    // [plane][word]
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t t[4];
        transpose4x4(table[half][w[j] & 0xFFu], table[half][(w[j] >> 8) & 0xFFu], table[half][(w[j] >> 16) & 0xFFu],
                     table[half][w[j] >> 24], t);
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k][j] = t[k];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int plane = 4 * half + k;
        if (plane < pl.count && QC_IN(pix * pl.count * c_pad + static_cast<size_t>(plane) * c_pad + c0 + 15, pixels * pl.count * c_pad))
          *reinterpret_cast<uint4*>(dst + static_cast<size_t>(plane) * c_pad) = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
      }
    }
  }
}

}  // namespace qc
