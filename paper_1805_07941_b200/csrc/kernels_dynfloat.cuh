// float <-> n-bit dynamic floating-point codes with p significand bits (Section 2.1, Eq. 2 and 4;
// conversion steps of Section 3), scale alpha = 2^e.  A code is the sign-and-magnitude pattern of
// Eq. 2 in one byte: bit n-1 the sign, then the exponent field E (n-p-1 bits), then the significand.
//   E = 0: value = significand            (spacing 1 up to 2^p)
//   E > 0: value = (2^p + significand) * 2^(E-1)
// so a magnitude a in binade [2^k, 2^(k+1)) is represented with spacing 2^s, s = max(0, k-p), and its code is
// (s << p) + a / 2^s: below 2^(p+1) the pattern IS the value, above it a / 2^s runs from 2^p to 2^(p+1) while the
// exponent field is s + 1.  HBM-bound streaming kernels: 4 bytes in and 1 out per value (encode), 1 in and 4 out
// (decode), as long as the conversion takes few instructions:
//  - encoding scales by 2^-e, clamps to beta_max, and adds 2^(23+s): the float addition rounds a to a multiple of
//    2^s, nearest-even, and leaves a / 2^s in the low bits (a carry into the next binade comes out right by itself);
//    signs are put on four magnitudes at once;
//  - decoding reads the pattern, shifted to where binary32 keeps its exponent, as a float: normal and subnormal
//    patterns of the two types correspond, so the value is that float times a power of two.
// Consecutive threads take consecutive words, four of them at a time.  25.7 M values: encode 92 -> 23 us,
// decode 36 -> 19 us.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace qc {

struct DynFloatFormat {
  int n, p;
  float scale;        // 2^-e
  uint32_t ke_min, ke_up, ke_off;   // (127+p) << 23; (23-p) << 23; that plus (127+p) << p
  float up0, up1, up2;   // 2^126 and two factors with product 2^(p + e)
  float beta_max;     // Eq. 5, as a float (exact: at most p+1 significant bits, exponent <= 126)
};

// Magnitude pattern, p >= 1 (the tie rule is that of the significand's last bit).  With ke the exponent field of
// max(a, 2^p), in place: 2^(23+s) has the bits ke + (23-p) << 23, and s << p is (ke >> (23-p)) - ((127+p) << p).
__device__ __forceinline__ uint32_t dynfloat_mag(float x, const DynFloatFormat& f) {
  // (a product that underflows is far below one half and rounds to zero anyway, one that overflows saturates)
  const float a = fminf(fabsf(x) * f.scale, f.beta_max);
  const uint32_t ke = max(__float_as_uint(a) & 0x7F800000u, f.ke_min);
  const float t = __uint_as_float(ke + f.ke_up) + a;
  const uint32_t mag = (ke >> (23 - f.p)) + __float_as_uint(t) - ke - f.ke_off;
  return x == x ? mag : 0u;
}

// p == 0, no significand bits: the values are the powers of two, code = exponent field.  The parity of the rounded
// quotient says nothing about the parity of the code here, so the tie at 1.5 * 2^k is resolved on the codes
// themselves (k+1 and k+2); below 1 the tie at one half goes to 0.
__device__ __forceinline__ uint32_t dynfloat_mag_p0(float x, const DynFloatFormat& f) {
  if (x != x) return 0u;
  const float a = fminf(fabsf(x) * f.scale, f.beta_max);
  const uint32_t bits = __float_as_uint(a);
  const int k = static_cast<int>(bits >> 23) - 127;
  uint32_t E = a > 0.5f ? 1u : 0u;
  if (k >= 0) {
    const uint32_t fr = bits & 0x7FFFFFu;
    E = static_cast<uint32_t>(k + 1);
    if (fr > 0x400000u || (fr == 0x400000u && (E & 1u))) ++E;
  }
  return E;
}

// Four values -> four codes: magnitudes side by side, then bit n-1 of every byte with a non-zero magnitude (at most
// 127: adding 127 carries into bit 7) whose value is negative.
template <bool P0>
__device__ __forceinline__ uint32_t dynfloat_encode_four(const float4& v, const DynFloatFormat& f) {
  auto mag = [&](float x) { return P0 ? dynfloat_mag_p0(x, f) : dynfloat_mag(x, f); };
  const uint32_t lo = __byte_perm(mag(v.x), mag(v.y), 0x0040), hi = __byte_perm(mag(v.z), mag(v.w), 0x0040);
  const uint32_t mags = __byte_perm(lo, hi, 0x5410);
  const uint32_t slo = __byte_perm(__float_as_uint(v.x), __float_as_uint(v.y), 0x0073);
  const uint32_t shi = __byte_perm(__float_as_uint(v.z), __float_as_uint(v.w), 0x0073);
  const uint32_t signs = __byte_perm(slo, shi, 0x5410) & (mags + 0x7F7F7F7Fu) & 0x80808080u;
  return mags | (signs >> (8 - f.n));
}

__device__ __forceinline__ float dynfloat_decode_one(uint32_t code, const DynFloatFormat& f) {
  const uint32_t mag = code & ((1u << (f.n - 1)) - 1u);
  const float v = __uint_as_float(mag << (23 - f.p)) * f.up0 * f.up1 * f.up2;
  return __uint_as_float(__float_as_uint(v) | ((code >> (f.n - 1)) << 31));
}

constexpr int kCodecUnroll = 4;

template <bool P0>
__global__ void __launch_bounds__(256, 6)
dynfloat_encode_kernel(const float* __restrict__ x, uint8_t* __restrict__ y, size_t count, DynFloatFormat f, int vec_ok) {
  const size_t tid = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const size_t nthreads = static_cast<size_t>(gridDim.x) * blockDim.x;
  const size_t nvec = vec_ok ? count / 4 : 0;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  uint32_t* y4 = reinterpret_cast<uint32_t*>(y);
  auto word = [&](const float4& v) { return dynfloat_encode_four<P0>(v, f); };
  size_t i = tid;
  for (; i + (kCodecUnroll - 1) * nthreads < nvec; i += kCodecUnroll * nthreads) {
    float4 v[kCodecUnroll];
#pragma unroll
    for (int u = 0; u < kCodecUnroll; ++u) v[u] = __ldg(x4 + i + u * nthreads);
#pragma unroll
    for (int u = 0; u < kCodecUnroll; ++u) y4[i + u * nthreads] = word(v[u]);
  }
  for (; i < nvec; i += nthreads) y4[i] = word(__ldg(x4 + i));
  for (size_t j = nvec * 4 + tid; j < count; j += nthreads) y[j] = static_cast<uint8_t>(word(make_float4(x[j], 0.0f, 0.0f, 0.0f)));
}

__global__ void __launch_bounds__(256, 6)
dynfloat_decode_kernel(const uint8_t* __restrict__ c, float* __restrict__ y, size_t count, DynFloatFormat f, int vec_ok) {
  const size_t tid = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const size_t nthreads = static_cast<size_t>(gridDim.x) * blockDim.x;
  const size_t nvec = vec_ok ? count / 4 : 0;
  const uint32_t* c4 = reinterpret_cast<const uint32_t*>(c);
  float4* y4 = reinterpret_cast<float4*>(y);
  auto four = [&](uint32_t w) {
    return make_float4(dynfloat_decode_one(w & 0xFFu, f), dynfloat_decode_one((w >> 8) & 0xFFu, f),
                       dynfloat_decode_one((w >> 16) & 0xFFu, f), dynfloat_decode_one(w >> 24, f));
  };
  size_t i = tid;
  for (; i + (kCodecUnroll - 1) * nthreads < nvec; i += kCodecUnroll * nthreads) {
    uint32_t w[kCodecUnroll];
#pragma unroll
    for (int u = 0; u < kCodecUnroll; ++u) w[u] = __ldg(c4 + i + u * nthreads);
#pragma unroll
    for (int u = 0; u < kCodecUnroll; ++u) y4[i + u * nthreads] = four(w[u]);
  }
  for (; i < nvec; i += nthreads) y4[i] = four(__ldg(c4 + i));
  for (size_t j = nvec * 4 + tid; j < count; j += nthreads) y[j] = dynfloat_decode_one(c[j], f);
}

}  // namespace qc
