// Host side of the weight conversions (Section 3 on the CPU): maxima, float -> beta, sums of magnitudes.  These passes
// run over every weight of a network at calibration (25.5 M in ResNet-50), so they are written four to sixteen values
// at a time with the vector instructions every x86-64 has; other hosts take the plain loops.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstdlib>

#if defined(__SSE2__)
#include <emmintrin.h>
#endif

namespace qc {

// float -> beta, any exponent: clamp to +-gamma = beta_max 2^e, scale by 2^-e, round to nearest even; NaN -> 0.
inline int8_t host_quantize_one(float v, int e, int n) {
  const float bmax = static_cast<float>((1 << (n - 1)) - 1);
  if (std::isnan(v)) return 0;
  const float gam = std::ldexp(bmax, e);
  v = std::fmin(std::fmax(v, -gam), gam);
  float r = std::nearbyint(std::ldexp(v, -e));
  r = std::fmin(std::fmax(r, -bmax), bmax);
  return static_cast<int8_t>(r);
}

// Largest finite |w[i]| (0 if none).
inline float host_max_abs(const float* w, size_t count) {
  float g = 0.0f;
  size_t i = 0;
#if defined(__SSE2__)
  const __m128 mask = _mm_castsi128_ps(_mm_set1_epi32(0x7fffffff)), top = _mm_set1_ps(3.402823466e+38f);
  __m128 m0 = _mm_setzero_ps(), m1 = m0;
  for (; i + 8 <= count; i += 8) {
    const __m128 a = _mm_and_ps(_mm_loadu_ps(w + i), mask), b = _mm_and_ps(_mm_loadu_ps(w + i + 4), mask);
    m0 = _mm_max_ps(m0, _mm_and_ps(a, _mm_cmple_ps(a, top)));      // (false for Inf and NaN: they count as 0)
    m1 = _mm_max_ps(m1, _mm_and_ps(b, _mm_cmple_ps(b, top)));
  }
  float lanes[4];
  _mm_storeu_ps(lanes, _mm_max_ps(m0, m1));
  for (float v : lanes) g = v > g ? v : g;
#endif
  for (; i < count; ++i) {
    const float a = std::fabs(w[i]);
    if (std::isfinite(a) && a > g) g = a;
  }
  return g;
}

// beta of `count` values at exponent e.
inline void host_quantize(const float* w, size_t count, int e, int n, int8_t* q) {
  size_t i = 0;
#if defined(__SSE2__)
  // |e| <= 100: gamma and 2^-e are normal, and a product that falls below the normal range is far below one half.
  // The conversion to integers rounds to nearest even, as nearbyint does, and |v| 2^-e <= beta_max needs no clamp.
  if (e >= -100 && e <= 100) {
    const float bmax = static_cast<float>((1 << (n - 1)) - 1);
    const __m128 gam = _mm_set1_ps(std::ldexp(bmax, e)), neg = _mm_set1_ps(-std::ldexp(bmax, e));
    const __m128 inv = _mm_set1_ps(std::ldexp(1.0f, -e));
    auto four = [&](const float* p) {
      __m128 v = _mm_loadu_ps(p);
      v = _mm_and_ps(v, _mm_cmpord_ps(v, v));                      // NaN -> 0
      v = _mm_min_ps(_mm_max_ps(v, neg), gam);
      return _mm_cvtps_epi32(_mm_mul_ps(v, inv));
    };
    for (; i + 16 <= count; i += 16) {
      const __m128i lo = _mm_packs_epi32(four(w + i), four(w + i + 4)), hi = _mm_packs_epi32(four(w + i + 8), four(w + i + 12));
      _mm_storeu_si128(reinterpret_cast<__m128i*>(q + i), _mm_packs_epi16(lo, hi));
    }
  }
#endif
  for (; i < count; ++i) q[i] = host_quantize_one(w[i], e, n);
}

// Sum of |w[i]|.
inline long long host_abs_sum(const int8_t* w, size_t count) {
  long long sum = 0;
  size_t i = 0;
#if defined(__SSE2__)
  __m128i acc = _mm_setzero_si128();
  const __m128i zero = _mm_setzero_si128();
  for (; i + 16 <= count; i += 16) {
    const __m128i v = _mm_loadu_si128(reinterpret_cast<const __m128i*>(w + i));
    const __m128i s = _mm_cmpgt_epi8(zero, v);                     // -1 where negative
    acc = _mm_add_epi64(acc, _mm_sad_epu8(_mm_sub_epi8(_mm_xor_si128(v, s), s), zero));   // (-128 -> 128 as unsigned)
  }
  long long lanes[2];
  _mm_storeu_si128(reinterpret_cast<__m128i*>(lanes), acc);
  sum = lanes[0] + lanes[1];
#endif
  for (; i < count; ++i) sum += std::abs(static_cast<int>(w[i]));
  return sum;
}

}  // namespace qc
