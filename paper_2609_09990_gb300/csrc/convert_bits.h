// Conversions between FP64, FP32, TF32 and BF16 by integer instructions, for
// the device (and the host, where they are compared with the ordinary ones).
// A conversion to or from FP64 takes the FP64 pipe 64 clocks a warp, as does
// an addition; these take the integer pipe and give the same bits.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define GBD_BOTH __host__ __device__ __forceinline__
#else
#define GBD_BOTH inline
#endif

namespace gbd {
namespace {

GBD_BOTH uint32_t float_bits(float x) {
  uint32_t u;
  memcpy(&u, &x, sizeof(u));
  return u;
}
GBD_BOTH float bits_float(uint32_t u) {
  float x;
  memcpy(&x, &u, sizeof(x));
  return x;
}

// to nearest, ties away from zero
GBD_BOTH float to_tf32(float x) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
#else   // of a finite value
  return bits_float((float_bits(x) + 0x1000u) & 0xFFFFE000u);
#endif
}

// x as FP64
GBD_BOTH double widen(float x) {
  const uint32_t u = float_bits(x), m = u & 0x7FFFFFFFu;
#ifdef __CUDA_ARCH__
  const int lead = __clz(m);
#else
  const int lead = m ? __builtin_clz(m) : 32;
#endif
  const int sh = m < 0x00800000u ? lead - 8 : 0;        // subnormal: to the leading one
  const uint32_t mm = m << sh;
  uint32_t hi = (mm >> 3) + ((896u - sh) << 20);
  hi += m >= 0x7F800000u ? 0x38000000u : 0u;            // infinities, NaN
  hi = (m ? hi : 0u) | (u & 0x80000000u);
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)(mm << 29));
#else
  const uint64_t b = (uint64_t)hi << 32 | (uint32_t)(mm << 29);
  double d;
  memcpy(&d, &b, sizeof(d));
  return d;
#endif
}

// TF32x3 of the FP64 value with the words xh, xl, for a finite one of ordinary
// size (else false): x rounded to FP32 and to TF32, and the rest x - hi (an
// integer of at most 43 bits in units of x's last place) likewise.
GBD_BOTH bool split_tf32(uint32_t xh, uint32_t xl, float* h, float* l) {
  const int e = (int)((xh >> 20) & 0x7FFu) - 896;          // exponent field of the FP32 value
  if (e < 80 || e > 250) return false;
  const uint32_t m23 = (xh & 0xFFFFFu) << 3 | xl >> 29, rest = xl << 3;
  uint32_t f = ((uint32_t)e << 23) + m23;
  f += (rest > 0x80000000u || (rest == 0x80000000u && (m23 & 1u))) ? 1u : 0u;   // to nearest even
  f = (f + 0x1000u) & 0xFFFFE000u;                          // to nearest, ties away
  const int64_t mx = (int64_t)((uint64_t)((xh & 0xFFFFFu) | 0x100000u) << 32 | xl);
  const int64_t mh = (int64_t)(f - ((uint32_t)e << 23) + 0x800000u) << 29;   // a carry into the exponent counts 2^23
  const uint32_t sg = xh & 0x80000000u;
  *h = bits_float(f | sg);
  *l = to_tf32((float)(sg ? mh - mx : mx - mh) * bits_float((uint32_t)(e - 52) << 23));
  return true;
}

// BF16, to nearest even, likewise
GBD_BOTH bool round_bf16(uint32_t xh, uint32_t xl, uint16_t* b) {
  const int e = (int)((xh >> 20) & 0x7FFu) - 896;
  if (e < 1 || e > 253) return false;
  const uint32_t v = (uint32_t)e << 7 | ((xh >> 13) & 0x7Fu), rest = xh << 19 | (xl ? 1u : 0u);
  *b = (uint16_t)((xh >> 31 << 15) | (v + ((rest > 0x80000000u || (rest == 0x80000000u && (v & 1u))) ? 1u : 0u)));
  return true;
}

}  // namespace
}  // namespace gbd
