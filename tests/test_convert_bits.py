"""The integer conversions of the tensor-core operands and sums (FP64 to the
TF32 pair and to BF16, FP32 to FP64) give the bits of the ordinary ones, on
the host: random mantissas, ends of runs, exact ties and one bit beside them,
every exponent they accept and those they leave to the ordinary conversion."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09990_gb300", "csrc")

PROGRAM = r"""
#include "convert_bits.h"
#include <cmath>
#include <cstdio>
#include <random>
using namespace gbd;
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static double real(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static long bad = 0, split = 0, rounded = 0;
static void check(uint64_t u) {
  const double x = real(u);
  const int e = (int)(u >> 52 & 0x7FF) - 896;
  float h, l;
  if (split_tf32((uint32_t)(u >> 32), (uint32_t)u, &h, &l)) {
    ++split;
    const float h2 = to_tf32((float)x), l2 = to_tf32((float)(x - (double)h2));
    bad += float_bits(h) != float_bits(h2) || float_bits(l) != float_bits(l2);
  } else {
    bad += e >= 80 && e <= 250;
  }
  uint16_t b;
  if (round_bf16((uint32_t)(u >> 32), (uint32_t)u, &b)) {
    ++rounded;
    const double y = bits_float((uint32_t)b << 16), dn = bits_float((uint32_t)(uint16_t)(b - 1) << 16),
                 up = bits_float((uint32_t)(uint16_t)(b + 1) << 16);
    const double d = std::fabs(x - y), a = std::fabs(x - dn), c = std::fabs(x - up);
    bad += d > a || d > c || ((d == a || d == c) && (b & 1));   // nearest, ties to even
  } else {
    bad += e >= 1 && e <= 253;
  }
}
int main() {
  std::mt19937_64 g(7);
  const uint64_t full = 0xFFFFFFFFFFFFFull;
  for (int e = 880; e < 1180; ++e)
    for (int i = 0; i < 8000; ++i) {
      uint64_t m = g() & full;
      const int k = g() % 5, at = g() % 52;
      if (k == 1) m &= ~0ull << at;                                     // ends in zeros: ties
      if (k == 2) m |= (1ull << at) - 1;                                // in ones
      if (k == 3) m = (m & ~0ull << at) + (1ull << at) - (g() % 3);     // beside a tie
      if (k == 4) m = full - (g() % 8);                                 // carries into the exponent
      check((g() & 1) << 63 | (uint64_t)e << 52 | (m & full));
    }
  for (uint64_t u : {0ull, 1ull << 63, 0x7FF0000000000000ull, 0xFFF0000000000000ull, 0x7FF8000000000000ull, 1ull, 0x7FEFFFFFFFFFFFFFull})
    check(u);
  for (uint64_t f = 0; f < 1ull << 32; f += 1 + g() % 2000) {
    const float x = bits_float((uint32_t)f);
    const double w = widen(x), o = (double)x;
    bad += !(bits(w) == bits(o) || (w != w && o != o));
  }
  for (uint32_t u : {0u, 0x80000000u, 1u, 0x80000001u, 0x7FFFFFu, 0x800000u, 0x7F7FFFFFu, 0x7F800000u, 0xFF800000u})
    bad += bits(widen(bits_float(u))) != bits((double)bits_float(u));
  bad += !(widen(bits_float(0x7FC00000u)) != widen(bits_float(0x7FC00000u)));
  std::printf("%ld wrong; %ld split, %ld rounded\n", bad, split, rounded);
  return bad || split < 1000000 || rounded < 1500000;
}
"""


def test_bit_for_bit(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
