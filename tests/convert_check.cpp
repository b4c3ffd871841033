// Host check of the FP64 <-> FP32 pair conversions
// (paper_2203_05665_gb300/csrc/h2_convert.hpp) against the plain forms: hi + lo
// within 2^-49 of the value, |lo| <= ulp(hi) / 2, hi and lo equal to the
// rounded ones except at ties of hi, widening exact for every kind of float.
// Exit status 0 on success.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "h2_convert.hpp"

static int bad = 0;

static void split(double v) {
  float hi, lo;
  h2::double_to_pair(v, hi, lo);
  const float ph = (float)v;
  if (!std::isfinite(v)) {
    bad += std::isnan(v) ? !std::isnan(hi) : hi != ph;
    return;
  }
  if (!std::isfinite(ph)) {
    bad += hi != ph;
    return;
  }
  const float pl = (float)(v - (double)ph);
  const double tiny = 1.5e-45;   // FP32's smallest step, below 2^-126
  if (std::fabs(((double)hi + (double)lo) - v) > std::ldexp(std::fabs(v), -49) + tiny) ++bad;
  if (std::fabs((double)lo) > 0.5 * (double)(std::nextafterf(std::fabs(hi), INFINITY) - std::fabs(hi)) + tiny) ++bad;
  if ((hi != ph || lo != pl) && std::fabs(v - (double)ph) != std::fabs(v - (double)hi)) ++bad;
  if (std::signbit(hi) != std::signbit(v)) ++bad;
}

static void wide(float f) {
  const double d = h2::widen(f), r = (double)f;
  if (std::isnan(f) ? !std::isnan(d) : h2::double_bits(d) != h2::double_bits(r)) ++bad;
}

int main() {
  std::mt19937_64 g(7);
  for (int e = -1074; e <= 1023; ++e)
    for (double m : {1.0, 1.0 + 0x1p-52, 2.0 - 0x1p-52, 1.0 + 0x1p-24, 1.0 + 0x1p-23, 1.0 + 3 * 0x1p-24,
                     2.0 - 0x1p-24, 2.0 - 0x1p-25, 1.0 + 0x1p-24 - 0x1p-52, 1.0 + 0x1p-24 + 0x1p-52, 1.5})
      split(std::ldexp(m, e)), split(-std::ldexp(m, e));
  for (int i = 0; i < 4000000; ++i) {
    split(h2::bits_double(g()));
    split(std::ldexp((double)(int64_t)g(), (int)(g() % 200) - 160));
    wide(h2::bits_float((uint32_t)g()));
  }
  for (double v : {0.0, -0.0, (double)INFINITY, -(double)INFINITY, (double)NAN}) split(v);
  for (uint32_t b : {0u, 1u, 0x7fffffu, 0x800000u, 0x7f7fffffu, 0x7f800000u, 0x7fc00000u})
    wide(h2::bits_float(b)), wide(h2::bits_float(b | 0x80000000u));
  std::printf("%d\n", bad);
  return bad != 0;
}
