// Host forms of the FP64 digit kernel's rules (csrc/kernels/f64_digits.h,
// csrc/core/f64_plan.h), for test_f64_rules.py.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <stdexcept>

#include "core/f64_plan.h"
#include "kernels/f64_digits.h"

using namespace dmrg;

static uint64_t bits(double x) {
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
}

// One chunk's sum of a[k] b[k] as the kernel forms it; returns 1 where it is computed
// again by multiply-adds.
extern "C" int f64_chunk(const double* a, const double* b, int K, double* out) {
  int ea = 1, eb = 1;
  for (int k = 0; k < K; ++k) {
    ea = std::max(ea, int(bits(a[k]) >> 52 & 0x7ff));
    eb = std::max(eb, int(bits(b[k]) >> 52 & 0x7ff));
  }
  float acc[8] = {};
  for (int k = 0; k < K; ++k) {
    const uint64_t x = f64_digits(uint32_t(bits(a[k]) >> 32), uint32_t(bits(a[k])), ea);
    const uint64_t y = f64_digits(uint32_t(bits(b[k]) >> 32), uint32_t(bits(b[k])), eb);
    for (int i = 0; i < 8; ++i)
      for (int j = 0; j < 8 - i; ++j)
        acc[i + j] += float((int(x >> (8 * (7 - i)) & 0xff) - 128) * (int(y >> (8 * (7 - j)) & 0xff) - 128));
  }
  int64_t hi;
  uint32_t lo;
  f64_combine(acc[0], acc[1], acc[2], acc[3], acc[4], acc[5], acc[6], acc[7], hi, lo);
  *out = f64_assemble(hi, lo, ea, eb, false);
  bool bad;
  int lead;
  f64_assemble_fast(hi, lo, ea, eb, false, &bad, &lead);
  if (!f64_weak(lead)) return 0;
  *out = 0.0;
  for (int k = 0; k < K; ++k) *out = std::fma(a[k], b[k], *out);
  return 1;
}

// 1 plain, 0 digits, -1 refused
extern "C" int f64_route(int forms, int small, int plain) {
  try {
    return f64_run_plain(forms, small, plain) ? 1 : 0;
  } catch (const std::logic_error&) {
    return -1;
  }
}
