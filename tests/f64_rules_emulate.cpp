// Host forms of the FP64 digit kernel's rules (csrc/kernels/f64_digits.h,
// csrc/core/f64_plan.h), for test_f64_rules.py.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <stdexcept>
#include <vector>

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

// Lists built into those of earlier plans, against fresh ones: 0, or the first that differs.
extern "C" int f64_reused_lists(int seed) {
  std::mt19937 g(static_cast<unsigned>(seed));
  auto rnd = [&](int lo, int hi) { return lo + int(g() % unsigned(hi - lo + 1)); };
  std::vector<double> at(64);
  F64PlanHost kept;
  for (int step = 0; step < 12; ++step) {
    std::vector<GemmProb> p;
    std::vector<GemmSeg> s;
    for (int i = rnd(0, 60); i > 0; --i) {
      GemmProb q{};
      q.C = &at[0];
      q.ldc = 200;
      q.M = rnd(step & 1, 90);
      q.N = rnd(step & 1, 90);
      q.alpha = rnd(0, 1) ? 1.0 : -0.5;
      q.accumulate = rnd(0, 1);
      q.s0 = int(s.size());
      for (int k = rnd(0, i % 7 ? 3 : 50); k > 0; --k)
        s.push_back(GemmSeg{&at[size_t(rnd(0, 3))], &at[size_t(rnd(0, 3))], 90, 90, rnd(step & 1, 40), rnd(0, 1), rnd(0, 1)});
      q.s1 = int(s.size());
      p.push_back(q);
    }
    const int what = rnd(1, 3);
    const F64PlanHost h = f64_build_plan(p, s, 4, what);
    f64_build_plan(kept, p, s, 4, what);
    auto differ = [](const auto& x, const auto& y) {
      return x.size() != y.size() || (x.size() && std::memcmp(x.data(), y.data(), x.size() * sizeof(x[0])));
    };
    if (differ(h.rowref, kept.rowref)) return 1;
    if (differ(h.colref, kept.colref)) return 2;
    if (differ(h.rows, kept.rows)) return 3;
    if (differ(h.units, kept.units)) return 4;
    if (differ(h.tiles, kept.tiles)) return 5;
    if (differ(h.pieces, kept.pieces)) return 6;
    if (differ(h.reds, kept.reds) || h.npart != kept.npart) return 7;
  }
  return 0;
}
