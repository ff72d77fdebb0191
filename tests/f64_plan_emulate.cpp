// Host interpreter of the FP64 tensor-core work list (csrc/core/f64_plan.h): walks the
// units and reductions as the kernel does, with the same digit arithmetic
// (kernels/f64_digits.h), and checks every operand access against the caller's arena.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "core/f64_plan.h"
#include "kernels/f64_digits.h"

using namespace dmrg;

namespace {
struct Bad {};
struct Octet { int s, k, n; };
}  // namespace

// The plain form (tiles): every element one chain of fused multiply-adds over its
// segments and k.  Returns 0, or the code of the first broken rule.
extern "C" int f64_emulate_plain(const GemmProb* p, int np, const GemmSeg* s, int ns, const double* lo,
                                 const double* hi, int what) {
  const F64PlanHost h = f64_build_plan(std::vector<GemmProb>(p, p + np), std::vector<GemmSeg>(s, s + ns), 4, what);
  if (h.tiles.empty()) return 0;
  if (h.pieces.size() != h.tiles.size() + 1) return 1;
  for (size_t i = 0; i < h.tiles.size(); ++i) {
    const F64Unit& u = h.tiles[i];
    if (h.pieces[i + 1] - h.pieces[i] != (u.rows + F64_PR - 1) / F64_PR * ((u.nt + F64_PC - 1) / F64_PC)) return 2;
    for (int r = 0; r < u.rows; ++r)
      for (int c = 0; c < u.nt; ++c) {
        int pos = u.pos0;
        while (pos + 1 < u.pos0 + u.npos && h.rows[size_t(pos) + 1].pre <= u.row0 + r) ++pos;
        const F64Row& R = h.rows[size_t(pos)];
        const int m = u.row0 + r - R.pre;
        if (m < 0 || m >= (R.m2 >> 1)) return 4;
        double acc = 0;
        for (int sg = 0; sg < u.nseg; ++sg) {
          const F64Ref &a = h.rowref[size_t(R.s0 + sg)], &b = h.colref[size_t(u.cs + sg)];
          for (int k = 0; k < (a.kt >> 1); ++k) {
            const double* x = a.p + ((a.kt & 1) ? int64_t(k) * a.ld + m : int64_t(m) * a.ld + k);
            const double* y = b.p + ((b.kt & 1) ? int64_t(k) * b.ld + u.n0 + c : int64_t(u.n0 + c) * b.ld + k);
            if (x < lo || x >= hi || y < lo || y >= hi) return 6;
            acc = std::fma(*x, *y, acc);
          }
        }
        double* o = u.trans ? R.C + m + int64_t(u.n0 + c) * R.ldc : R.C + int64_t(m) * R.ldc + u.n0 + c;
        *o = (R.m2 & 1) ? *o + R.alpha * acc : R.alpha * acc;
      }
  }
  return 0;
}

// returns 0, or the code of the first broken rule; stat3 = units, reductions, log2 of
// the largest digit sum among the weights that have to be exact
extern "C" int f64_emulate(const GemmProb* p, int np, const GemmSeg* s, int ns, int nsm, const double* lo,
                           const double* hi, double* stat3) {
  const F64PlanHost h = f64_build_plan(std::vector<GemmProb>(p, p + np), std::vector<GemmSeg>(s, s + ns), nsm);
  std::vector<double> part(size_t(h.npart), NAN);
  double top = 0;
  auto at = [&](const F64Ref& f, int r, int k) {
    const double* x = f.p + ((f.kt & 1) ? int64_t(k) * f.ld + r : int64_t(r) * f.ld + k);
    if (x < lo || x >= hi) throw Bad();
    return *x;
  };
  auto find = [&](int pos0, int npos, int rr) {
    int pos = pos0;
    while (pos + 1 < pos0 + npos && h.rows[size_t(pos) + 1].pre <= rr) ++pos;
    return pos;
  };
  auto field = [](double x) {
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return int((b >> 52) & 0x7ff);
  };
  auto digits = [](double x, int e, int* d) {
    uint64_t b;
    std::memcpy(&b, &x, 8);
    const uint64_t y = f64_digits(uint32_t(b >> 32), uint32_t(b), e);
    for (int j = 0; j < 8; ++j) d[j] = int((y >> (8 * (7 - j))) & 0xff) - 128;
  };
  try {
    for (const F64Unit& u : h.units) {
      if (u.rows < 1 || u.rows > F64_TM || u.nt < 1 || u.nt > F64_TN || u.npos < 1 || u.npos > F64_TM) return 2;
      std::vector<Octet> oc;
      for (int sg = u.sg, k = u.k0; int(oc.size()) < u.noct; k = 0, ++sg) {
        if (sg >= u.nseg) return 3;
        const int K = h.colref[size_t(u.cs + sg)].kt >> 1;
        for (; k < K && int(oc.size()) < u.noct; k += 8) oc.push_back({sg, k, std::min(8, K - k)});
      }
      for (int r = 0; r < u.rows; ++r) {
        const int pos = find(u.pos0, u.npos, u.row0 + r);
        const F64Row& R = h.rows[size_t(pos)];
        const int m = u.row0 + r - R.pre;
        if (m < 0 || m >= (R.m2 >> 1)) return 4;
        for (int c = 0; c < u.nt; ++c) {
          double* out = u.part >= 0 ? &part.at(size_t(u.part + int64_t(F64_TM) * c + r))
                                    : (u.trans ? R.C + m + int64_t(u.n0 + c) * R.ldc : R.C + int64_t(m) * R.ldc + u.n0 + c);
          const double alpha = u.part >= 0 ? 1.0 : R.alpha;
          for (size_t o0 = 0; o0 == 0 || o0 < oc.size(); o0 += F64_CHUNK) {
            const size_t o1 = std::min(oc.size(), o0 + F64_CHUNK);
            int ea = 1, eb = 1;
            std::vector<double> x, y;
            for (size_t o = o0; o < o1; ++o)
              for (int k = 0; k < oc[o].n; ++k) {
                const F64Ref &fa = h.rowref[size_t(R.s0 + oc[o].s)], &fb = h.colref[size_t(u.cs + oc[o].s)];
                if ((fa.kt >> 1) != (fb.kt >> 1)) return 5;
                x.push_back(at(fa, m, oc[o].k + k));
                y.push_back(at(fb, u.n0 + c, oc[o].k + k));
                ea = std::max(ea, field(x.back()));
                eb = std::max(eb, field(y.back()));
              }
            double v = 0;
            if (ea == F64_SPECIAL || eb == F64_SPECIAL) {
              for (size_t k = 0; k < x.size(); ++k) v = std::fma(x[k], y[k], v);
            } else if (!x.empty()) {
              int64_t acc[8] = {};
              for (size_t k = 0; k < x.size(); ++k) {
                int a[8], b[8];
                digits(x[k], ea, a);
                digits(y[k], eb, b);
                for (int i = 0; i < 8; ++i)
                  for (int j = 0; j < 8 - i; ++j) acc[i + j] += a[i] * b[j];
              }
              for (int w = 0; w < 6; ++w) top = std::max(top, std::fabs(double(acc[w])));
              int64_t H;
              uint32_t L;
              float f[8];
              for (int w = 0; w < 8; ++w) f[w] = float(acc[w]);
              f64_combine(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], H, L);
              v = f64_assemble(H, L, ea, eb, false);
              bool bad;
              const double w = f64_assemble_fast(H, L, ea, eb, true, &bad);
              if (!bad && !(w == -v)) return 8;
              if (bad && std::fabs(v) > 1e-307 && std::fabs(v) < 4e307) return 9;
            }
            v *= alpha;
            const bool old = o0 > 0 || (u.part < 0 && (R.m2 & 1));
            *out = old ? *out + v : v;
          }
        }
      }
    }
    for (const F64Red& t : h.reds)
      for (int r = 0; r < t.rows; ++r)
        for (int c = 0; c < t.nt; ++c) {
          double v = part.at(size_t(t.part + int64_t(F64_TM) * c + r));
          for (int q = 1; q < t.nparts; ++q) v += part.at(size_t(t.part + (int64_t(q) * t.n16 + c) * F64_TM + r));
          int pos = t.pos0;
          while (h.rows[size_t(pos)].pre + (h.rows[size_t(pos)].m2 >> 1) <= t.row0 + r) ++pos;
          const F64Row& R = h.rows[size_t(pos)];
          const int m = t.row0 + r - R.pre;
          double* out = t.trans ? R.C + m + int64_t(t.n0 + c) * R.ldc : R.C + int64_t(m) * R.ldc + t.n0 + c;
          *out = (R.m2 & 1) ? *out + R.alpha * v : R.alpha * v;
        }
  } catch (const Bad&) {
    return 6;
  } catch (...) {
    return 7;
  }
  stat3[0] = double(h.units.size());
  stat3[1] = double(h.reds.size());
  stat3[2] = top > 0 ? std::log2(top) : 0;
  return 0;
}

// the rule that sends a launch to the plain kernel, on sizes alone
extern "C" int f64_emulate_small(int np, const int* M, const int* N, const int* nseg, int ns, const int* K) {
  std::vector<GemmProb> p(static_cast<size_t>(np));
  std::vector<GemmSeg> s(static_cast<size_t>(ns));
  for (int k = 0; k < ns; ++k) s[size_t(k)].K = K[k];
  int at = 0;
  for (int i = 0; i < np; ++i) {
    p[size_t(i)].M = M[i];
    p[size_t(i)].N = N[i];
    p[size_t(i)].s0 = at;
    p[size_t(i)].s1 = at += nseg[i];
  }
  return f64_small(p, s) ? 1 : 0;
}
