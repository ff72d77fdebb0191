// FP64 numbers as eight signed 8-bit digits, and back: the number format of the
// tensor-core FP64 product (f64_tc.cu).  Plain integer arithmetic, usable on the
// host and on the device.
//
// With e the largest biased exponent of a row (at least 1; |x| < 2^(e - 1022) for
// every x of it), x is taken as the integer X = trunc(x / 2^(e - 1084)), |X| < 2^62,
// and X = sum_j d_j 2^(8 (7 - j)) with digits d_j in [-128, 127], |d_0| <= 64.  The
// 53 bits of an element within 2^9 of the row's largest are kept whole; what a
// smaller one loses is below 2^-62 of the row's largest.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define F64_HD __host__ __device__ __forceinline__
#else
#define F64_HD inline
#endif

namespace dmrg {

constexpr int F64_DIGITS = 8;
constexpr int F64_SPECIAL = 0x7ff;   // exponent field of infinities and NaN

// the eight digits of x, each biased by 128, digit j in byte 7 - j (hi, lo: the
// words of x; e: the row's exponent, >= x's own and >= 1)
F64_HD uint64_t f64_digits(uint32_t hi, uint32_t lo, int e) {
  const int ef = int((hi >> 20) & 0x7ffu);
  const uint32_t mh = (hi & 0xfffffu) | (ef ? 0x100000u : 0u);
  const uint64_t m = ((uint64_t(mh) << 32) | lo) << 9;
  int d = e - (ef ? ef : 1);
  d = d > 63 ? 63 : d;
  const uint64_t x = m >> d;   // below 2^62; 0 once d > 61
  const uint64_t s = (hi >> 31) ? uint64_t(0) - x : x;
  return s + 0x8080808080808080ull;
}

F64_HD int f64_clz32(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz(int(x));
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
// upper word of (hi:lo) << n, n < 32
F64_HD uint32_t f64_shl(uint32_t hi, uint32_t lo, int n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, n);
#else
  return n ? (hi << n) | (lo >> (32 - n)) : hi;
#endif
}
F64_HD double f64_bits(uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double r;
  std::memcpy(&r, &b, 8);
  return r;
#endif
}

// mant 2^(E - 1075) outside the range of normal results, in two steps (apart, so that
// no FP64 instruction enters the common path by speculation)
#if defined(__CUDACC__)
static __host__ __device__ __noinline__
#else
inline
#endif
double f64_scale(uint64_t mant, int E) {
  const int q = E - 1075;
  int q1 = q / 2, q2 = q - q1;
  q1 = q1 < -1000 ? -1000 : (q1 > 1000 ? 1000 : q1);
  q2 = q2 < -1000 ? -1000 : (q2 > 1000 ? 1000 : q2);
  return double(mant) * f64_bits(uint64_t(q1 + 1023) << 52) * f64_bits(uint64_t(q2 + 1023) << 52);
}

F64_HD int f64_rint(float x) {
#if defined(__CUDA_ARCH__)
  return __float2int_rn(x);
#else
  return int(std::lrintf(x));
#endif
}

// The product sum of a chunk: a[w] = sum_k sum_{i + j = w} da_i db_j (exact integers for
// w < 6; |a[0]| < 2^20, |a[1]| < 2^22, |a[2]| < 2^23, the others below 2^25), so
// sum_k Xa Xb = 2^56 (V + what the weights above 7 hold) with V = sum_w a[w] 2^(8 (7 - w)),
// given as hi 2^32 + lo (weight 7 rounded into weight 6: 2^-60 of the largest product).
// Shifts and adds only: a 64-bit integer multiply-add runs on the slow FP64 pipe.
F64_HD void f64_combine(float a0, float a1, float a2, float a3, float a4, float a5, float a6, float a7, int64_t& hi,
                        uint32_t& lo) {
  const int32_t p01 = f64_rint(a0) * 256 + f64_rint(a1), p23 = f64_rint(a2) * 256 + f64_rint(a3);
  const int64_t g = int64_t((uint64_t(int64_t(p01)) << 16)) + p23;
  const int64_t t = int64_t(uint64_t(int64_t(f64_rint(a4))) << 16) + int64_t(uint64_t(int64_t(f64_rint(a5))) << 8) +
                    f64_rint(a7 * 0.00390625f + a6);
  hi = g + int32_t(uint64_t(t) >> 24);   // |t| < 2^43: 24 of its bits go to lo
  lo = uint32_t(t) << 8;
}

// A sum too small for its digits: |V| < 2^F64_WEAK, where a product of the row's and the
// column's largest elements has |V| of 2^66 to 2^68.  V is off by at most 578 k + 2^14
// (weights above 7: below 450 a product; elements cut at 2^-62 of the largest: below 128;
// the sums of weights 6 and 7 in FP32), so a sum of terms that are each far below the
// largest row element times the largest column element has lost bits that plain
// multiply-adds keep.  Such sums are computed again, plainly; the others are within
// 2^-36 of their own value and, as a rule (errors of either sign), within 2^-44.
// lead: the leading zero bits of |V| as 96 bits.
constexpr int F64_WEAK = 54;
F64_HD bool f64_weak(int lead) { return lead >= 96 - F64_WEAK; }

// The double nearest to (hi 2^32 + lo) 2^(ea + eb - 2112), its sign flipped when `flip`
// (integer instructions only in the normal range: an FP64 one costs 16 times as much
// here).
//
// f64_assemble_fast: without branches, so that several elements' chains interleave;
// *bad is set where the result is not a normal number below 2^1023 or zero; *lead: the
// leading zero bits of |V|.
F64_HD double f64_assemble_fast(int64_t hi, uint32_t c0, int ea, int eb, bool flip, bool* bad, int* lead = nullptr) {
  const bool neg = hi < 0;
  // |V| as three words
  const uint64_t m = neg ? ~uint64_t(hi) + (c0 == 0 ? 1 : 0) : uint64_t(hi);
  uint32_t a = uint32_t(m >> 32), b = uint32_t(m), c = neg ? 0u - c0 : c0;
  // leading zero words out
  const bool z1 = a == 0;
  a = z1 ? b : a;
  b = z1 ? c : b;
  c = z1 ? 0u : c;
  const bool z2 = a == 0;
  a = z2 ? b : a;
  b = z2 ? 0u : b;
  const int lz = f64_clz32(a);
  const int zeros = (z1 ? 32 : 0) + (z2 ? 32 : 0) + lz;
  if (lead) *lead = zeros;
  const int E = ea + eb - 994 - zeros;
  // (w1:w0) 2^(E - 1086): the top bit of w1 set; 53 bits kept, rounded to nearest
  const uint32_t w1 = f64_shl(a, b, lz), w0 = f64_shl(b, c, lz);
  const uint64_t mant = ((uint64_t(w1 >> 11) << 32) | f64_shl(w1, w0, 21)) + ((w0 >> 10) & 1u);
  const uint64_t sign = neg != flip ? uint64_t(1) << 63 : 0;
  *bad = a != 0 && uint32_t(E - 1) >= 2045u;
  return f64_bits(a != 0 ? sign | ((uint64_t(uint32_t(E - 1)) << 52) + mant) : 0);
}

F64_HD double f64_assemble(int64_t hi, uint32_t lo, int ea, int eb, bool flip) {
  uint32_t a = uint32_t(uint64_t(hi) >> 32), b = uint32_t(hi), c = lo;   // V as three words
  const bool neg = hi < 0;
  if (neg) {
    const uint64_t m = ~uint64_t(hi) + (c == 0 ? 1 : 0);
    a = uint32_t(m >> 32);
    b = uint32_t(m);
    c = 0u - c;
  }
  int E = ea + eb - 994;
  if (a == 0) {
    a = b;
    b = c;
    c = 0;
    E -= 32;
    if (a == 0) {
      a = b;
      b = 0;
      E -= 32;
      if (a == 0) return 0.0;
    }
  }
  const int lz = f64_clz32(a);
  E -= lz;
  // (w1:w0) 2^(E - 1086): the top bit of w1 set; 53 bits kept, rounded to nearest
  const uint32_t w1 = f64_shl(a, b, lz), w0 = f64_shl(b, c, lz);
  const uint64_t mant = ((uint64_t(w1 >> 11) << 32) | f64_shl(w1, w0, 21)) + ((w0 >> 10) & 1u);
  const uint64_t sign = uint64_t(neg != flip) << 63;
  if (uint32_t(E - 1) < 2045u) return f64_bits(sign | ((uint64_t(uint32_t(E - 1)) << 52) + mant));
  const double r = f64_scale(mant, E);
  return neg != flip ? -r : r;
}

}  // namespace dmrg
