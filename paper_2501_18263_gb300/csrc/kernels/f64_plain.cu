// FP64 grouped GEMM by plain multiply-adds: every output element is one chain of FMAs
// over its segments and k in order, so a result does not depend on tiles or on the
// number of SMs.  Used where the rounding sequence is part of the result (a Davidson
// solve bounded in its iterations amplifies a difference of one rounding to percents
// within ten iterations) and for products too small for the tensor-core form.
//
// An FP64 warp instruction holds its SM quarter's pipe for 64 clocks, so loads are
// cheap beside it: one output per lane, a warp per 8 x 4 piece (any ragged tile is cut
// with little waste), operands straight from the L1, the next eight k of both operands
// loaded while the last eight are multiplied.  Measured: FP64 sigma of L = 32, D = 512
// 53 ms (34 ms at 2 multiply-adds per clock and SM), of L = 16, D = 128 2.3 ms against
// 203.8 and 10.6 ms for 64 x 64 tiles, whose warps idled on ragged edges and whose few
// tiles left SMs without work; results are bit-identical to those tiles'.
#include "f64_tc.h"

namespace dmrg {
namespace {

constexpr int PLAIN_WARPS = 4;

__device__ __forceinline__ F64Ref load_ref(const F64Ref* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return F64Ref{reinterpret_cast<const double*>((uint64_t(uint32_t(v.y)) << 32) | uint32_t(v.x)), v.z, v.w};
}

__global__ void __launch_bounds__(32 * PLAIN_WARPS) gemm_f64_plain_kernel(
    const F64Unit* __restrict__ tiles, const int* __restrict__ pieces, int ntiles, int npieces,
    const F64Row* __restrict__ rows, const F64Ref* __restrict__ rowref, const F64Ref* __restrict__ colref) {
  const int pc = blockIdx.x * PLAIN_WARPS + int(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (pc >= npieces) return;
  int lo = 0, hi = ntiles - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pieces[mid] <= pc) lo = mid;
    else hi = mid - 1;
  }
  const F64Unit u = tiles[lo];
  const int i = pc - pieces[lo], nc = (u.nt + F64_PC - 1) / F64_PC;
  const int r = F64_PR * (i / nc) + (lane >> 2), c = F64_PC * (i % nc) + (lane & 3);
  const bool on = r < u.rows && c < u.nt;
  const int rr = u.row0 + min(r, u.rows - 1), n = u.n0 + min(c, u.nt - 1);
  int a = u.pos0, b = u.pos0 + u.npos - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (rows[mid].pre <= rr) a = mid;
    else b = mid - 1;
  }
  const F64Row R = rows[a];
  const int m = rr - R.pre;
  const F64Ref* ra = rowref + R.s0;
  const F64Ref* rb = colref + u.cs;

  // iterator over (segment, k) in steps of eight k; the next segment's operand records
  // are loaded a segment ahead
  int s = 0, k = 0, K = 0;
  const double *pa = nullptr, *pb = nullptr;
  int64_t sa = 0, sb = 0;
  F64Ref na{}, nb{};
  auto enter = [&]() {   // segment s from the loaded records, records of s + 1 on their way
    K = na.kt >> 1;
    pa = na.p + ((na.kt & 1) ? int64_t(m) : int64_t(m) * na.ld);
    sa = (na.kt & 1) ? na.ld : 1;
    pb = nb.p + ((nb.kt & 1) ? int64_t(n) : int64_t(n) * nb.ld);
    sb = (nb.kt & 1) ? nb.ld : 1;
    k = 0;
    if (s + 1 < u.nseg) {
      na = load_ref(ra + s + 1);
      nb = load_ref(rb + s + 1);
    }
  };
  // the next batch's addresses and count; its elements are loaded one by one between
  // the multiply-adds of the batch before, in the shadow of each other's pipe time
  const double *qa = nullptr, *qb = nullptr;
  int64_t ta = 0, tb = 0;
  auto open = [&]() -> int {
    if (s >= u.nseg) return 0;
    qa = pa;
    qb = pb;
    ta = sa;
    tb = sb;
    const int cnt = min(8, K - k);
    pa += 8 * sa;
    pb += 8 * sb;
    k += 8;
    if (k >= K && ++s < u.nseg) enter();
    return cnt;
  };
  double acc = 0.0;
  if (u.nseg > 0) {
    na = load_ref(ra);
    nb = load_ref(rb);
    enter();
    double x[8], y[8];
    int cnt = open();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      x[j] = j < cnt ? __ldg(qa) : 0.0;
      y[j] = j < cnt ? __ldg(qb) : 0.0;
      qa += ta;
      qb += tb;
    }
    while (cnt > 0) {
      const int next = open();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j < cnt) acc = fma(x[j], y[j], acc);
        x[j] = j < next ? __ldg(qa) : 0.0;
        y[j] = j < next ? __ldg(qb) : 0.0;
        qa += ta;
        qb += tb;
      }
      cnt = next;
    }
  }
  if (!on) return;
  const double v = R.alpha * acc;
  double* o = u.trans ? R.C + m + int64_t(n) * R.ldc : R.C + int64_t(m) * R.ldc + n;
  *o = (R.m2 & 1) ? *o + v : v;
}

}  // namespace

void launch_gemm_f64_plain(const F64Unit* tiles, const int* pieces, int ntiles, int npieces, const F64Row* rows,
                           const F64Ref* rowref, const F64Ref* colref, cudaStream_t st) {
  if (npieces <= 0) return;
  gemm_f64_plain_kernel<<<unsigned((npieces + PLAIN_WARPS - 1) / PLAIN_WARPS), 32 * PLAIN_WARPS, 0, st>>>(
      tiles, pieces, ntiles, npieces, rows, rowref, colref);
}

}  // namespace dmrg
