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
// 50 ms (34 ms at 2 multiply-adds per clock and SM), of L = 16, D = 128 1.2 ms against
// 203.8 and 10.6 ms for 64 x 64 tiles, whose warps idled on ragged edges and whose few
// tiles left SMs without work; results are bit-identical to those tiles'.
//
// Long sums (F64_LONG octets and more) have few pieces and segments of a handful of k,
// whose addresses take a warp longer than their multiply-adds: there each piece has two
// warps, one that copies the operands of 16 k at a time, packed over segment borders,
// into shared memory (cp.async), and one that only multiplies (L = 16, D = 128: 1.8 ms
// with one warp for both).
#include "../exec_errors.h"
#include "f64_tc.h"
#include "tc.cuh"

namespace dmrg {
namespace {

constexpr int PLAIN_WARPS = 4;

__device__ __forceinline__ F64Ref load_ref(const F64Ref* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return F64Ref{reinterpret_cast<const double*>((uint64_t(uint32_t(v.y)) << 32) | uint32_t(v.x)), v.z, v.w};
}

// the tile of piece pc (prefix sums `pieces`) among tiles [t0, t1)
__device__ __forceinline__ int find_tile(const int* __restrict__ pieces, int t0, int t1, int pc) {
  int lo = t0, hi = t1 - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pieces[mid] <= pc) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// the problem of stack row rr among those of a tile
__device__ __forceinline__ int find_row(const F64Row* __restrict__ rows, const F64Unit& u, int rr) {
  int a = u.pos0, b = u.pos0 + u.npos - 1;
  while (a < b) {
    const int mid = (a + b + 1) >> 1;
    if (rows[mid].pre <= rr) a = mid;
    else b = mid - 1;
  }
  return a;
}

// ---- long sums.  Four pairs of warps per CTA: warp w < 4 multiplies, warp w + 4 loads.
constexpr int LK = 16;                       // k per buffer
constexpr int LRING = 4;                     // buffers
constexpr int LBUF = LK * (F64_PR + F64_PC); // doubles of a buffer: k-major, 8 rows then 4 columns

__global__ void __launch_bounds__(64 * PLAIN_WARPS) gemm_f64_long_kernel(
    const F64Unit* __restrict__ tiles, const int* __restrict__ pieces, int ntiles, int npieces,
    const F64Row* __restrict__ rows, const F64Ref* __restrict__ rowref, const F64Ref* __restrict__ colref, int* err) {
  __shared__ __align__(16) double buf[PLAIN_WARPS][LRING][LBUF];
  __shared__ uint64_t bars[PLAIN_WARPS][2 * LRING];
  __shared__ int cnts[PLAIN_WARPS][LRING];
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, w = warp & (PLAIN_WARPS - 1);
  if (threadIdx.x < PLAIN_WARPS * LRING) {
    const int pw = threadIdx.x / LRING, r = threadIdx.x % LRING;
    mbar_init(saddr(&bars[pw][r]), 33);          // full: every lane's copies, and the count
    mbar_init(saddr(&bars[pw][LRING + r]), 1);   // empty
  }
  if (threadIdx.x == 0) abort_word = 0;
  __syncthreads();
  const int pc = blockIdx.x * PLAIN_WARPS + w;
  if (pc >= npieces) return;
  const F64Unit u = tiles[find_tile(pieces, 0, ntiles, pc)];
  const int i = pc - pieces[find_tile(pieces, 0, ntiles, pc)], nc = (u.nt + F64_PC - 1) / F64_PC;
  const int r0 = F64_PR * (i / nc), c0 = F64_PC * (i % nc);
  auto full = [&](int r) { return saddr(&bars[w][r]); };
  auto empty = [&](int r) { return saddr(&bars[w][LRING + r]); };

  if (warp >= PLAIN_WARPS) {
    // ---- loads: lane = (k of the buffer, half of the rows and columns)
    const int kl = lane & (LK - 1), hf = lane / LK;
    int m[4], n[2];
    const F64Ref* ra[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rr = u.row0 + min(r0 + 4 * hf + q, u.rows - 1), a = find_row(rows, u, rr);
      m[q] = rr - rows[a].pre;
      ra[q] = rowref + rows[a].s0;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) n[q] = u.n0 + min(c0 + 2 * hf + q, u.nt - 1);
    const F64Ref* rb = colref + u.cs;
    int s = 0, k0 = 0;
    for (int step = 0;; ++step) {
      const int r = step % LRING;
      // the buffer's k: segment and place of each, from the lengths of the next 32 segments
      const int K = s + lane < u.nseg ? rb[s + lane].kt >> 1 : 0;
      int pre = K - (lane == 0 ? k0 : 0);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, pre, d);
        if (lane >= d) pre += v;
      }
      const int cnt = min(LK, __shfl_sync(0xffffffffu, pre, 31));
      int j = 0;   // segments of the window that end at or before this k
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
        if (__shfl_sync(0xffffffffu, pre, j + d - 1) <= kl) j += d;
      const int before = __shfl_sync(0xffffffffu, pre, max(j - 1, 0));
      const int sj = s + j, k = j == 0 ? k0 + kl : kl - before;
      const bool on = kl < cnt;
      if (step >= LRING && !mbar_wait_warp(empty(r), ((step / LRING) - 1) & 1, abort_flag, err, 21)) break;
      if (on) {
        const uint32_t dst = saddr(&buf[w][r][kl * (F64_PR + F64_PC)]);
        auto copy = [&](const F64Ref& f, int row, int at) {
          const double* p = f.p + ((f.kt & 1) ? int64_t(k) * f.ld + row : int64_t(row) * f.ld + k);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 8u * uint32_t(at)), "l"(p) : "memory");
        };
        F64Ref fa[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) fa[q] = load_ref(ra[q] + sj);
        const F64Ref fb = load_ref(rb + sj);
#pragma unroll
        for (int q = 0; q < 4; ++q) copy(fa[q], m[q], 4 * hf + q);
#pragma unroll
        for (int q = 0; q < 2; ++q) copy(fb, n[q], F64_PR + 2 * hf + q);
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full(r)) : "memory");
      if (lane == 0) {
        cnts[w][r] = cnt;
        mbar_arrive(full(r));
      }
      __syncwarp();
      if (cnt == 0) break;
      // the k after the buffer's last one (every full buffer's last lane knows it)
      const int last = cnt - 1;
      const int sl = __shfl_sync(0xffffffffu, sj, last), kn = __shfl_sync(0xffffffffu, k, last) + 1;
      const bool done = kn >= __shfl_sync(0xffffffffu, K, sl - s);
      s = done ? sl + 1 : sl;
      k0 = done ? 0 : kn;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // none in flight at exit
  } else {
    // ---- multiply-adds
    const int r = r0 + (lane >> 2), c = c0 + (lane & 3);
    double acc = 0.0;
    for (int step = 0;; ++step) {
      const int b = step % LRING;
      if (!mbar_wait_warp(full(b), (step / LRING) & 1, abort_flag, err, 22)) return;
      const int cnt = cnts[w][b];
      if (cnt == 0) break;
      const double* x = &buf[w][b][lane >> 2];
      const double* y = &buf[w][b][F64_PR + (lane & 3)];
      if (cnt == LK) {
#pragma unroll
        for (int k = 0; k < LK; ++k) acc = fma(x[k * (F64_PR + F64_PC)], y[k * (F64_PR + F64_PC)], acc);
      } else {
        for (int k = 0; k < cnt; ++k) acc = fma(x[k * (F64_PR + F64_PC)], y[k * (F64_PR + F64_PC)], acc);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(b));
    }
    if (r < u.rows && c < u.nt) {
      const int rr = u.row0 + r;
      const F64Row R = rows[find_row(rows, u, rr)];
      const int m = rr - R.pre, n = u.n0 + c;
      const double v = R.alpha * acc;
      double* o = u.trans ? R.C + m + int64_t(n) * R.ldc : R.C + int64_t(m) * R.ldc + n;
      *o = (R.m2 & 1) ? *o + v : v;
    }
  }
}

// ---- short sums: one warp per piece
__global__ void __launch_bounds__(32 * PLAIN_WARPS) gemm_f64_plain_kernel(
    const F64Unit* __restrict__ tiles, const int* __restrict__ pieces, int t0, int ntiles, int npieces,
    const F64Row* __restrict__ rows, const F64Ref* __restrict__ rowref, const F64Ref* __restrict__ colref) {
  const int pc = pieces[t0] + blockIdx.x * PLAIN_WARPS + int(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (pc >= npieces) return;
  const int tl = find_tile(pieces, t0, ntiles, pc);
  const F64Unit u = tiles[tl];
  const int i = pc - pieces[tl], nc = (u.nt + F64_PC - 1) / F64_PC;
  const int r = F64_PR * (i / nc) + (lane >> 2), c = F64_PC * (i % nc) + (lane & 3);
  const bool on = r < u.rows && c < u.nt;
  const int rr = u.row0 + min(r, u.rows - 1), n = u.n0 + min(c, u.nt - 1);
  const F64Row R = rows[find_row(rows, u, rr)];
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

void launch_gemm_f64_plain(const F64Unit* tiles, const int* pieces, int nlong, int plong, int ntiles, int npieces,
                           const F64Row* rows, const F64Ref* rowref, const F64Ref* colref, int* err,
                           cudaStream_t st) {
  if (plong > 0)
    gemm_f64_long_kernel<<<unsigned((plong + PLAIN_WARPS - 1) / PLAIN_WARPS), 64 * PLAIN_WARPS, 0, st>>>(
        tiles, pieces, nlong, plong, rows, rowref, colref, err);
  if (npieces > plong)
    gemm_f64_plain_kernel<<<unsigned((npieces - plong + PLAIN_WARPS - 1) / PLAIN_WARPS), 32 * PLAIN_WARPS, 0, st>>>(
        tiles, pieces, nlong, ntiles, npieces, rows, rowref, colref);
}

}  // namespace dmrg
