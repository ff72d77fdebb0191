// Divide-and-conquer symmetric tridiagonal eigensolver (Cuppen, "A divide and
// conquer method for the symmetric tridiagonal eigenproblem", Numer. Math. 36
// (1981); eigenvectors by Gu and Eisenstat, "A divide-and-conquer algorithm for the
// symmetric tridiagonal eigenproblem", SIAM J. Matrix Anal. Appl. 16 (1995)).
//
// T is torn at every block boundary: with beta = T[b-1, b] and rho = |beta|,
// T = diag(T_1, T_2) + rho v v^T, v = e_{b-1} + sign(beta) e_b, where T_1, T_2 have
// their corner diagonal entries lowered by rho.  The leaves (at most 32 rows) are
// solved by implicit QL on one warp each.  A merge of two solved blocks with
// eigenpairs (D_i, Q_i) is the eigenproblem of D + rho z z^T, z = Q^T v (the last
// row of Q_1, sign(beta) times the first row of Q_2):
//  1. z normalised (rho takes ||z||^2), D sorted;
//  2. deflation: a component with rho |z_i| <= tol keeps (d_i, column i); of two
//     close poles a plane rotation zeroes the earlier z and keeps it when the
//     coupling it leaves, |(d_i - d_p) c s|, is below tol
//     (tol = 8 eps max(max |d|, rho));
//  3. the k roots of 1 + rho sum_i z_i^2 / (d_i - lambda) = 0, root j in
//     (d_j, d_{j+1}) (the last in (d_k, d_k + rho sum z^2)), each as an offset tau
//     from its nearer pole, by bisection on the bit patterns of tau, evaluated only
//     where a rational interpolation leaves f's sign in doubt (one warp per root, the
//     sums over the lanes);
//  4. z recomputed from the roots, zh_i^2 = prod_j (lambda_j - d_i) /
//     (rho prod_{l != i} (d_l - d_i)), so that the eigenvectors u_j = zh / (d - lambda_j)
//     are orthogonal to working accuracy;
//  5. the new eigenvectors Q [u_j] by an FP64 GEMM per merge.
// Every difference d_i - lambda_j is formed as (d_i - d_org(j)) - tau_j.
#include "tridiag_dc.h"

#include <cstdint>

namespace dmrg {
namespace {

__device__ __forceinline__ double dc_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// the sums of four values in six additions: each half of the warp takes two of them,
// each quarter one (an FP64 addition of a warp holds its pipe for 64 clocks, a select
// and a shuffle do not)
__device__ __forceinline__ void dc_warp_sum4(double& a, double& b, double& c, double& d) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  const double x = (h ? c : a) + __shfl_xor_sync(full, h ? a : c, 16);
  const double y = (h ? d : b) + __shfl_xor_sync(full, h ? b : d, 16);
  double v = (q ? y : x) + __shfl_xor_sync(full, q ? x : y, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
  a = __shfl_sync(full, v, 0);
  b = __shfl_sync(full, v, 8);
  c = __shfl_sync(full, v, 16);
  d = __shfl_sync(full, v, 24);
}

__device__ __forceinline__ int dc_find(const int* pre, int nj, int x) {
  int lo = 0, hi = nj - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// ---- leaves: one warp each, lane r holds row r of the leaf's eigenvectors in
// shared memory; the lanes look for negligible couplings, run the QL recurrences of one
// iteration (the rotations recorded by lane 0), then every lane applies them to its row.
// More than 60 iterations for one eigenvalue: *err = 9.
//
// Bound by the chain of dependent FP64 instructions, about 900 rotations of a hypot and
// two quotients for 32 rows.  The leaves of the density matrices of one bond at L = 24,
// D = 1024: 2.32 ms with one lane at work on both quotients and on the search for
// negligible couplings, 2.04 with the search on the lanes, 1.74 now.  A corrected
// reciprocal square root in place of hypot and quotients took 1.34, but its last bits let
// a coupling fall below its threshold an iteration earlier or later now and then, and
// every iteration turns the signs of eigenvectors around.  For the same reason what is
// fused here is written out and not left to the compiler.
constexpr int DC_LEAF_WARPS = 4;

__global__ void __launch_bounds__(32 * DC_LEAF_WARPS) dc_leaf_kernel(const DcLeaf* __restrict__ leaves, int nl,
                                                                    int* err) {
  __shared__ double zsm[DC_LEAF_WARPS][DC_LEAF][DC_LEAF + 1];
  __shared__ double dsm[DC_LEAF_WARPS][DC_LEAF], esm[DC_LEAF_WARPS][DC_LEAF];
  __shared__ double rc[DC_LEAF_WARPS][DC_LEAF], rs[DC_LEAF_WARPS][DC_LEAF];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int li = blockIdx.x * DC_LEAF_WARPS + w;
  if (li >= nl) return;
  const DcLeaf lf = leaves[li];
  const int s = lf.s, o = lf.o, n = lf.n;
  double (*Zl)[DC_LEAF + 1] = zsm[w];
  double* dd = dsm[w];
  double* ee = esm[w];
  if (lane < s) {
    double dv = lf.d[o + lane];
    if (lane == 0 && o > 0) dv -= fabs(lf.e[o - 1]);             // tear above the leaf
    if (lane == s - 1 && o + s < n) dv -= fabs(lf.e[o + s - 1]);  // tear below it
    dd[lane] = dv;
    ee[lane] = lane < s - 1 ? lf.e[o + lane] : 0.0;
    for (int c = 0; c < s; ++c) Zl[lane][c] = (c == lane) ? 1.0 : 0.0;
  }
  __syncwarp();
  const double eps = 2.220446049250313e-16;
  int l = 0, iter = 0;
  double tnorm = 0.0;
  if (lane < s) tnorm = fabs(dd[lane]) + fabs(ee[lane]) + (lane ? fabs(ee[lane - 1]) : 0.0);
#pragma unroll
  for (int of = 16; of > 0; of >>= 1) tnorm = fmax(tnorm, __shfl_xor_sync(0xffffffffu, tnorm, of));
  for (;;) {
    bool small = true;
    if (lane < s - 1)
      small = fabs(ee[lane]) <= eps * (fabs(dd[lane]) + fabs(dd[lane + 1])) || fabs(ee[lane]) <= eps * tnorm;
    const unsigned cut = __ballot_sync(0xffffffffu, small);
    while (l < s && (cut >> l & 1u)) {
      ++l;
      iter = 0;
    }
    if (l >= s) break;
    if (++iter > 60) {
      if (lane == 0) atomicExch(err, 9);
      break;
    }
    const int mm = __ffs(int(cut & (~0u << l))) - 1;   // the row s - 1 is always in cut
    // the recurrences, on every lane; an instruction of the warp takes as long for two of
    // the quotients (products) as for one, so lane 0 forms the sine's, lane 1 the cosine's
    double g = (dd[l + 1] - dd[l]) / (2.0 * ee[l]);
    double r = hypot(g, 1.0);
    g = dd[mm] - dd[l] + ee[l] / (g + (g >= 0.0 ? r : -r));
    double sn = 1.0, c = 1.0, p = 0.0;
    double dn = dd[mm], di = dd[mm - 1], ei = ee[mm - 1];
    const double dl = dd[l];
    __syncwarp();   // read by every lane before lane 0 writes
    int i = mm - 1;
    for (; i >= l; --i) {
      const int ip = i > l ? i - 1 : l;
      const double dnext = dd[ip], enext = ee[ip];
      const double fb = __dmul_rn(lane ? c : sn, ei);
      const double f = __shfl_sync(0xffffffffu, fb, 0), b = __shfl_sync(0xffffffffu, fb, 1);
      r = hypot(f, g);
      if (r == 0.0) {
        if (lane == 0) {
          ee[i + 1] = 0.0;
          dd[i + 1] = dn - p;
        }
        break;
      }
      const double q = (lane ? g : f) / r;
      sn = __shfl_sync(0xffffffffu, q, 0);
      c = __shfl_sync(0xffffffffu, q, 1);
      g = dn - p;
      const double rn = fma(2.0 * c, b, __dmul_rn(di - g, sn));
      p = __dmul_rn(sn, rn);
      __syncwarp();   // (the next entries are read)
      if (lane == 0) {
        ee[i + 1] = r;
        dd[i + 1] = __dadd_rn(g, p);
        rc[w][mm - 1 - i] = c;
        rs[w][mm - 1 - i] = sn;
      }
      g = fma(c, rn, -b);
      dn = di;
      di = dnext;
      ei = enext;
    }
    if (lane == 0) {
      if (i < l) {
        dd[l] = dl - p;
        ee[l] = g;
      }
      ee[mm] = 0.0;
    }
    __syncwarp();
    const int nrot = mm - 1 - i, first = mm - 1;
    if (lane < s) {
      // rotation q mixes columns i = first - q and i + 1 of row `lane`
      double zi1 = Zl[lane][first + 1];
      for (int q = 0; q < nrot; ++q) {
        const int i = first - q;
        const double c = rc[w][q], sn = rs[w][q];
        const double zi = Zl[lane][i];
        Zl[lane][i + 1] = fma(c, zi1, __dmul_rn(sn, zi));
        zi1 = fma(c, zi, -__dmul_rn(sn, zi1));
      }
      if (nrot > 0) Zl[lane][first - nrot + 1] = zi1;
    }
    __syncwarp();
  }
  if (lane < s) {
    lf.d[o + lane] = dd[lane];
    // column c of the leaf is column o + c of Z, rows o .. o + s - 1
    for (int c = 0; c < s; ++c) lf.Z[int64_t(o + c) * n + o + lane] = Zl[lane][c];
  }
}

// ---- merge step 1-2: one CTA per merge.  z from the two blocks' boundary rows,
// normalised; poles sorted (rank of each); deflation on one thread (sequential
// over the sorted poles, as the pairing with the previous kept pole requires); its chain
// of roots and quotients, one per pole, was most of 1.10 ms of the four levels (as at step 3), now
// 0.30: only pairs that come near the tolerance take them.
constexpr int DC_PREP_THREADS = 256;

__device__ double dc_block_sum(double v, double* red) {
  v = dc_warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    double x = lane < int(blockDim.x >> 5) ? red[lane] : 0.0;
    x = dc_warp_sum(x);
    if (lane == 0) red[32] = x;
  }
  __syncthreads();
  return red[32];
}

__global__ void __launch_bounds__(DC_PREP_THREADS) dc_prep_kernel(const DcMerge* __restrict__ ms) {
  __shared__ double red[34];
  const DcMerge m = ms[blockIdx.x];
  const int s = m.s, s1 = m.s1, o = m.o, n = m.n;
  const double beta = m.e[o + s1 - 1];
  const double sg = beta >= 0.0 ? 1.0 : -1.0;
  // z_i (column i of the two blocks) into gc temporarily, d into gs
  double part = 0.0;
  for (int i = threadIdx.x; i < s; i += blockDim.x) {
    const double zi = i < s1 ? m.Z[int64_t(o + i) * n + (o + s1 - 1)] : sg * m.Z[int64_t(o + i) * n + (o + s1)];
    m.gc[i] = zi;
    m.gs[i] = m.d[o + i] + 0.0;   // no -0.0: the order below is on bit patterns
    part += zi * zi;
  }
  const double nz2 = dc_block_sum(part, red);
  const double inv = nz2 > 0.0 ? 1.0 / sqrt(nz2) : 0.0;
  // rank sort (ties by index) on integers that order as the doubles do: an FP64
  // comparison holds the pipe as long as a multiply-add
  auto key = [](double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
  };
  for (int i = threadIdx.x; i < s; i += blockDim.x) {
    const double di = m.gs[i];
    const long long ki = key(di);
    int r = 0;
    for (int j = 0; j < s; ++j) {
      const long long kj = key(m.gs[j]);
      r += (kj < ki) || (kj == ki && j < i);
    }
    m.ds[r] = di;
    m.zs[r] = m.gc[i] * inv;
    m.perm[r] = i;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double rho = fabs(beta) * nz2;
    const double dmax = fmax(fabs(m.ds[0]), fabs(m.ds[s - 1]));
    const double tol = 8.0 * 2.220446049250313e-16 * fmax(dmax, rho);
    // a pair is looked at closely only if |(d_i - d_p) z_i z_p| <= tol (z_i^2 + z_p^2)
    // up to rounding, which takes no root and no division
    const double near = tol > 1e-280 ? 1.000001 * tol : 1e300;
    int ng = 0, p = -1;
    double zp = 0.0, dp = 0.0, zi = m.zs[0], di = m.ds[0];
    for (int i = 0; i < s; ++i) {
      const int in = i + 1 < s ? i + 1 : i;
      const double znext = m.zs[in], dnext = m.ds[in];
      if (rho * fabs(zi) <= tol) {   // deflated: (ds_i, column i) stays an eigenpair
        m.gp[2 * i + 1] = -1;        // mark (the pair slots double as flags below)
      } else {
        m.gp[2 * i + 1] = 0;
        if (p >= 0 && fabs((di - dp) * zi * zp) <= near * (zi * zi + zp * zp)) {
          const double t = hypot(zp, zi);
          const double c = zi / t, sn = -zp / t;
          if (fabs((di - dp) * c * sn) <= tol) {
            // rotate columns p, i so that z_p = 0; pole p deflates
            const double a = dp * c * c + di * sn * sn;
            di = dp * sn * sn + di * c * c;
            zi = t;
            m.ds[p] = a;
            m.ds[i] = di;
            m.zs[p] = 0.0;
            m.zs[i] = t;
            m.gp[2 * p + 1] = -1;
            m.gc[ng] = c;
            m.gs[ng] = sn;
            m.gp[2 * ng] = p | (i << 16);
            ++ng;
          }
        }
        p = i;
        zp = zi;
        dp = di;
      }
      zi = znext;
      di = dnext;
    }
    m.cnt[1] = ng;
    m.rho[0] = rho;
  }
  __syncthreads();
  if (threadIdx.x < 32) {   // the poles that are kept, in order
    const int lane = threadIdx.x;
    int k = 0;
    for (int i0 = 0; i0 < s; i0 += 32) {
      const int i = i0 + lane;
      const bool keep = i < s && m.gp[2 * i + 1] == 0;
      const unsigned b = __ballot_sync(0xffffffffu, keep);
      if (keep) {
        const int at = k + __popc(b & ((1u << lane) - 1u));
        m.ndp[at] = i;
        m.dk[at] = m.ds[i];
        m.zk[at] = m.zs[i];
      }
      k += __popc(b);
    }
    if (lane == 0) m.cnt[0] = k;
  }
}

// ---- merge step 3: one warp per root (pre_s: prefix sums of the merges' s; root
// slots past k exit).  f(lambda) rises from -inf to +inf between poles; the root is
// bracketed on the half of (d_j, d_{j+1}) where it lies, as bit patterns of tau
// (non-negative doubles order like their bit patterns), and bisected down to adjacent
// doubles, at most 63 halvings.  The value it ends at is part of the result: near a
// root f's sign flickers with its rounding, and a last bit of tau can decide a later
// deflation, hence an eigenvector's sign.  So the halvings are always these, but f is
// only evaluated where its sign is in doubt:
//  - with n the sum of the poles up to j (negated) and p = 1 + that of the others, n
//    falls and p grows with lambda, so n > (1 + delta) p proves f < 0, rounding
//    included, for every smaller lambda of the bracket too (delta: twice the relative
//    error of a sum of k terms), and p > (1 + delta) n the same for f > 0;
//  - the first few points are those of c + s_1 / (d_j - x) + s_2 / (d_{j+1} - x) with
//    the values and slopes of the two sums (Bunch, Nielsen and Sorensen, Numer. Math.
//    31 (1978)); two more, just outside the stretch in doubt, close it from both sides.
// Bound by FP64 divisions, one per pole and evaluation.  16 evaluations a root instead
// of 63: the four levels of the same matrices 3.44 -> 1.09 ms (0.70 for the rational
// points alone, which end at another of the neighbouring doubles).
__global__ void __launch_bounds__(256) dc_secular_kernel(const DcMerge* __restrict__ ms, int nm,
                                                         const int* __restrict__ pre_s) {
  const int gw = int((threadIdx.x >> 5) * gridDim.x + blockIdx.x), lane = threadIdx.x & 31;
  if (gw >= pre_s[nm]) return;
  const int mi = dc_find(pre_s, nm, gw);
  const DcMerge m = ms[mi];
  const int j = gw - pre_s[mi];
  const int k = m.cnt[0];
  if (j >= k) return;
  const double rho = m.rho[0];
  const double* dk = m.dk;
  const double* zk = m.zk;
  const double a = dk[j];
  double b;
  if (j + 1 < k) {
    b = dk[j + 1];
  } else {
    double z2 = 0.0;
    for (int i = lane; i < k; i += 32) z2 += zk[i] * zk[i];
    b = a + rho * dc_warp_sum(z2);
  }
  const bool last = j + 1 == k;
  // the sums over the poles up to j (p1) and past it (p2) and their derivatives, at the
  // point t from dorg; neg and pos of them
  double p1, p2, q1, q2, neg, pos;
  auto sums = [&](double dorg, double t) {
    p1 = p2 = q1 = q2 = 0.0;
    for (int i = lane; i < k; i += 32) {
      const double z = zk[i], q = z / ((dk[i] - dorg) - t);
      const bool left = i <= j;
      p1 = fma(left ? z : 0.0, q, p1);
      p2 = fma(left ? 0.0 : z, q, p2);
      q1 = fma(left ? q : 0.0, q, q1);
      q2 = fma(left ? 0.0 : q, q, q2);
    }
    dc_warp_sum4(p1, p2, q1, q2);
    neg = -rho * p1;
    pos = 1.0 + rho * p2;
  };
  const double over = 1.0 + (k * 0.0625 + 32.0) * 2.220446049250313e-16;   // 1 + delta
  const double mid = 0.5 * (a + b);
  sums(0.0, mid);
  bool upper = last || pos > neg * over;   // f(mid) > 0
  if (!upper && !(neg > pos * over)) {
    double fm = 0.0;
    for (int i = lane; i < k; i += 32) fm += zk[i] * zk[i] / (dk[i] - mid);
    upper = 1.0 + rho * dc_warp_sum(fm) > 0.0;
  }
  const int og = upper ? j : j + 1;
  const double sgn = upper ? 1.0 : -1.0;
  const double hi = last ? b - a : upper ? mid - a : b - mid;
  const double dorg = dk[og];
  long long ilo = 0, ihi = __double_as_longlong(hi);
  long long in = 0, out = ihi;   // the root is known to be further out than `in`, nearer than `out`
  auto mark = [&](long long at) {   // false: f's sign is in doubt there
    const bool l = neg > pos * over, r = pos > neg * over;
    if (sgn > 0.0 ? l : r) in = at > in ? at : in;
    if (sgn > 0.0 ? r : l) out = at < out ? at : out;
    return l || r;
  };
  long long x = last ? __double_as_longlong(mid - a) : ihi;   // the point of the sums
  bool doubt = false;
  double est = -1.0;
  for (int it = 0; it < 14 && out - in > 16; ++it) {
    const double t = sgn * __longlong_as_double(x);
    const double d1 = (a - dorg) - t, d2 = (b - dorg) - t;
    const double s1 = rho * q1, s2 = rho * q2, f = pos - neg;
    double eta;
    if (last) {
      eta = d1 + s1 * d1 * d1 / (f - s1 * d1);
    } else {
      const double c = f - s1 * d1 - s2 * d2;
      const double A = (d1 + d2) * f - d1 * d2 * (s1 + s2), B = d1 * d2 * f;
      const double disc = sqrt(fabs(A * A - 4.0 * B * c));
      eta = A <= 0.0 ? (A - disc) / (2.0 * c) : 2.0 * B / (A + disc);
    }
    const double tn = sgn * (t + eta);
    const long long xn = tn > 0.0 ? __double_as_longlong(tn) : 0;
    const long long step = xn > x ? xn - x : x - xn;
    if (tn > 0.0 && (doubt || step <= 64)) {
      est = tn;
      break;
    }
    x = xn > in && xn < out ? xn : in + ((out - in) >> 1);   // (a NaN goes to the middle)
    sums(dorg, sgn * __longlong_as_double(x));
    doubt = !mark(x);
  }
  if (est > 0.0) {
    const double w = 1.5 * (over - 1.0) * fmax(neg, pos) / (rho * (q1 + q2));
    for (int side = 0; side < 2; ++side) {
      double ww = w;
      for (int tries = 0; tries < 3; ++tries, ww *= 8.0) {
        const double t = side ? est + ww : est - ww;
        const long long at = t > 0.0 ? __double_as_longlong(t) : 0;
        if (at <= in || at >= out) break;
        sums(dorg, sgn * __longlong_as_double(at));
        mark(at);
        if (side ? out == at : in == at) break;
      }
    }
  }
  while (ihi - ilo > 1) {
    const long long im = ilo + ((ihi - ilo) >> 1);
    bool up = im <= in;
    if (!up && im < out) {
      const double t = sgn * __longlong_as_double(im);
      double f = 0.0;
      for (int i = lane; i < k; i += 32) f += zk[i] * zk[i] / ((dk[i] - dorg) - t);
      f = 1.0 + rho * dc_warp_sum(f);
      up = (f < 0.0) == (sgn > 0.0);
    }
    if (up) ilo = im;
    else ihi = im;
  }
  if (lane == 0) {
    m.org[j] = og;
    m.tau[j] = sgn * __longlong_as_double(ihi);
  }
}

// ---- merge steps 4a and 4b: one CTA per 32 roots, lane = root.  Their products and
// norms are chains in the order of the poles (their rounding is part of the result, as
// above), their terms are divisions: the CTA's warps fill tiles of DZ_T poles x 32
// roots in shared memory, one warp runs down the finished tile while the others fill the
// next.  The same levels: 0.68 -> 0.10 and 0.54 -> 0.11 ms against a thread per root.
// (pre_w: prefix sums of the merges' ceil(s / 32); CTAs past k exit.)
constexpr int DZ_T = 64;
constexpr int DZ_WARPS = 8;

// zh_i from the roots: lambda_j - d_i = tau_j - (d_i - d_org(j)); every factor paired
// with a pole gap, that of j = i with rho
__global__ void __launch_bounds__(32 * DZ_WARPS) dc_zhat_kernel(const DcMerge* __restrict__ ms, int nm,
                                                                const int* __restrict__ pre_w) {
  __shared__ double tile[2][DZ_T][32];
  const int mi = dc_find(pre_w, nm, int(blockIdx.x));
  const DcMerge m = ms[mi];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = m.cnt[0], i0 = 32 * (int(blockIdx.x) - pre_w[mi]);
  if (i0 >= k) return;
  const int i = min(i0 + lane, k - 1);
  const double di = m.dk[i];
  auto fill = [&](int t, int wf, int nw) {   // tile t, by warps wf, wf + nw, ..
    for (int jj = wf; jj < DZ_T && DZ_T * t + jj < k; jj += nw) {
      const int j = DZ_T * t + jj;
      tile[t & 1][jj][lane] = j == i ? 1.0 : (m.tau[j] - (di - m.dk[m.org[j]])) / (m.dk[j] - di);
    }
  };
  const int nt = (k + DZ_T - 1) / DZ_T;
  double prod = 1.0;
  fill(0, w, DZ_WARPS);
  if (w == 0) prod = (m.tau[i] - (di - m.dk[m.org[i]])) / m.rho[0];
  __syncthreads();
  for (int t = 0; t < nt; ++t) {
    if (w == 0) {
      for (int jj = 0; jj < DZ_T && DZ_T * t + jj < k; ++jj) prod *= tile[t & 1][jj][lane];
    } else if (t + 1 < nt) {
      fill(t + 1, w - 1, DZ_WARPS - 1);
    }
    __syncthreads();
  }
  if (w == 0 && i0 + lane < k) m.zh[i] = copysign(sqrt(fmax(prod, 0.0)), m.zk[i]);
}

// column j of U (k x k, column-major), normalised
__global__ void __launch_bounds__(32 * DZ_WARPS) dc_ucol_kernel(const DcMerge* __restrict__ ms, int nm,
                                                                const int* __restrict__ pre_w) {
  __shared__ double tile[2][DZ_T][33];
  __shared__ double inv[32];
  const int mi = dc_find(pre_w, nm, int(blockIdx.x));
  const DcMerge m = ms[mi];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = m.cnt[0], j0 = 32 * (int(blockIdx.x) - pre_w[mi]);
  if (j0 >= k) return;
  const int j = min(j0 + lane, k - 1);
  const double dorg = m.dk[m.org[j]], tj = m.tau[j];
  auto fill = [&](int t, int wf, int nw) {
    for (int ii = wf; ii < DZ_T && DZ_T * t + ii < k; ii += nw) {
      const int i = DZ_T * t + ii;
      tile[t & 1][ii][lane] = m.zh[i] / ((m.dk[i] - dorg) - tj);
    }
  };
  const int nt = (k + DZ_T - 1) / DZ_T;
  double nrm = 0.0;
  fill(0, w, DZ_WARPS);
  __syncthreads();
  for (int t = 0; t < nt; ++t) {
    if (w == 0) {
      for (int ii = 0; ii < DZ_T && DZ_T * t + ii < k; ++ii) {
        const double v = tile[t & 1][ii][lane];
        nrm = fma(v, v, nrm);
      }
    } else {
      if (t + 1 < nt) fill(t + 1, w - 1, DZ_WARPS - 1);
      for (int c = w - 1; c < 32 && j0 + c < k; c += DZ_WARPS - 1)   // unscaled, along the column
        for (int ii = lane; ii < DZ_T && DZ_T * t + ii < k; ii += 32)
          m.U[int64_t(j0 + c) * k + DZ_T * t + ii] = tile[t & 1][ii][c];
    }
    __syncthreads();
  }
  if (w == 0) inv[lane] = 1.0 / sqrt(nrm);
  __syncthreads();
  for (int c = w; c < 32 && j0 + c < k; c += DZ_WARPS) {
    double* u = m.U + int64_t(j0 + c) * k;
    const double s = inv[c];
    for (int i = lane; i < k; i += 32) u[i] *= s;
  }
}

// ---- merge step 5a: Qp = the two blocks' eigenvectors (block diagonal), columns
// in sorted order, then the deflation rotations; one thread per (merge, row)
__global__ void __launch_bounds__(256) dc_qp_kernel(const DcMerge* __restrict__ ms, int nm,
                                                    const int* __restrict__ pre_s) {
  const int g = int(blockIdx.x * blockDim.x + threadIdx.x);
  if (g >= pre_s[nm]) return;
  const int mi = dc_find(pre_s, nm, g);
  const DcMerge m = ms[mi];
  const int r = g - pre_s[mi];
  const int s = m.s, s1 = m.s1, o = m.o, n = m.n;
  const bool top = r < s1;
  for (int c = 0; c < s; ++c) {
    const int src = m.perm[c];
    m.Qp[int64_t(c) * s + r] = ((src < s1) == top) ? m.Z[int64_t(o + src) * n + o + r] : 0.0;
  }
  const int ng = m.cnt[1];
  for (int q = 0; q < ng; ++q) {
    const int pr = m.gp[2 * q], p = pr & 0xffff, i = pr >> 16;
    const double c = m.gc[q], sn = m.gs[q];
    double* qp = m.Qp + int64_t(p) * s + r;
    double* qi = m.Qp + int64_t(i) * s + r;
    const double a = *qp, b = *qi;
    *qp = c * a + sn * b;
    *qi = -sn * a + c * b;
  }
}

// ---- merge step 5b: the new eigenvectors of the non-deflated poles,
// Z[:, o + ndp[j]] = Qp[:, ndp] U[:, j] (s x k times k x k), 32 x 32 tiles
// (pre_t: prefix sums of the merges' ceil(s / DC_TILE)^2 tiles; tiles past k exit).
// FP64 multiply-adds at two per clock and SM bound it once every SM has tiles: 64 x 64
// ones left most idle.  The same levels: 0.97 -> 0.51 ms.
constexpr int DG_T = DC_TILE, DG_K = 16, DG_E = DG_T / 16;   // DG_E x DG_E results a thread

__global__ void __launch_bounds__(256) dc_gemm_kernel(const DcMerge* __restrict__ ms, int nm,
                                                      const int* __restrict__ pre_t) {
  __shared__ double As[DG_K][DG_T + 1];
  __shared__ double Bs[DG_K][DG_T + 1];
  const int mi = dc_find(pre_t, nm, int(blockIdx.x));
  const DcMerge m = ms[mi];
  const int s = m.s, k = m.cnt[0], o = m.o, n = m.n;
  const int ntc = (s + DG_T - 1) / DG_T;
  const int t = int(blockIdx.x) - pre_t[mi];
  const int r0 = (t / ntc) * DG_T, c0 = (t % ntc) * DG_T;
  if (c0 >= k) return;
  const int tr = threadIdx.x & 15, tc = threadIdx.x >> 4;
  double acc[DG_E][DG_E];
#pragma unroll
  for (int i = 0; i < DG_E; ++i)
#pragma unroll
    for (int j = 0; j < DG_E; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < k; k0 += DG_K) {
    for (int e = threadIdx.x; e < DG_T * DG_K; e += blockDim.x) {
      const int rr = e % DG_T, kk = e / DG_T;
      const int r = r0 + rr, kq = k0 + kk;
      As[kk][rr] = (r < s && kq < k) ? m.Qp[int64_t(m.ndp[kq]) * s + r] : 0.0;
    }
    for (int e = threadIdx.x; e < DG_T * DG_K; e += blockDim.x) {
      const int kk = e % DG_K, cc = e / DG_K;
      const int c = c0 + cc, kq = k0 + kk;
      Bs[kk][cc] = (c < k && kq < k) ? m.U[int64_t(c) * k + kq] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < DG_K; ++kk) {
      double a[DG_E], b[DG_E];
#pragma unroll
      for (int i = 0; i < DG_E; ++i) a[i] = As[kk][tr + 16 * i];
#pragma unroll
      for (int j = 0; j < DG_E; ++j) b[j] = Bs[kk][tc + 16 * j];
#pragma unroll
      for (int i = 0; i < DG_E; ++i)
#pragma unroll
        for (int j = 0; j < DG_E; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < DG_E; ++j) {
    const int c = c0 + tc + 16 * j;
    if (c >= k) continue;
    double* zc = m.Z + int64_t(o + m.ndp[c]) * n + o;
#pragma unroll
    for (int i = 0; i < DG_E; ++i) {
      const int r = r0 + tr + 16 * i;
      if (r < s) zc[r] = acc[i][j];
    }
  }
}

// ---- merge step 5c: eigenvalues of the merged block; deflated columns copied
// from Qp.  One CTA per (merge, sorted position).
__global__ void __launch_bounds__(128) dc_finish_kernel(const DcMerge* __restrict__ ms, int nm,
                                                        const int* __restrict__ pre_s) {
  const int mi = dc_find(pre_s, nm, int(blockIdx.x));
  const DcMerge m = ms[mi];
  const int c = int(blockIdx.x) - pre_s[mi];
  const int s = m.s, o = m.o, n = m.n, k = m.cnt[0];
  if (m.gp[2 * c + 1] == -1) {   // deflated
    if (threadIdx.x == 0) m.d[o + c] = m.ds[c];
    const double* src = m.Qp + int64_t(c) * s;
    double* dst = m.Z + int64_t(o + c) * n + o;
    for (int r = threadIdx.x; r < s; r += blockDim.x) dst[r] = src[r];
  } else if (threadIdx.x == 0) {
    // c = ndp[j] for one j (ndp ascending): the root j
    int lo = 0, hi = k - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (m.ndp[mid] < c) lo = mid + 1;
      else hi = mid;
    }
    m.d[o + c] = m.dk[m.org[lo]] + m.tau[lo];
  }
}

}  // namespace

void launch_dc_leaves(const DcLeaf* leaves, int nleaves, int* err, cudaStream_t st) {
  if (nleaves <= 0) return;
  const unsigned g = unsigned((nleaves + DC_LEAF_WARPS - 1) / DC_LEAF_WARPS);
  dc_leaf_kernel<<<g, 32 * DC_LEAF_WARPS, 0, st>>>(leaves, nleaves, err);
}

void launch_dc_merges(const DcMerge* m, int nmerge, const int* pre_s, int total, const int* pre_w, int wtotal,
                      const int* pre_t, int ttotal, cudaStream_t st) {
  if (nmerge <= 0) return;
  dc_prep_kernel<<<unsigned(nmerge), DC_PREP_THREADS, 0, st>>>(m);
  dc_secular_kernel<<<unsigned((total + 7) / 8), 256, 0, st>>>(m, nmerge, pre_s);
  dc_zhat_kernel<<<unsigned(wtotal), 32 * DZ_WARPS, 0, st>>>(m, nmerge, pre_w);
  dc_ucol_kernel<<<unsigned(wtotal), 32 * DZ_WARPS, 0, st>>>(m, nmerge, pre_w);
  dc_qp_kernel<<<unsigned((total + 255) / 256), 256, 0, st>>>(m, nmerge, pre_s);
  dc_gemm_kernel<<<unsigned(ttotal), 256, 0, st>>>(m, nmerge, pre_t);
  dc_finish_kernel<<<unsigned(total), 128, 0, st>>>(m, nmerge, pre_s);
}

}  // namespace dmrg
