// FP64 grouped GEMM on the 5th-generation tensor cores (tcgen05 + TMEM).
//
// The FP64 units of this GPU run two multiply-adds per clock and SM, the tensor cores
// 4096 16-bit ones, so an FP64 product is computed from exact small-integer products
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59
// (2012)): every row of A and every column of B is scaled by its largest exponent
// over a chunk of K and written as eight signed 8-bit digits (f64_digits.h).  A digit
// is exact in FP16, a product of two in FP32, and so are the sums over a chunk (at
// most 192 k) of the digit products of equal weight (0 to 5; those of weights 6 and 7,
// worth 2^-56 and less of the largest product, may round), so that
//   acc[w] = sum_k sum_{i + j = w} dA_i dB_j,   w = 0 .. 7,
// gives A B up to 2^-58 a k of the row's largest element times the column's (each up to
// the power of two above it); the 36 products per k replace one FP64 multiply-add.  The
// accumulators are combined in integers, rounded once to FP64 and added over the chunks
// in FP64.  The error is normwise: an element 2^9 or more below its row's largest is held
// in fewer than 53 bits.  Elements of C whose chunk sum comes out far below what its row
// and column could give (f64_weak; FINE only), and rows or columns with an infinity or a
// NaN, are computed by plain FP64 multiply-adds.
//
// One tile: 128 rows (TMEM lanes) x up to 64 columns, eight accumulators of 64 TMEM
// columns.  With B's digits stored one after the other along N, one MMA of digit i of
// A with digits 0 .. 7 - i of B (N up to 256) adds into the accumulators i .. 7 at
// once: at most 12 instead of 36 MMAs per 16 k, and A's digits are read from shared
// memory 12 instead of 36 times.
//
// One persistent CTA per SM; its registers are dealt out again by warpgroup:
//   warps 0-11   converters: per chunk a first pass over the operands finds the rows'
//                exponents, a second (out of the L1 and L2) writes the digits into a ring
//                of four 16-k stages in the tensor core's core-matrix layout.  Bound by
//                instruction issue, about 50 per element
//   warp 12      TMEM allocation and the MMA issuer (one lane)
//   warp 13      reads the work list ahead of the others: which problem each row
//                belongs to, the octets of each chunk (a ring of four slots)
//   warps 16-23  drain: TMEM -> integers -> FP64 -> C (64 bytes of a row at a time
//                through shared memory where C is row-major), two warps per TMEM lane
//                quarter
// Tiles of at most 32 columns use half of TMEM and are double-buffered.
//
// Measured (FP64 sigma at the centre bond of L = 32, D = 512, 20.5 G multiply-adds in
// ragged blocks of 1 to 140 rows): 14.1 ms, against 203.8 ms for 64 x 64 tiles of FP64
// multiply-adds without stacking or a split of long sums, and 50 ms for the plain pieces
// of f64_plain.cu; relative error against 64 bits 6e-16 (plain: 1e-15) at L = 8, D = 64.
// Small sums computed again cost 0.6 ms of it (about one element in 5000 of dense
// operators; with the line of f64_weak at 2^52 13.9 ms, 2^56 14.9, 2^58 18.8, 2^60 31).
#include <cuda_fp16.h>

#include <atomic>
#include <cstdint>

#include "../exec_errors.h"
#include "f64_digits.h"
#include "f64_tc.h"
#include "tc.cuh"

namespace dmrg {
namespace {

constexpr int CONV = 12;                         // converter warps
constexpr int DRAIN = 8;                         // drain warps
constexpr int W_MMA = CONV, W_HEAD = CONV + 1, W_DRAIN = CONV + 4;
constexpr int THREADS = 32 * (W_DRAIN + DRAIN);
// registers per thread: the launch's 80 x 24 warps are dealt out as 88 to converters
// and drain warps and 40 to the others (12 x 88 + 4 x 40 + 8 x 88 = 24 x 80)
constexpr int REGS = 80;
constexpr int STAGES = 4;
constexpr int SLOTS = 4;
constexpr int A_BYTES = F64_DIGITS * F64_TM * 32;   // digits x rows x 16 k x 2 bytes
constexpr int B_BYTES = F64_DIGITS * F64_TN * 32;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int STG_LD = 9;                        // doubles per staged row (8 columns)

// one chunk of a unit, written by the header warp (expo by the converters)
struct Slot {
  int noct;            // octets; 0: a problem without segments, -1: no more chunks
  int first;           // first chunk of its unit (pos is written then)
  int ci;              // chunk of the unit
  int rows, n0, nt, cs, trans;
  int pad[2];
  int64_t part;
  int2 oct[F64_CHUNK]; // segment; 16 x first k + length
  int s0[F64_TM];      // per row: its problem's first segment, its row there
  int m[F64_TM];
  int pos[F64_TM];     // and its problem
  int expo[F64_TM + F64_TN];   // high words of the largest magnitudes
};
constexpr int STG_OFF = STAGES * STAGE_BYTES;
constexpr int PTR_OFF = STG_OFF + DRAIN * 32 * STG_LD * 8;
constexpr int SLOT_OFF = PTR_OFF + DRAIN * 32 * 8;
constexpr int BAR_OFF = SLOT_OFF + SLOTS * int(sizeof(Slot));
constexpr int SMEM_BYTES = BAR_OFF + 256;
constexpr uint32_t TMEM_COLS = 512;
static_assert(sizeof(Slot) % 8 == 0 && SMEM_BYTES <= 232448, "shared memory layout");
static_assert(F64_DIGITS * F64_TN <= int(TMEM_COLS), "accumulators");
static_assert(CONV * 88 + 4 * 40 + DRAIN * 88 <= (THREADS / 32) * REGS, "register split");

// no-swizzle K-major layout: core matrices of 8 rows x 16 bytes, the two of a 16-k
// stage 128 bytes apart (LBO), 8-row groups 256 bytes apart (SBO)
__device__ __forceinline__ uint64_t f64_sdesc(uint32_t addr) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) | (static_cast<uint64_t>(128u >> 4) << 16) |
         (static_cast<uint64_t>(256u >> 4) << 32) | (static_cast<uint64_t>(1) << 46);
}

// kind::f16, FP16 x FP16 -> FP32, M = 128
__device__ __forceinline__ uint32_t f64_idesc(int n) {
  return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(F64_TM >> 4) << 24);
}

// the MMAs of one 16-k stage of an N-column tile: digit i of A with digits j .. of B, as
// many as fit N = 256, into the accumulators i + j ..; every operand a constant away
// from the stage's descriptors (computing them per MMA took ten times the MMAs' time)
template <int N>
__device__ __forceinline__ void stage_mmas(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  constexpr int PER = 256 / N < F64_DIGITS ? 256 / N : F64_DIGITS;
#pragma unroll
  for (int i = 0; i < F64_DIGITS; ++i)
#pragma unroll
    for (int j = 0; j < F64_DIGITS - i; j += PER) {
      const int nd = PER < F64_DIGITS - i - j ? PER : F64_DIGITS - i - j;
      mma(d + uint32_t((i + j) * N), a + uint64_t(i * F64_TM * 2), b + uint64_t(j * N * 2), f64_idesc(nd * N),
          i == 0 ? acc : 1u);
    }
}

// TMEM 32 lanes x 4 columns of the eight accumulators (n columns apart) and the wait
__device__ __forceinline__ void tmem_ld8x4(uint32_t t, uint32_t n, float (&v)[8][4]) {
  uint32_t a[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%33];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%34];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%35];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%36];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%37];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%38];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%39];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]),
        "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(a[16]),
        "=r"(a[17]), "=r"(a[18]), "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]), "=r"(a[24]),
        "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]), "=r"(a[31])
      : "r"(t), "r"(t + n), "r"(t + 2 * n), "r"(t + 3 * n), "r"(t + 4 * n), "r"(t + 5 * n), "r"(t + 6 * n),
        "r"(t + 7 * n)
      : "memory");
#pragma unroll
  for (int w = 0; w < 8; ++w)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[w][i] = __uint_as_float(a[4 * w + i]);
}

// the problem (position in `rows`) of stack row `row`, one row per lane, among the
// npos problems from pos0 (warp-collective)
__device__ __forceinline__ int locate(const F64Row* __restrict__ rows, int pos0, int npos, int row) {
  const int lane = threadIdx.x & 31;
  int pos = pos0;
  for (int b = 1; b < npos; b += 32) {
    const int v = b + lane < npos ? rows[pos0 + b + lane].pre : INT32_MAX;
    int j = 0;   // entries <= row (the entries ascend)
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
      if (__shfl_sync(0xffffffffu, v, j + s - 1) <= row) j += s;
    if (__shfl_sync(0xffffffffu, v, 31) <= row) j = 32;
    pos += j;
  }
  return pos;
}

// one element's sum over the slot's octets by plain FP64 multiply-adds, a k per lane
// (warp-collective, the sum on every lane): rows or columns that hold an infinity or a
// NaN, and sums too small for their digits.  Twelve octets at a time, all their records
// loaded before any element: it is bound by the two latencies
__device__ __noinline__ double chunk_dot(const Slot* S, const F64Ref* __restrict__ ra, const F64Ref* __restrict__ rb,
                                         int m, int n, int nOct) {
  const int lane = threadIdx.x & 31, kl = lane & 7;
  double acc = 0.0;
#pragma unroll 1
  for (int h = 0; h < nOct; h += 12) {
    int2 e[3];
    int4 fa[3], fb[3];
    double x[3], y[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      e[q] = S->oct[h + 4 * q + (lane >> 3)];   // octets past the last have no k
      fa[q] = __ldg(reinterpret_cast<const int4*>(ra + e[q].x));
      fb[q] = __ldg(reinterpret_cast<const int4*>(rb + e[q].x));
    }
    auto at = [](const int4& f, int r, int k) {
      const double* p = reinterpret_cast<const double*>((uint64_t(uint32_t(f.y)) << 32) | uint32_t(f.x));
      return __ldg(p + ((f.w & 1) ? int64_t(k) * f.z + r : int64_t(r) * f.z + k));
    };
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int k = (e[q].y >> 4) + kl;
      const bool on = kl < (e[q].y & 15);
      x[q] = on ? at(fa[q], m, k) : 0.0;
      y[q] = on ? at(fb[q], n, k) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) acc = fma(x[q], y[q], acc);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
  return acc;
}

__device__ __noinline__ double assemble_any(int64_t hi, uint32_t lo, int ea, int eb, bool flip) {
  return f64_assemble(hi, lo, ea, eb, flip);
}

// an 8-row group of a tile's rows or columns, as a converter lane sees it
struct Group {
  const F64Ref* ref;   // the lane's row: its operands by segment
  int row;             // and its index there
  uint32_t dst;        // byte offset of the lane's piece of the group in a stage
  uint32_t dig;        // bytes from one digit to the next
  int ex;              // place of the row's exponent
  bool val;            // the row exists
};

// the operand records of the B octets from o for the lane's row
template <int B>
__device__ __forceinline__ void load_refs(const Group& g, const int2* oct, int o, int4 (&f)[B]) {
#pragma unroll
  for (int j = 0; j < B; ++j) f[j] = __ldg(reinterpret_cast<const int4*>(g.ref + oct[o + j].x));
}

// and the lane's k pair in each of them
template <int B>
__device__ __forceinline__ void load_pairs(const Group& g, const int2* oct, int o, int kp, const int4 (&f)[B],
                                           double (&x)[B][2]) {
#pragma unroll
  for (int j = 0; j < B; ++j) {
    const int e = oct[o + j].y, k = (e >> 4) + 2 * kp, n = g.val ? (e & 15) - 2 * kp : 0;
    const bool t = f[j].w & 1;
    const double* p = reinterpret_cast<const double*>((uint64_t(uint32_t(f[j].y)) << 32) | uint32_t(f[j].x)) +
                      (int64_t(t ? k : g.row) * f[j].z + (t ? g.row : k));
    x[j][0] = n > 0 ? __ldg(p) : 0.0;
    x[j][1] = n > 1 ? __ldg(p + (t ? f[j].z : 1)) : 0.0;
  }
}

// both, all records first, so that a batch pays each of the two latencies once
template <int B>
__device__ __forceinline__ void load_octets(const Group& g, const int2* oct, int o, int kp, double (&x)[B][2]) {
  int4 f[B];
  load_refs<B>(g, oct, o, f);
  load_pairs<B>(g, oct, o, kp, f, x);
}

// the digits of two neighbouring elements of a row, digit w to address a + w stride:
// a biased digit b as the FP16 number 1024 + b, less 1152
__device__ __forceinline__ void store_digits(double x0, double x1, int e, uint32_t a, uint32_t stride) {
  const uint64_t d0 = f64_digits(uint32_t(__double2hiint(x0)), uint32_t(__double2loint(x0)), e);
  const uint64_t d1 = f64_digits(uint32_t(__double2hiint(x1)), uint32_t(__double2loint(x1)), e);
  const __half2 bias = __half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));   // 1152
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t w0 = uint32_t(h ? d0 : d0 >> 32), w1 = uint32_t(h ? d1 : d1 >> 32);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const uint32_t u = __byte_perm(w0, w1, p ? 0x5410u : 0x7632u);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t b = __byte_perm(u, 0x64646464u, q ? 0x4240u : 0x4341u);
        const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&b), bias);
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(a + stride * uint32_t(4 * h + 2 * p + q)),
                     "r"(*reinterpret_cast<const uint32_t*>(&d))
                     : "memory");
      }
    }
  }
}

template <bool FINE>
__global__ void __maxnreg__(REGS)
    gemm_f64_tc_kernel(const F64Unit* __restrict__ units, int nunits, const F64Row* __restrict__ rows,
                       const F64Ref* __restrict__ rowref, const F64Ref* __restrict__ colref,
                       double* __restrict__ part, int* next, int* err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  Slot* slots = reinterpret_cast<Slot*>(smem + SLOT_OFF);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + BAR_OFF);
  constexpr int NBAR = 2 * STAGES + 4 + 3 * SLOTS + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NBAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert(NBAR * 8 + 8 <= 256, "barriers");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = gridDim.x;
  auto full = [&](int s) { return saddr(&bars[s]); };
  auto empty = [&](int s) { return saddr(&bars[STAGES + s]); };
  auto acc_full = [&](int b) { return saddr(&bars[2 * STAGES + b]); };
  auto acc_empty = [&](int b) { return saddr(&bars[2 * STAGES + 2 + b]); };
  auto slot_full = [&](int e) { return saddr(&bars[2 * STAGES + 4 + e]); };
  auto slot_empty = [&](int e) { return saddr(&bars[2 * STAGES + 4 + SLOTS + e]); };
  auto ex_full = [&](int e) { return saddr(&bars[2 * STAGES + 4 + 2 * SLOTS + e]); };
  const uint32_t mma_fin = saddr(&bars[NBAR - 1]);

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full(s), CONV);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), DRAIN);
    }
    for (int e = 0; e < SLOTS; ++e) {
      mbar_init(slot_full(e), 1);
      mbar_init(slot_empty(e), CONV + 1 + DRAIN);
      mbar_init(ex_full(e), CONV);
    }
    mbar_init(mma_fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp < CONV) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    // ---- converters.  A lane holds row rl of an 8-row group and the k pair kp of an
    // octet, so that a warp reads 64 bytes of each of 8 rows (or 8 consecutive rows at
    // each k) and writes each digit of an 8 x 8 piece as one 128-byte core matrix.  The
    // groups of a chunk, times its octets, are dealt out over all converter warps; the
    // exponents meet in the slot.  The exponents of chunk c + 1 are taken before the
    // digits of chunk c are written, so that no warp waits for the others' maxima.
    const int rl = lane >> 2, kp = lane & 3;
    auto group = [&](const Slot& S, int ga, int g) {
      Group q;
      if (g < ga) {
        const int r = 8 * g + rl;
        q.val = r < S.rows;
        q.row = S.m[r];
        q.ref = rowref + S.s0[r];
        q.dst = uint32_t(g * 256 + lane * 4);
        q.dig = F64_TM * 32;
        q.ex = r;
      } else {
        const int c = 8 * (g - ga) + rl;
        q.val = c < S.nt;
        q.row = S.n0 + min(c, S.nt - 1);
        q.ref = colref + S.cs;
        q.dst = uint32_t(A_BYTES + (g - ga) * 256 + lane * 4);
        q.dig = uint32_t((S.nt + 15) & ~15) * 32;
        q.ex = F64_TM + c;
      }
      return q;
    };
    int step = 0;
    bool stop = false, more = true;
    for (int chunk = 0; !stop; ++chunk) {
      // exponents of chunk `chunk`
      if (more) {
        const int sl = chunk % SLOTS;
        if (!mbar_wait_warp(slot_full(sl), (chunk / SLOTS) & 1, abort_flag, err, 11)) break;
        Slot& S = slots[sl];
        const int nOct = S.noct;
        more = nOct >= 0;
        if (nOct > 0) {
          const int ga = (S.rows + 7) >> 3, G8 = ga + ((S.nt + 7) >> 3), nb = (nOct + 7) >> 3;
#pragma unroll 1
          for (int i = warp; i < G8 * nb; i += CONV) {
            const int g = nb == 1 ? i : nb == 2 ? i >> 1 : (i * 171) >> 9, o = 8 * (i - g * nb);
            const Group q = group(S, ga, g);
            int mx = 0;
            auto widen = [&](double v) { mx = max(mx, __double2hiint(v) & 0x7fffffff); };
            if (nOct - o <= 4) {
              double x[4][2];
              load_octets<4>(q, S.oct, o, kp, x);
#pragma unroll
              for (int j = 0; j < 8; ++j) widen(x[j >> 1][j & 1]);
            } else {
              double x[8][2];
              load_octets<8>(q, S.oct, o, kp, x);
#pragma unroll
              for (int j = 0; j < 16; ++j) widen(x[j >> 1][j & 1]);
            }
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            if (kp == 0) atomicMax(&S.expo[q.ex], mx);
          }
        }
        if (more) {
          __syncwarp();
          if (lane == 0) mbar_arrive(ex_full(sl));
        }
      }
      if (chunk == 0) continue;
      // digits of the chunk before
      const int sl = (chunk - 1) % SLOTS;
      Slot& S = slots[sl];
      const int nOct = S.noct;
      if (nOct < 0) break;
      if (nOct > 0) {
        if (!mbar_wait_warp(ex_full(sl), ((chunk - 1) / SLOTS) & 1, abort_flag, err, 18)) break;
        const int ga = (S.rows + 7) >> 3, G8 = ga + ((S.nt + 7) >> 3), nst = (nOct + 1) >> 1;
        // items (stage, group): elements loaded one item ahead, operand records two
        int t = 0, g = warp, step0 = step;
        auto next = [&](int& t, int& g) {
          g += CONV;
          while (g >= G8) {
            g -= G8;
            ++t;
          }
        };
        while (g >= G8) {
          g -= G8;
          ++t;
        }
        int t1 = t, g1 = g;
        next(t1, g1);
        Group q{}, q1{};
        int4 f1[2];
        double x[2][2];
        if (t < nst) {
          q = group(S, ga, g);
          load_octets<2>(q, S.oct, 2 * t, kp, x);
        }
        if (t1 < nst) {
          q1 = group(S, ga, g1);
          load_refs<2>(q1, S.oct, 2 * t1, f1);
        }
        int done = 0;   // stages this warp has arrived at
        while (!stop) {
          // arrive at the stages before the next item's
          for (; done < min(t, nst); ++done, ++step) {
            const int st = step % STAGES;
            if (step >= STAGES && !mbar_wait_warp(empty(st), ((step / STAGES) - 1) & 1, abort_flag, err, 12)) {
              stop = true;
              break;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(full(st));
          }
          if (stop || t >= nst) break;
          const int st = (step0 + t) % STAGES;
          if (step0 + t >= STAGES &&
              !mbar_wait_warp(empty(st), (((step0 + t) / STAGES) - 1) & 1, abort_flag, err, 12)) {
            stop = true;
            break;
          }
          int t2 = t1, g2 = g1;
          next(t2, g2);
          double y[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
          if (t1 < nst) load_pairs<2>(q1, S.oct, 2 * t1, kp, f1, y);
          Group q2 = q1;
          if (t2 < nst) {
            q2 = group(S, ga, g2);
            load_refs<2>(q2, S.oct, 2 * t2, f1);
          }
          const int e = max(S.expo[q.ex] >> 20, 1);
          const uint32_t d = saddr(smem + st * STAGE_BYTES) + q.dst;
#pragma unroll 1
          for (int j = 0; j < 2; ++j)   // rolled: the loop body stays small for the instruction cache
            store_digits(j ? x[1][0] : x[0][0], j ? x[1][1] : x[0][1], e, d + 128u * j, q.dig);
          q = q1;
          q1 = q2;
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j >> 1][j & 1] = y[j >> 1][j & 1];
          t = t1;
          t1 = t2;
          g1 = g2;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(slot_empty(sl));
    }
  } else if (warp < W_DRAIN) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == W_MMA) {
      // ---- MMA issuer
      if (lane == 0) {
        int step = 0, tog = 0;
        int used0 = 0, used1 = 0;
        for (int chunk = 0;; ++chunk) {
          const int sl = chunk % SLOTS;
          if (!mbar_wait(slot_full(sl), (chunk / SLOTS) & 1, abort_flag, err, 13)) goto mma_done;
          const int nOct = slots[sl].noct, n = (slots[sl].nt + 15) & ~15;
          mbar_arrive(slot_empty(sl));
          if (nOct < 0) break;
          if (nOct == 0) continue;
          const bool wide = n > 32;
          const int b0 = wide ? 0 : tog;
          if (!wide) tog ^= 1;
          if (b0 == 0) {
            if (used0 > 0 && !mbar_wait(acc_empty(0), (used0 - 1) & 1, abort_flag, err, 14)) goto mma_done;
            ++used0;
          }
          if (b0 == 1 || wide) {
            if (used1 > 0 && !mbar_wait(acc_empty(1), (used1 - 1) & 1, abort_flag, err, 14)) goto mma_done;
            ++used1;
          }
          const uint32_t d = tmem + 256u * b0;
          for (int t = 0; t < (nOct + 1) >> 1; ++t, ++step) {
            const int st = step % STAGES;
            if (!mbar_wait(full(st), (step / STAGES) & 1, abort_flag, err, 15)) goto mma_done;
            fence_after();
            const uint32_t base = saddr(smem + st * STAGE_BYTES);
            const uint64_t da = f64_sdesc(base), db = f64_sdesc(base + A_BYTES);
            const uint32_t acc = t > 0;
            if (n == 16) stage_mmas<16>(d, da, db, acc);
            else if (n == 32) stage_mmas<32>(d, da, db, acc);
            else if (n == 48) stage_mmas<48>(d, da, db, acc);
            else stage_mmas<64>(d, da, db, acc);
            mma_commit(empty(st));
          }
          mma_commit(acc_full(b0));
        }
        goto mma_end;
      mma_done:
        *abort_flag = 1;
      mma_end:
        // every MMA this thread issued has finished before TMEM is released
        mma_commit(mma_fin);
        mbar_wait_exit(mma_fin, 0, err);
      }
      __syncwarp();
    } else if (warp == W_HEAD) {
      // ---- header: the work list, up to SLOTS chunks ahead
      int chunk = 0;
      bool stop = false;
      for (int ui = blockIdx.x; ui < nunits && !stop;) {
        // the next unit is claimed while this one is read
        int nx = 0;
        if (lane == 0) nx = G + atomicAdd(next, 1);
        const F64Unit* u = units + ui;
        const int nseg = u->nseg, cs = u->cs, urows = u->rows;
        int s = u->sg, k0 = u->k0, left = u->noct, ci = 0;
        int rs0[F64_TM / 32] = {}, rm[F64_TM / 32] = {};   // the lane's rows of the unit
        do {
          // lane o: segment, first k and length of the chunk's octet o
          const int nOct = min(F64_CHUNK, left);
          int os = s, ok = 0, oc = 0;
          if (nOct > 0) {
            const int K = s + lane < nseg ? colref[cs + s + lane].kt >> 1 : 0;
            int pre = max((K - (lane == 0 ? k0 : 0) + 7) >> 3, 0);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const int v = __shfl_up_sync(0xffffffffu, pre, d);
              if (lane >= d) pre += v;
            }
            const int o = min(lane, nOct - 1);
            int j = 0;   // inclusive counts <= o
#pragma unroll
            for (int d = 16; d > 0; d >>= 1)
              if (__shfl_sync(0xffffffffu, pre, j + d - 1) <= o) j += d;
            const int before = __shfl_sync(0xffffffffu, pre, max(j - 1, 0));
            const int Kj = __shfl_sync(0xffffffffu, K, j);
            ok = j == 0 ? k0 + 8 * o : 8 * (o - before);
            os = s + j;
            oc = lane < nOct ? min(8, Kj - ok) : 0;
            s = __shfl_sync(0xffffffffu, os, nOct - 1);
            k0 = __shfl_sync(0xffffffffu, ok, nOct - 1) + 8;
            if (k0 >= __shfl_sync(0xffffffffu, Kj, nOct - 1)) {
              ++s;
              k0 = 0;
            }
          }
          const int sl = chunk % SLOTS;
          if (chunk >= SLOTS && !mbar_wait_warp(slot_empty(sl), ((chunk / SLOTS) - 1) & 1, abort_flag, err, 16)) {
            stop = true;
            break;
          }
          Slot& S = slots[sl];
          if (lane < F64_CHUNK) S.oct[lane] = make_int2(os, ok * 16 + oc);
          for (int i = lane; i < F64_TM + F64_TN; i += 32) S.expo[i] = 0;
          if (ci == 0) {
            const int pos0 = u->pos0, npos = u->npos, row0 = u->row0;
#pragma unroll
            for (int i = 0; i < F64_TM / 32; ++i) {
              const int r = lane + 32 * i, rr = row0 + min(r, urows - 1);
              const int pos = locate(rows, pos0, npos, rr);
              S.pos[r] = pos;
              rs0[i] = rows[pos].s0;
              rm[i] = rr - rows[pos].pre;
            }
          }
#pragma unroll
          for (int i = 0; i < F64_TM / 32; ++i) {
            S.s0[lane + 32 * i] = rs0[i];
            S.m[lane + 32 * i] = rm[i];
          }
          if (lane == 0) {
            S.noct = nOct;
            S.first = ci == 0;
            S.ci = ci;
            S.rows = urows;
            S.n0 = u->n0;
            S.nt = u->nt;
            S.cs = cs;
            S.trans = u->trans;
            S.part = u->part;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(slot_full(sl));
          ++chunk;
          ++ci;
          left -= nOct;
        } while (left > 0);
        ui = __shfl_sync(0xffffffffu, nx, 0);
      }
      // the last CTA to get here clears the counters for the next launch
      if (lane == 0 && atomicAdd(next + 1, 1) == G - 1) {
        next[0] = 0;
        next[1] = 0;
      }
      const int sl = chunk % SLOTS;
      if (!stop && (chunk < SLOTS || mbar_wait_warp(slot_empty(sl), ((chunk / SLOTS) - 1) & 1, abort_flag, err, 16))) {
        if (lane == 0) {
          slots[sl].noct = -1;
          mbar_arrive(slot_full(sl));
        }
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
    // ---- drain
    const int dw = warp - W_DRAIN, half = dw >> 2, quarter = warp & 3;
    const int r = quarter * 32 + lane;
    const uint32_t tq = tmem + (uint32_t(quarter * 32) << 16);
    double* stg = reinterpret_cast<double*>(smem + STG_OFF) + dw * 32 * STG_LD;
    uint64_t* ptrs = reinterpret_cast<uint64_t*>(smem + PTR_OFF) + dw * 32;
    int tog = 0, seen0 = 0, seen1 = 0;
    // the lane's row: place of its output, its factor (alpha = +-1 apart from others),
    // whether C is added to
    double* out = nullptr;
    int64_t cstr = 0;
    double alpha = 1.0;
    int m = 0, s0 = 0;
    bool rv = false, flip = false, any_other = false, acc0 = false, direct = false;
    for (int chunk = 0;; ++chunk) {
      const int sl = chunk % SLOTS;
      if (!mbar_wait_warp(slot_full(sl), (chunk / SLOTS) & 1, abort_flag, err, 17)) break;
      Slot& S = slots[sl];
      const int nOct = S.noct;
      if (nOct < 0) break;
      const int nt = S.nt, n16 = (nt + 15) & ~15, nrows = S.rows;
      if (S.first) {
        const F64Row R = rows[S.pos[r]];
        const int64_t pt = S.part;
        m = S.m[r];
        s0 = R.s0;
        rv = r < nrows;
        direct = pt >= 0 || S.trans;
        cstr = pt >= 0 ? F64_TM : R.ldc;   // stride of a column (direct)
        out = pt >= 0 ? part + pt + r
                      : (S.trans ? R.C + m + int64_t(S.n0) * R.ldc : R.C + int64_t(m) * R.ldc + S.n0);
        alpha = pt >= 0 ? 1.0 : R.alpha;
        const long long ab = __double_as_longlong(alpha);
        flip = ab == __double_as_longlong(-1.0);
        any_other = __any_sync(0xffffffffu, ab != __double_as_longlong(1.0) && !flip);
        acc0 = pt < 0 && (R.m2 & 1);
      }
      const bool old = S.ci > 0 || acc0;
      const bool any_old = __any_sync(0xffffffffu, old);
      const bool wide = n16 > 32;
      const int b0 = wide ? 0 : tog;
      int ea = 1;
      bool special = false;   // a row or column of the tile holds an infinity or a NaN
      if (nOct > 0) {
        if (!wide) tog ^= 1;
        if (!mbar_wait_warp(ex_full(sl), (chunk / SLOTS) & 1, abort_flag, err, 18) ||
            !mbar_wait_warp(acc_full(b0), (b0 ? seen1 : seen0) & 1, abort_flag, err, 19))
          break;
        ++(b0 ? seen1 : seen0);
        fence_after();
        ea = rv ? max(S.expo[r] >> 20, 1) : 1;
        special = __any_sync(0xffffffffu, ea == F64_SPECIAL ||
                                              (lane < nt && (S.expo[F64_TM + lane] >> 20) == F64_SPECIAL) ||
                                              (lane + 32 < nt && (S.expo[F64_TM + 32 + lane] >> 20) == F64_SPECIAL));
      }
      if (!direct) {
        // row pointers for the staged stores; bit 0: add to C
        ptrs[lane] = reinterpret_cast<uint64_t>(out) | (old ? 1u : 0u);
        __syncwarp();
      }
      // (a quarter without rows has nothing to do)
      for (int cb = half * (n16 >> 1); cb < (half + 1) * (n16 >> 1) && cb < nt && quarter * 32 < nrows; cb += 8) {
#pragma unroll 1
        for (int hh = 0; hh < 8; hh += 4) {
          double v[4] = {0.0, 0.0, 0.0, 0.0};
          if (nOct > 0) {
            float a[8][4];
            bool bad = false;
            uint32_t again = 0;   // elements that digits do not give (well enough)
            __syncwarp();   // the stores of the columns before diverge; the load is .aligned
            tmem_ld8x4(tq + 256u * b0 + uint32_t(cb + hh), uint32_t(n16), a);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              bool bd;
              int64_t hi;
              uint32_t lo;
              f64_combine(a[0][i], a[1][i], a[2][i], a[3][i], a[4][i], a[5][i], a[6][i], a[7][i], hi, lo);
              int lead;
              v[i] = f64_assemble_fast(hi, lo, ea, max(S.expo[F64_TM + min(cb + hh + i, nt - 1)] >> 20, 1), flip, &bd,
                                       &lead);
              bad |= bd && rv;
              if (FINE && f64_weak(lead)) again |= 1u << i;
            }
            if (__any_sync(0xffffffffu, bad)) {   // results outside the normal range
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                int64_t hi;
                uint32_t lo;
                f64_combine(a[0][i], a[1][i], a[2][i], a[3][i], a[4][i], a[5][i], a[6][i], a[7][i], hi, lo);
                v[i] = assemble_any(hi, lo, ea, max(S.expo[F64_TM + min(cb + hh + i, nt - 1)] >> 20, 1), flip);
              }
            }
            if (special || (FINE && __any_sync(0xffffffffu, again != 0))) {
              const int xa = rv ? S.expo[r] : 0;
#pragma unroll
              for (int i = 0; i < 4; ++i) {   // (a sum of nothing but zeros is one)
                const int xb = S.expo[F64_TM + min(cb + hh + i, nt - 1)];
                const bool sp = (xa >> 20) == F64_SPECIAL || (xb >> 20) == F64_SPECIAL;
                const bool terms = (xa != 0 && xb != 0) || __double_as_longlong(v[i]) << 1 != 0;
                if (!rv || cb + hh + i >= nt || !(sp || terms)) again &= ~(1u << i);
                else if (sp) again |= 1u << i;
              }
              for (uint32_t left = __ballot_sync(0xffffffffu, again != 0); left; left &= left - 1) {
                const int l = __ffs(int(left)) - 1;
                const uint32_t todo = __shfl_sync(0xffffffffu, again, l);
                const int ml = __shfl_sync(0xffffffffu, m, l), sl0 = __shfl_sync(0xffffffffu, s0, l);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  if (!(todo >> i & 1u)) continue;
                  const double x = chunk_dot(&S, rowref + sl0, colref + S.cs, ml, S.n0 + cb + hh + i, nOct);
                  if (lane == l) v[i] = flip ? -x : x;
                }
              }
            }
          }
          if (any_other) {   // factors other than +-1 (warp-uniform)
            asm volatile("" ::: "memory");   // kept a branch: FP64 instructions are slow
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] *= flip ? 1.0 : alpha;
          }
          if (direct) {
            if (rv) {
              double* p = out + int64_t(cb + hh) * cstr;
              if (any_old) {
                double c[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) c[i] = old && cb + hh + i < nt ? p[i * cstr] : 0.0;
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] += c[i];
              }
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (cb + hh + i < nt) p[i * cstr] = v[i];
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) stg[lane * STG_LD + hh + i] = v[i];
          }
        }
        if (!direct) {
          // 8 columns of 32 rows through shared memory: 64 bytes of 4 rows per store
          __syncwarp();
          const int cc = lane & 7;
          double v[8];
          double* p[8];
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            const int sr = 4 * it + (lane >> 3);
            const uint64_t po = ptrs[sr];
            v[it] = stg[sr * STG_LD + cc];
            const bool on = quarter * 32 + sr < nrows && cb + cc < nt;
            p[it] = on ? reinterpret_cast<double*>(po & ~uint64_t(1)) + cb + cc : nullptr;
            if (any_old && on && (po & 1)) v[it] += *p[it];
          }
#pragma unroll
          for (int it = 0; it < 8; ++it)
            if (p[it]) *p[it] = v[it];
          __syncwarp();
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) {
        if (nOct > 0) {
          mbar_arrive(acc_empty(b0));
          if (wide) mbar_arrive(acc_empty(1));
        }
        mbar_arrive(slot_empty(sl));
      }
      if (*abort_flag) break;
    }
  }
  fence_before();
  __syncthreads();
  if (warp == W_MMA) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// C = alpha * (sum of a split tile's partial sums, in K order) (+ C)
__global__ void __launch_bounds__(256) gemm_f64_reduce_kernel(const F64Red* __restrict__ reds,
                                                              const F64Row* __restrict__ rows,
                                                              const double* __restrict__ part) {
  const F64Red t = reds[blockIdx.x];
  const int64_t stride = int64_t(F64_TM) * t.n16;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < F64_TM * t.nt; e += gridDim.y * 256) {
    const int r = e & (F64_TM - 1), c = e / F64_TM;
    if (r >= t.rows) continue;
    const double* p = part + t.part + e;
    double s = p[0];
#pragma unroll 4
    for (int q = 1; q < t.nparts; ++q) s += p[q * stride];
    int pos = t.pos0;
    while (rows[pos].pre + (rows[pos].m2 >> 1) <= t.row0 + r) ++pos;
    const F64Row R = rows[pos];
    const int m = t.row0 + r - R.pre;
    double* o = t.trans ? R.C + m + int64_t(t.n0 + c) * R.ldc : R.C + int64_t(m) * R.ldc + t.n0 + c;
    s *= R.alpha;
    *o = (R.m2 & 1) ? *o + s : s;
  }
}

}  // namespace

namespace {

template <bool FINE>
void launch_tc(const F64Unit* units, int nunits, const F64Row* rows, const F64Ref* rowref, const F64Ref* colref,
               double* part, int* next, int* err, int nsm, cudaStream_t st) {
  // the shared-memory opt-in is a per-device attribute of the kernel (devices past 63
  // set it on every launch)
  static std::atomic<uint64_t> attr_set{0};
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = (dev >= 0 && dev < 64) ? (uint64_t(1) << dev) : 0;
  if (!bit || !(attr_set.load(std::memory_order_relaxed) & bit)) {
    // the register split in the kernel draws on exactly REGS registers per thread
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, gemm_f64_tc_kernel<FINE>) != cudaSuccess || fa.numRegs != REGS)
      throw CudaError("gemm_f64_tc_kernel: built with another register count");
    if (cudaFuncSetAttribute(gemm_f64_tc_kernel<FINE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) ==
        cudaSuccess)
      attr_set.fetch_or(bit, std::memory_order_relaxed);
  }
  const int grid = nunits < nsm ? nunits : nsm;
  gemm_f64_tc_kernel<FINE><<<grid, THREADS, SMEM_BYTES, st>>>(units, nunits, rows, rowref, colref, part, next, err);
}

}  // namespace

void launch_gemm_f64_tc(const F64Unit* units, int nunits, const F64Row* rows, const F64Ref* rowref,
                        const F64Ref* colref, double* part, const F64Red* reds, int nreds, int* next, int* err, int nsm,
                        bool fine, cudaStream_t st) {
  if (nunits <= 0) return;
  if (fine) launch_tc<true>(units, nunits, rows, rowref, colref, part, next, err, nsm, st);
  else launch_tc<false>(units, nunits, rows, rowref, colref, part, next, err, nsm, st);
  if (nreds > 0) gemm_f64_reduce_kernel<<<dim3(unsigned(nreds), 4), 256, 0, st>>>(reds, rows, part);
}

}  // namespace dmrg
