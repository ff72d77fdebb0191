// Work list of the tensor-core FP64 grouped GEMM (f64_tc.cu), built on the host from
// the problems and segments of Exec::gemm_plan.
//
// Row side and column side.  A tile has up to 128 rows (the tensor core's lanes) and
// up to 64 columns.  Problems of one launch that multiply by the same column side --
// the same list of B operands, e.g. the same psi block for every operator's rows --
// are stacked into one tall group so that their short rows fill the lanes; problems
// that share their A list are stacked the same way with the two sides exchanged
// (C^T = B^T A^T).  Every problem takes the orientation that needs fewer lanes.
//
// K runs over all segments of a problem, in octets (8 consecutive k of one segment,
// the last of a segment padded with zeros).  A chunk is at most 24 octets: up to 192 k
// the digit sums of the weights that matter are exact in the tensor core's FP32
// accumulators.  Long sums are split over units (ranges of whole chunks), whose
// partial sums are added in a fixed order by a second kernel.
#pragma once
#include <cstdint>
#include <memory>
#include <new>
#include <utility>
#include <vector>

#include "../exec.h"

namespace dmrg {

constexpr int F64_TM = 128;          // rows of a tile
constexpr int F64_TN = 64;           // most columns of a tile
constexpr int F64_CHUNK = 24;        // octets of a chunk
constexpr int F64_PR = 8, F64_PC = 4;   // rows and columns of a piece
constexpr int F64_LONG = 32;         // octets from which a plain sum counts as long (any line from 16 to 64 gives the same
                                     // time; none: GEMMs of the L = 16, D = 128 Davidson 24.6 -> 37.5 ms)

// operand of one segment, seen from its side: element (r, k) at p[r ld + k] (kt even)
// or p[k ld + r] (kt odd); K = kt / 2
struct F64Ref {
  const double* p;
  int ld, kt;
};
// one problem at its place in a group: rows [pre, pre + m2 / 2) of the stack, the
// operands of its segments at s0, accumulate flag in bit 0 of m2
struct F64Row {
  double* C;
  double alpha;
  int ldc, s0, pre, m2;
};
// one unit: a tile (stack rows row0 .., columns n0 ..) and a range of noct octets that
// begins at k0 of segment sg; part >= 0: the unit's sum goes to that place of the
// partial sums (column-major, 128 rows), otherwise to C
struct F64Unit {
  int pos0, npos;    // problems the tile's rows belong to
  int row0, rows, n0, nt;
  int cs, nseg;      // column operands: refs cs .. cs + nseg - 1
  int sg, k0, noct;
  int trans;         // 1: sides exchanged, C(row, col) at C[row + col ldc]
  int64_t part;
};
struct F64Red {
  int pos0, row0, rows, n0, nt, trans, nparts, n16;
  int64_t part;
};

// vectors whose resize leaves new elements as they are (each is written once, by the
// plan).  With these, one pass for the plain form and lists kept from plan to plan, the
// host lists of preparing a bond of L = 20, D = 256 take 12 ms of 400 instead of 31
template <class T>
struct F64Alloc : std::allocator<T> {
  template <class U>
  struct rebind { using other = F64Alloc<U>; };
  template <class U>
  void construct(U* p) noexcept { ::new (static_cast<void*>(p)) U; }
  template <class U, class... A>
  void construct(U* p, A&&... a) { ::new (static_cast<void*>(p)) U{std::forward<A>(a)...}; }
};
template <class T>
using F64List = std::vector<T, F64Alloc<T>>;

struct F64PlanHost {
  F64List<F64Ref> rowref, colref;
  F64List<F64Row> rows;
  F64List<F64Unit> units;
  // the tiles unsplit, longest sum first, and the prefix sums of their 8 x 4 pieces
  // (the plain FP64 kernel: one warp per piece)
  F64List<F64Unit> tiles;
  F64List<int> pieces;
  std::vector<F64Red> reds;
  int64_t npart = 0;   // doubles of the partial sums
  void clear() {   // empty, the memory kept
    rowref.clear(); colref.clear(); rows.clear(); units.clear();
    tiles.clear(); pieces.clear(); reds.clear();
    npart = 0;
  }
  size_t capacity_bytes() const {
    return (rowref.capacity() + colref.capacity()) * sizeof(F64Ref) + rows.capacity() * sizeof(F64Row) +
           (units.capacity() + tiles.capacity()) * sizeof(F64Unit) + pieces.capacity() * sizeof(int) +
           reds.capacity() * sizeof(F64Red);
  }
};

// what: F64_UNITS the tensor-core form, F64_TILES the plain one (alone, its problems
// are not stacked), or both
enum { F64_UNITS = 1, F64_TILES = 2 };
F64PlanHost f64_build_plan(const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s, int nsm,
                           int what = F64_UNITS | F64_TILES);
// the same into the lists of an earlier plan
void f64_build_plan(F64PlanHost& out, const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s, int nsm, int what);

// true for a launch that is faster in plain multiply-adds: a digit unit's latency (fill
// the pipeline, one chunk, drain) is longer than what little there is to compute.  The work is counted as the plain kernel pays for it, pieces of 8 x 4 and
// whole octets.  Sigma at L = 10, D = 100 / L = 6, D = 16 / L = 18, D = 24, one path
// only -> this rule: 294 -> 272, 99 -> 76, 248 -> 239 us; any line between 1.5e6 and
// 8e6 gives these times, with k counted without the octets' padding 1e6 is already too
// much (L = 24, D = 16: 300 -> 347 us).  A sum of more than F64_SMALL_K is one warp's
// chain (64 clocks per k) and goes to the units, which split it.
constexpr double F64_SMALL_MAC = 3e6;
constexpr int64_t F64_SMALL_K = 512;
bool f64_small(const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s);

// whether a run of a plan built for `forms` (GEMM_ANY, GEMM_PLAIN) goes to the plain
// kernel; throws std::logic_error when the form asked for is not among them (the plan
// may hold no work in it, and C would keep its old contents)
bool f64_run_plain(int forms, bool small, bool plain);

}  // namespace dmrg
