// Shared memory of the tridiagonal reduction (exec_cuda.cu), by the largest order of a
// batch: 40 scalars and three vectors, or, past order 9670, where three do not fit in an
// SM's 227 KB, two; the third (the row at work, then its reflector: read once a row by
// every warp) is then a CTA's own stretch of global memory.  Plain C++.
#pragma once
#include <cstddef>
#include <stdexcept>

namespace dmrg {

struct SyevShared {
  size_t bytes;
  int len;    // doubles of a vector
  bool far;   // the third vector lies in global memory
};

inline SyevShared syev_shared(int n) {
  constexpr size_t most = 227 * 1024;
  const int len = n + 2 > 4 ? n + 2 : 4;
  auto bytes = [&](int vectors) { return sizeof(double) * (size_t(vectors) * size_t(len) + 40); };
  if (bytes(3) <= most) return {bytes(3), len, false};
  if (bytes(2) <= most) return {bytes(2), len, true};
  throw std::runtime_error("syev: matrix too large for the shared-memory workspace");
}

}  // namespace dmrg
