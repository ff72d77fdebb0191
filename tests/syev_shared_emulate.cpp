// Shared memory of the eigensolver's reduction (csrc/kernels/syev_shared.h): vectors in
// shared memory (2 or 3) for order n, -1 where the order is refused; its bytes.
#include "kernels/syev_shared.h"

extern "C" int syev_vectors(int n, long* bytes) {
  try {
    const dmrg::SyevShared s = dmrg::syev_shared(n);
    *bytes = long(s.bytes);
    return s.len < n + 2 ? -2 : s.far ? 2 : 3;
  } catch (const std::runtime_error&) {
    return -1;
  }
}
