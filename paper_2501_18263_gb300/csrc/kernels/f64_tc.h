// Tensor-core FP64 grouped GEMM shared by exec_cuda.cu and f64_tc.cu.
#pragma once
#include <cuda_runtime.h>

#include "../core/f64_plan.h"

namespace dmrg {

// one launch over the units of a plan and, when some are split over K, one over its
// reductions; err is a device int that receives a nonzero code when a bounded wait
// gives up; fine: sums too small for their digits are computed again by multiply-adds
// (f64_weak); next: two device ints of the plan, zero before its first launch, through
// which the CTAs claim units (zero again when the launch ends)
void launch_gemm_f64_tc(const F64Unit* units, int nunits, const F64Row* rows, const F64Ref* rowref,
                        const F64Ref* colref, double* part, const F64Red* reds, int nreds, int* next, int* err, int nsm,
                        bool fine, cudaStream_t st);

// the same problems by plain FP64 multiply-adds, every element's terms in the order of
// its segments and k: tiles (the first nlong, with plong pieces, are long sums) and the
// prefix sums of their pieces (npieces the last)
void launch_gemm_f64_plain(const F64Unit* tiles, const int* pieces, int nlong, int plong, int ntiles, int npieces,
                           const F64Row* rows, const F64Ref* rowref, const F64Ref* colref, int* err,
                           cudaStream_t st);

}  // namespace dmrg
