// FP64 deflation projection on the tensor cores by integer digits (deflate_oz.cu).
#pragma once

#include "deflate.cuh"

namespace dtr {

// Queues what the digits need of V into D->vexp (defl_oz_space_bytes(k) bytes, device); scratch: 12 k bytes; bad[0] (device):
// some column cannot be written in integers, bad[1]: some FP32 or BF16 entries have more bits than their column's integers.
size_t defl_oz_space_bytes(int k);
int defl_oz_setup(const dtr_defl_s *D, void *scratch, int *bad, cudaStream_t st);
size_t defl_oz_scratch_bytes(int k, int b);
// Partial sums as k_defl_partial's, over *chunks (<= max_chunks) chunks of sites.
int defl_oz_contract(const dtr_defl_s *D, const double2 *Z, int b, void *scratch, int max_chunks, double2 *partial,
                     int *chunks, cudaStream_t st);
// x = V W (W column-major k x b); needs no contraction before it.
int defl_oz_expand(const dtr_defl_s *D, const double2 *W, int b, void *scratch, double2 *x, cudaStream_t st);
// Two device ints each: either is set where the digits would not do, and the FP64 kernel has to run.  Entries that the
// integers cannot hold (not finite, a column below 2^-800), blocks too graded for fixed point (deflate_oz.cu).
const int *defl_oz_contract_flags(const void *scratch);
const int *defl_oz_expand_flags(const void *scratch);

}  // namespace dtr
