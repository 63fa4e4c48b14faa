// FP64 deflation projection on the tensor cores by integer digits (deflate_oz.cu).
#pragma once

#include "deflate.cuh"

namespace dtr {

// Queues the exponents of V's columns into D->vexp (k ints, device); *bad (device): some column cannot be written in
// integers.
int defl_oz_setup(const dtr_defl_s *D, int *bad, cudaStream_t st);
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
