// FP64 deflation projection on the tensor cores by exact integer digits (deflate_oz.cu).
#pragma once

#include "deflate.cuh"

namespace dtr {

// Exponents of V's columns into D->vexp (k + 1 ints, device); D->vexp_ok: every column can be written in integers.
int defl_oz_setup(dtr_defl_s *D, cudaStream_t st);
size_t defl_oz_scratch_bytes(int k, int b);
// partial sums as k_defl_partial's, over *chunks (<= max_chunks) chunks of sites.  Entries that the integers cannot hold
// (not finite, or a column below 2^-800) set the int at the start of scratch and leave partial alone.
int defl_oz_contract(const dtr_defl_s *D, const double2 *Z, int b, void *scratch, int max_chunks, double2 *partial,
                     int *chunks, cudaStream_t st);
// x = V W (W column-major k x b), after defl_oz_contract on the same scratch; the same flag.
int defl_oz_expand(const dtr_defl_s *D, const double2 *W, int b, void *scratch, double2 *x, cudaStream_t st);

}  // namespace dtr
