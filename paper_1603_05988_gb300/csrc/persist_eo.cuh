// Persistent batched BiCGStab on the red-black Schur complement (persist_eo.cu).
#pragma once

#include "eo_core.cuh"
#include "persist.cuh"

namespace dtr {

// S: storage of the Krylov vectors (float, __half, __nv_bfloat16); arithmetic and the iterate are FP32.
// Fields are half-lattice [h][12][b], b >= 2 (see eo_core.cuh).
template <typename S> struct EoArgs {
  const float2 *U;                                // FP32 links [site][mu][3][3]
  float2 *x;                                      // even sites, interleaved complex
  typename Pair2<S>::T *r, *rhat, *p, *v, *t;     // even sites
  float4 *w;                                      // odd sites, FP32: S p = D p - H w / 2 cancels down to the smallest
                                                  // eigenvalue, so a w rounded to 11 bits would cost its digits
  Geom g;
  int b, logp;                                    // columns; log2(b / 2)
  float diag, wscale;                             // D = 4 + m0, 1 / (2 D)
  Scal *sc;
  double2 *partial;
  GridSync *gs;
  int max_iters;
  int grid;                                       // requested CTAs (0 = all co-resident)
};
template <typename S> int launch_persistent_eo(const EoArgs<S> &ea, cudaStream_t st);

}  // namespace dtr
