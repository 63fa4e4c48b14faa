// Persistent batched BiCGStab on the red-black Schur complement (persist_eo.cu).
#pragma once

#include "eo_core.cuh"
#include "persist.cuh"

namespace dtr {

// S: storage of the Krylov vectors (float, __half, __nv_bfloat16); arithmetic and the iterate are FP32.
// Fields are half-lattice [h][12][b / 2] pairs, b >= 2 (see eo_core.cuh).
template <typename S> struct EoArgs {
  const float2 *U;                                // FP32 links [site][mu][kLink32]
  float4 *x;                                      // even sites
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

// Plain FP64 BiCGStab with true-residual restarts (persist_eo64.cu).  x and z are whole-lattice fields [site][12][b],
// the others half-lattice ones [h][12][b], b >= 1.
struct Eo64Args {
  const double2 *U;                       // FP64 links [site][mu][3][3]
  double2 *x;                             // initial guess in, solution out; gs->x_nonzero 0 says that it is zero (it must
                                          // be: the iterations add to it), and the first residual is z
  const double2 *z;
  double2 *r, *rhat, *p, *v, *t, *w, *ro;  // w, ro on the odd sites
  Geom g;
  int b, logb;
  double diag;
  Scal *sc;
  double2 *partial;
  GridSync *gs;
  int max_iters, max_cycles;
  int grid;
};
int launch_persistent_eo64(const Eo64Args &ea, cudaStream_t st);

}  // namespace dtr
