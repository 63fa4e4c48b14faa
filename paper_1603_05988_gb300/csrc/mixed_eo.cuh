// The mixed solvers' defect-correction cycle on the red-black Schur complement (mixed_eo.cu).
#pragma once

#include "persist_eo.cuh"
#include "reduce.cuh"

namespace dtr {

// Device buffers of one block's cycles.  Fields "both" are [parity][h][12][bi] float2 (even sites first), "half"
// [h][12][bi] in the storage of the Krylov vectors; bi = max(b, 2) columns.
struct EoBufs {
  float2 *rf;                        // both: scaled residual
  float2 *e;                         // both: the cycle's correction
  void *r, *rhat, *p, *v, *t, *w;    // half
};
inline int eo_width(int b) { return b < 2 ? 2 : b; }
size_t eo_scratch_bytes(int64_t V, int b);
// hands out the buffers in eo_scratch_bytes bytes from a 256-byte-aligned address
EoBufs eo_carve(char *w, int64_t V, int b);

// Schur complement usable: it divides by D = 4 + m0, and entries of w = H p / (2 D) stay within 8 of p's down to
// |D| = 1/2.
inline bool eo_usable(double m0) { return (4.0 + m0) * (4.0 + m0) >= 0.25; }

// rf = hs * scale * r64 and the inner problem r = rhat = p = rf_e + H rf_o / (2 D), e = 0, then the inner BiCGStab;
// store 0 FP32, 1 FP16, 2 BF16.  kernels: launches added (without the profiling kernel).
int eo_inner(const dtr_gauge_s *gauge, const EoBufs &B, const Geom &g, int b, double m0, const double2 *r64,
             const Scal *outer, Scal *inner, const Reduce &red, GridSync *gs, double inner_tol2, int maxiter,
             double hs, int store, int grid, cudaStream_t st, int *kernels);
// e on the odd sites, x64 += e / (hs * scale); counters and the choice of the next residual as k_mixed_accum.
void eo_accum(const dtr_gauge_s *gauge, const EoBufs &B, const Geom &g, int b, double m0, double2 *x, Scal *outer,
              const Scal *inner, double hs, GridSync *gs, int allow_update, cudaStream_t st);

}  // namespace dtr
