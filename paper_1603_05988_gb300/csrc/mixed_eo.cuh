// The mixed solvers' defect correction on the red-black Schur complement (mixed_eo.cu).
#pragma once

#include "persist_eo.cuh"
#include "reduce.cuh"

namespace dtr {

// Device buffers of one block's cycles, all in the pair layout of eo_core.cuh over bi = max(b, 2) columns: "both" is
// [parity][h][12][bi / 2] float4 (even sites first), "half" [h][12][bi / 2] in the storage of the Krylov vectors, but w,
// on the odd sites, in FP32.
struct EoBufs {
  float4 *rhi, *rlo;               // both: the residual times base, in double-float
  float4 *e;                       // both: the cycle's correction times base * fac
  void *r, *rhat, *p, *v, *t, *w;  // half
  float4 *xhi, *xlo;               // both: x times base, for the true residual (the memory of r .. v)
};
inline int eo_width(int b) { return b < 2 ? 2 : b; }
size_t eo_scratch_bytes(int64_t V, int b);
// hands out the buffers in eo_scratch_bytes bytes from a 256-byte-aligned address
EoBufs eo_carve(char *w, int64_t V, int b);

// Schur complement usable: it divides by D = 4 + m0, and ||w|| = ||H p|| / (2 |D|) stays within 8 ||p|| down to |D| = 1/2.
// At |D| <= 2 BiCGStab converged on neither system (4^4 to 8^3 x 16, eps 0.2 and 0.7, every storage), so the line's
// place there decides nothing but which kernels run out of iterations.
inline bool eo_usable(double m0) { return (4.0 + m0) * (4.0 + m0) >= 0.25; }

struct EoSolve {
  const dtr_gauge_s *gauge;
  Geom g;
  int b;
  double m0;
  double2 *x;        // FP64 iterate, [site][12][b]
  const double2 *z;
  EoBufs B;
  Scal *outer, *inner;
  Reduce red;
  GridSync *gs;
  double hs;         // norm that the inner right-hand sides are scaled to (within a factor of 2 below)
  int grid;          // CTAs of the persistent kernel (0: all SMs): a lane's share, which its other kernels keep to as well
};

// Residual of the initial guess; the caller says that x is zero, or the device finds out.  All add up to *kernels.
void eo_first_resid(const EoSolve &S, int x_is_zero, cudaStream_t st);
// Inner BiCGStab of one cycle; store 0 FP32, 1 FP16, 2 BF16.
int eo_inner(const EoSolve &S, double inner_tol2, int maxiter, int store, int grid, cudaStream_t st, int *kernels);
// e on the odd sites, x += e / (base * fac); counters, and with choose the next residual (gs->sel)
void eo_accum(const EoSolve &S, int choose, cudaStream_t st);
// residual -= A e / fac in double-float, run if gs->sel is 1 (one kernel)
void eo_update(const EoSolve &S, cudaStream_t st);
// residual = z - A x (three kernels), run if *run_flag == run_if (NULL: always)
void eo_true_resid(const EoSolve &S, int restart, const int *run_flag, int run_if, cudaStream_t st);

}  // namespace dtr
