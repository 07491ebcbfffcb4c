// FP64 line recurrences (Pade derivatives) and polynomial P1 solves (k_rec64.cu), shared by the 2D and
// 3D grids and by the reverse pass.
#pragma once

#include "ms_internal.h"

namespace ms {

// Shortest line (rows of A) the recurrences take: its last segment (16 rows) starts beyond the rows that
// the first end corrects.
constexpr int kRecMinLine = 16 + kRecWarm + 2;

// The end correction of a closure's lines (transposed: of A^{-T}).
void line_ends(int closure, int kind, bool transposed, LineEnds* e);

// x = scale * y, y the polynomial p(T) b / p_0 in Horner form, y <- b + q[k] T y for k = m-1 .. 1,
// p(t) ~ 1 / (D - t) with the relative error of the Chebyshev polynomial of degree m on the spectrum
// [c - s, c + s] of T: 1 / T_m((D - c) / s) <= tol.
// At least degree mmin; false if kChebMax is not enough.
bool cheb_coefs(double D, double c, double s, double tol, Cheb* p, int mmin = 2);

// out (+)= scale * delta in along a line (App. A.1), or its transpose: `axis_stride_*` between points
// of a line, n0 lines apart by s0_*, n1 apart by s1_*.  Output r (0 .. rows-1) goes to point r + out_off
// of out_len; lines [lo, hi) of the n0 are live.  Without accumulation every other point is set to 0.
struct LineArgs {
  const double* in;
  double* out;
  int M;  // rows of A
  int out_len, out_off;
  int n0, n1, lo, hi;
  size_t in_sa, in_s0, in_s1, out_sa, out_s0, out_s1;
  double scale;
  int accumulate;
};
// Up to kLineBatch independent derivatives in one launch, with the same M and ends, all along the
// contiguous axis (in_sa == 1) or all across it.
constexpr int kLineBatch = 3;
void launch_line64(const LineArgs* a, int count, const LineEnds& e, bool transposed, cudaStream_t st);
// Derivatives along x (contiguous) and y of one half-step that do not depend on one another, with equal M:
// one launch where the lines are cut into short segments; false (nothing launched) otherwise.
bool launch_line64_pair(const LineArgs& x, const LineArgs& y, const LineEnds& e, bool transposed, cudaStream_t st);

// P1 x = b for one or two 2D fields in one launch; upd (if not NULL) gains upd_scale x, out (if not
// NULL) receives x (0 on the walls).  b may not be out.
struct Cheb2dField {
  const double* b;
  double* out;
  double* upd;
  Shape s;
  const double* b2 = nullptr;  // with cheb2d64_tiles only: b + b2 is the right-hand side
};
// Whether the solve of `pts` points runs all its levels in one launch (k_cheb2d64).
inline bool cheb2d64_tiles(long pts) { return pts <= 300000; }
// buf: two work planes per field, all distinct from each other and from b and out.  On the grid's stream; every
// launch is marked for the profiler as `kind`.  Returns the number of launches.
int launch_cheb2d64(ms_grid* g, int kind, const Cheb2dField* f, int nf, double* const (*buf)[2], const Cheb& p,
                    double bscale, double upd_scale);

// The same for up to three 3D components; buf: two work arrays per component, in which every wall point
// of a Dirichlet axis may hold anything (they are not read).
constexpr int kCheb3dBatch = 3;
struct Cheb3dField {
  const double* b;
  const double* y;  // set by the launcher
  double* out;
  double* upd;
  int n[3], bc[3];
};
int launch_cheb3d64(ms_grid* g, int kind, const Cheb3dField* f, double* const (*buf)[2], int count, const Cheb& p,
                    double bscale, double upd_scale);

}  // namespace ms
