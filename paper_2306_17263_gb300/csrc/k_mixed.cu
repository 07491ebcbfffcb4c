// MS_FP32_REFINED: the step of Sec. 3.4 in FP32 arithmetic with accuracy won back by
// exact coefficients, float-float intermediates where the scheme cancels, and refinement.
//
// Scaling.  Every operator is applied in an integer-coefficient form so that FP32 adds
// rounding noise, and coherent errors of coefficients below the solve's tolerance:
//   G~ = 12 G = (12 beta) u + L u                  (filter of Eq. "eq:ell", L = h^2 Delta_h)
//   y  = A^{-1} (D1~ G~)                           (Pade of App. A.1, D1~ the plain difference)
//   6 P~ x = b,  6 P~ = 6 c1 h^2 - 6 Lx - 6 Ly - Lx Ly   (P1 of Def. "def:operatorsP" times 6 h^2)
// Coefficients that are not exact in FP32 (12 beta, explicit rows of A^{-1}, the end corrections, the last
// level of the solve and the final scale) are carried as hi + lo pairs.  One FP32 number each are rho of the
// recurrences (1.1e-9 off, its gain at theta = 0 exact: an error of theta^2 times that), the decaying vector of the
// end corrections (6e-11) and the earlier levels of the solve, a Chebyshev polynomial ((36 / D)^2 2^-25, 1.4e-11 at
// the stability limit).  Long runs at 64^2 to 256^2 drift by 1e-10 of omega T and less against FP64.  A small term
// that is added to a large one again and again the same way is a coherent error too: the filter's low part, the
// farther rows of the end corrections and the far taps of explicit rows join small partial sums first.  With these
// scalings the increments are
//   E += (12 Z / r) x_E,   H_x += (12 / (r Z)) x_Hx,   H_y += (12 / (r Z)) x_Hy.
//
// Cancellation.  The Pade derivative of a resolved field is a difference of nearly equal
// values (|D1 G| ~ theta |G|, theta = pi k h), so an FP32 rounding of G at the level of |G|
// would be amplified by 1/theta in every step.  The kernels therefore take the first
// differences of the float-float state, (hi_{m+1} - hi_m) + (lo_{m+1} - lo_m), filter the
// differences (the filter commutes with D1~), and only then apply the well-conditioned A^{-1}.
// The last level of the solve is added to the state apart from the right-hand side, so that no rounding of the
// solution itself shrinks every increment the same way.  The state is a float-float pair updated with
// error-free transformations.
//
// Kernels (k_tiled.cu): the derivatives along both axes, then the solve and the update, per half-step,
// i.e. four launches per time step.
#include <cmath>
#include <string>

#include "k_fp64.cuh"
#include "k_mixed.cuh"
#include "k_tiled.cuh"

namespace ms {

namespace {
thread_local std::string g_mixed_err;

struct Split {
  float hi, lo;
};
Split split(double v) {
  Split s;
  s.hi = (float)v;
  s.lo = (float)(v - (double)s.hi);
  return s;
}
}  // namespace

const char* mixed_last_error() { return g_mixed_err.c_str(); }

MixedConsts mixed_consts(const ms_grid* g) {
  const double c1h2 = g->c1 * g->h * g->h;
  const Split cb = split(12.0 * g->beta);
  const Split d = split(6.0 * c1h2);
  const Split sE = split(12.0 * g->Z / g->desc.r);
  const Split sH = split(12.0 / (g->desc.r * g->Z));
  MixedConsts k;
  k.cb_hi = cb.hi;
  k.cb_lo = cb.lo;
  k.d_hi = d.hi;
  k.d_lo = d.lo;
  k.omega = (float)(2.0 / (12.0 * c1h2 + 32.0));
  k.sE_hi = sE.hi;
  k.sE_lo = sE.lo;
  k.sH_hi = sH.hi;
  k.sH_lo = sH.lo;
  return k;
}

ms_status step_mixed(ms_grid* g, int* nl) {
  const double N1 = g->N + 1.0, Nd = g->N;
  const double ne = N1 * N1, nh = Nd * N1;  // points of E_z and of each H component
  // Step 1: b on E_z in two planes, then the E solve and update
  walk_d(g, 0);
  // recorded bytes: the state each launch must touch (8 B per point per float-float read or
  // write), the algorithmic bytes of a step being 48 B per cell (each component read and written
  // once); the right-hand-side planes are intermediates and are not counted
  prof_mark(g, KK_CURL32, 16.0 * nh);                        // H_x, H_y (hi, lo) read
  // sources in the units of b: 6 h^2 P1 x = s b, s the planes' factor, with E += (12 Z / r) x, so
  // b = (h^3 r^2 / (2 Z)) R / s; H += (12 / (r Z)) x, b = (h^3 r^2 Z / 2) R / s
  const double hr2 = g->h * g->h * g->h * g->desc.r * g->desc.r / plane_rhs_scale(g);
  const double scale_e = hr2 / (2.0 * g->Z), scale_h = hr2 * g->Z / 2.0;
  if (g->nsrc) {
    launch_src_time(g, scale_e, scale_h);
    prof_mark(g, KK_SRC, 0.0);
    *nl += 1;
    if (g->d_walldata) {
      launch_wall_data(g);
      prof_mark(g, KK_SRC, 8.0 * 12.0 * N1);
      *nl += 1;
    }
    launch_src_e32(g, g->s32[4], g->ld32, scale_e);
    prof_mark(g, KK_SRC, 8.0 * ne);
    *nl += 1;
  }
  walk_s(g, 0);
  prof_mark(g, KK_SOLVE32, 16.0 * ne);                       // E_z (hi, lo) read and written
  // Step 2: b_x and b_y, then both H solves and updates
  walk_d(g, 1);
  prof_mark(g, KK_CURL32, 8.0 * ne);                         // E_z (hi, lo) read
  if (g->nsrc) {
    launch_src_h32(g, g->s32[2], g->s32[3], g->ld32, scale_h);
    prof_mark(g, KK_SRC, 16.0 * nh);
    *nl += 1;
  }
  walk_s(g, 1);
  prof_mark(g, KK_SOLVE32, 16.0 * 2.0 * nh);                 // H_x, H_y (hi, lo) read and written
  if (g->nsrc) {
    launch_tick(g);
    prof_mark(g, KK_SRC, 0.0);
    *nl += 1;
  }
  *nl += 4;
  return MS_OK;
}

ms_status mixed_setup(ms_grid* g) {
  std::string err;
  for (int kind = 0; kind < 2; ++kind) {
    const int M = (kind == HALF_TO_NODE) ? g->N - 1 : g->N;
    PadeTable& t = g->pade32[kind];
    if (build_pade_table(M, g->desc.closure, kind, 1e-12, &t, &err, /*of_differences=*/true) != 0) {
      g_mixed_err = err;
      return MS_EINVAL;
    }
    // the band kernels (tracked form) hold half-widths up to kBand32Max
    if (t.K > kBand32Max) {
      g_mixed_err = "FP32 Pade band half-width outside the range the kernels hold";
      return MS_EUNSUPPORTED;
    }
    if (g->N > kTinyN && g->desc.scheme != MS_SCHEME_C4_DE) continue;  // the walks take the recurrences
    std::vector<float> whi(t.w.size()), wlo(t.w.size());
    for (size_t k = 0; k < t.w.size(); ++k) {
      Split s = split(t.w[k]);
      whi[k] = s.hi;
      wlo[k] = s.lo;
    }
    if (dev_malloc(&t.d_whi, whi.size() * sizeof(float)) != cudaSuccess ||
        dev_malloc(&t.d_wlo, wlo.size() * sizeof(float)) != cudaSuccess) {
      g_mixed_err = "cudaMalloc of FP32 Pade tables failed";
      return MS_ENOMEM;
    }
    if (cudaMemcpy(t.d_whi, whi.data(), whi.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(t.d_wlo, wlo.data(), wlo.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) {
      g_mixed_err = "copy of FP32 Pade tables failed";
      return MS_ECUDA;
    }
  }
  const ms_status wk = walk_setup(g);
  if (wk != MS_OK) {
    g_mixed_err = "the FP32 solve polynomial needs too high a degree";
    return wk;
  }
  // state and right-hand-side planes in one allocation
  const size_t pl = plane_floats(g->N);
  if (dev_malloc(&g->slab32, 10 * pl * sizeof(float)) != cudaSuccess) {
    g_mixed_err = "cudaMalloc of the FP32 planes failed";
    return MS_ENOMEM;
  }
  if (cudaMemsetAsync(g->slab32, 0, 10 * pl * sizeof(float), g->stream) != cudaSuccess) {
    g_mixed_err = "clearing the FP32 planes failed";
    return MS_ECUDA;
  }
  for (int f = 0; f < 3; ++f) {
    g->hi[f] = g->slab32 + f * pl + plane_origin(f);
    g->lo[f] = g->slab32 + (3 + f) * pl + plane_origin(f);
  }
  g->s32[2] = g->slab32 + 6 * pl + plane_origin(HX);
  g->s32[3] = g->slab32 + 7 * pl + plane_origin(HY);
  g->s32[4] = g->slab32 + 8 * pl + plane_origin(EZ);
  g->s32[1] = g->slab32 + 9 * pl + plane_origin(EZ);
  return MS_OK;
}

void mixed_teardown(ms_grid* g) {
  for (int k = 0; k < 2; ++k) {
    dev_free(g->pade32[k].d_whi);
    dev_free(g->pade32[k].d_wlo);
    g->pade32[k].d_whi = g->pade32[k].d_wlo = nullptr;
  }
  dev_free(g->slab32);
  g->slab32 = nullptr;
}

}  // namespace ms
