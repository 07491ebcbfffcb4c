// Three-dimensional compact scheme: six components on the staggered unit cube (Eq. "eq:meshes"),
// boundary types of Table "tab:bc", Step 1 / Step 2 of Sec. 3.4 with
//   curl_h = [[0, -d_z, d_y], [d_z, 0, -d_x], [-d_y, d_x, 0]],
// the 7-point filter of Eq. "eq:ell" (Delta_h = D_xx + D_yy + D_zz) and the 19-point
// P1 = -(Delta_h + (h^2/6) Upsilon_h) + kappa^2 (1 + 2/r^2), Upsilon_h = D_zz D_xx + D_yy D_zz
// + D_xx D_yy (Def. "def:operatorsP").  Every component is Dirichlet (stored wall zeros) along
// the axes on which it sits on nodes and Neumann (even ghosts) along its half-node axes.
//
// MS_FP64: filter, Pade recurrences (k_rec64.cu; bands on short lines) and polynomial solves, up to three
// components per launch.
// MS_FP32_REFINED: the arithmetic of the 2D FP32 path (k_mixed.cu) carried to 3D: float-float
// state; each half-step first filters its three source components once into float-float
// G = 12 beta u + L u (k_ffilt3d32), then per axis the two Pade terms by walking warps (k_walk3d32,
// k_walkx3d32): first differences of G along the line (the filter commutes with the difference under the
// ghost rules) and A^{-1} by two first-order recurrences, accumulating the right-hand side (short lines
// by explicit table rows, k_short3d32); the solve (k_lev3d32) is a Chebyshev
// polynomial in Horner form, one level per launch.  The three components of a half-step share launches
// (14 per step).  The transform solver (k_transform.cu) is followed by Richardson sweeps (k_sweep3d32).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "grid3d.cuh"
#include "k_fp64.cuh"
#include "k_pdl.cuh"
#include "k_rec64.cuh"
#include "k_tiled.cuh"
#include "k_src3.cuh"
#include "k_transform.cuh"
#include "k_walk_dev.cuh"

namespace ms {

Shape3 field_shape3(int N, int c) {
  Shape3 s;
  for (int a = 0; a < 3; ++a) {
    const bool node = (c < 3) ? (a != c % 3) : (a == c % 3);
    s.bc[a] = node ? DIR : NEU;
    s.n[a] = node ? N + 1 : N;
  }
  return s;
}

struct Grid3D {
  Shape3 sh[6];
  double* f64[6] = {};
  float* hi[6] = {};
  float* lo[6] = {};
  double* s64[9] = {};  // FP64: G[3], R[3], and, with G again, the work planes of the solves; FP32 grids use [0], [1]
  double* slab64 = nullptr;  // FP64: storage of s64 (one allocation: each takes as long as many steps of a small grid)
  float* s32[3] = {};   // FP32: R
  float* gh[3] = {};    // FP32: filtered components G~ (hi, lo) of one half-step, slot c % 3
  float* gl[3] = {};
  double* dview[6] = {};  // FP32_REFINED grids: FP64 copy of the state for the diagnostics
  size_t nmax = 0;      // points of the largest component
  int solver = MS_SOLVER_RICHARDSON;  // FP32_REFINED: P1 solve by Richardson sweeps or by transforms
  TransformSolver* ts = nullptr;       // made when the transform solver is first selected
  int ts_sweeps = 0;                   // refinement sweeps after a transform solve
};

namespace {

thread_local std::string g_err3;

ms_status fail3(ms_status s, const std::string& m) {
  set_last_error(m.c_str());
  return s;
}

#define MS3_CUDA(call)                                                                            \
  do {                                                                                            \
    cudaError_t e_ = (call);                                                                      \
    if (e_ != cudaSuccess) return fail3(MS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define MS3_TRY(expr)           \
  do {                          \
    ms_status s_ = (expr);      \
    if (s_ != MS_OK) return s_; \
  } while (0)

__device__ __forceinline__ bool unk3(const Shape3& s, int i, int j, int k) {
  return interior(s.bc[0], i, s.n[0]) && interior(s.bc[1], j, s.n[1]) && interior(s.bc[2], k, s.n[2]);
}

__device__ __forceinline__ size_t at3(const Shape3& s, int i, int j, int k) {
  return ((size_t)k * s.n[1] + j) * s.n[0] + i;
}

dim3 grid3(const Shape3& s, dim3 blk) {
  return dim3((s.n[0] + blk.x - 1) / blk.x, (s.n[1] + blk.y - 1) / blk.y, s.n[2]);
}

// ---------------------------------------------------------------------------------------
// FP64 kernels

// G = beta u + (1/12) L u, L = h^2 Delta_h (7 points), 0 at wall points; three components per launch.
struct Filter3d64Args {
  const double* u[3];
  double* G[3];
  Shape3 s[3];
  int nz;  // planes of the largest component
};
__global__ void k_filter3d64(Filter3d64Args A, double c0) {
  pdl_wait();
  const int f = blockIdx.z / A.nz, k = blockIdx.z - f * A.nz;
  const Shape3& s = A.s[f];
  const double* __restrict__ u = A.u[f];
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= s.n[0] || j >= s.n[1] || k >= s.n[2]) return;
  const size_t p = at3(s, i, j, k);
  if (!unk3(s, i, j, k)) {
    A.G[f][p] = 0.0;
    return;
  }
  const double nb = (u[at3(s, clampi(i - 1, s.n[0]), j, k)] + u[at3(s, clampi(i + 1, s.n[0]), j, k)]) +
                    (u[at3(s, i, clampi(j - 1, s.n[1]), k)] + u[at3(s, i, clampi(j + 1, s.n[1]), k)]) +
                    (u[at3(s, i, j, clampi(k - 1, s.n[2]))] + u[at3(s, i, j, clampi(k + 1, s.n[2]))]);
  A.G[f][p] = fma(c0, u[p], nb * (1.0 / 12.0));  // c0 = beta - 6/12
}

// Pade band along AXIS (App. A.1): out[o] (+)= scale * sum_t W(r, t) in[r - left + t], r = o - out_off,
// at every point of the output component; the two other coordinates are shared with the input.
template <int AXIS>
__global__ void k_pade3d64(const double* __restrict__ in, double* __restrict__ out, Shape3 so, Shape3 si,
                           const double* __restrict__ tab, int rows, int n_in, int left, int K, int B,
                           int all_explicit, int out_off, double scale, int accumulate) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
  if (x >= so.n[0] || y >= so.n[1]) return;
  const size_t po = at3(so, x, y, z);
  const int o = AXIS == 0 ? x : (AXIS == 1 ? y : z);
  const int r = o - out_off;
  double v = 0.0;
  if (r >= 0 && r < rows) {
    const double* w = pade_row_ptr(tab, r, rows, K, B, all_explicit);
    size_t base, stride;
    if (AXIS == 0) {
      base = at3(si, 0, y, z);
      stride = 1;
    } else if (AXIS == 1) {
      base = at3(si, x, 0, z);
      stride = (size_t)si.n[0];
    } else {
      base = at3(si, x, y, 0);
      stride = (size_t)si.n[0] * si.n[1];
    }
    const int k0 = r - left;
    for (int t = 0; t < 2 * K + 2; ++t) {
      const int kk = k0 + t;
      if (kk < 0 || kk >= n_in) continue;
      v = fma(w[t], in[base + (size_t)kk * stride], v);
    }
    v *= scale;
  }
  out[po] = accumulate ? out[po] + v : v;
}

__global__ void k_zero_walls3d64(double* __restrict__ u, Shape3 s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
  if (i >= s.n[0] || j >= s.n[1]) return;
  if (!unk3(s, i, j, k)) u[at3(s, i, j, k)] = 0.0;
}

// Superposition of separable modes: out = sum_q coef[q] tx[q][i] ty[q][j] tz[q][k].
__global__ void k_mode_field3(double* __restrict__ out, Shape3 s, const double* __restrict__ tx,
                              const double* __restrict__ ty, const double* __restrict__ tz,
                              const double* __restrict__ coef, int nm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
  if (i >= s.n[0] || j >= s.n[1]) return;
  double v = 0.0;
  for (int q = 0; q < nm; ++q)
    v += coef[q] * tx[(size_t)q * s.n[0] + i] * ty[(size_t)q * s.n[1] + j] * tz[(size_t)q * s.n[2] + k];
  out[at3(s, i, j, k)] = unk3(s, i, j, k) ? v : 0.0;
}

// ---------------------------------------------------------------------------------------
// FP32_REFINED kernels

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// (hi, lo) += (s_hi + s_lo) x with error-free transformations (two-product by FMA, Knuth two-sum), on two
// independent pairs at once.
__device__ __forceinline__ void ff_add_scaled3_2(float2& hi, float2& lo, float2 x, float2 s_hi, float2 s_lo) {
  const float2 p = mul2(s_hi, x);
  float2 e = fma2(s_hi, x, neg2(p));
  e = fma2(s_lo, x, e);
  const float2 s = add2(hi, p);
  const float2 bb = sub2(s, hi);
  const float2 err = add2(sub2(hi, sub2(s, bb)), sub2(p, bb));
  const float2 l = add2(lo, add2(err, e));
  const float2 h2 = add2(s, l);
  lo = sub2(l, sub2(h2, s));
  hi = h2;
}

__device__ __forceinline__ void cp4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Float-float filter of one component, Eq. "eq:ell" in the units of the FP32 step:
//   G = 12 beta u + L u,  L = h^2 Delta_h (7 points),
// with even ghosts on Neumann axes and the stored wall zeros on Dirichlet axes; G = 0 at wall
// points.  12 beta u is an exact two-product of the hi parts plus the cross terms; L u, a sum of
// first differences each taken of the float-float values (so FP32 holds it to its own relative
// accuracy), joins the low word, and two-sum renormalises the pair.  The Pade terms below then
// difference G: D1 G = (12 beta + L') D1 u, the filter commuting with the difference under the
// ghost rules (zero differences beyond the ends of a Neumann line, even ones on a Dirichlet line).
// A thread takes two rows of one column and marches along z with the planes below and above in
// registers, the next plane fetched ahead (no shared memory; the neighbour rows and columns come from L1):
// three components at 256^3 in 205 us, 75^3 in 13; planes through a ring in shared memory took 182 to 213 us
// and 21.
// The tile form before it, 32 x 16 tiles of three planes in shared memory, issued 112 instructions per 32
// points, 70 us per component at 256^3.
constexpr int FY3 = 8;
struct Filter3d32Args {  // the three components of a half-step
  const float *hi[3], *lo[3];
  float *gh[3], *gl[3];
  Shape3 s[3];
  int nz, zc;  // marches along z of the largest component, planes per march
};
__global__ void __launch_bounds__(32 * FY3, 4) k_ffilt3d32(const __grid_constant__ Filter3d32Args A, float cb_hi,
                                                          float cb_lo) {
  pdl_wait();
  const int which = blockIdx.z / A.nz, kz = blockIdx.z - which * A.nz;
  const float* __restrict__ hi = A.hi[which];
  const float* __restrict__ lo = A.lo[which];
  float* __restrict__ gh = A.gh[which];
  float* __restrict__ gl = A.gl[which];
  const Shape3& s = A.s[which];
  const int n0 = s.n[0], n1 = s.n[1], n2 = s.n[2];
  const int i = blockIdx.x * 32 + threadIdx.x, j = 2 * (blockIdx.y * FY3 + threadIdx.y);
  const int k0 = kz * A.zc, k1 = min(k0 + A.zc, n2);
  if (i >= n0 || j >= n1 || k0 >= k1) return;
  const bool two = j + 1 < n1, ux = interior(s.bc[0], i, n0);
  const bool u[2] = {ux && interior(s.bc[1], j, n1), ux && interior(s.bc[1], j + 1, n1)};
  const unsigned sz = n0 * n1;
  // rows j - 1 .. j + 2 of the column, and left and right of rows j, j + 1 (clamped: even ghosts; results
  // on walls are set to 0)
  unsigned om[4], ol[2], orr[2];
#pragma unroll
  for (int r = 0; r < 4; ++r) om[r] = clampi(j - 1 + r, n1) * n0 + i;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    ol[t] = om[t + 1] - i + clampi(i - 1, n0);
    orr[t] = om[t + 1] - i + clampi(i + 1, n0);
  }
  float hm[4], lm[4], hl[2], hr[2], sl[2];  // one plane: the column (hi, lo), left and right (hi, sum of lo)
  auto fetch = [&](int k) {
    const float* __restrict__ ph = hi + (size_t)clampi(k, n2) * sz;
    const float* __restrict__ pl = lo + (size_t)clampi(k, n2) * sz;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      hm[r] = ph[om[r]];
      lm[r] = pl[om[r]];
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      hl[t] = ph[ol[t]];
      hr[t] = ph[orr[t]];
      sl[t] = pl[ol[t]] + pl[orr[t]];
    }
  };
  float hz[2], lz[2];            // plane below
  float hc[4], lc[4], xl[2], xr[2], xs[2];  // plane k
  fetch(k0 - 1);
  hz[0] = hm[1];
  hz[1] = hm[2];
  lz[0] = lm[1];
  lz[1] = lm[2];
  auto shift = [&]() {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      hc[r] = hm[r];
      lc[r] = lm[r];
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      xl[t] = hl[t];
      xr[t] = hr[t];
      xs[t] = sl[t];
    }
  };
  fetch(k0);
  shift();
  fetch(k0 + 1);
  unsigned g[2] = {k0 * sz + om[1], k0 * sz + (two ? om[2] : om[1])};
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const bool uz = interior(s.bc[2], k, n2);
    float G[2], E[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const float c = hc[t + 1], d = lc[t + 1];
      // first differences of the hi parts; the lo parts as one sum
      const float lap = (((xl[t] - c) + (xr[t] - c)) + ((hc[t] - c) + (hc[t + 2] - c))) + ((hz[t] - c) + (hm[t + 1] - c));
      const float lol = fmaf(-6.0f, d, (xs[t] + (lc[t] + lc[t + 2])) + (lz[t] + lm[t + 1]));
      const float p = __fmul_rn(cb_hi, c);
      float e = fmaf(cb_hi, c, -p);
      e = fmaf(cb_hi, d, e);
      e = fmaf(cb_lo, c, e);
      const float x = __fadd_rn(e, lap + lol);
      const float h = __fadd_rn(p, x), bb = __fsub_rn(h, p);
      const bool live = uz && u[t];
      G[t] = live ? h : 0.0f;
      E[t] = live ? __fadd_rn(__fsub_rn(p, __fsub_rn(h, bb)), __fsub_rn(x, bb)) : 0.0f;
      hz[t] = c;
      lz[t] = d;
    }
    shift();
    if (k + 1 < k1) fetch(k + 2);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (t == 0 || two) {
        gh[g[t]] = G[t];
        gl[g[t]] = E[t];
      }
      g[t] += sz;
    }
  }
}

// Planes per march along z for nz planes of `cols` tiles: 16 (two more come in), fewer where that leaves SMs
// idle (75^3: levels of three components 28 to 31 us with 16, 17 us with 4).
int march_planes(int cols, int nz) {
  int zc = 16;
  while (zc > 4 && cols * ((nz + zc - 1) / zc) < 4 * 152) zc /= 2;
  return zc;
}

struct TermArgs {
  const float* gh;
  const float* gl;
  float* R;
  Shape3 ss, sd;
  float sign;
  int accumulate;
};
struct TermArgs2 {  // the two terms of a half-step along one axis
  TermArgs t[2];
  int nz;  // planes of the larger component
};

// Pade terms y = A^{-1} D1 G, R (+)= sign y, on lines shorter than kWalk3Min rows (grids of up to 16 cells, all
// end rows): a thread sums its explicit table row over the differences of G, hi and lo parts apart, taps
// farthest first.  Without accumulation points that no band row reaches get 0.  Indices are 32-bit.
__global__ void k_short3d32(const __grid_constant__ TermArgs2 A, int axis, int out_off, int M,
                            const float* __restrict__ whi, const float* __restrict__ wlo, int K, int B,
                            int all_explicit) {
  pdl_wait();
  const int which = blockIdx.z / A.nz;
  const TermArgs& T = A.t[which];
  const Shape3 &ss = T.ss, &sd = T.sd;
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z - which * A.nz;
  if (x >= sd.n[0] || y >= sd.n[1] || z >= sd.n[2]) return;
  const size_t pd = at3(sd, x, y, z);
  const int r = (axis == 0 ? x : (axis == 1 ? y : z)) - out_off;
  if (!unk3(sd, x, y, z) || r < 0 || r >= M) {
    if (!T.accumulate) T.R[pd] = 0.0f;
    return;
  }
  const int sa = axis == 0 ? 1 : (axis == 1 ? ss.n[0] : ss.n[0] * ss.n[1]);
  const size_t ps = at3(ss, axis == 0 ? 0 : x, axis == 1 ? 0 : y, axis == 2 ? 0 : z);
  const float* __restrict__ h = T.gh + ps;
  const float* __restrict__ l = T.gl + ps;
  auto diff = [&](int m) { return (h[(m + 1) * sa] - h[m * sa]) + (l[(m + 1) * sa] - l[m * sa]); };
  const float* wh = pade_row_ptr(whi, r, M, K, B, all_explicit);
  const float* wl = pade_row_ptr(wlo, r, M, K, B, all_explicit);
  float acc = 0.0f, lo = 0.0f;
  for (int dist = K + 1; dist >= 1; --dist) {
    for (int side = 1; side >= -1; side -= 2) {
      const int m = r + side * dist, t = m - r + K;
      if (t < 0 || t > 2 * K + 1 || m < 0 || m >= M) continue;
      const float d = diff(m);
      acc = fmaf(__ldg(wh + t), d, acc);
      lo = fmaf(__ldg(wl + t), d, lo);
    }
  }
  const float d = diff(r);
  lo = fmaf(__ldg(wl + K), d, lo);
  acc = fmaf(__ldg(wh + K), d, acc + lo);
  T.R[pd] = T.accumulate ? T.R[pd] + T.sign * acc : T.sign * acc;
}

// Pade terms along y and z on lines of at least kWalk3Min rows: the walk along y of the 2D step
// (k_tiled.cu) on the filtered G.  A lane takes one x and walks down its segment of a line, every access
// coalesced; forward recurrence with the walk, backward over groups of eight rows, the closure's end rows
// as a rank-one correction.  45 warp instructions per 32 points, where a tile form with the differences in
// shared memory issued 115: two terms at 256^3 take 88 us (3.0 to 4.6 TB/s), bound by the loads a warp has in
// flight, and took 130 to 185 us.  Shorter lines are all end rows (k_short3d32).
constexpr int kWalk3Min = 16, kW3Warps = 4;
struct Walk3Term {
  const float* gh;
  const float* gl;
  float* R;
  int nx, nq;               // lines: x, and the other transverse index
  unsigned sa, sq, da, dq;  // strides along the line and between the nq, in source and destination
  int out_len;
  float sign;
  int accumulate;
};
struct Walk3Args {
  Walk3Term t[2];
  int M, off;
  float g[4], gl[4], v[kEnd], sc_hi, sc_lo;
  int nxt, nq, nseg, chunk, rb;  // x tiles, lines along q (largest), segments as in k_tiled.cu
};

// Group of eight differences m0 .. m0 + 7 along a line from the filtered points after them: the forward
// values z, and the rows m0 - 7 .. m0 of the result (in the units of the scaled recurrences) by the backward
// recurrence.  `first`, `final`: the result rows are the first or last eight of the line.
template <bool EDGE>
__device__ __forceinline__ void walk3_group(const Walk3Args& A, const float (&ch)[8], const float (&cl)[8], float& h0,
                                            float& l0, float& z, float (&zp)[7], float (&y)[8], int m0, bool first,
                                            bool final) {
  float zc[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    float d = (ch[t] - h0) + (cl[t] - l0);
    if (EDGE) d = (m0 + t >= 0 && m0 + t < A.M) ? d : 0.0f;
    h0 = ch[t];
    l0 = cl[t];
    zc[t] = z = fmaf(kRhoF, z, d);
  }
  float acc = zc[7];
#pragma unroll
  for (int t = 6; t >= 1; --t) acc = fmaf(kRhoF, acc, zc[t]);
  const float ynext = acc;  // of the row after the group
  y[7] = acc = fmaf(kRhoF, acc, zc[0]);
#pragma unroll
  for (int t = 6; t >= 0; --t) y[t] = acc = fmaf(kRhoF, acc, zp[t]);
  if (EDGE && (first || final)) {
    const float zr[8] = {zp[0], zp[1], zp[2], zp[3], zp[4], zp[5], zp[6], zc[0]};
    if (first) end_rows<false>(y, zr, ynext, end_phi(A, y[0], y[1], y[2], y[3]), A.v);
    if (final) end_rows<true>(y, zr, ynext, end_phi(A, y[7], y[6], y[5], y[4]), A.v);
  }
#pragma unroll
  for (int t = 0; t < 7; ++t) zp[t] = zc[t + 1];
}

template <bool EDGE>
__device__ __forceinline__ void walk3_segment(const Walk3Args& A, const Walk3Term& T, int x, int q, int seg) {
  const bool live = x < T.nx, last = seg == A.nseg - 1;
  const int M = A.M, r0 = last ? A.rb : seg * A.chunk, r1 = last ? M : min(r0 + A.chunk, A.rb);
  const float* __restrict__ ph = T.gh + (size_t)q * T.sq + min(x, T.nx - 1);
  const float* __restrict__ pl = T.gl + (size_t)q * T.sq + min(x, T.nx - 1);
  float* __restrict__ Rq = T.R + (size_t)q * T.dq + min(x, T.nx - 1);
  auto row = [&](int r) { return (unsigned)(EDGE ? min(max(r, 0), M) : r) * T.sa; };
  const int ms = r0 - 9;
  float h0 = ph[row(ms)], l0 = pl[row(ms)];
  float nh[8], nl[8], old[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    nh[t] = ph[row(ms + 1 + t)];
    nl[t] = pl[row(ms + 1 + t)];
  }
  float z = 0.0f, zp[7] = {};
  const int ngrp = 2 + (r1 - r0 + 7) / 8;
  float* bp = Rq + (unsigned)(r0 + A.off) * T.da;
  for (int gi = 0; gi < ngrp; ++gi) {
    const int m0 = ms + 8 * gi;
    float ch[8], cl[8], y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      ch[t] = nh[t];
      cl[t] = nl[t];
    }
    if (gi + 1 < ngrp) {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        nh[t] = ph[row(m0 + 9 + t)];
        nl[t] = pl[row(m0 + 9 + t)];
      }
    }
    const int left = gi < 2 ? 0 : min(8, r1 - (r0 + 8 * (gi - 2)));
    if (T.accumulate) {
#pragma unroll
      for (int t = 0; t < 8; ++t) old[t] = t < left ? bp[(unsigned)t * T.da] : 0.0f;
    }
    walk3_group<EDGE>(A, ch, cl, h0, l0, z, zp, y, m0, seg == 0 && gi == 2, last && gi == ngrp - 1);
    if (gi < 2) continue;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float v = fmaf(A.sc_hi, y[t], A.sc_lo * y[t]);
      if (live && t < left) bp[(unsigned)t * T.da] = T.accumulate ? fmaf(T.sign, v, old[t]) : T.sign * v;
    }
    bp += 8u * T.da;
  }
  if (live && !T.accumulate) {  // wall points of the line
    if (seg == 0)
      for (int r = 0; r < A.off; ++r) Rq[(unsigned)r * T.da] = 0.0f;
    if (last)
      for (int r = M + A.off; r < T.out_len; ++r) Rq[(unsigned)r * T.da] = 0.0f;
  }
}

__global__ void __launch_bounds__(32 * kW3Warps, 7) k_walk3d32(const __grid_constant__ Walk3Args A) {
  pdl_wait();
  int item = blockIdx.x * kW3Warps + (threadIdx.x >> 5);
  const int xt = item % A.nxt;
  item /= A.nxt;
  const int seg = item % A.nseg;
  item /= A.nseg;
  const int which = item / A.nq, q = item - which * A.nq;
  if (which > 1) return;
  const Walk3Term& T = A.t[which];
  if (q >= T.nq || 32 * xt >= T.nx) return;
  const int x = 32 * xt + (threadIdx.x & 31);
  const int r0 = seg == A.nseg - 1 ? A.rb : seg * A.chunk, r1 = seg == A.nseg - 1 ? A.M : min(r0 + A.chunk, A.rb);
  if (r0 >= 10 && r1 + 18 <= A.M) walk3_segment<false>(A, T, x, q, seg);
  else walk3_segment<true>(A, T, x, q, seg);
}

// The same walk for the terms along x: a lane takes a row of the component (x, all rows of a plane stack
// being equally long), 32 rows per warp, and sixteen points of every row at a time come through tiles in
// shared memory, filled by cp.async along x kAX tiles ahead; the results go back through the tile just read and
// leave along x.  Two accumulating terms at 256^3: 142 and 121 us (200 and 180 us with two tiles ahead, for the
// warps their shared memory leaves out; 166 us by tiles of 64 x 32).  In Walk3Term, nx counts the rows, sq and
// dq are their strides.
constexpr int kAX = 1, kRX = kAX + 1, kXW = 16, kXS = kXW + 1, kWXWarps = 2;  // tile stride odd: no bank conflicts
template <bool EDGE>
__device__ __forceinline__ void walk3x_segment(const Walk3Args& A, const Walk3Term& T, int row0, int seg,
                                               float (*tile)[2][32 * kXS]) {
  const int lane = threadIdx.x & 31, xr = lane & (kXW - 1), rs = lane / kXW * 16;  // rows rs .. rs + 15
  const int cap = min(31, T.nx - 1 - row0);  // last row of the warp
  const bool last = seg == A.nseg - 1;
  const int M = A.M, r0 = last ? A.rb : seg * A.chunk, r1 = last ? M : min(r0 + A.chunk, A.rb);
  const float* __restrict__ ph = T.gh + (size_t)row0 * T.sq;
  const float* __restrict__ pl = T.gl + (size_t)row0 * T.sq;
  float* __restrict__ R = T.R + (size_t)row0 * T.dq + A.off;
  const int ms = r0 - 9, ngrp = 2 + (r1 - r0 + 7) / 8, ntile = (ngrp + 1) / 2;
  auto fetch = [&](int c) {
    if (c < ntile) {
      const int x = min(max(ms + 1 + kXW * c + xr, 0), M);
      float* dh = tile[c % kRX][0] + rs * kXS + xr;
      float* dl = tile[c % kRX][1] + rs * kXS + xr;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const unsigned o = (unsigned)min(rs + i, cap) * T.sq + x;
        cp4(dh + i * kXS, ph + o);
        cp4(dl + i * kXS, pl + o);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < kAX; ++c) fetch(c);
  const unsigned o0 = (unsigned)min(lane, cap) * T.sq + max(ms, 0);
  float h0 = ph[o0], l0 = pl[o0];
  float z = 0.0f, zp[7] = {};
  for (int c = 0; c < ntile; ++c) {
    __syncwarp();  // the tile read last is free
    fetch(c + kAX);
    const int rw = r0 + kXW * (c - 1) + xr;  // result row of the lane when writing
    const bool out = c > 0 && rw < r1;
    float old[16];
    if (T.accumulate) {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        old[i] = out && rs + i <= cap ? R[(unsigned)(rs + i) * T.dq + rw] : 0.0f;
    }
    asm volatile("cp.async.wait_group %0;" ::"n"(kAX) : "memory");
    __syncwarp();
    float* th = tile[c % kRX][0] + lane * kXS;
    const float* tl = tile[c % kRX][1] + lane * kXS;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int gi = 2 * c + u;
      if (gi >= ngrp) break;
      float ch[8], cl[8], y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        ch[t] = th[8 * u + t];
        cl[t] = tl[8 * u + t];
      }
      walk3_group<EDGE>(A, ch, cl, h0, l0, z, zp, y, ms + 8 * gi, seg == 0 && gi == 2, last && gi == ngrp - 1);
#pragma unroll
      for (int t = 0; t < 8; ++t) th[8 * u + t] = T.sign * fmaf(A.sc_hi, y[t], A.sc_lo * y[t]);
    }
    if (c == 0) continue;
    __syncwarp();
    const float* tw = tile[c % kRX][0] + rs * kXS + xr;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (out && rs + i <= cap)
        R[(unsigned)(rs + i) * T.dq + rw] = T.accumulate ? tw[i * kXS] + old[i] : tw[i * kXS];
  }
  if (lane <= cap && !T.accumulate) {  // wall points of the lines
    float* __restrict__ Rl = T.R + (size_t)(row0 + lane) * T.dq;
    if (seg == 0)
      for (int r = 0; r < A.off; ++r) Rl[r] = 0.0f;
    if (last)
      for (int r = M + A.off; r < T.out_len; ++r) Rl[r] = 0.0f;
  }
}

__global__ void __launch_bounds__(32 * kWXWarps) k_walkx3d32(const __grid_constant__ Walk3Args A) {
  __shared__ float tiles[kWXWarps][kRX][2][32 * kXS];
  pdl_wait();
  int item = blockIdx.x * kWXWarps + (threadIdx.x >> 5);
  const int seg = item % A.nseg;  // the segments of a line share its sectors in L2
  item /= A.nseg;
  const int which = item / A.nxt, row0 = 32 * (item - which * A.nxt);
  if (which > 1) return;
  const Walk3Term& T = A.t[which];
  if (row0 >= T.nx) return;
  const int r0 = seg == A.nseg - 1 ? A.rb : seg * A.chunk, r1 = seg == A.nseg - 1 ? A.M : min(r0 + A.chunk, A.rb);
  if (r0 >= 10 && r1 + 18 <= A.M) walk3x_segment<false>(A, T, row0, seg, tiles[threadIdx.x >> 5]);
  else walk3x_segment<true>(A, T, row0, seg, tiles[threadIdx.x >> 5]);
}

// The solve of a half-step: 6 h^2 P1 = D - T with D = 6 c1 h^2 + 24 and, from the 19-point stencil,
// T y = 2 e + c + (2 y + e)_{z-1} + (2 y + e)_{z+1}, e and c the sums over the four edge and the four
// corner neighbours in the plane, spectrum [-8, 24].  The Chebyshev polynomial of k_rec64.cu in Horner
// form, y <- b + q T y, to a relative error of 1e-10, one level per launch for the three components; T y
// is 24 / D of D y at most (2e-3 at r = 0.4, 7e-3 at the stability limit), so a level rounds the increment at 1e-10
// to 4e-10 of itself, and the last level's q T y enters the state apart from b.  A block takes a tile of 32 x 16 columns and marches along z; the
// planes come through a ring in shared memory filled by cp.async kA3 planes ahead (loads straight
// into registers, one plane ahead, left the march waiting for them: 180 to 225 us per level of three
// components at 256^3), and a thread keeps e, c and q = 2 y + e of its four rows in registers as two pairs:
// 32 instructions per 32 points, 75 with two rows and scalar operations, 84 in a Richardson sweep with its
// residual.  Three components at 256^3: 107 us for the first level, 147 a middle one, 213 the last one
// (127, 170, 240 with two rows; 195 to 280 per sweep), 3.8, 4.1 and 4.7 TB/s: bound by loads in flight.
constexpr int L3Y = 4, L3T = 32 * L3Y;  // warps (of four rows) and threads per block
constexpr int kA3 = 3, kR3 = kA3 + 1;   // a power of two of slots
constexpr int S3W = 34, S3N = S3W * (4 * L3Y + 2), S3P = (S3N + L3T - 1) / L3T;  // a staged plane, per thread
struct Lev3d32Args {
  const float* b[3];
  const float* y[3];
  float* out[3];         // iterate (not LAST)
  float *hi[3], *lo[3];  // state (LAST)
  Shape3 s[3];
  float q;                       // of this level (not LAST)
  float s_hi, s_lo, l_hi, l_lo;  // increment scale s, s q (LAST)
  int nz, zc;  // marches along z of the largest component, planes per march
};

// FIRST: y is b itself.
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(L3T, LAST ? 5 : 7) k_lev3d32(const __grid_constant__ Lev3d32Args A) {
  __shared__ float ring[kR3][S3N];
  pdl_wait();
  const int which = blockIdx.z / A.nz, kz = blockIdx.z - which * A.nz;
  const Shape3& s = A.s[which];
  const int n0 = s.n[0], n1 = s.n[1], n2 = s.n[2];
  const int d0 = s.bc[0] == DIR, d1 = s.bc[1] == DIR, d2 = s.bc[2] == DIR;
  const int i0 = d0 + blockIdx.x * 32, j0 = d1 + blockIdx.y * 4 * L3Y;
  const int k0 = d2 + kz * A.zc, k1 = min(k0 + A.zc, n2 - d2);
  if (i0 >= n0 - d0 || j0 >= n1 - d1 || k0 >= k1) return;  // block-uniform
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
  const int i = i0 + tx, j = j0 + 4 * ty;
  const int rows = i < n0 - d0 ? min(4, n1 - d1 - j) : 0;  // the thread's unknowns
  const unsigned sz = n0 * n1;  // points per component fit 31 bits (n <= 512)
  const float* __restrict__ y = A.y[which];
  const float* __restrict__ b = A.b[which];
  float* __restrict__ out = A.out[which];
  float* __restrict__ shi = A.hi[which];
  float* __restrict__ slo = A.lo[which];
  // staged points of the thread: ghosts of a Neumann axis mirror (clamped), walls of a Dirichlet axis hold
  // zeros (b: the terms write them; y: the level before)
  unsigned po[S3P];
#pragma unroll
  for (int q = 0; q < S3P; ++q) {
    const int e = min(tid + q * L3T, S3N - 1), r = e / S3W, c = e - r * S3W;
    po[q] = clampi(j0 - 1 + r, n1) * n0 + clampi(i0 - 1 + c, n0);
  }
  const bool tail = tid + (S3P - 1) * L3T < S3N;
  const int S = k1 - k0 + 2;  // planes k0 - 1 .. k1
  auto fetch = [&](int st) {
    if (st < S) {
      const float* __restrict__ p = y + (size_t)clampi(k0 - 1 + st, n2) * sz;
      float* d = ring[st % kR3] + tid;
#pragma unroll
      for (int q = 0; q < S3P; ++q)
        if (q < S3P - 1 || tail) cp4(d + q * L3T, p + po[q]);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int t = 0; t < kA3; ++t) fetch(t);
  // per-point operands two planes ahead; point rows t and t + 2 of the thread are halves of a pair
  const unsigned own = j * n0 + i;
  float2 b1[2] = {}, b2[2] = {}, h1[2] = {}, h2[2] = {}, l1[2] = {}, l2[2] = {};
  auto load = [&](const float* __restrict__ p, float2(&v)[2]) {
    if (rows > 0) v[0].x = p[0];
    if (rows > 1) v[1].x = p[n0];
    if (rows > 2) v[0].y = p[2 * n0];
    if (rows > 3) v[1].y = p[3 * n0];
  };
  auto store = [&](float* __restrict__ p, const float2(&v)[2]) {
    if (rows > 0) p[0] = v[0].x;
    if (rows > 1) p[n0] = v[1].x;
    if (rows > 2) p[2 * n0] = v[0].y;
    if (rows > 3) p[3 * n0] = v[1].y;
  };
  float2 qm[2] = {}, q0[2] = {}, u0[2] = {}, m0[2] = {};  // q of planes k - 1, k; 2 e + c and y of plane k
  const float2 two = bc2(2.0f), q = bc2(A.q);
  const float2 s_hi = bc2(A.s_hi), n_hi = bc2(-A.s_hi), s_lo = bc2(A.s_lo), l_hi = bc2(A.l_hi), l_lo = bc2(A.l_lo);
  unsigned g = k0 * sz + own;
#pragma unroll 4
  for (int st = 0; st < S; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kA3 - 1) : "memory");
    __syncthreads();  // plane st is there for every thread, and the slot read last is free
    fetch(st + kA3);
    const float* r = ring[st % kR3] + (4 * ty) * S3W + tx;
    float2 bc[2], hc[2], lc[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      bc[t] = FIRST ? m0[t] : b1[t];
      b1[t] = b2[t];
      hc[t] = h1[t];
      h1[t] = h2[t];
      lc[t] = l1[t];
      l1[t] = l2[t];
    }
    if (k0 + st < k1) {  // used two planes on
      const unsigned p = (k0 + st) * sz + own;
      if (!FIRST) load(b + p, b2);
      if (LAST) {
        load(shi + p, h2);
        load(slo + p, l2);
      }
    }
    float ms[6], xs[6];
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      ms[t] = r[t * S3W + 1];
      xs[t] = r[t * S3W] + r[t * S3W + 2];
    }
    float2 m[4], x[4], v[2];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      m[t] = make_float2(ms[t], ms[t + 2]);
      x[t] = make_float2(xs[t], xs[t + 2]);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const float2 e = add2(x[t + 1], add2(m[t], m[t + 2]));
      const float2 qn = fma2(two, m[t + 1], e);
      const float2 T = add2(u0[t], add2(qm[t], qn));
      if (LAST) ff_add_scaled(hc[t], lc[t], bc[t], T, s_hi, n_hi, s_lo, l_hi, l_lo);
      else v[t] = fma2(q, T, bc[t]);
      qm[t] = q0[t];
      q0[t] = qn;
      u0[t] = fma2(two, e, add2(x[t], x[t + 2]));
      m0[t] = m[t + 1];
    }
    if (st >= 2) {
      if (LAST) {
        store(shi + g, hc);
        store(slo + g, lc);
      } else {
        store(out + g, v);
      }
      g += sz;
    }
  }
  if (!LAST && rows > 0) {
    // zeros on the walls the next level reads: those next to the thread's points, corners included
    const int jl = j + rows - 1;
    const int di0 = d0 && i == 1 ? -1 : 0, di1 = d0 && i == n0 - 2 ? 1 : 0;
    const int dj0 = d1 && j == 1 ? -1 : 0, dj1 = d1 && jl == n1 - 2 ? 1 : 0;
    const int dk0 = d2 && k0 == 1 ? -1 : 0, dk1 = d2 && k1 == n2 - 1 ? 1 : 0;
    if (di0 | di1 | dj0 | dj1 | dk0 | dk1)
      for (int k = k0 + dk0; k < k1 + dk1; ++k)
        for (int jj = j + dj0; jj <= jl + dj1; ++jj)
          for (int ii = i + di0; ii <= i + di1; ++ii)
            if (k < k0 || k >= k1 || jj < j || jj > jl || ii != i) out[((size_t)k * n1 + jj) * n0 + ii] = 0.0f;
  }
}

// One sweep of the FP32 Richardson iteration on 6 h^2 P1 x = b (6h^2 P1 = d - 6(Lx + Ly + Lz)
// - (LxLy + LyLz + LzLx), d = 6 c1 h^2 as hi + lo), x_{k+1} = x_k + omega (b - 6 h^2 P1 x_k): the
// refinement after a transform solve.  LAST: the state (hi, lo) += s x + s corr (two separate
// error-free additions) instead of writing x.
// A block of SWX x SWT threads takes a tile of SWX x SWY points and marches SWZ planes along z;
// a thread takes rows j and j + SWT of one column, and every operation acts on that pair at once
// (paired FP32 instructions).  The iterate on planes z-1, z, z+1 over the tile with a one-point
// halo in x and y sits in a ring in shared memory as pairs: pair row pr holds tile rows pr - 1 and
// pr - 1 + SWT, so a shift in x or y is the same shift of both halves.  The next plane is
// fetched into registers, and the per-point operands (b, the state) of the next plane too, while
// the current one is computed.  Tiles cover the unknowns only: halo points past a Neumann end
// are its even ghosts (clamped), walls of a Dirichlet axis are taken as zeros without a load, so
// no sweep reads or writes a wall point.
constexpr int SWX = 32, SWT = 8, SWY = 2 * SWT, SWZ = 16;
constexpr int SWXP = SWX + 2, SWRP = SWT + 2;  // pair rows of a staged plane
constexpr int SWN = SWRP * SWXP;               // staged pairs per plane
static_assert(SWN <= 2 * SWX * SWT, "two staged pairs per thread");

template <bool LAST>
__global__ void __launch_bounds__(SWX * SWT, LAST ? 4 : 5) k_sweep3d32(const float* __restrict__ b, const float* __restrict__ xin,
                                                            float* __restrict__ xout, Shape3 s, float d_hi, float d_lo,
                                                            float omega, float* __restrict__ shi,
                                                            float* __restrict__ slo, float s_hi, float s_lo) {
  __shared__ float2 xs[3][SWRP][SWXP];
  const int n0 = s.n[0], n1 = s.n[1], n2 = s.n[2];
  // tiles cover the unknowns only: index u along an axis is point u + lo (lo = 1 on a Dirichlet
  // axis, whose walls are read as the zeros they hold, without a load)
  const int lo0 = s.bc[0] == DIR, lo1 = s.bc[1] == DIR, lo2 = s.bc[2] == DIR;
  const int nu0 = n0 - 2 * lo0, nu1 = n1 - 2 * lo1, nu2 = n2 - 2 * lo2;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int iu = blockIdx.x * SWX + tx, ju = blockIdx.y * SWY + ty;  // rows ju and ju + SWT
  const int k0 = blockIdx.z * SWZ, k1 = min(k0 + SWZ, nu2);
  const bool in0 = iu < nu0 && ju < nu1, in1 = iu < nu0 && ju + SWT < nu1;
  const int sz = n0 * n1;
  const float* X0 = xin;
  // position q along an axis of n points: false where the value is a wall zero, else the point
  // (even ghosts of a Neumann axis clamped)
  auto place = [](int q, int n, int dir, int* at) {
    if (dir) {
      *at = q;
      return q > 0 && q < n - 1;
    }
    *at = clampi(q, n);
    return true;
  };
  // plane loader: thread t stages pairs t and t + 256 (< SWN), at offsets fixed for the march
  const int t1 = ty * SWX + tx, t2 = t1 + SWX * SWT;
  const bool has2 = t2 < SWN;
  auto pair_off = [&](int e, int half, bool* live) {
    const int row = e / SWXP, col = e - row * SWXP;
    int y, x;
    const bool ly = place(lo1 + blockIdx.y * SWY + row - 1 + half * SWT, n1, lo1, &y);
    const bool lx = place(lo0 + blockIdx.x * SWX + col - 1, n0, lo0, &x);
    *live = ly && lx;
    return *live ? y * n0 + x : 0;
  };
  bool v1a, v1b, v2a, v2b;
  const int o1a = pair_off(t1, 0, &v1a), o1b = pair_off(t1, 1, &v1b);
  const int o2a = pair_off(has2 ? t2 : t1, 0, &v2a), o2b = pair_off(has2 ? t2 : t1, 1, &v2b);
  float2 ra = make_float2(0.0f, 0.0f), rb = make_float2(0.0f, 0.0f);
  auto fetch = [&](int ku) {  // plane of unknown index ku (-1 .. nu2)
    int z;
    const bool lz = place(lo2 + ku, n2, lo2, &z);
    const float* P = X0 + (lz ? z : 0) * sz;
    ra = make_float2(lz && v1a ? P[o1a] : 0.0f, lz && v1b ? P[o1b] : 0.0f);
    if (has2) rb = make_float2(lz && v2a ? P[o2a] : 0.0f, lz && v2b ? P[o2b] : 0.0f);
  };
  const float2 om2 = bc2(omega);
  auto stage = [&](float2(*pl)[SWXP]) {
    float2* f = &pl[0][0];
    f[t1] = ra;
    if (has2) f[t2] = rb;
  };
  // per-point operands of the next plane
  float2 bq = make_float2(0.0f, 0.0f), hq = bq, lq = bq;
  const int dj = SWT * n0;
  auto fetch_pt = [&](int p) {
    if (in0) {
      bq.x = b[p];
      if (LAST) {
        hq.x = shi[p];
        lq.x = slo[p];
      }
    }
    if (in1) {
      bq.y = b[p + dj];
      if (LAST) {
        hq.y = shi[p + dj];
        lq.y = slo[p + dj];
      }
    }
  };
  float2(*Zm)[SWXP] = xs[0];
  float2(*Z0)[SWXP] = xs[1];
  float2(*Zp)[SWXP] = xs[2];
  fetch(k0 - 1);
  stage(Zm);
  fetch(k0);
  stage(Z0);
  fetch(k0 + 1);
  int p = (lo2 + k0) * sz + (lo1 + ju) * n0 + lo0 + iu;
  fetch_pt(p);
  const int c0 = tx + 1, r0 = ty + 1;  // halo coordinates in the pair layout
  const float2 m2 = bc2(-2.0f), m6 = bc2(-6.0f), ndh2 = bc2(-d_hi), ndl2 = bc2(-d_lo), sh2 = bc2(s_hi), sl2 = bc2(s_lo);
  for (int k = k0; k < k1; ++k, p += sz) {
    stage(Zp);
    __syncthreads();
    if (k + 1 < k1) fetch(k + 2);
    const float2 bc = bq, hc = hq, lc = lq;
    if (k + 1 < k1) fetch_pt(p + sz);
    // second differences as a + b - 2 v: the residual's dominant term d x enters exactly, so
    // the rounding of these sums is far below an ulp of the residual
    auto LX = [&](const float2(*Pl)[SWXP], int rr) { return fma2(m2, Pl[rr][c0], add2(Pl[rr][c0 - 1], Pl[rr][c0 + 1])); };
    auto LY = [&](const float2(*Pl)[SWXP]) { return fma2(m2, Pl[r0][c0], add2(Pl[r0 - 1][c0], Pl[r0 + 1][c0])); };
    const float2 x = Z0[r0][c0];
    const float2 lx = LX(Z0, r0), ly = LY(Z0);
    const float2 lz = fma2(m2, x, add2(Zm[r0][c0], Zp[r0][c0]));
    const float2 lxly = fma2(m2, lx, add2(LX(Z0, r0 - 1), LX(Z0, r0 + 1)));
    const float2 lxlz = fma2(m2, lx, add2(LX(Zm, r0), LX(Zp, r0)));
    const float2 lylz = fma2(m2, ly, add2(LY(Zm), LY(Zp)));
    const float2 rest = fma2(m6, add2(add2(lx, ly), lz), neg2(add2(add2(lxly, lylz), lxlz)));
    // b - d x with the product exact: b - d_hi x, then - d_lo x, one rounding each
    const float2 res = sub2(fma2(ndl2, x, fma2(ndh2, x, bc)), rest);
    if (LAST) {
      const float2 corr = mul2(om2, res);
      float2 h = hc, l = lc;
      ff_add_scaled3_2(h, l, x, sh2, sl2);
      ff_add_scaled3_2(h, l, corr, sh2, sl2);
      if (in0) {
        shi[p] = h.x;
        slo[p] = l.x;
      }
      if (in1) {
        shi[p + dj] = h.y;
        slo[p + dj] = l.y;
      }
    } else {
      const float2 xn = fma2(om2, res, x);
      if (in0) xout[p] = xn.x;
      if (in1) xout[p + dj] = xn.y;
    }
    __syncthreads();  // the slot of plane k - 1 is staged again as plane k + 2
    float2(*t)[SWXP] = Zm;
    Zm = Z0;
    Z0 = Zp;
    Zp = t;
  }
}

dim3 sweep_grid3(const Shape3& s) {  // tiles over the unknowns
  const int nu0 = s.n[0] - 2 * (s.bc[0] == DIR), nu1 = s.n[1] - 2 * (s.bc[1] == DIR), nu2 = s.n[2] - 2 * (s.bc[2] == DIR);
  return dim3((nu0 + SWX - 1) / SWX, (nu1 + SWY - 1) / SWY, (nu2 + SWZ - 1) / SWZ);
}

__global__ void k_split3(const double* __restrict__ v, float* __restrict__ hi, float* __restrict__ lo, size_t n) {
  const size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float h = (float)v[p];
  hi[p] = h;
  lo[p] = (float)(v[p] - (double)h);
}

__global__ void k_join3(const float* __restrict__ hi, const float* __restrict__ lo, double* __restrict__ v, size_t n) {
  const size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  v[p] = (double)hi[p] + (double)lo[p];
}

// ---------------------------------------------------------------------------------------
// Host launchers

const dim3 kBlk(32, 8, 1);

// G[c] = filtered u[c] for the components c0 .. c0 + 2.
void filter3d64(ms_grid* g, int c0, double* const* u, double* const* G) {
  Filter3d64Args A;
  A.nz = 0;
  double pts = 0.0;
  int nx = 0, ny = 0;
  for (int c = 0; c < 3; ++c) {
    const Shape3& s = g->g3->sh[c0 + c];
    A.u[c] = u[c];
    A.G[c] = G[c];
    A.s[c] = s;
    A.nz = s.n[2] > A.nz ? s.n[2] : A.nz;
    nx = s.n[0] > nx ? s.n[0] : nx;
    ny = s.n[1] > ny ? s.n[1] : ny;
    pts += (double)s.size();
  }
  launch_pdl(k_filter3d64, dim3((nx + 31) / 32, (ny + 7) / 8, 3 * A.nz), kBlk, 0, g->stream, A, g->beta - 0.5);
  prof_mark(g, KK_FILTER3D64, 16.0 * pts);
}

// out (+)= scale * delta_axis(in), in of component shape si, out of shape so
struct Pade3d64 {
  int axis;
  Shape3 si, so;
  const double* in;
  double* out;
  double scale;
  int accumulate;
};

LineArgs line_of(const Pade3d64& q, const PadeTable& t) {
  const int P = q.axis == 0 ? 1 : 0, Q = q.axis == 2 ? 1 : 2;  // the two other axes
  auto stride = [](const Shape3& s, int a) { return a == 0 ? (size_t)1 : (a == 1 ? (size_t)s.n[0] : (size_t)s.n[0] * s.n[1]); };
  LineArgs a{};
  a.in = q.in;
  a.out = q.out;
  a.M = t.M;
  a.out_len = q.so.n[q.axis];
  a.out_off = q.si.bc[q.axis] == NEU && q.so.bc[q.axis] == DIR ? 1 : 0;
  a.n0 = q.so.n[P];
  a.n1 = q.so.n[Q];
  a.lo = 0;
  a.hi = a.n0;
  a.in_sa = stride(q.si, q.axis);
  a.in_s0 = stride(q.si, P);
  a.in_s1 = stride(q.si, Q);
  a.out_sa = stride(q.so, q.axis);
  a.out_s0 = stride(q.so, P);
  a.out_s1 = stride(q.so, Q);
  a.scale = q.scale;
  a.accumulate = q.accumulate;
  return a;
}

// Up to three independent derivatives of one kind (all with axis 0 or none), in one launch; lines
// shorter than kRecMinLine take the band kernel, one launch each.  Returns the number of launches.
int pade3d64(ms_grid* g, const Pade3d64* q, int count) {
  const PadeTable& t = g->pade[q[0].si.bc[q[0].axis] == NEU ? HALF_TO_NODE : NODE_TO_HALF];
  auto bytes = [&](int k) {
    return 8.0 * ((double)q[k].si.size() + (q[k].accumulate ? 2.0 : 1.0) * (double)q[k].so.size());
  };
  if (t.M >= kRecMinLine) {
    LineArgs a[kLineBatch];
    double b = 0.0;
    for (int k = 0; k < count; ++k) {
      a[k] = line_of(q[k], t);
      b += bytes(k);
    }
    launch_line64(a, count, t.ends, false, g->stream);
    prof_mark(g, KK_PADE3D64, b);
    return 1;
  }
  for (int k = 0; k < count; ++k) {
    const LineArgs a = line_of(q[k], t);
    const Shape3 &so = q[k].so, &si = q[k].si;
    const dim3 grd = grid3(so, kBlk);
    if (q[k].axis == 0)
      k_pade3d64<0><<<grd, kBlk, 0, g->stream>>>(q[k].in, q[k].out, so, si, t.d_w, t.rows, t.n_in, t.left, t.K, t.B,
                                                  t.all_explicit, a.out_off, q[k].scale, q[k].accumulate);
    else if (q[k].axis == 1)
      k_pade3d64<1><<<grd, kBlk, 0, g->stream>>>(q[k].in, q[k].out, so, si, t.d_w, t.rows, t.n_in, t.left, t.K, t.B,
                                                  t.all_explicit, a.out_off, q[k].scale, q[k].accumulate);
    else
      k_pade3d64<2><<<grd, kBlk, 0, g->stream>>>(q[k].in, q[k].out, so, si, t.d_w, t.rows, t.n_in, t.left, t.K, t.B,
                                                  t.all_explicit, a.out_off, q[k].scale, q[k].accumulate);
    prof_mark(g, KK_PADE3D64, bytes(k));
  }
  return count;
}

// R[c] = s (d_{c+1} G_{c+2} - d_{c+2} G_{c+1}) on the components cd0 + c, G of the components cs0 + c.
// The first launch writes with axes across x only (the terms of axis 1, 2, 1), then the term of axis 2
// and the two of axis 0 add to it.
int curl3d64(ms_grid* g, int cs0, int cd0, double* const* G, double* const* R, double s) {
  Grid3D* G3 = g->g3;
  auto term = [&](int c, int axis, int acc) {
    const int p1 = (c + 1) % 3, p2 = (c + 2) % 3;
    const int src = axis == p1 ? p2 : p1;
    return Pade3d64{axis, G3->sh[cs0 + src], G3->sh[cd0 + c], G[src], R[c], axis == p1 ? s : -s, acc};
  };
  const Pade3d64 first[3] = {term(0, 1, 0), term(1, 2, 0), term(2, 1, 0)};
  const Pade3d64 second[1] = {term(0, 2, 1)};
  const Pade3d64 third[2] = {term(1, 0, 1), term(2, 0, 1)};
  return pade3d64(g, first, 3) + pade3d64(g, second, 1) + pade3d64(g, third, 2);
}

// x = P1^{-1} b for the components c0 .. c0 + 2; upd[c] += upd_scale x, and, if out is set, out[c] is the
// work plane that holds x (its wall points are not written).
void solve3d64(ms_grid* g, int c0, double* const* b, double* const* upd, double upd_scale, const double** out, int* nl) {
  Grid3D* G3 = g->g3;
  Cheb3dField f[3];
  double* buf[3][2];
  const int m = g->cheb64.m;
  for (int c = 0; c < 3; ++c) {
    const Shape3& s = G3->sh[c0 + c];
    buf[c][0] = G3->s64[c];
    buf[c][1] = G3->s64[6 + c];
    f[c].b = b[c];
    f[c].out = nullptr;
    f[c].upd = upd ? upd[c] : nullptr;
    if (out) {
      f[c].out = buf[c][m & 1];
      out[c] = f[c].out;
    }
    for (int a = 0; a < 3; ++a) {
      f[c].n[a] = s.n[a];
      f[c].bc[a] = s.bc[a];
    }
  }
  *nl += launch_cheb3d64(g, KK_SWEEP3D64, f, buf, 3, g->cheb64, 6.0 * g->h * g->h, upd_scale);
}

ms_status step3d64(ms_grid* g) {
  Grid3D* G3 = g->g3;
  int nl = 0;
  double** G = G3->s64;      // G[0..2]
  double** R = G3->s64 + 3;  // R[0..2]
  const double s_he = g->kappa2 * g->Z / g->h, s_eh = g->kappa2 / (g->Z * g->h);
  if (g->src3) {  // time factors of this step's source terms
    src3_time(g);
    prof_mark(g, KK_SRC, 0.0);
    nl += 1;
  }
  auto add_src = [&](int c0) {
    if (!g->src3) return;
    for (int c = 0; c < 3; ++c) {
      src3_add(g, c0 + c, R[c]);
      prof_mark(g, KK_SRC, 16.0 * (double)G3->sh[c0 + c].size());
      nl += 1;
    }
  };
  // Step 1: R_e = kappa^2 Z (d_{e+1} G_{e+2} - d_{e+2} G_{e+1}) on E_e, P1 E* = R, E += h_tau E*
  filter3d64(g, 3, G3->f64 + 3, G);
  nl += 1 + curl3d64(g, 3, 0, G, R, s_he);
  add_src(0);
  solve3d64(g, 0, R, G3->f64, g->ht, nullptr, &nl);
  // Step 2: R_h = -(kappa^2/Z)(d_{h+1} G_{E,h+2} - d_{h+2} G_{E,h+1}) on H_h
  filter3d64(g, 0, G3->f64, G);
  nl += 1 + curl3d64(g, 0, 3, G, R, -s_eh);
  add_src(3);
  solve3d64(g, 3, R, G3->f64 + 3, g->ht, nullptr, &nl);
  if (g->src3) {  // the device step index advances with the step
    launch_tick(g);
    prof_mark(g, KK_SRC, 0.0);
    nl += 1;
  }
  g->launches_per_step = nl;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("3D FP64 step: ") + cudaGetErrorString(e));
  return MS_OK;
}

// FP32_REFINED: G (hi, lo) = 12 beta u + L u of the components c0 .. c0 + 2 into the filter buffers.
void filter3d32(ms_grid* g, int c0, float cb_hi, float cb_lo) {
  Grid3D* G3 = g->g3;
  Filter3d32Args A;
  int nx = 0, ny = 0;
  int nz = 0;
  double pts = 0.0;
  for (int c = 0; c < 3; ++c) {
    const Shape3& s = G3->sh[c0 + c];
    A.hi[c] = G3->hi[c0 + c];
    A.lo[c] = G3->lo[c0 + c];
    A.gh[c] = G3->gh[c];
    A.gl[c] = G3->gl[c];
    A.s[c] = s;
    nx = s.n[0] > nx ? s.n[0] : nx;
    ny = s.n[1] > ny ? s.n[1] : ny;
    nz = s.n[2] > nz ? s.n[2] : nz;
    pts += (double)s.size();
  }
  const int tx = (nx + 31) / 32, ty = (ny + 2 * FY3 - 1) / (2 * FY3);
  A.zc = march_planes(3 * tx * ty, nz);
  A.nz = (nz + A.zc - 1) / A.zc;
  launch_pdl(k_ffilt3d32, dim3(tx, ty, 3 * A.nz), dim3(32, FY3), 0, g->stream, A, cb_hi, cb_lo);
  prof_mark(g, KK_FILT3D32, 16.0 * pts);  // state hi + lo in, G hi + lo out
}

// FP32_REFINED: one Pade term y = A^{-1} D1 G of source component cs (G made by filter3d32) along an
// axis, added with `sign` into R of component cd (or written to it).
struct Term3 {
  int cs, cd;
  float sign;
  int accumulate;
};

// The two terms of a half-step along one axis in one launch.  Returns the number of launches issued.
int terms3d32(ms_grid* g, int axis, const Term3& q0, const Term3& q1) {
  Grid3D* G3 = g->g3;
  const int kind = (G3->sh[q0.cs].bc[axis] == NEU) ? HALF_TO_NODE : NODE_TO_HALF;
  const PadeTable& t = g->pade32[kind];
  const int off = (kind == HALF_TO_NODE) ? 1 : 0;
  const Term3* q[2] = {&q0, &q1};
  if (t.M >= kWalk3Min) {
    const int Q = axis == 2 ? 1 : 2;
    auto stride = [](const Shape3& s, int a) { return a == 0 ? 1u : (a == 1 ? (unsigned)s.n[0] : (unsigned)(s.n[0] * s.n[1])); };
    Walk3Args A;
    A.M = t.M;
    A.off = off;
    set_ends(g->walk.ends[kind], &A);
    const double sc = walk_rhs_scale();  // (1 - rho)^2, rho the FP32 root
    A.sc_hi = (float)sc;
    A.sc_lo = (float)(sc - (double)A.sc_hi);
    A.nxt = A.nq = 0;
    double bytes = 0.0;
    for (int k = 0; k < 2; ++k) {
      Walk3Term& a = A.t[k];
      const Shape3& ss = G3->sh[q[k]->cs];
      const Shape3& sd = G3->sh[q[k]->cd];
      a.gh = G3->gh[q[k]->cs % 3];
      a.gl = G3->gl[q[k]->cs % 3];
      a.R = G3->s32[q[k]->cd % 3];
      a.nx = axis ? sd.n[0] : sd.n[1] * sd.n[2];
      a.nq = axis ? sd.n[Q] : 1;
      a.sa = stride(ss, axis);
      a.sq = stride(ss, axis ? Q : 1);
      a.da = stride(sd, axis);
      a.dq = stride(sd, axis ? Q : 1);
      a.out_len = sd.n[axis];
      a.sign = q[k]->sign;
      a.accumulate = q[k]->accumulate;
      A.nxt = std::max(A.nxt, (a.nx + 31) / 32);
      A.nq = std::max(A.nq, a.nq);
      bytes += 4.0 * (2.0 * (double)ss.size() + (a.accumulate ? 2.0 : 1.0) * (double)sd.size());
    }
    // segments of about 64 rows (16 more warm up each), shorter where that leaves SMs idle: steps with 24 and 64
    // rows, us: 75^3 131, 142; 100^3 273, 275; 128^3 345, 342; 160^3 581, 564; 256^3 1986, 1911
    const int rows = 2 * A.nxt * A.nq * (t.M / 64) >= 4000 ? 64 : 24;
    line_segments(t.M, rows, &A.nseg, &A.chunk, &A.rb);
    const int items = 2 * A.nxt * A.nq * A.nseg;
    if (axis) launch_pdl(k_walk3d32, dim3((items + kW3Warps - 1) / kW3Warps), dim3(32 * kW3Warps), 0, g->stream, A);
    else launch_pdl(k_walkx3d32, dim3((items + kWXWarps - 1) / kWXWarps), dim3(32 * kWXWarps), 0, g->stream, A);
    prof_mark(g, KK_TERM3D32, bytes);
    return 1;
  }
  TermArgs2 A;
  int nx = 0, ny = 0;
  A.nz = 0;
  double bytes = 0.0;
  for (int k = 0; k < 2; ++k) {
    TermArgs& a = A.t[k];
    a.gh = G3->gh[q[k]->cs % 3];
    a.gl = G3->gl[q[k]->cs % 3];
    a.R = G3->s32[q[k]->cd % 3];
    a.ss = G3->sh[q[k]->cs];
    a.sd = G3->sh[q[k]->cd];
    a.sign = q[k]->sign;
    a.accumulate = q[k]->accumulate;
    nx = std::max(nx, a.sd.n[0]);
    ny = std::max(ny, a.sd.n[1]);
    A.nz = std::max(A.nz, a.sd.n[2]);
    // G hi + lo in, R out (read too when accumulating)
    bytes += 4.0 * (2.0 * (double)a.ss.size() + (a.accumulate ? 2.0 : 1.0) * (double)a.sd.size());
  }
  launch_pdl(k_short3d32, dim3((nx + 31) / 32, (ny + 3) / 4, 2 * A.nz), dim3(32, 4), 0, g->stream, A, axis, off, t.M,
             (const float*)t.d_whi, (const float*)t.d_wlo, t.K, t.B, (int)t.all_explicit);
  prof_mark(g, KK_TERM3D32, bytes);
  return 1;
}

// Transform solve (tensor cores) of component c followed by ts_sweeps Richardson sweeps with the
// exact residual, the last of which updates the state.
void solve3d32_ts(ms_grid* g, int c, float d_hi, float d_lo, float omega, float s_hi, float s_lo, int* nl) {
  Grid3D* G3 = g->g3;
  const Shape3& s = G3->sh[c];
  const float* b = G3->s32[c % 3];
  float* buf[2] = {G3->gh[c % 3], G3->gl[c % 3]};  // the filter's planes are free by now
  *nl += ts_solve(*G3->ts, s, b, buf[0], 6.0f * (float)(g->c1 * g->h * g->h), g->stream, g);
  const dim3 grd = sweep_grid3(s), blk(SWX, SWT, 1);
  const int R = G3->ts_sweeps;
  for (int k = 0; k < R; ++k) {
    const float* xin = buf[k & 1];
    float* xo = buf[(k + 1) & 1];
    if (k == R - 1)
      k_sweep3d32<true><<<grd, blk, 0, g->stream>>>(b, xin, xo, s, d_hi, d_lo, omega, G3->hi[c], G3->lo[c],
                                                           s_hi, s_lo);
    else
      k_sweep3d32<false><<<grd, blk, 0, g->stream>>>(b, xin, xo, s, d_hi, d_lo, omega, G3->hi[c], G3->lo[c],
                                                            s_hi, s_lo);
    prof_mark(g, KK_SWEEP3D32, 4.0 * (double)s.size() * (2.0 + (k == R - 1 ? 4.0 : 1.0)));
  }
  *nl += R;
}

// The solves and updates of the components c0 .. c0 + 2 from s32; the filter buffers, free by now,
// hold the iterates.
void solve3d32(ms_grid* g, int c0, const MixedConsts& k, int* nl) {
  Grid3D* G3 = g->g3;
  const bool e = c0 == 0;
  if (G3->solver == MS_SOLVER_TRANSFORM_TC) {
    for (int c = 0; c < 3; ++c)
      solve3d32_ts(g, c0 + c, k.d_hi, k.d_lo, k.omega, e ? k.sE_hi : k.sH_hi, e ? k.sE_lo : k.sH_lo, nl);
    return;
  }
  const Cheb& p = g->walk.cheb;
  Lev3d32Args A;
  int tx = 0, ty = 0, nz = 0;
  double pts = 0.0;
  for (int c = 0; c < 3; ++c) {
    const Shape3& s = G3->sh[c0 + c];
    A.s[c] = s;
    A.b[c] = G3->s32[c];
    A.hi[c] = G3->hi[c0 + c];
    A.lo[c] = G3->lo[c0 + c];
    int u[3];
    for (int a = 0; a < 3; ++a) u[a] = s.n[a] - 2 * (s.bc[a] == DIR);
    tx = std::max(tx, (u[0] + 31) / 32);
    ty = std::max(ty, (u[1] + 4 * L3Y - 1) / (4 * L3Y));
    nz = std::max(nz, u[2]);
    pts += (double)s.size();
  }
  const double s = (e ? 12.0 * g->Z / g->desc.r : 12.0 / (g->desc.r * g->Z)) * p.p0;
  const Split sp = split(s), lp = split(s * p.q[1]);
  A.s_hi = sp.hi;
  A.s_lo = sp.lo;
  A.l_hi = lp.hi;
  A.l_lo = lp.lo;
  A.zc = march_planes(3 * tx * ty, nz);
  A.nz = (nz + A.zc - 1) / A.zc;
  const dim3 grd(tx, ty, 3 * A.nz), blk(32, L3Y);
  for (int l = p.m - 1; l >= 1; --l) {
    const int step = p.m - 1 - l;
    A.q = (float)p.q[l];
    for (int c = 0; c < 3; ++c) {
      float* buf[2] = {G3->gh[c], G3->gl[c]};
      A.y[c] = step == 0 ? A.b[c] : buf[(step + 1) & 1];
      A.out[c] = buf[step & 1];
    }
    const bool first = step == 0, last = l == 1;
    if (first && last) launch_pdl(k_lev3d32<true, true>, grd, blk, 0, g->stream, A);
    else if (first) launch_pdl(k_lev3d32<true, false>, grd, blk, 0, g->stream, A);
    else if (last) launch_pdl(k_lev3d32<false, true>, grd, blk, 0, g->stream, A);
    else launch_pdl(k_lev3d32<false, false>, grd, blk, 0, g->stream, A);
    prof_mark(g, KK_SWEEP3D32, 4.0 * pts * ((step == 0 ? 1.0 : 2.0) + (l == 1 ? 4.0 : 1.0)));
  }
  *nl += p.m - 1;
}

ms_status step3d32(ms_grid* g) {
  const MixedConsts k = mixed_consts(g);
  int nl = 0;
  Grid3D* G3 = g->g3;
  if (g->src3) {
    src3_time(g);
    prof_mark(g, KK_SRC, 0.0);
    nl += 1;
  }
  // c0: first component of the half-step's fields, cs: of its sources; R_c = sign (D_{c+1} G_{c+2} -
  // D_{c+2} G_{c+1}) axis by axis, source terms in the units of b, the solves
  auto half = [&](int c0, int cs, float sign) {
    filter3d32(g, cs, k.cb_hi, k.cb_lo);
    nl += 1;
    nl += terms3d32(g, 2, Term3{cs + 1, c0 + 0, -sign, 0}, Term3{cs + 0, c0 + 1, sign, 0});
    nl += terms3d32(g, 1, Term3{cs + 2, c0 + 0, sign, 1}, Term3{cs + 0, c0 + 2, -sign, 0});
    nl += terms3d32(g, 0, Term3{cs + 2, c0 + 1, -sign, 1}, Term3{cs + 1, c0 + 2, sign, 1});
    if (g->src3)
      for (int c = 0; c < 3; ++c) {
        src3_add(g, c0 + c, G3->s32[c]);
        prof_mark(g, KK_SRC, 8.0 * (double)G3->sh[c0 + c].size());
        nl += 1;
      }
    solve3d32(g, c0, k, &nl);
  };
  half(0, 3, 1.0f);   // Step 1: E from H
  half(3, 0, -1.0f);  // Step 2: H from the updated E
  if (g->src3) {
    launch_tick(g);
    prof_mark(g, KK_SRC, 0.0);
    nl += 1;
  }
  g->launches_per_step = nl;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("3D FP32 step: ") + cudaGetErrorString(e));
  return MS_OK;
}

// Largest |h_tau lambda|^2 / 4 over the 3D Fourier symbol at CFL number r (units h = 1).
double max_amp2_3d(double r) {
  const double k2 = 24.0 / (r * r), beta = 1.0 + 2.0 / (r * r);
  const int n = 48;
  std::vector<double> mu(n), dd(n);
  for (int a = 0; a < n; ++a) {
    const double t = M_PI * (a + 1) / n;
    mu[a] = 4.0 * std::sin(t / 2) * std::sin(t / 2);
    const double d = 2.0 * std::sin(t / 2) * 12.0 / (11.0 + std::cos(t));
    dd[a] = d * d;
  }
  double worst = 0.0;
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < n; ++b)
      for (int c = 0; c < n; ++c) {
        const double s1 = mu[a] + mu[b] + mu[c], s2 = mu[a] * mu[b] + mu[b] * mu[c] + mu[c] * mu[a];
        const double gg = k2 * (beta - s1 / 12.0) / (k2 * beta + s1 - s2 / 6.0);
        const double v = r * r * gg * gg * (dd[a] + dd[b] + dd[c]);
        if (v > worst) worst = v;
      }
  return worst;
}

// The polynomial of the FP64 solves: 6 h^2 P1 = D - T, T in [-8, 24] (k_rec64.cu).
ms_status cheb3d64(ms_grid* g) {
  if (!cheb_coefs(6.0 * g->c1 * g->h * g->h + 24.0, 8.0, 16.0, 1e-17, &g->cheb64))
    return fail3(MS_ENOTCONV, "the FP64 solve polynomial needs too high a degree");
  return MS_OK;
}

template <typename T>
ms_status alloc3(T** p, size_t n) {
  cudaError_t e = dev_malloc((void**)p, n * sizeof(T) + 256);
  if (e != cudaSuccess) {
    *p = nullptr;
    return fail3(MS_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  return MS_OK;
}

ms_status store3(ms_grid* g, int c, const double* dev) {
  Grid3D* G3 = g->g3;
  const Shape3& s = G3->sh[c];
  if (g->desc.precision == MS_FP64) {
    if (dev != G3->f64[c])
      MS3_CUDA(cudaMemcpyAsync(G3->f64[c], dev, s.size() * sizeof(double), cudaMemcpyDeviceToDevice, g->stream));
    k_zero_walls3d64<<<grid3(s, kBlk), kBlk, 0, g->stream>>>(G3->f64[c], s);
  } else {
    double* tmp = G3->s64[0];
    if (dev != tmp) MS3_CUDA(cudaMemcpyAsync(tmp, dev, s.size() * sizeof(double), cudaMemcpyDeviceToDevice, g->stream));
    k_zero_walls3d64<<<grid3(s, kBlk), kBlk, 0, g->stream>>>(tmp, s);
    k_split3<<<(unsigned)((s.size() + 255) / 256), 256, 0, g->stream>>>(tmp, G3->hi[c], G3->lo[c], s.size());
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("store: ") + cudaGetErrorString(e));
  return MS_OK;
}

// FP64 view of component c: the FP64 array, or hi + lo joined into dst.
const double* view3(ms_grid* g, int c, double* dst) {
  Grid3D* G3 = g->g3;
  if (g->desc.precision == MS_FP64) return G3->f64[c];
  const size_t n = G3->sh[c].size();
  k_join3<<<(unsigned)((n + 255) / 256), 256, 0, g->stream>>>(G3->hi[c], G3->lo[c], dst, n);
  return dst;
}

// Exact modes (component c) into out, t_E / t_H (see the oracle's mode: sine on node axes,
// cosine on half axes; H = -(1/(Z omega)) curl(E shape) sin(omega t)).
ms_status exact3(ms_grid* g, const ms_mode3* modes, int nm, double tE, double tH, int c, double* out) {
  const int N = g->N;
  const Shape3& s = g->g3->sh[c];
  std::vector<double> host;
  const size_t ox = 0, oy = (size_t)nm * s.n[0], oz = oy + (size_t)nm * s.n[1], oc = oz + (size_t)nm * s.n[2];
  host.assign(oc + nm, 0.0);
  auto sin_node = [&](int k, int i) {
    if (i == 0 || i == N) return 0.0;
    long q = ((long)k * i) % (2L * N);
    return std::sin(M_PI * (double)q / N);
  };
  auto cos_half = [&](int k, int i) {
    long q = ((long)k * (2L * i + 1)) % (4L * N);
    return std::cos(M_PI * (double)q / (2.0 * N));
  };
  for (int q = 0; q < nm; ++q) {
    const int kk[3] = {modes[q].m, modes[q].n, modes[q].p};
    const size_t off[3] = {ox, oy, oz};
    for (int a = 0; a < 3; ++a)
      for (int i = 0; i < s.n[a]; ++i)
        host[off[a] + (size_t)q * s.n[a] + i] = (s.bc[a] == DIR) ? sin_node(kk[a], i) : cos_half(kk[a], i);
    const double a = M_PI * kk[0], b = M_PI * kk[1], cc = M_PI * kk[2];
    const double w = std::sqrt(a * a + b * b + cc * cc);
    const double Ax = modes[q].ax, Ay = modes[q].ay, Az = modes[q].az;
    const double ce = std::cos(w * tE), sh = -std::sin(w * tH) / (g->Z * w);
    const double amp[6] = {Ax * ce, Ay * ce, Az * ce, sh * (Az * b - Ay * cc), sh * (Ax * cc - Az * a),
                           sh * (Ay * a - Ax * b)};
    host[oc + q] = amp[c];
  }
  if (host.size() > g->modetab_cap) {
    dev_free(g->d_modetab);
    g->d_modetab = nullptr;
    g->modetab_cap = 0;
    MS3_TRY(alloc3(&g->d_modetab, host.size()));
    g->modetab_cap = host.size();
  }
  MS3_CUDA(cudaMemcpyAsync(g->d_modetab, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice, g->stream));
  k_mode_field3<<<grid3(s, kBlk), kBlk, 0, g->stream>>>(out, s, g->d_modetab + ox, g->d_modetab + oy,
                                                         g->d_modetab + oz, g->d_modetab + oc, nm);
  MS3_CUDA(cudaGetLastError());
  MS3_CUDA(cudaStreamSynchronize(g->stream));  // the host table is released on return
  return MS_OK;
}

ms_status check_modes3(const ms_mode3* modes, int nm) {
  if (nm < 0 || (nm > 0 && !modes)) return fail3(MS_EINVAL, "invalid modes");
  for (int q = 0; q < nm; ++q) {
    const ms_mode3& m = modes[q];
    if (m.m < 1 || m.n < 1 || m.p < 1) return fail3(MS_EINVAL, "mode indices must be >= 1");
    const double dot = m.ax * m.m + m.ay * m.n + m.az * m.p;
    const double scale = std::fabs(m.ax * m.m) + std::fabs(m.ay * m.n) + std::fabs(m.az * m.p);
    if (std::fabs(dot) > 1e-12 * (scale > 0 ? scale : 1.0))
      return fail3(MS_EINVAL, "mode polarisation must satisfy A . (m, n, p) = 0 (divergence-free E)");
  }
  return MS_OK;
}

}  // namespace

// Rows of 3D sources: indices >= 0 with at least two >= 1, (ax, ay, az) . (m, n, p) = 0, finite
// values; off resonance (omega^2 != pi^2 |k|^2) when a driven solution is asked for.
ms_status check_sources3(const ms_source3* src, int nsrc, bool need_off_resonance) {
  if (nsrc < 0 || nsrc > 64 || (nsrc > 0 && !src)) return fail3(MS_EINVAL, "invalid sources (0 <= nsrc <= 64)");
  for (int q = 0; q < nsrc; ++q) {
    const ms_source3& s = src[q];
    if (s.m < 0 || s.n < 0 || s.p < 0 || s.m > 1000000 || s.n > 1000000 || s.p > 1000000)
      return fail3(MS_EINVAL, "source indices must be in [0, 1e6]");
    if ((s.m > 0) + (s.n > 0) + (s.p > 0) < 2) return fail3(MS_EINVAL, "a source needs at least two nonzero indices");
    if (!std::isfinite(s.ax) || !std::isfinite(s.ay) || !std::isfinite(s.az) || !std::isfinite(s.omega))
      return fail3(MS_EINVAL, "non-finite source");
    const double dot = s.ax * s.m + s.ay * s.n + s.az * s.p;
    const double scale = std::fabs(s.ax * s.m) + std::fabs(s.ay * s.n) + std::fabs(s.az * s.p);
    if (std::fabs(dot) > 1e-12 * (scale > 0 ? scale : 1.0))
      return fail3(MS_EINVAL, "source polarisation must satisfy (ax, ay, az) . (m, n, p) = 0 (div J = 0)");
    if (need_off_resonance) {
      const double k2 = M_PI * M_PI * ((double)s.m * s.m + (double)s.n * s.n + (double)s.p * s.p);
      if (std::fabs(s.omega * s.omega - k2) <= 1e-12 * (k2 > 1 ? k2 : 1.0) || s.omega == 0.0)
        return fail3(MS_EINVAL, "driven solution needs 0 < omega^2 != pi^2 (m^2 + n^2 + p^2)");
    }
  }
  return MS_OK;
}

ms_status mode_field3_tables(ms_grid* g, int c, const std::vector<double>& tq, const std::vector<double>& coef,
                             double* out) {
  const Shape3& s = g->g3->sh[c];
  const int nm = (int)coef.size(), per = s.n[0] + s.n[1] + s.n[2];
  const size_t oy = (size_t)nm * s.n[0], oz = oy + (size_t)nm * s.n[1], oc = oz + (size_t)nm * s.n[2];
  std::vector<double> host(oc + nm, 0.0);
  for (int q = 0; q < nm; ++q) {
    for (int i = 0; i < s.n[0]; ++i) host[(size_t)q * s.n[0] + i] = tq[(size_t)q * per + i];
    for (int j = 0; j < s.n[1]; ++j) host[oy + (size_t)q * s.n[1] + j] = tq[(size_t)q * per + s.n[0] + j];
    for (int k = 0; k < s.n[2]; ++k) host[oz + (size_t)q * s.n[2] + k] = tq[(size_t)q * per + s.n[0] + s.n[1] + k];
    host[oc + q] = coef[q];
  }
  if (host.size() > g->modetab_cap) {
    dev_free(g->d_modetab);
    g->d_modetab = nullptr;
    g->modetab_cap = 0;
    MS3_TRY(alloc3(&g->d_modetab, host.size()));
    g->modetab_cap = host.size();
  }
  MS3_CUDA(cudaMemcpyAsync(g->d_modetab, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice, g->stream));
  k_mode_field3<<<grid3(s, kBlk), kBlk, 0, g->stream>>>(out, s, g->d_modetab, g->d_modetab + oy, g->d_modetab + oz,
                                                         g->d_modetab + oc, nm);
  MS3_CUDA(cudaGetLastError());
  MS3_CUDA(cudaStreamSynchronize(g->stream));  // the host table is released on return
  return MS_OK;
}


double stability_limit_3d() {
  static double cached = 0.0;
  if (cached > 0.0) return cached;
  double lo = 0.3, hi = 1.0;
  for (int it = 0; it < 50; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (max_amp2_3d(mid) <= 4.0) lo = mid;
    else hi = mid;
  }
  cached = lo;
  return cached;
}

ms_status create_grid3d(const ms_grid_desc* d, ms_grid** out) {
  if (d->n < 4 || d->n > 512) return fail3(MS_EINVAL, "3D grids need 4 <= n <= 512");
  if (!(d->z_imp > 0.0) || !std::isfinite(d->z_imp)) return fail3(MS_EINVAL, "z_imp must be positive");
  if (!(d->r > 0.0) || !std::isfinite(d->r)) return fail3(MS_EINVAL, "r must be positive");
  if (d->precision != MS_FP64 && d->precision != MS_FP32_REFINED) return fail3(MS_EINVAL, "unknown precision");
  if (d->closure != MS_CLOSURE_PAPER && d->closure != MS_CLOSURE_REFLECT) return fail3(MS_EINVAL, "unknown closure");
  if (d->scheme != MS_SCHEME_C4) return fail3(MS_EUNSUPPORTED, "3D grids run the compact scheme only");
  const double rmax = stability_limit_3d();
  if (d->r >= rmax) {
    char buf[160];
    snprintf(buf, sizeof buf, "r = %.6g is at or above the stability limit %.6g of the 3D scheme", d->r, rmax);
    return fail3(MS_ECFL, buf);
  }
  ms_grid* g = new ms_grid();
  g->g3 = new Grid3D();
  Grid3D* G3 = g->g3;
  g->desc = *d;
  g->N = d->n;
  g->Z = d->z_imp;
  g->h = 1.0 / d->n;
  g->ht = d->r * g->h;
  g->kappa2 = 24.0 / (g->ht * g->ht);
  g->beta = 1.0 + g->kappa2 * g->h * g->h / 12.0;
  g->c1 = g->kappa2 * g->beta;
  auto cleanup = [&](ms_status s) {
    ms_destroy(g);
    return s;
  };
  for (int c = 0; c < 6; ++c) {
    G3->sh[c] = field_shape3(g->N, c);
    if (G3->sh[c].size() > G3->nmax) G3->nmax = G3->sh[c].size();
  }
  if (d->stream) {
    g->stream = (cudaStream_t)d->stream;
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cleanup(fail3(MS_ECUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e)));
    g->own_stream = true;
  }
  std::string err;
  ms_status s = MS_OK;
  if (d->precision == MS_FP64) {
    for (int kind = 0; kind < 2 && s == MS_OK; ++kind) {
      const int M = (kind == HALF_TO_NODE) ? g->N - 1 : g->N;
      PadeTable& t = g->pade[kind];
      if (build_pade_table(M, d->closure, kind, 1e-18, &t, &err) != 0) return cleanup(fail3(MS_EINVAL, err));
      if (M >= kRecMinLine) continue;  // longer lines take the recurrences
      s = alloc3(&t.d_w, t.w.size());
      if (s == MS_OK && cudaMemcpy(t.d_w, t.w.data(), t.w.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
        s = fail3(MS_ECUDA, "copy of Pade tables failed");
    }
    if (s == MS_OK) s = cheb3d64(g);
    for (int c = 0; c < 6 && s == MS_OK; ++c) s = alloc3(&G3->f64[c], G3->sh[c].size());
    const size_t pl = (G3->nmax + 31) / 32 * 32;
    if (s == MS_OK) s = alloc3(&G3->slab64, 9 * pl);
    for (int k = 0; k < 9 && s == MS_OK; ++k) G3->s64[k] = G3->slab64 + k * pl;
  } else {
    for (int kind = 0; kind < 2 && s == MS_OK; ++kind) {
      const int M = (kind == HALF_TO_NODE) ? g->N - 1 : g->N;
      PadeTable& t = g->pade32[kind];
      if (build_pade_table(M, d->closure, kind, 1e-12, &t, &err, /*of_differences=*/true) != 0)
        return cleanup(fail3(MS_EINVAL, err));
      if (M >= kWalk3Min) continue;  // longer lines take the walks
      std::vector<float> whi(t.w.size()), wlo(t.w.size());
      for (size_t q = 0; q < t.w.size(); ++q) {
        whi[q] = (float)t.w[q];
        wlo[q] = (float)(t.w[q] - (double)whi[q]);
      }
      s = alloc3(&t.d_whi, whi.size());
      if (s == MS_OK) s = alloc3(&t.d_wlo, wlo.size());
      if (s == MS_OK && (cudaMemcpy(t.d_whi, whi.data(), whi.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
                         cudaMemcpy(t.d_wlo, wlo.data(), wlo.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess))
        s = fail3(MS_ECUDA, "copy of FP32 Pade tables failed");
    }
    for (int kind = 0; kind < 2; ++kind) line_ends(d->closure, kind, false, &g->walk.ends[kind]);
    // the solve polynomial to 1e-10 (below the FP32 rounding noise, which is not coherent)
    if (s == MS_OK && !cheb_coefs(6.0 * g->c1 * g->h * g->h + 24.0, 8.0, 16.0, 1e-10, &g->walk.cheb))
      s = fail3(MS_ENOTCONV, "the FP32 solve polynomial needs too high a degree");
    for (int c = 0; c < 6 && s == MS_OK; ++c) s = alloc3(&G3->hi[c], G3->sh[c].size());
    for (int c = 0; c < 6 && s == MS_OK; ++c) s = alloc3(&G3->lo[c], G3->sh[c].size());
    for (int k = 0; k < 3 && s == MS_OK; ++k) s = alloc3(&G3->s32[k], G3->nmax);
    for (int k = 0; k < 3 && s == MS_OK; ++k) s = alloc3(&G3->gh[k], G3->nmax);
    for (int k = 0; k < 3 && s == MS_OK; ++k) s = alloc3(&G3->gl[k], G3->nmax);
    for (int k = 0; k < 2 && s == MS_OK; ++k) s = alloc3(&G3->s64[k], G3->nmax);
  }
  if (s == MS_OK) s = alloc3(&g->d_result, 8);
  if (s == MS_OK) {
    const int b = reduce_blocks(G3->nmax);
    s = alloc3(&g->d_partial, (size_t)b * 4);
    g->partial_cap = b;
  }
  if (s != MS_OK) return cleanup(s);
  for (int c = 0; c < 6; ++c) {
    const size_t n = G3->sh[c].size();
    if (G3->f64[c]) cudaMemsetAsync(G3->f64[c], 0, n * sizeof(double), g->stream);
    if (G3->hi[c]) cudaMemsetAsync(G3->hi[c], 0, n * sizeof(float), g->stream);
    if (G3->lo[c]) cudaMemsetAsync(G3->lo[c], 0, n * sizeof(float), g->stream);
  }
  for (int k = 0; k < 9; ++k)
    if (G3->s64[k]) cudaMemsetAsync(G3->s64[k], 0, G3->nmax * sizeof(double), g->stream);
  for (int k = 0; k < 3; ++k)
    if (G3->s32[k]) cudaMemsetAsync(G3->s32[k], 0, G3->nmax * sizeof(float), g->stream);
  cudaError_t e = cudaStreamSynchronize(g->stream);
  if (e != cudaSuccess) return cleanup(fail3(MS_ECUDA, std::string("create: ") + cudaGetErrorString(e)));
  *out = g;
  return MS_OK;
}

// Accuracy of one transform solve relative to the solution (bf16 three-product split: about 16
// correct bits per pass over six passes, measured at up to 2e-5 on random data), which fixes the
// refinement sweeps: ts_accuracy * rho^R <= 1e-10, the target of the polynomial solve.
constexpr double kTsAccuracy = 5e-5;

ms_status set_solver3d(ms_grid* g, int solver) {
  Grid3D* G3 = g->g3;
  if (solver == MS_SOLVER_RICHARDSON) {
    G3->solver = solver;
    return MS_OK;
  }
  if (!G3->ts) {
    G3->ts = new TransformSolver();
    std::string err;
    const int rc = ts_setup(g->N, G3->ts, &err);
    if (rc != 0) {
      ts_free(G3->ts);
      delete G3->ts;
      G3->ts = nullptr;
      return fail3(rc == -2 ? MS_ENOMEM : MS_ECUDA, err);
    }
  }
  int R = 0;
  MS3_TRY(ms_solver_sweeps(3, g->desc.r, MS_FP32_REFINED, 1e-10 / kTsAccuracy, &R));
  G3->ts_sweeps = R;
  G3->solver = solver;
  return MS_OK;
}

ms_status transform_solve3d(ms_grid* g, int c, const float* b, float* x) {
  Grid3D* G3 = g->g3;
  if (!G3->ts) {  // set the solver up without selecting it
    const int keep = G3->solver;
    MS3_TRY(set_solver3d(g, MS_SOLVER_TRANSFORM_TC));
    G3->solver = keep;
  }
  ts_solve(*G3->ts, G3->sh[c], b, x, 6.0f * (float)(g->c1 * g->h * g->h), g->stream, g);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("transform solve: ") + cudaGetErrorString(e));
  return MS_OK;
}

ms_status transform_status3d(ms_grid* g) {
  Grid3D* G3 = g->g3;
  if (!G3 || !G3->ts) return MS_OK;
  int flag = 0;
  if (cudaMemcpy(&flag, G3->ts->d_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail3(MS_ECUDA, "reading the transform solver's status failed");
  if (flag) {
    cudaMemset(G3->ts->d_err, 0, sizeof(int));
    return fail3(MS_ETIMEOUT, "a transform GEMM gave up waiting for its tensor-core MMAs; its output is invalid");
  }
  return MS_OK;
}

void destroy_grid3d(ms_grid* g) {
  Grid3D* G3 = g->g3;
  if (!G3) return;
  src3_free(g);
  if (G3->ts) {
    ts_free(G3->ts);
    delete G3->ts;
    G3->ts = nullptr;
  }
  for (int c = 0; c < 6; ++c) {
    dev_free(G3->f64[c]);
    dev_free(G3->hi[c]);
    dev_free(G3->lo[c]);
    dev_free(G3->dview[c]);
  }
  dev_free(G3->slab64);
  for (int k = 0; k < 9 && !G3->slab64; ++k) dev_free(G3->s64[k]);
  for (int k = 0; k < 3; ++k) dev_free(G3->s32[k]);
  for (int k = 0; k < 3; ++k) {
    dev_free(G3->gh[k]);
    dev_free(G3->gl[k]);
  }
  for (int k = 0; k < 2; ++k) {
    dev_free(g->pade32[k].d_whi);
    dev_free(g->pade32[k].d_wlo);
    g->pade32[k].d_whi = g->pade32[k].d_wlo = nullptr;
  }
  delete G3;
  g->g3 = nullptr;
}

int state_arrays3d(ms_grid* g, double** f64, float** hi, float** lo, size_t* n) {
  Grid3D* G3 = g->g3;
  for (int c = 0; c < 6; ++c) {
    f64[c] = G3->f64[c];
    hi[c] = G3->hi[c];
    lo[c] = G3->lo[c];
    n[c] = G3->sh[c].size();
  }
  return 6;
}

ms_status step3d(ms_grid* g) { return g->desc.precision == MS_FP64 ? step3d64(g) : step3d32(g); }

ms_status set_fields3d(ms_grid* g, const double* const* comps, int host) {
  for (int c = 0; c < 6; ++c)
    if (!comps[c]) return fail3(MS_EINVAL, "NULL component");
  Grid3D* G3 = g->g3;
  for (int c = 0; c < 6; ++c) {
    const size_t n = G3->sh[c].size();
    if (host) {
      double* tmp = G3->s64[0];
      MS3_CUDA(cudaMemcpyAsync(tmp, comps[c], n * sizeof(double), cudaMemcpyHostToDevice, g->stream));
      MS3_TRY(store3(g, c, tmp));
    } else {
      MS3_TRY(store3(g, c, comps[c]));
    }
  }
  if (host) MS3_CUDA(cudaStreamSynchronize(g->stream));
  return MS_OK;
}

ms_status get_fields3d(ms_grid* g, double* const* comps, int host) {
  for (int c = 0; c < 6; ++c)
    if (!comps[c]) return fail3(MS_EINVAL, "NULL component");
  Grid3D* G3 = g->g3;
  for (int c = 0; c < 6; ++c) {
    const size_t n = G3->sh[c].size();
    if (g->desc.precision == MS_FP64) {
      MS3_CUDA(cudaMemcpyAsync(comps[c], G3->f64[c], n * sizeof(double),
                               host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, g->stream));
    } else if (host) {
      const double* v = view3(g, c, G3->s64[0]);
      MS3_CUDA(cudaMemcpyAsync(comps[c], v, n * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
      MS3_CUDA(cudaStreamSynchronize(g->stream));  // s64[0] is reused by the next component
    } else {
      view3(g, c, comps[c]);
    }
  }
  MS3_CUDA(cudaGetLastError());
  if (host) MS3_CUDA(cudaStreamSynchronize(g->stream));
  return MS_OK;
}

// FP64 components for the diagnostics.  An FP64 grid gives its state; an FP32_REFINED grid joins
// its float-float state into FP64 copies, and on the first call builds what the FP64 kernels need
// (FP64 Pade tables, the FP64 polynomial, FP64 scratch), kept until the grid is destroyed.
ms_status diag_view3d(ms_grid* g, double** f) {
  Grid3D* G3 = g->g3;
  if (g->desc.precision == MS_FP64) {
    for (int c = 0; c < 6; ++c) f[c] = G3->f64[c];
    return MS_OK;
  }
  std::string err;
  for (int kind = 0; kind < 2; ++kind) {
    PadeTable& t = g->pade[kind];
    if (t.d_w || t.M >= kRecMinLine) continue;
    const int M = (kind == HALF_TO_NODE) ? g->N - 1 : g->N;
    if (build_pade_table(M, g->desc.closure, kind, 1e-18, &t, &err) != 0) return fail3(MS_EINVAL, err);
    if (M >= kRecMinLine) continue;
    MS3_TRY(alloc3(&t.d_w, t.w.size()));
    if (cudaMemcpy(t.d_w, t.w.data(), t.w.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess)
      return fail3(MS_ECUDA, "copy of Pade tables failed");
  }
  if (!g->cheb64.m) MS3_TRY(cheb3d64(g));
  for (int k = 0; k < 9; ++k)
    if (!G3->s64[k]) MS3_TRY(alloc3(&G3->s64[k], G3->nmax));
  for (int c = 0; c < 6; ++c) {
    const size_t n = G3->sh[c].size();
    if (!G3->dview[c]) MS3_TRY(alloc3(&G3->dview[c], n));
    k_join3<<<(unsigned)((n + 255) / 256), 256, 0, g->stream>>>(G3->hi[c], G3->lo[c], G3->dview[c], n);
    f[c] = G3->dview[c];
  }
  return MS_OK;
}

// Discrete energy of a 3D grid: W = h^3 [Z^-1 sum E.E + Z (sum H.H - h_tau sum H*.H)], H* the Step 2
// increment that the current E gives (P1^{-1} of the H right-hand side), computed in FP64 with the
// step's own filter, Pade and solve kernels but not added to H.
ms_status energy3d(ms_grid* g, double* W) {
  Grid3D* G3 = g->g3;
  double* f[6];
  MS3_TRY(diag_view3d(g, f));
  double** G = G3->s64;  // G[0..2]: filtered E
  double** R = G3->s64 + 3;
  const double* X[3];  // the increments
  const double s_eh = g->kappa2 / (g->Z * g->h);
  int nl = 0;
  filter3d64(g, 0, f, G);
  for (int c = 0; c < 3; ++c) {
    const size_t n = G3->sh[c].size();
    launch_dot(f[c], f[c], n, g->d_partial, reduce_blocks(n), g->d_result, 0, c > 0, g->stream);
  }
  curl3d64(g, 0, 3, G, R, -s_eh);
  for (int c = 0; c < 3; ++c) {  // walls of the work planes, which the solve does not write
    MS3_CUDA(cudaMemsetAsync(G3->s64[c], 0, G3->nmax * sizeof(double), g->stream));
    MS3_CUDA(cudaMemsetAsync(G3->s64[6 + c], 0, G3->nmax * sizeof(double), g->stream));
  }
  solve3d64(g, 3, R, nullptr, 0.0, X, &nl);
  for (int hc = 0; hc < 3; ++hc) {
    const size_t n = G3->sh[3 + hc].size();
    const double* Hc = f[3 + hc];
    launch_dot(Hc, Hc, n, g->d_partial, reduce_blocks(n), g->d_result, 1, hc > 0, g->stream);
    launch_dot(X[hc], Hc, n, g->d_partial, reduce_blocks(n), g->d_result, 2, hc > 0, g->stream);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("3D energy: ") + cudaGetErrorString(e));
  double r[3];
  MS3_CUDA(cudaMemcpyAsync(r, g->d_result, sizeof r, cudaMemcpyDeviceToHost, g->stream));
  MS3_CUDA(cudaStreamSynchronize(g->stream));
  *W = g->h * g->h * g->h * (r[0] / g->Z + g->Z * (r[1] - g->ht * r[2]));
  return MS_OK;
}

// Pade divergence of H on the N^3 cell centres of a 3D grid (in FP64): div_h H = sum_a delta_a H_a,
// each a node -> half-node derivative along its own axis; *norm = sqrt(h^3 sum div^2).
ms_status divergence3d(ms_grid* g, double* norm) {
  Grid3D* G3 = g->g3;
  double* f[6];
  MS3_TRY(diag_view3d(g, f));
  const int N = g->N;
  Shape3 sc;  // cell centres: N points on every axis, no walls
  for (int a = 0; a < 3; ++a) {
    sc.n[a] = N;
    sc.bc[a] = NEU;
  }
  double* div = G3->s64[0];
  const double sc_h = 1.0 / g->h;
  for (int a = 0; a < 3; ++a) {
    const Pade3d64 q{a, G3->sh[3 + a], sc, f[3 + a], div, sc_h, a > 0};
    pade3d64(g, &q, 1);
  }
  const size_t n = sc.size();
  launch_dot(div, div, n, g->d_partial, reduce_blocks(n), g->d_result, 0, 0, g->stream);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(MS_ECUDA, std::string("3D divergence: ") + cudaGetErrorString(e));
  double r;
  MS3_CUDA(cudaMemcpyAsync(&r, g->d_result, sizeof r, cudaMemcpyDeviceToHost, g->stream));
  MS3_CUDA(cudaStreamSynchronize(g->stream));
  *norm = std::sqrt(g->h * g->h * g->h * r);
  return MS_OK;
}

}  // namespace ms

using namespace ms;

extern "C" {

ms_status ms_init_modes3(ms_grid* g, const ms_mode3* modes, int nmodes) {
  if (!g || !g->g3) return fail3(MS_EINVAL, "ms_init_modes3 needs a 3D grid");
  MS3_TRY(check_modes3(modes, nmodes));
  double* tmp = g->g3->s64[1];
  for (int c = 0; c < 6; ++c) {
    MS3_TRY(exact3(g, modes, nmodes, 0.0, 0.5 * g->ht, c, tmp));
    MS3_TRY(store3(g, c, tmp));
  }
  g->step = 0;
  if (g->d_step) MS3_CUDA(cudaMemcpy(g->d_step, &g->step, sizeof(long), cudaMemcpyHostToDevice));
  MS3_CUDA(cudaStreamSynchronize(g->stream));
  return MS_OK;
}

ms_status ms_init_driven3(ms_grid* g, const ms_source3* src, int nsrc) {
  if (!g || !g->g3) return fail3(MS_EUNSUPPORTED, "ms_init_driven3 needs a 3D grid");
  MS3_TRY(check_sources3(src, nsrc, true));
  double* tmp = g->g3->s64[1];
  for (int c = 0; c < 6; ++c) {
    MS3_TRY(exact_driven3(g, src, nsrc, 0.0, 0.5 * g->ht, c, tmp));
    MS3_TRY(store3(g, c, tmp));
  }
  g->step = 0;
  if (g->d_step) MS3_CUDA(cudaMemcpy(g->d_step, &g->step, sizeof(long), cudaMemcpyHostToDevice));
  MS3_CUDA(cudaStreamSynchronize(g->stream));
  return MS_OK;
}

ms_status ms_error_vs_exact3(ms_grid* g, const ms_mode3* modes, int nmodes, double* l2_abs, double* l2_rel,
                             double* max_abs, double* sum_abs) {
  if (!g || !g->g3) return fail3(MS_EINVAL, "ms_error_vs_exact3 needs a 3D grid");
  MS3_TRY(check_modes3(modes, nmodes));
  Grid3D* G3 = g->g3;
  const double tE = g->step * g->ht, tH = (g->step + 0.5) * g->ht;
  for (int c = 0; c < 6; ++c) {
    const size_t n = G3->sh[c].size();
    MS3_TRY(exact3(g, modes, nmodes, tE, tH, c, G3->s64[1]));
    const double* v = view3(g, c, G3->s64[0]);
    launch_err_reduce(v, G3->s64[1], n, g->d_partial, reduce_blocks(n), g->d_result, c > 0, g->stream);
  }
  double r[4];
  MS3_CUDA(cudaMemcpyAsync(r, g->d_result, sizeof r, cudaMemcpyDeviceToHost, g->stream));
  MS3_CUDA(cudaStreamSynchronize(g->stream));
  const double h3 = g->h * g->h * g->h;
  if (l2_abs) *l2_abs = std::sqrt(h3 * r[0]);
  if (l2_rel) *l2_rel = r[1] > 0.0 ? std::sqrt(r[0] / r[1]) : 0.0;
  if (max_abs) *max_abs = r[2];
  if (sum_abs) *sum_abs = r[3];
  return MS_OK;
}

}  // extern "C"
