// Reverse (adjoint) pass of the FP32_REFINED step in FP32 arithmetic with a float-float adjoint
// state.
//
// The FP32_REFINED forward step, in the units of k_mixed.cu, is
//   S1: E   += sE P~_E^{-1} (Y_x F~ H_y - Y_y F~ H_x),
//   S2: H_x += sH P~_Hx^{-1} (-Y_y F~ E),   H_y += sH P~_Hy^{-1} (Y_x F~ E),
// with P~ = 6 h^2 P1 (Def. "def:operatorsP"), F~ = 12 beta + L the filter of Eq. "eq:ell" on the
// source grid, Y = A^{-1} D the Pade derivative of App. A.1 (D the first differences of a line),
// sE = 12 Z / r, sH = 12 / (r Z).  F~ and P~ are symmetric on the unknowns (Dirichlet zeros, even Neumann
// ghosts), so the transposed step M^T = S1^T S2^T is
//   S2^T: l_E  += sH F~_E (-Y_y^T P~^{-1} l_Hx + Y_x^T P~^{-1} l_Hy),
//   S1^T: l_Hy += sE F~_Hy Y_x^T P~_E^{-1} l_E,   l_Hx += -sE F~_Hx Y_y^T P~_E^{-1} l_E,
// with Y^T = D^T A^{-T}: (Y^T u)_j = v_{j-1} - v_j, v = A^{-T} u, v_{-1} = v_M = 0.
//
// Precision.  D^T takes the difference of two nearly equal values of a smooth v, which would
// amplify an FP32 rounding of v by 1 / (pi k h).  A^{-1} and the difference commute on the infinite line,
// so the difference is taken first, of the float-float u, and A^{-1} is applied to it in FP32: with
// e_j = u_{j-1} - u_j (u_{-1} = u_M = 0, zero beyond the line) and w the infinite-line solution for e,
// (Y^T u)_j = w_j + k_j w_0 near the first end and its mirror image at the last (the end rows of A^{-T}
// change v by a multiple of its first value, and w_0 = (rho - 1) v_0).  The difference of the high parts is
// kept apart from that of the low parts, the recurrences' rho z and the end correction, all small beside it, until w
// itself is rounded: one rounding of w's size per value, as in a float-float A^{-1} whose result is differenced.
//   u is a pair (l_hi, uc) over the value of the solve's polynomial at t = 36, where smooth fields sit, so that
// uc, the rest, holds only what (T - 36) makes of them: its rounding, which the difference amplifies too, is that of
// a second difference.  As p_0 (l_hi, l_lo + q T y) before, uc was 36 / D of l_hi (1.8e-2 at r = 0.65) and a step's
// derivatives at 2048^2 were off by 1.3e-7 of themselves, 5.3e-8 by the Richardson solve before that, 3.2e-8 now
// (1024^2, r = 0.5: 3.5e-8, 3.6e-8, 2.6e-8).
//   The filter and the scaling act on the difference, a well-conditioned FP32 value, and the result is added to l
// with error-free transformations.  The step is the transpose of the FP64 operator up to this rounding.  Gradients
// after 2000 steps at 1024^2 stand 1.9e-8 from the FP64 reverse pass (bands and sweeps: 2.2e-8).
//
// Kernels, six launches per reverse step, the walks of k_tiled.cu turned round: solve (k_solve_pair),
// both transposed derivatives into planes (k_walk_dT), filter and update (k_filter_update), for the H
// fields and then for E_z: 43 us per step at 1024^2, 124 at 2048^2.  The band form before it (separate sweeps,
// transposed bands in float-float, one kernel per operator, 18 launches) took 165 and 506 us.
#include <string>
#include <vector>

#include "k_fp64.cuh"
#include "k_mixed.cuh"
#include "k_rec64.cuh"
#include "k_tiled.cuh"
#include "k_walk_dev.cuh"

namespace ms {

struct Adj32 {
  float* slab = nullptr;
  float* lh[3] = {};  // adjoint state (l_E, l_Hx, l_Hy), hi parts
  float* ll[3] = {};  // lo parts
  float* uc[3] = {};  // low parts of the solutions, u = gain (l_hi + uc)
  float* py[3] = {};  // transposed derivatives along y (E_z, H_x) and ...
  float* px[3] = {};  // ... along x (E_z, H_y)
  Graph g1, gk;
};

namespace {

ms_status a32fail(ms_status s, const std::string& m) {
  set_last_error(m.c_str());
  return s;
}

void free_graph32(Graph* gr) {
  if (gr->exec) cudaGraphExecDestroy(gr->exec);
  if (gr->graph) cudaGraphDestroy(gr->graph);
  *gr = Graph{};
}

constexpr int kEndT = 16;   // rows the end correction reaches (its vector decays from the fourth row on)
constexpr int TOUT = 104;   // columns a warp writes along x (12 on each side: carries and end rows)
constexpr int THALO = 12;

// ---- solve ---------------------------------------------------------------------------------

// (Four blocks per SM with three levels: with five, 124 bytes of spills.)

template <int P>
__global__ void __launch_bounds__(32 * WPB, P <= 2 ? 5 : 4) k_solve_pair(const __grid_constant__ SArgs A,
                                                                         const __grid_constant__ SArgs B, int na) {
  __shared__ float4 ring[WPB][4 * kRing * 32];
  pdl_wait();
  const int w = threadIdx.x >> 5, b = blockIdx.x;
  if (b < na) s_item<P, true>(A, ring[w], b * WPB + w);
  else s_item<P, true>(B, ring[w], (b - na) * WPB + w);
}

// ---- transposed derivatives ----------------------------------------------------------------

// Along y: lines are the columns 1 .. ncol-2, inputs u_0 .. u_{M-1}, outputs 0 .. M, written negated.
struct YTArgs {
  const float* uh;  // row of u_0, column 0
  const float* ul;
  float* b;         // row of output 0
  int ld, ncol, M;
  float k[kEndT], kl[kEndT];  // end correction, in pairs
  int nstrip, nseg, chunk, end;  // segments: 0 down from the first end, 1 up from the last (`end` rows
                                 // each), the others `chunk` rows down between them
};

// Along x, rows 1 .. nrows of E_z- or H_y-shaped fields; pointers at column m = 0.
struct XTArgs {
  const float* uh;
  const float* ul;
  float* b;
  int ld, M;     // inputs per line
  int from_h;    // input u_i at column i of H_y, output j at column j - 1 of E_z; else u_i at column i of
                 // E_z, output j at column j of H_y
  float k[kEndT], kl[kEndT];
  int nrows, nstrip, nblk, rows;
};

// A segment of 32 columns: y of e = differences of u, groups of eight rows (k_tiled.cu).  UP: the segment
// walks up from the last end, rows and sign mirrored.  EDGE: rows may lie beyond the line.
template <bool EDGE>
__device__ __forceinline__ void yt_segment(const YTArgs& A, int strip, int seg) {
  const int lane = threadIdx.x & 31;
  const int col = 1 + 32 * strip + lane;
  const bool live = col <= A.ncol - 2;
  const int cc = min(col, A.ncol - 2);
  const int M = A.M, R = M + 1;
  const bool up = seg == 1;
  const int r0 = seg < 2 ? 0 : A.end + (seg - 2) * A.chunk;
  const int r1 = seg < 2 ? A.end : min(r0 + A.chunk, R - A.end);
  const ptrdiff_t st = up ? -(ptrdiff_t)A.ld : (ptrdiff_t)A.ld;
  const float* ph = A.uh + cc + (up ? (size_t)(M - 1) * A.ld : 0);  // logical row i at ph[i * st]
  const float* pl = A.ul + cc + (up ? (size_t)(M - 1) * A.ld : 0);
  float* bp = A.b + cc + (up ? (ptrdiff_t)M * A.ld : 0) + (ptrdiff_t)r0 * st;
  const float sign = up ? 1.0f : -1.0f;  // results are written negated; the mirror changes the sign
  auto get = [&](const float* p, int i) { return EDGE ? ((i >= 0 && i < M) ? p[i * st] : 0.0f) : p[i * st]; };
  const int ms = r0 - 9;
  float h0 = get(ph, ms - 1), l0 = get(pl, ms - 1);  // u_{m-1}
  float nh[8], nl[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    nh[t] = get(ph, ms + t);
    nl[t] = get(pl, ms + t);
  }
  float z = 0.0f, ep[7] = {}, gp[7] = {}, w0 = 0.0f, w0l = 0.0f;
  const int ngrp = 2 + (r1 - r0 + 7) / 8;
  for (int gi = 0; gi < ngrp; ++gi) {
    const int m0 = ms + 8 * gi;
    float ch[8], cl[8], ec[8], gc[8], zc[8], y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      ch[t] = nh[t];
      cl[t] = nl[t];
    }
    if (gi + 1 < ngrp) {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        nh[t] = get(ph, m0 + 8 + t);
        nl[t] = get(pl, m0 + 8 + t);
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      ec[t] = h0 - ch[t];
      gc[t] = fmaf(kRhoF, z, l0 - cl[t]);
      h0 = ch[t];
      l0 = cl[t];
      zc[t] = z = ec[t] + gc[t];
    }
    float acc = zc[7];
#pragma unroll
    for (int t = 6; t >= 1; --t) acc = fmaf(kRhoF, acc, zc[t]);
    const float ynext = acc;
    y[7] = acc = ec[0] + fmaf(kRhoF, acc, gc[0]);
#pragma unroll
    for (int t = 6; t >= 0; --t) y[t] = acc = ep[t] + fmaf(kRhoF, acc, gp[t]);
    if (EDGE && seg < 2 && gi >= 2 && gi < 2 + kEndT / 8) {  // the first end's rows
      float n[8];                                             // y less e
#pragma unroll
      for (int t = 0; t < 8; ++t) n[t] = fmaf(kRhoF, t < 7 ? y[t < 7 ? t + 1 : t] : ynext, t < 7 ? gp[t < 7 ? t : 0] : gc[0]);
      if (gi == 2) {
        w0 = y[0];
        w0l = n[0] - (w0 - ep[0]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int j = 8 * (gi - 2) + t;
        y[t] = (t < 7 ? ep[t < 7 ? t : 0] : ec[0]) + fmaf(A.k[j], w0, fmaf(A.kl[j], w0, fmaf(A.k[j], w0l, n[t])));
      }
    }
#pragma unroll
    for (int t = 0; t < 7; ++t) {
      ep[t] = ec[t + 1];
      gp[t] = gc[t + 1];
    }
    if (gi < 2) continue;
    if (live) {
      const int left = r1 - (r0 + 8 * (gi - 2));
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t < left) bp[t * st] = sign * y[t];
    }
    bp += 8 * st;
  }
}

__device__ __forceinline__ void yt_item(const YTArgs& A, int item) {
  if (item >= A.nstrip * A.nseg) return;
  const int seg = item / A.nstrip, strip = item - seg * A.nstrip;
  // rows of u: r0 - 10 .. r1 + 15
  if (seg >= 2 && A.end + (seg - 2) * A.chunk >= 10 && min(A.end + (seg - 1) * A.chunk, A.M + 1 - A.end) + 15 < A.M)
    yt_segment<false>(A, strip, seg);
  else yt_segment<true>(A, strip, seg);
}

template <bool FROM_H, bool EDGE>
__device__ __forceinline__ void xt_block(const XTArgs& A, float4* ring, int strip, int blk) {
  const int lane = threadIdx.x & 31;
  const int m_s = TOUT * strip - THALO, m0 = m_s + 4 * lane;
  const int M = A.M, o = FROM_H ? 1 : 0;  // output index j = column + o
  const int Mo = M + 1 - 2 * o;           // columns written: the unknown ones of E_z (0 .. M-2), all of H_y
  const int j0 = 1 + blk * A.rows, j1 = min(j0 + A.rows, 1 + A.nrows);
  const size_t ld = A.ld;
  const bool ok = !EDGE || (m0 >= -4 && m0 + 8 <= A.ld);
  const bool out = lane >= THALO / 4 && lane < (THALO + TOUT) / 4 && (!EDGE || (m0 >= 0 && m0 < Mo));
  bool inu[4] = {true, true, true, true}, ine[4] = {true, true, true, true};
  float kl[4] = {}, kr[4] = {}, kll[4] = {}, krl[4] = {};
  bool left = false, right = false;
  int ll = 0, el = 0, lr = 0, er = 0;  // lane and element of output 0 and of output M
  if (EDGE) {
    left = strip == 0;
    right = M - o <= m_s + 127;
    ll = (-o - m_s) >> 2;
    el = (-o - m_s) & 3;
    lr = (M - o - m_s) >> 2;
    er = (M - o - m_s) & 3;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int m = m0 + q, j = m + o, r = M - j;
      inu[q] = m >= 0 && m < M;
      ine[q] = j >= 0 && j <= M;
      kl[q] = (left && j >= 0 && j < kEndT) ? A.k[j & (kEndT - 1)] : 0.0f;
      kr[q] = (right && r >= 0 && r < kEndT) ? A.k[r & (kEndT - 1)] : 0.0f;
      kll[q] = (left && j >= 0 && j < kEndT) ? A.kl[j & (kEndT - 1)] : 0.0f;
      krl[q] = (right && r >= 0 && r < kEndT) ? A.kl[r & (kEndT - 1)] : 0.0f;
    }
  }
  const size_t off = ok ? m0 : 0;
  const float* fh = A.uh + (size_t)j0 * ld + off;
  const float* fl = A.ul + (size_t)j0 * ld + off;
  int todo = j1 - j0;
  auto fetch = [&](int slot) {
    if (todo > 0) {
      cp16(ring + (2 * slot) * 32 + lane, fh, ok);
      cp16(ring + (2 * slot + 1) * 32 + lane, fl, ok);
    }
    cp_commit();
    fh += ld;
    fl += ld;
    --todo;
  };
#pragma unroll
  for (int t = 0; t < kAhead; ++t) fetch(t);
  float* bp = A.b + (size_t)j0 * ld + m0;
  int rd = 0, wr = kAhead;
  for (int jj = j0; jj < j1; ++jj, bp += ld) {
    cp_wait<kAhead - 1>();
    const float4 H = ring[(2 * rd) * 32 + lane], L = ring[(2 * rd + 1) * 32 + lane];
    fetch(wr);
    rd = rd == kRing - 1 ? 0 : rd + 1;
    wr = wr == kRing - 1 ? 0 : wr + 1;
    float h[4] = {H.x, H.y, H.z, H.w}, l[4] = {L.x, L.y, L.z, L.w}, e[4], d[4], y[4];
    if (EDGE) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        h[q] = inu[q] ? h[q] : 0.0f;
        l[q] = inu[q] ? l[q] : 0.0f;
      }
    }
    // e of output j = u_{j-1} - u_j
    if (FROM_H) {  // j = column + 1
      const float hn = __shfl_down_sync(kFull, h[0], 1), ln = __shfl_down_sync(kFull, l[0], 1);
      const float hq[5] = {h[0], h[1], h[2], h[3], hn}, lq[5] = {l[0], l[1], l[2], l[3], ln};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        e[q] = hq[q] - hq[q + 1];
        l[q] = lq[q] - lq[q + 1];
      }
    } else {  // j = column
      const float hp = __shfl_up_sync(kFull, h[3], 1), lp = __shfl_up_sync(kFull, l[3], 1);
      const float hq[5] = {hp, h[0], h[1], h[2], h[3]}, lq[5] = {lp, l[0], l[1], l[2], l[3]};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        e[q] = hq[q] - hq[q + 1];
        l[q] = lq[q] - lq[q + 1];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (EDGE) {
        e[q] = ine[q] ? e[q] : 0.0f;
        l[q] = ine[q] ? l[q] : 0.0f;
      }
      d[q] = e[q] + l[q];
    }
    float t = fmaf(kRhoF, fmaf(kRhoF, fmaf(kRhoF, d[0], d[1]), d[2]), d[3]);
    float c1 = __shfl_up_sync(kFull, t, 1), c2 = __shfl_up_sync(kFull, t, 2);
    if (EDGE) {
      c1 = lane < 1 ? 0.0f : c1;
      c2 = lane < 2 ? 0.0f : c2;
    }
    float c = fmaf(kR4, c2, c1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      l[q] = fmaf(kRhoF, c, l[q]);
      c = d[q] = e[q] + l[q];
    }
    t = fmaf(kRhoF, fmaf(kRhoF, fmaf(kRhoF, d[3], d[2]), d[1]), d[0]);
    c1 = __shfl_down_sync(kFull, t, 1);
    c2 = __shfl_down_sync(kFull, t, 2);
    if (EDGE) {
      c1 = lane > 30 ? 0.0f : c1;
      c2 = lane > 29 ? 0.0f : c2;
    }
    c = fmaf(kR4, c2, c1);
    float n[4];  // y less e
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      n[q] = fmaf(kRhoF, c, l[q]);
      c = y[q] = e[q] + n[q];
    }
    if (EDGE) {
      auto pick = [&](const float(&v)[4], int e) { return e == 0 ? v[0] : (e == 1 ? v[1] : (e == 2 ? v[2] : v[3])); };
      // c += (k + kl) (w + wl), w + wl = output 0 (or M) of the infinite line
      auto end = [&](const float(&k)[4], const float(&kl)[4], float(&c)[4], int lane0, int el0) {
        const float pe = pick(e, el0), pn = pick(n, el0);
        const float w = pe + pn;
        const float wh = __shfl_sync(kFull, w, lane0), wl = __shfl_sync(kFull, pn - (w - pe), lane0);
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = fmaf(k[q], wh, fmaf(kl[q], wh, fmaf(k[q], wl, c[q])));
      };
      float c4[4] = {n[0], n[1], n[2], n[3]};
      if (left) end(kl, kll, c4, ll, el);
      if (right) end(kr, krl, c4, lr, er);
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = e[q] + c4[q];
    }
    if (out) *reinterpret_cast<float4*>(bp) = make_float4(y[0], y[1], y[2], y[3]);  // (pads: never read unmasked)
  }
}

template <bool FROM_H>
__device__ __forceinline__ void xt_item(const XTArgs& A, float4* ring, int item) {
  if (item >= A.nstrip * A.nblk) return;
  const int blk = item / A.nstrip, strip = item - blk * A.nstrip;
  if (strip == 0 || A.M <= TOUT * strip - THALO + 128) xt_block<FROM_H, true>(A, ring, strip, blk);
  else xt_block<FROM_H, false>(A, ring, strip, blk);
}

template <bool FROM_H>
__global__ void __launch_bounds__(32 * WPB) k_walk_dT(const __grid_constant__ YTArgs Y, const __grid_constant__ XTArgs X,
                                                      int nyb) {
  __shared__ float4 ring[WPB][2 * kRing * 32];
  pdl_wait();
  const int w = threadIdx.x >> 5, b = blockIdx.x;
  if (b < nyb) yt_item(Y, b * WPB + w);
  else xt_item<FROM_H>(X, ring[w], (b - nyb) * WPB + w);
}

// ---- filter and update ---------------------------------------------------------------------

// l (hi, lo) += s (12 beta y + L y) at the unknowns of a field, y = px + py there (E_z; the H fields have one of
// them), 0 on Dirichlet walls, mirrored across Neumann ones.  Bound by memory: a lane takes four columns of a row.
// rho of the recurrences is an FP32 number, off by d = 1.1e-9, which multiplies a derivative's symbol along its line
// by 1 + kRhoErr L to first order (its gain at theta = 0 is exact); 12 beta y takes that back: without it the
// gradient after 2000 steps at 32^2 was off by 2.3e-6, 1.1e-6 of it rounding.
constexpr double kRho = -0.045548849896677730860604;  // -11 + sqrt(120)
constexpr double kRhoErr = ((double)kRhoF - kRho) * (1.0 + kRho) / ((1.0 - kRho) * (1.0 - kRho) * (1.0 - kRho));
struct FArgs {
  const float* px;  // derivative along x, at column m = 0 of row 0 (E_z, H_y)
  const float* py;  // along y (E_z, H_x)
  float* lh;
  float* ll;
  int ld, M, u0, u1;
  float c_hi, c_lo, s_hi, s_lo;  // 12 beta s, s
  float r;                       // -12 beta s kRhoErr
};
struct FArgs2 {
  FArgs f[2];
};
constexpr int FY = 8;
// F: the field (E_z has both parts, H_x the one along y, H_y the one along x).
template <int F>
__device__ __forceinline__ void filter_update4(const FArgs& A) {
  constexpr bool PX = F != HX, PY = F != HY;
  const int m0 = 4 * (blockIdx.x * 32 + threadIdx.x), j = A.u0 + blockIdx.y * FY + threadIdx.y;
  if (m0 >= A.M || j >= A.u1) return;
  const size_t ld = A.ld;
  const int M = A.M;
  // rows above and below: 0 beyond a Dirichlet wall, the row itself across a Neumann one
  constexpr bool neu_x = F == HY, neu_y = F == HX;
  const int ja = j > A.u0 ? j - 1 : j, jb = j + 1 < A.u1 ? j + 1 : j;
  const bool oka = j > A.u0 || neu_y, okb = j + 1 < A.u1 || neu_y;
  struct Row {
    float v[4];
  };
  auto row = [&](bool part, const float* p, int r, bool ok) {
    const float4 a = part && ok ? ld4(p + r * ld + m0) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    return Row{{a.x, a.y, a.z, a.w}};
  };
  auto one = [&](bool part, const float* p, int m) { return part ? p[j * ld + m] : 0.0f; };
  const Row x = row(PX, A.px, j, true), xa = row(PX, A.px, ja, oka), xb = row(PX, A.px, jb, okb);
  const Row z = row(PY, A.py, j, true), za = row(PY, A.py, ja, oka), zb = row(PY, A.py, jb, okb);
  auto sum = [&](float a, float b) { return PX && PY ? a + b : (PX ? a : b); };
  // columns beside the four, and those past the field
  const bool in0 = m0 > 0, in1 = m0 + 4 < M;
  const float xl = in0 ? one(PX, A.px, m0 - 1) : (neu_x ? x.v[0] : 0.0f), xr = in1 ? one(PX, A.px, m0 + 4) : 0.0f;
  const float zl = in0 ? one(PY, A.py, m0 - 1) : 0.0f, zr = in1 ? one(PY, A.py, m0 + 4) : 0.0f;
  float* ph = A.lh + j * ld + m0;
  float* pl = A.ll + j * ld + m0;
  const float4 H = ld4(ph), L = ld4(pl);
  float h[4] = {H.x, H.y, H.z, H.w}, lo[4] = {L.x, L.y, L.z, L.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (m0 + q >= M) continue;  // the pads keep their zeros
    const bool wall = m0 + q == M - 1;
    const float xq = x.v[q], zq = z.v[q], y = sum(xq, zq);
    const float lx = q ? x.v[q ? q - 1 : 0] : xl, lz = q ? z.v[q ? q - 1 : 0] : zl;
    const float rx = wall ? (neu_x ? xq : 0.0f) : (q < 3 ? x.v[q < 3 ? q + 1 : 0] : xr);
    const float rz = wall ? 0.0f : (q < 3 ? z.v[q < 3 ? q + 1 : 0] : zr);
    // an exact two-product of 12 beta s y; s L y, first differences, joins its error term
    const float ly = (sum(xa.v[q], za.v[q]) - y) + (sum(xb.v[q], zb.v[q]) - y);
    const float lap = ((sum(lx, lz) - y) + (sum(rx, rz) - y)) + ly;
    float along = PX ? (lx - xq) + (rx - xq) : ly;
    if (PX && PY) along += (za.v[q] - zq) + (zb.v[q] - zq);
    const float p = __fmul_rn(A.c_hi, y);
    float e = fmaf(A.c_hi, y, -p);
    e = fmaf(A.c_lo, y, e);
    if (PX && PY) {  // what px + py rounds away
      const float yb = __fsub_rn(y, xq);
      e = fmaf(A.c_hi, __fadd_rn(__fsub_rn(xq, __fsub_rn(y, yb)), __fsub_rn(zq, yb)), e);
    }
    e = fmaf(A.s_hi, lap, fmaf(A.s_lo, lap, fmaf(A.r, along, e)));
    const float u = __fadd_rn(h[q], p);
    const float bb = __fsub_rn(u, h[q]);
    const float err = __fadd_rn(__fsub_rn(h[q], __fsub_rn(u, bb)), __fsub_rn(p, bb));
    const float l2 = __fadd_rn(lo[q], __fadd_rn(err, e));
    const float h2 = __fadd_rn(u, l2);
    lo[q] = __fsub_rn(l2, __fsub_rn(h2, u));
    h[q] = h2;
  }
  *reinterpret_cast<float4*>(ph) = make_float4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<float4*>(pl) = make_float4(lo[0], lo[1], lo[2], lo[3]);
}

template <bool OF_H>
__global__ void __launch_bounds__(32 * FY) k_filter_update(const __grid_constant__ FArgs2 A) {
  pdl_wait();
  if (!OF_H) filter_update4<EZ>(A.f[0]);
  else if (blockIdx.z == 0) filter_update4<HX>(A.f[0]);
  else filter_update4<HY>(A.f[1]);
}

// ---- host ----------------------------------------------------------------------------------

int blocks_of(int items) { return (items + WPB - 1) / WPB; }

// The end correction of the transposed derivative: v = y + t (y_0) with t the vector of the closure's
// A^{-T} (LineEnds), t_{-1} = -rho, so k_j = (t_{j-1} - t_j) / (rho - 1) on w_0 = (rho - 1) y_0.
void end_rows_T(int closure, int kind, float* k, float* kl) {
  LineEnds e;
  line_ends(closure, kind, true, &e);
  const double rho = (double)kRhoF;
  double prev = -rho;
  for (int j = 0; j < kEndT; ++j) {
    const double t = j < kRecWarm ? e.v[j] : 0.0;
    const Split p = split((prev - t) / (rho - 1.0));
    k[j] = p.hi;
    kl[j] = p.lo;
    prev = t;
  }
}

// H (from_h: solutions of H_x and H_y into the E_z planes) or E_z (into the H_x and H_y planes).
void derivatives_T(ms_grid* g, bool from_h) {
  Adj32* A = g->adj32;
  const int N = g->N;
  const int kind = from_h ? NODE_TO_HALF : HALF_TO_NODE;
  YTArgs y{};
  XTArgs x{};
  const int ys = from_h ? HX : EZ, yd = from_h ? EZ : HX, xs = from_h ? HY : EZ, xd = from_h ? EZ : HY;
  y.ld = x.ld = g->ld32;
  y.M = x.M = from_h ? N : N - 1;
  const size_t row1 = from_h ? 0 : y.ld;  // E_z: u_0 at row 1
  y.uh = A->lh[ys] + row1;
  y.ul = A->uc[ys] + row1;
  y.b = A->py[yd];
  y.ncol = N + 1;
  end_rows_T(g->desc.closure, kind, y.k, y.kl);
  for (int j = 0; j < kEndT; ++j) {
    x.k[j] = y.k[j];
    x.kl[j] = y.kl[j];
  }
  y.nstrip = (N - 1 + 31) / 32;
  const int R = y.M + 1;
  const int rows = y.nstrip * (R / 64) >= 1500 ? 64 : 32;
  y.end = R >= 4 * rows ? rows : 16;
  const int mid = R - 2 * y.end;
  const int K = mid > 0 ? (mid + rows - 1) / rows : 0;
  y.chunk = K ? ((mid + K - 1) / K + 7) / 8 * 8 : 8;
  y.nseg = 2 + (mid > 0 ? (mid + y.chunk - 1) / y.chunk : 0);
  x.from_h = from_h;
  x.uh = A->lh[xs] + (from_h ? 0 : 1);
  x.ul = A->uc[xs] + (from_h ? 0 : 1);
  x.b = A->px[xd] + (from_h ? 1 : 0);
  x.nrows = N - 1;
  const int Mo = from_h ? N - 1 : N;
  x.nstrip = (Mo + TOUT - 1) / TOUT;
  const int br = x.nstrip * (N / 8) < 1216 ? 4 : 8;
  x.nblk = (x.nrows + br - 1) / br;
  x.rows = (x.nrows + x.nblk - 1) / x.nblk;
  const int nyb = blocks_of(y.nstrip * y.nseg);
  const dim3 grd(nyb + blocks_of(x.nstrip * x.nblk)), blk(32 * WPB);
  if (from_h) launch_pdl(k_walk_dT<true>, grd, blk, 0, g->stream, y, x, nyb);
  else launch_pdl(k_walk_dT<false>, grd, blk, 0, g->stream, y, x, nyb);
}

// The solve's polynomial p about t = 36, where the smoothest fields sit: p(t) = gain (1 + q (t - 36) r(t)), with r in
// the Horner form of the levels, coefficients r[l] of level l + 1.
struct PairPoly {
  double gain, q, r[kChebMax];
};
PairPoly pair_poly(const Cheb& c) {
  long double p[kChebMax + 1] = {c.p0}, gain = 0.0L, h = 0.0L;
  for (int k = 1; k < c.m; ++k) p[k] = p[k - 1] * (long double)c.q[k];
  for (int k = c.m - 1; k >= 0; --k) gain = 36.0L * gain + p[k];
  PairPoly out{};
  out.gain = (double)gain;
  // 1 - p / gain = (36 - t) h(t), q r = h, by synthetic division from the constant term
  for (int k = 0; k < c.m - 1; ++k) {
    const long double n = ((k ? 0.0L : 1.0L) - p[k] / gain + h) / 36.0L;
    if (k == 0) out.q = (double)n;
    else out.r[c.m - 2 - k] = (double)(n / h);
    h = n;
  }
  return out;
}

// u = P~^{-1} l over the gain of its polynomial for the H fields or E_z: uc.
void solve_pair(ms_grid* g, bool of_h) {
  Adj32* A = g->adj32;
  SArgs a[2];
  int nb[2] = {0, 0};
  const int nf = of_h ? 2 : 1;
  const PairPoly poly = pair_poly(g->walk.cheb);
  for (int k = 0; k < nf; ++k) {
    const int f = of_h ? (k ? HY : HX) : EZ, mc = f == HY ? 0 : 1;
    a[k] = make_s(g, f, A->lh[f], nullptr, nf);
    a[k].hi = nullptr;
    const Split q = split(poly.q);
    a[k].l_hi = q.hi;
    a[k].l_lo = q.lo;
    for (int l = 0; l < g->walk.cheb.m - 2; ++l) a[k].q[l] = (float)poly.r[l];
    a[k].lo = A->ll[f] + mc;
    a[k].out = A->uc[f] + mc;
    nb[k] = blocks_of(a[k].nstrip * a[k].nblk);
  }
  if (nf == 1) a[1] = a[0];
  const dim3 grd(nb[0] + nb[1]), blk(32 * WPB);
  const int P = g->walk.cheb.m - 1;
  if (P == 2) launch_pdl(k_solve_pair<2>, grd, blk, 0, g->stream, a[0], a[1], nb[0]);
  else if (P == 3) launch_pdl(k_solve_pair<3>, grd, blk, 0, g->stream, a[0], a[1], nb[0]);
  else launch_pdl(k_solve_pair<4>, grd, blk, 0, g->stream, a[0], a[1], nb[0]);
}

FArgs filter_args(ms_grid* g, int f) {
  Adj32* A = g->adj32;
  const int N = g->N, mc = f == HY ? 0 : 1;
  FArgs a{};
  a.px = f == HX ? nullptr : A->px[f] + mc;
  a.py = f == HY ? nullptr : A->py[f] + mc;
  a.lh = A->lh[f] + mc;
  a.ll = A->ll[f] + mc;
  a.ld = g->ld32;
  a.M = f == HY ? N : N - 1;
  a.u0 = f == HX ? 0 : 1;
  a.u1 = N;
  const double sc = (f == EZ ? 12.0 / (g->desc.r * g->Z) : 12.0 * g->Z / g->desc.r) * pair_poly(g->walk.cheb).gain *
                    walk_rhs_scale();
  const double c = 12.0 * g->beta * sc;
  const Split cp = split(c), sp = split(sc);
  a.c_hi = cp.hi;
  a.c_lo = cp.lo;
  a.s_hi = sp.hi;
  a.s_lo = sp.lo;
  a.r = (float)(-c * kRhoErr);
  return a;
}

void filter_update(ms_grid* g, bool of_h) {
  FArgs2 A;
  A.f[0] = filter_args(g, of_h ? HX : EZ);
  A.f[1] = filter_args(g, of_h ? HY : EZ);
  const dim3 grd((g->N + 127) / 128, (g->N + FY - 1) / FY, of_h ? 2 : 1), blk(32, FY);
  if (of_h) launch_pdl(k_filter_update<true>, grd, blk, 0, g->stream, A);
  else launch_pdl(k_filter_update<false>, grd, blk, 0, g->stream, A);
}

// One transposed step on the float-float adjoint state.
void adjoint_step32(ms_grid* g) {
  solve_pair(g, true);       // S2^T: u_H = P~^{-1} l_H; y_E = Y_x^T u_Hy - Y_y^T u_Hx; l_E += sH F~ y_E
  derivatives_T(g, true);
  filter_update(g, false);
  solve_pair(g, false);      // S1^T: u_E = P~^{-1} l_E; y_Hy = Y_x^T u_E, y_Hx = -Y_y^T u_E; l_H += sE F~ y_H
  derivatives_T(g, false);
  filter_update(g, true);
}

ms_status capture32(ms_grid* g, Graph* gr, int steps) {
  if (gr->exec) return MS_OK;
  if (cudaStreamBeginCapture(g->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
    return a32fail(MS_ECUDA, "cudaStreamBeginCapture failed");
  for (int q = 0; q < steps; ++q) adjoint_step32(g);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(g->stream, &graph);
  if (e != cudaSuccess) return a32fail(MS_ECUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(e));
  e = cudaGraphInstantiate(&gr->exec, graph, 0);
  if (e != cudaSuccess) {
    cudaGraphDestroy(graph);
    return a32fail(MS_ECUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e));
  }
  gr->graph = graph;
  gr->steps = steps;
  return MS_OK;
}

}  // namespace

ms_status adjoint32_setup(ms_grid* g) {
  if (g->adj32) return MS_OK;
  Adj32* A = new Adj32();
  g->adj32 = A;
  const size_t pl = plane_floats(g->N);
  constexpr int kPlanes = 13;
  if (dev_malloc(&A->slab, kPlanes * pl * sizeof(float)) != cudaSuccess) {
    adjoint32_teardown(g);
    return a32fail(MS_ENOMEM, "cudaMalloc of the FP32 adjoint planes failed");
  }
  if (cudaMemsetAsync(A->slab, 0, kPlanes * pl * sizeof(float), g->stream) != cudaSuccess) {
    adjoint32_teardown(g);
    return a32fail(MS_ECUDA, "clearing the FP32 adjoint planes failed");
  }
  float* next = A->slab;
  auto plane = [&](int f) {
    float* p = next + plane_origin(f);
    next += pl;
    return p;
  };
  for (int f = 0; f < 3; ++f) {
    A->lh[f] = plane(f);
    A->ll[f] = plane(f);
    A->uc[f] = plane(f);
  }
  A->py[EZ] = plane(EZ);
  A->px[EZ] = plane(EZ);
  A->py[HX] = plane(HX);
  A->px[HY] = plane(HY);
  return MS_OK;
}

void adjoint32_teardown(ms_grid* g) {
  Adj32* A = g->adj32;
  if (!A) return;
  free_graph32(&A->g1);
  free_graph32(&A->gk);
  dev_free(A->slab);
  delete A;
  g->adj32 = nullptr;
}

// The adjoint state from / to FP64 arrays (device), three fields.
void adjoint32_load(ms_grid* g, const double* const* l) {
  for (int f = 0; f < 3; ++f) launch_split2d(l[f], g->adj32->lh[f], g->adj32->ll[f], g->ld32, g->sh[f], g->stream);
}
void adjoint32_store(ms_grid* g, double* const* l) {
  for (int f = 0; f < 3; ++f) launch_join2d(g->adj32->lh[f], g->adj32->ll[f], g->ld32, l[f], g->sh[f], g->stream);
}

// (M^T)^nsteps on the float-float adjoint state, replaying captured chunks of 16 steps.
ms_status adjoint32_steps(ms_grid* g, long nsteps) {
  Adj32* A = g->adj32;
  const int chunk = 16;
  if (nsteps >= chunk) {
    ms_status s = capture32(g, &A->gk, chunk);
    if (s != MS_OK) return s;
  }
  if (nsteps % chunk) {
    ms_status s = capture32(g, &A->g1, 1);
    if (s != MS_OK) return s;
  }
  long left = nsteps;
  for (; left >= chunk; left -= chunk)
    if (cudaGraphLaunch(A->gk.exec, g->stream) != cudaSuccess) return a32fail(MS_ECUDA, "cudaGraphLaunch failed");
  for (; left > 0; --left)
    if (cudaGraphLaunch(A->g1.exec, g->stream) != cudaSuccess) return a32fail(MS_ECUDA, "cudaGraphLaunch failed");
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return a32fail(MS_ECUDA, std::string("FP32 adjoint steps: ") + cudaGetErrorString(e));
  return MS_OK;
}

}  // namespace ms
