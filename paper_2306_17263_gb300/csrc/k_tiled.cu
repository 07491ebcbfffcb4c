// FP32_REFINED step of 2D grids.  Two launches per half-step, both made of warps that walk along y with
// everything they carry in registers and the rows ahead in a ring in shared memory of each warp's own: no barriers.
//
//   walk_d : the Pade derivatives (App. A.1, Eq. "eq:lhs") of the filtered source into right-hand-side
//            planes, one plane per axis.  Along y a lane takes one column (30 of 32 lanes write, the
//            outer two hold the neighbour columns of the filter) and walks down its segment of the line.
//            Along x a lane takes four adjacent columns of a row (a warp 128, of which it writes 112)
//            and walks down a block of rows, carrying the differences of the rows above and below.
//   walk_s : the solve of P1 (Def. "def:operatorsP") and the float-float update E += h_tau E* /
//            H += h_tau H*.  A lane takes four adjacent columns (a warp 128, of which it writes 120)
//            and walks down a block of rows; the levels of the solve follow one another a row apart,
//            so no iterate is stored and the state is read and written once.
//
// Differences are taken on the float-float state, delta_m = (hi_{m+1} - hi_m) + (lo_{m+1} - lo_m), and
// filtered, d = 12 beta delta + L delta (the filter of Eq. "eq:ell" commutes with the difference: D1
// (12 beta + L) u = (12 beta + L') D1 u with the ghost rules below); L delta, the sum of the four neighbours less 4
// delta, is formed on its own, small as it is, before the low part of 12 beta joins it: that part is about an ulp of
// the neighbours' sum and would be rounded the same way everywhere (1e-9 of the filter at r = 0.68).  A^{-1} d is the two first-order
// recurrences A factors into, z_i = d_i + rho z_{i-1} and y_i = z_i + rho y_{i+1}, up to the factor (1 -
// rho)^2 that the increment scales carry, each z and y rounded once.  Along y the forward one follows the
// walk and the backward one runs over groups of eight rows from seven rows beyond (|rho|^8 = 2e-11);
// along x a lane runs both over its four columns and takes the carries of two lanes on either side.  The closure's
// end rows change the solution by a multiple of the decaying vector rho^i (LineEnds) in the first and the last
// eight rows of a line (end_rows).
//
// Ghost rules of the difference along a line: a source that is Neumann along it (H_y along x, H_x along
// y; even ghost u(-1) = u(0), Cor. "cor:ghost_cor") has zero differences beyond the ends; one that is
// Dirichlet (E_z, zero at the wall, filter zero there) even ones (delta_{-1} = delta_0).  Across the line
// every source is Dirichlet with stored zeros.
//
// The solve is the Chebyshev polynomial of k_rec64.cu, 6 h^2 P1 = D - T with T = (L_x + 6)(L_y + 6), in
// Horner form y <- b + q T y to a relative error of 1e-10: five operations per point and level.  T y is
// 36 / D of D y at most (7e-3 at r = 0.5, 2.2e-2 at the stability limit), so an FP32 level rounds the increment at
// 4e-10 to 1.3e-9 of itself, and the last level's q T y enters the state apart from b, never rounded into it.
//
// Why walks: both kernels of the tile form this replaces (64 x 64 tiles in shared memory) were bound by
// instruction issue, 140-150 warp instructions per 32 points and field.  Derivative along x and solve in
// one walk (no plane between them) was tried: 146 registers leave 12 warps per SM, and with a chain of
// eight shuffles per row it ran 66 us for E_z at 2048^2.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "k_fp64.cuh"
#include "k_pdl.cuh"
#include "k_rec64.cuh"
#include "k_tiled.cuh"
#include "k_walk_dev.cuh"

namespace ms {

// Arguments of a derivative along y: lines are the columns 1 .. ncol-2 of the source.
struct YArgs {
  const float* sh;  // source, point (0, 0)
  const float* sl;
  float* b;         // destination plane, row of output 0, column 0
  int ld, ncol, M, even;
  float cb_hi, cb_lo;  // 12 beta
  float g[4], gl[4], v[kEnd];  // end correction, g in pairs
  int nstrip, nseg, chunk, rb;  // column strips; segments of `chunk` rows, the last one [rb, M)
  // grids of at most kTinyN cells: explicit rows of A^{-1}, both derivatives of the half-step
  int tiny, step, N;
  const float *th[2], *tl[2];  // sources of the derivatives along x and y: Step 1 H_y, H_x; Step 2 E_z
  float* tb[2];                // destinations of those along y and x
  const float *whi, *wlo;
  int K;
  int filter;
};

// Arguments of a derivative along x; pointers at column m = 0 (the first unknown one) of row 0.
struct XArgs {
  const float* sh;  // source
  const float* sl;
  float* b;         // destination plane
  int ld, M;        // outputs 0 .. M-1 of every row
  int u0, u1;       // rows u0 .. u1-1
  float cb_hi, cb_lo;
  float g[4], gl[4], v[kEnd];
  int nstrip, nblk, rows;
};

namespace {

// ---- derivative along y --------------------------------------------------------------------------------

// One segment of 32 columns.  Rows m = r0 - 9 .. are pushed through the recurrences in groups of eight;
// the y of a group lags its last row by seven, so the first two groups only warm up.  EDGE: rows of the
// walk may lie beyond the line's ends.
template <bool FILTER, bool EDGE>
__device__ __forceinline__ void y_segment(const YArgs& A, int strip, int seg) {
  const int lane = threadIdx.x & 31;
  const int col = YOUT * strip + lane;
  const bool live = lane >= 1 && lane <= YOUT && col <= A.ncol - 2;
  const bool last = seg == A.nseg - 1;
  const int r0 = last ? A.rb : seg * A.chunk, r1 = last ? A.M : min(r0 + A.chunk, A.rb);
  const size_t ld = A.ld;
  const int cc = min(col, A.ncol - 1);
  const float* ph = A.sh + cc;
  const float* pl = A.sl + cc;
  auto row = [&](int r) { return EDGE ? (size_t)min(max(r, 0), A.M) * ld : (size_t)r * ld; };
  const int ms = r0 - 9;
  // u at rows ms - 1, ms, ms + 1 -> delta_{ms-1}, delta_ms
  float h1 = ph[row(ms + 1)], l1 = pl[row(ms + 1)];
  float dm, d0;
  {
    const float hm = ph[row(ms - 1)], lm = pl[row(ms - 1)], h0 = ph[row(ms)], l0 = pl[row(ms)];
    dm = (h0 - hm) + (l0 - lm);
    d0 = (h1 - h0) + (l1 - l0);
  }
  float z = 0.0f, zp[7] = {};  // z of the last row; of the seven rows before a group
  float nh[8], nl[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    nh[t] = ph[row(ms + 2 + t)];
    nl[t] = pl[row(ms + 2 + t)];
  }
  float* bp = A.b + (size_t)r0 * ld + col;
  const int ngrp = 2 + (r1 - r0 + 7) / 8;
  for (int gidx = 0; gidx < ngrp; ++gidx) {
    const int m0 = ms + 8 * gidx;
    float ch[8], cl[8], zc[8], y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      ch[t] = nh[t];
      cl[t] = nl[t];
    }
    if (gidx + 1 < ngrp) {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        nh[t] = ph[row(m0 + 10 + t)];
        nl[t] = pl[row(m0 + 10 + t)];
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int m = m0 + t;
      float dp = (ch[t] - h1) + (cl[t] - l1);  // delta_{m+1}
      h1 = ch[t];
      l1 = cl[t];
      float d;
      if (FILTER) {
        const float a = __shfl_up_sync(kFull, d0, 1), b = __shfl_down_sync(kFull, d0, 1);
        float um = dm, up = dp;
        if (EDGE && A.even) {
          um = m == 0 ? d0 : um;
          up = m == A.M - 1 ? d0 : up;
        }
        d = fmaf(A.cb_hi, d0, fmaf(A.cb_lo, d0, fmaf(-4.0f, d0, (a + b) + (um + up))));
      } else {
        d = d0;
      }
      if (EDGE) d = (m >= 0 && m < A.M) ? d : 0.0f;
      dm = d0;
      d0 = dp;
      z = fmaf(kRhoF, z, d);
      zc[t] = z;
    }
    // backward from the group's last row: seven rows of warm-up, then the rows r0 + 8 (gidx - 2) .. + 7
    float acc = zc[7];
#pragma unroll
    for (int t = 6; t >= 1; --t) acc = fmaf(kRhoF, acc, zc[t]);
    const float ynext = acc;  // of the row after the group
    y[7] = acc = fmaf(kRhoF, acc, zc[0]);
#pragma unroll
    for (int t = 6; t >= 0; --t) y[t] = acc = fmaf(kRhoF, acc, zp[t]);
    if (EDGE && gidx >= 2) {
      const float zr[8] = {zp[0], zp[1], zp[2], zp[3], zp[4], zp[5], zp[6], zc[0]};
      if (seg == 0 && gidx == 2) end_rows<false>(y, zr, ynext, end_phi(A, y[0], y[1], y[2], y[3]), A.v);
      if (last && gidx == ngrp - 1) end_rows<true>(y, zr, ynext, end_phi(A, y[7], y[6], y[5], y[4]), A.v);
    }
#pragma unroll
    for (int t = 0; t < 7; ++t) zp[t] = zc[t + 1];
    if (gidx < 2) continue;
    if (live) {
      const int left = r1 - (r0 + 8 * (gidx - 2));
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t < left) bp[(size_t)t * ld] = -y[t];
    }
    bp += 8 * ld;
  }
}

// Lines of at most 16 rows (grids of up to kTinyN cells): outputs from the explicit rows of A^{-1}.  A warp
// takes two lines of one axis, a lane one difference and one output; the differences of a line come from the
// lanes of its half.  A step is bound by the latency of its launches, so the lines go over as many warps as
// there are (8^2 and 16^2: 14 and 17 us per step; 49 and 212 with one warp for a whole half-step).
__device__ __forceinline__ void tiny_item(const YArgs& A, int item) {
  const int N = A.N, M = A.M, K = A.K, rs = 2 * K + 2, per = N / 2;  // items per axis
  if (item >= 2 * per) return;
  const int axis = item >= per, r = threadIdx.x & 15;  // axis 0: lines are rows of the source, 1 columns
  const int c = 1 + 2 * (item - axis * per) + ((threadIdx.x >> 4) & 1), cc = min(c, N - 1);
  const float *h = A.th[axis], *l = A.tl[axis];
  const size_t sm = axis == 0 ? 1 : A.ld, sc = axis == 0 ? A.ld : 1;
  auto delta = [&](int line) {
    const size_t p = line * sc + r * sm;
    return r < M ? (h[p + sm] - h[p]) + (l[p + sm] - l[p]) : 0.0f;
  };
  float d = delta(cc);
  if (A.filter) {
    const float x = d, up = delta(cc - 1), dn = delta(cc + 1);
    float a = __shfl_up_sync(kFull, x, 1, 16), b = __shfl_down_sync(kFull, x, 1, 16);
    if (r == 0) a = A.even ? x : 0.0f;
    if (r == M - 1) b = A.even ? x : 0.0f;
    const float lap = ((a - x) + (b - x)) + ((up - x) + (dn - x));
    d = fmaf(A.cb_hi, x, fmaf(A.cb_lo, x, lap));
  }
  // farthest taps first: added after the nearest ones, those beyond the sixth would round away in every sum
  const float *wh = A.whi + r * rs, *wl = A.wlo + r * rs;
  float hi = 0.0f, lo = 0.0f;
#pragma unroll 8
  for (int q = 2 * K + 1; q >= 0; --q) {
    const int m = r + ((q & 1) ? (q + 1) / 2 : -(q / 2)), t = m - r + K;
    const float x = __shfl_sync(kFull, d, m & 15, 16);
    if (r >= M || m < 0 || m >= M) continue;
    lo = fmaf(wl[t], x, lo);
    hi = fmaf(wh[t], x, q ? hi : hi + lo);
  }
  if (r >= M || c >= N) return;
  const int o = r + (A.step == 0);
  if (axis == 0) A.tb[1][(size_t)c * A.ld + o] = hi;
  else A.tb[0][(size_t)o * A.ld + c] = -hi;
}

template <bool FILTER>
__device__ __forceinline__ void y_item(const YArgs& A, int item) {
  if (A.tiny) {
    tiny_item(A, item);
    return;
  }
  if (item >= A.nstrip * A.nseg) return;
  const int seg = item / A.nstrip, strip = item - seg * A.nstrip;
  const int r0 = seg == A.nseg - 1 ? A.rb : seg * A.chunk;
  const int r1 = seg == A.nseg - 1 ? A.M : min(r0 + A.chunk, A.rb);
  // rows the walk touches: r0 - 10 .. the end of its last group and of the next one's loads
  if (r0 >= 10 && r1 + 18 <= A.M) y_segment<FILTER, false>(A, strip, seg);
  else y_segment<FILTER, true>(A, strip, seg);
}

// ---- derivative along x --------------------------------------------------------------------

// One block of rows of one 128-column strip.  SE: the source is E_z (delta_m ends at its column m, even
// beyond the ends).  EDGE: the strip sees an end of the lines; lanes beyond it hold zeros.
template <bool SE, bool FILTER, bool EDGE>
__device__ __forceinline__ void x_block(const XArgs& A, float4* ring, int strip, int blk) {
  const int lane = threadIdx.x & 31;
  const int m_s = XOUT * strip - XHALO, m0 = m_s + 4 * lane;
  const int M = A.M;
  const int j0 = A.u0 + blk * A.rows, j1 = min(j0 + A.rows, A.u1);
  const size_t ld = A.ld;
  const bool ok = !EDGE || (m0 >= -4 && m0 + 8 <= A.ld);  // the lane's columns lie in the row
  const bool out = lane >= XHALO / 4 && lane < (XHALO + XOUT) / 4 && (!EDGE || (m0 < M && m0 >= 0));
  const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  auto load = [&](const float* p, int row) { return ok ? ld4(p + (size_t)row * ld + m0) : zero4; };
  // edge strips: masks, and the end corrections' coefficients at the lane's columns
  bool in[4] = {true, true, true, true}, first[4] = {}, lastc[4] = {};
  float vl[4] = {}, vr[4] = {}, gr[4] = {}, grl[4] = {};
  int la = 0, lb = 0;
  bool right = false;
  if (EDGE) {
    right = M - 1 <= m_s + 127;
    la = (M - 1 - m_s) >> 2;
    lb = (M - 4 - m_s) >> 2;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int m = m0 + k, e = M - 1 - m;
      in[k] = m >= 0 && m < M;
      first[k] = m == 0;
      lastc[k] = e == 0;
      vl[k] = (strip == 0 && m >= 0 && m < kEnd) ? A.v[m & 7] : 0.0f;
      vr[k] = (right && e >= 0 && e < kEnd) ? A.v[e & 7] : 0.0f;
      gr[k] = (right && e >= 0 && e < 4) ? A.g[e & 3] : 0.0f;
      grl[k] = (right && e >= 0 && e < 4) ? A.gl[e & 3] : 0.0f;
    }
  }
  // differences of one source row
  auto diff = [&](const float4& h, const float4& l, float(&d)[4]) {
    if (SE) {
      const float hp = __shfl_up_sync(kFull, h.w, 1), lp = __shfl_up_sync(kFull, l.w, 1);
      d[0] = (h.x - hp) + (l.x - lp);
      d[1] = (h.y - h.x) + (l.y - l.x);
      d[2] = (h.z - h.y) + (l.z - l.y);
      d[3] = (h.w - h.z) + (l.w - l.z);
    } else {
      const float hn = __shfl_down_sync(kFull, h.x, 1), ln = __shfl_down_sync(kFull, l.x, 1);
      d[0] = (h.y - h.x) + (l.y - l.x);
      d[1] = (h.z - h.y) + (l.z - l.y);
      d[2] = (h.w - h.z) + (l.w - l.z);
      d[3] = (hn - h.w) + (ln - l.w);
    }
  };
  // ring: [slot][hi, lo of row jj + 1][lane]
  const size_t off = ok ? m0 : 0;
  const float* fh = A.sh + (size_t)(j0 + 1) * ld + off;
  const float* fl = A.sl + (size_t)(j0 + 1) * ld + off;
  int left = j1 - j0;  // rows to fetch (the last is row j1 <= u1)
  auto fetch = [&](int slot) {
    if (left > 0) {
      cp16(ring + (2 * slot) * 32 + lane, fh, ok);
      cp16(ring + (2 * slot + 1) * 32 + lane, fl, ok);
    }
    cp_commit();
    fh += ld;
    fl += ld;
    --left;
  };
#pragma unroll
  for (int t = 0; t < kAhead; ++t) fetch(t);
  float dm[4], d0[4];
  {
    const float4 ah = load(A.sh, j0 - 1), al = load(A.sl, j0 - 1), bh = load(A.sh, j0), bl = load(A.sl, j0);
    diff(ah, al, dm);
    diff(bh, bl, d0);
  }
  const float2 cb_hi = bc2(A.cb_hi), cb_lo = bc2(A.cb_lo);
  float* bp = A.b + (size_t)j0 * ld + m0;
  int rd = 0, wr = kAhead;  // slots of rows jj + 1 and jj + 1 + kAhead
  for (int jj = j0; jj < j1; ++jj, bp += ld) {
    float dp[4], d[4], y[4];
    cp_wait<kAhead - 1>();
    const float4 ch = ring[(2 * rd) * 32 + lane], cl = ring[(2 * rd + 1) * 32 + lane];
    fetch(wr);
    rd = rd == kRing - 1 ? 0 : rd + 1;
    wr = wr == kRing - 1 ? 0 : wr + 1;
    diff(ch, cl, dp);
    if (FILTER) {
      const float a = __shfl_up_sync(kFull, d0[3], 1), e = __shfl_down_sync(kFull, d0[0], 1);
      float l[4] = {a, d0[0], d0[1], d0[2]}, r[4] = {d0[1], d0[2], d0[3], e};
      if (EDGE) {  // zero differences beyond the ends of a Neumann source, even ones of E_z
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          l[k] = first[k] ? (SE ? d0[k] : 0.0f) : l[k];
          r[k] = lastc[k] ? (SE ? d0[k] : 0.0f) : r[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 4; k += 2) {
        const float2 x = make_float2(d0[k], d0[k + 1]);
        const float2 nb = add2(make_float2(l[k] + r[k], l[k + 1] + r[k + 1]),
                               add2(make_float2(dm[k], dm[k + 1]), make_float2(dp[k], dp[k + 1])));
        const float2 v = fma2(cb_hi, x, fma2(cb_lo, x, fma2(bc2(-4.0f), x, nb)));
        d[k] = v.x;
        d[k + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) d[k] = d0[k];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (EDGE) d[k] = in[k] ? d[k] : 0.0f;
      dm[k] = d0[k];
      d0[k] = dp[k];
    }
    // forward: the carry of the two lanes before (eight terms) from their local chains, then the chain with
    // it, so that every z is rounded once at its own size; backward the same
    float t = fmaf(kRhoF, fmaf(kRhoF, fmaf(kRhoF, d[0], d[1]), d[2]), d[3]);
    float c1 = __shfl_up_sync(kFull, t, 1), c2 = __shfl_up_sync(kFull, t, 2);
    if (EDGE) {
      c1 = lane < 1 ? 0.0f : c1;
      c2 = lane < 2 ? 0.0f : c2;
    }
    float c = fmaf(kR4, c2, c1);
#pragma unroll
    for (int k = 0; k < 4; ++k) c = d[k] = fmaf(kRhoF, c, d[k]);
    t = fmaf(kRhoF, fmaf(kRhoF, fmaf(kRhoF, d[3], d[2]), d[1]), d[0]);
    c1 = __shfl_down_sync(kFull, t, 1);
    c2 = __shfl_down_sync(kFull, t, 2);
    if (EDGE) {
      c1 = lane > 30 ? 0.0f : c1;
      c2 = lane > 29 ? 0.0f : c2;
    }
    c = fmaf(kR4, c2, c1);
    const float ynext = c;
#pragma unroll
    for (int k = 3; k >= 0; --k) c = y[k] = fmaf(kRhoF, c, d[k]);
    if (EDGE) {  // as end_rows
      float n[4] = {kRhoF * y[1], kRhoF * y[2], kRhoF * y[3], kRhoF * ynext};
      if (strip == 0) {  // columns 0 .. 3 are lane 2's
        const float phi = __shfl_sync(kFull, end_phi(A, y[0], y[1], y[2], y[3]), XHALO / 4);
#pragma unroll
        for (int k = 0; k < 4; ++k) n[k] = fmaf(vl[k], phi, n[k]);
      }
      if (right) {
        const float lo = fmaf(grl[0], y[0], fmaf(grl[1], y[1], fmaf(grl[2], y[2], grl[3] * y[3])));
        const float part = fmaf(gr[0], y[0], fmaf(gr[1], y[1], fmaf(gr[2], y[2], fmaf(gr[3], y[3], lo))));
        const float pa = __shfl_sync(kFull, part, la), pb = __shfl_sync(kFull, part, lb);
        const float phi = la == lb ? pa : pa + pb;
#pragma unroll
        for (int k = 0; k < 4; ++k) n[k] = fmaf(vr[k], phi, n[k]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) y[k] = d[k] + n[k];
    }
    if (out) *reinterpret_cast<float4*>(bp) = make_float4(y[0], y[1], y[2], y[3]);  // (pads: never read unmasked)
  }
}

template <bool SE, bool FILTER>
__device__ __forceinline__ void x_item(const XArgs& A, float4* ring, int item) {
  if (item >= A.nstrip * A.nblk) return;
  const int blk = item / A.nstrip, strip = item - blk * A.nstrip;
  if (strip == 0 || A.M - 1 <= XOUT * strip - XHALO + 127) x_block<SE, FILTER, true>(A, ring, strip, blk);
  else x_block<SE, FILTER, false>(A, ring, strip, blk);
}

// The two derivatives of a half-step: blocks [0, nyb) along y, the others along x.
template <bool SE, bool FILTER>
__global__ void __launch_bounds__(32 * WPB) k_walk_d(const __grid_constant__ YArgs Y, const __grid_constant__ XArgs X,
                                                     int nyb) {
  __shared__ float4 ring[WPB][2 * kRing * 32];
  pdl_wait();
  const int w = threadIdx.x >> 5, b = blockIdx.x;
  if (b < nyb) y_item<FILTER>(Y, b * WPB + w);
  else x_item<SE, FILTER>(X, ring[w], (b - nyb) * WPB + w);
}

// One or two fields: blocks [0, na) solve the first.
template <int P>
__global__ void __launch_bounds__(32 * WPB, P <= 3 ? 5 : 4) k_walk_s(const __grid_constant__ SArgs A, const __grid_constant__ SArgs B,
                                                     int na) {
  __shared__ float4 ring[WPB][4 * kRing * 32];
  pdl_wait();
  const int w = threadIdx.x >> 5, b = blockIdx.x;
  if (b < na) s_item<P>(A, ring[w], b * WPB + w);
  else s_item<P>(B, ring[w], (b - na) * WPB + w);
}

// ---- batches -------------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ void copy_args(T* dst, const T* src) {
  static_assert(sizeof(T) % 4 == 0, "argument structs are made of 4-byte words");
  const int* s = reinterpret_cast<const int*>(src);
  int* d = reinterpret_cast<int*>(dst);
  for (int k = threadIdx.x; k < (int)(sizeof(T) / 4); k += 32 * WPB) d[k] = s[k];
  __syncthreads();
}

// Entry e of a work list: argument work[2 e], its items work[2 e + 1] .. + WPB - 1 on the warps of a block.
// Derivatives: arguments below ny are walks along y, the others along x (ny is that of both half-steps'
// lists).
template <bool SE>
__global__ void __launch_bounds__(32 * WPB) k_batch_d(const YArgs* __restrict__ ya, const XArgs* __restrict__ xa, int ny,
                                                      const int* __restrict__ work, int n) {
  __shared__ union {
    YArgs y;
    XArgs x;
  } sA;
  __shared__ float4 ring[WPB][2 * kRing * 32];
  pdl_wait();
  for (int e = blockIdx.x; e < n; e += gridDim.x) {
    const int arg = work[2 * e], item = work[2 * e + 1] + (threadIdx.x >> 5);
    if (arg < ny) {
      copy_args(&sA.y, ya + arg);
      y_item<true>(sA.y, item);
    } else {
      copy_args(&sA.x, xa + (arg - ny));
      x_item<SE, true>(sA.x, ring[threadIdx.x >> 5], item);
    }
    __syncthreads();
  }
}

template <int P>
__global__ void __launch_bounds__(32 * WPB, P <= 3 ? 5 : 4) k_batch_s(const SArgs* __restrict__ args, const int* __restrict__ work, int n) {
  __shared__ SArgs sA;
  __shared__ float4 ring[WPB][4 * kRing * 32];
  pdl_wait();
  for (int e = blockIdx.x; e < n; e += gridDim.x) {
    copy_args(&sA, args + work[2 * e]);
    s_item<P>(sA, ring[threadIdx.x >> 5], work[2 * e + 1] + (threadIdx.x >> 5));
    __syncthreads();
  }
}

// ---- host ----------------------------------------------------------------------------------

YArgs make_y(const ms_grid* g, int step, float* plane0, float* plane1, const float* src_hi, const float* src_lo) {
  YArgs a{};
  const int N = g->N;
  const int src = step == 0 ? HX : EZ;
  const int kind = step == 0 ? HALF_TO_NODE : NODE_TO_HALF;
  a.sh = src_hi ? src_hi : g->hi[src];
  a.sl = src_hi ? src_lo : g->lo[src];
  a.ld = g->ld32;
  a.b = plane0 + (step == 0 ? a.ld : 0);  // output r at row r + 1 (E_z), r (H_x)
  a.ncol = N + 1;
  a.M = step == 0 ? N - 1 : N;
  a.even = step == 1;
  const Split c = split(12.0 * g->beta);
  a.cb_hi = c.hi;
  a.cb_lo = c.lo;
  set_ends(g->walk.ends[kind], &a);
  a.nstrip = (N - 1 + YOUT - 1) / YOUT;
  // Rows per segment: 16 more warm up its recurrences, so long segments do less work, but a grid wants
  // about ten warps per SM, and small grids short walks.  Steps with 16, 32 and 64 rows, us: 256^2 17.5, 19.4, 22.8;
  // 512^2 22.6, 23.5, 26.8; 777^2 28.4, 28.8, 31.2; 1024^2 34.0, 33.3, 36.0; 1536^2 56.9, 55.1, 55.0; 2048^2 86.9,
  // 82.8, 81.4.  The choice depends on N alone: a cavity of a batch takes the segments of a single grid, and with
  // them its rounding.
  line_segments(a.M, a.nstrip * (a.M / 64) >= 1500 ? 64 : (N > 320 ? 32 : 16), &a.nseg, &a.chunk, &a.rb);
  a.tiny = N <= kTinyN;
  a.step = step;
  a.N = N;
  if (a.tiny) {
    a.th[0] = step == 0 ? g->hi[HY] : a.sh;
    a.tl[0] = step == 0 ? g->lo[HY] : a.sl;
    a.th[1] = a.sh;
    a.tl[1] = a.sl;
    a.tb[0] = plane0;
    a.tb[1] = plane1;
    a.whi = g->pade32[kind].d_whi;
    a.wlo = g->pade32[kind].d_wlo;
    a.K = g->pade32[kind].K;
    a.nstrip = 1;
    a.nseg = 2 * (N / 2);  // two lines of one axis per item
  }
  a.filter = src_hi == nullptr;
  return a;
}

// The derivative along x of a half-step: into E_z (step 0), H_y (step 1).
XArgs make_x(const ms_grid* g, int step, float* plane, const float* src_hi, const float* src_lo) {
  XArgs a{};
  const int N = g->N;
  const int ms = step == 0 ? 0 : 1, md = step == 0 ? 1 : 0;  // column of m = 0 in source and destination
  const int src = step == 0 ? HY : EZ;
  a.ld = g->ld32;
  a.sh = (src_hi ? src_hi : g->hi[src]) + ms;
  a.sl = (src_hi ? src_lo : g->lo[src]) + ms;
  a.b = plane ? plane + md : nullptr;
  a.M = step == 0 ? N - 1 : N;
  a.u0 = 1;
  a.u1 = N;
  const Split c = split(12.0 * g->beta);
  a.cb_hi = c.hi;
  a.cb_lo = c.lo;
  set_ends(g->walk.ends[step == 0 ? HALF_TO_NODE : NODE_TO_HALF], &a);
  a.nstrip = N <= kTinyN ? 0 : (a.M + XOUT - 1) / XOUT;
  // Rows per block, 4 and 8, us per step: 256^2 17.5, 18.0; 512^2 23.5, 22.8; 777^2 28.8, 29.2; 1024^2 33.0, 33.3;
  // 1280^2 44.4, 43.9; 2048^2 82.3, 81.3.
  const int rows = a.nstrip * (N / 8) < 1216 ? 4 : 8;
  a.nblk = (N - 1 + rows - 1) / rows;
  a.rows = (N - 1 + a.nblk - 1) / a.nblk;
  return a;
}

// Rows per block of a solve launch, warps(rows) in all: P rows above and below are computed twice, but a launch
// wants `most` warps, about thirteen per SM, and small ones are bound by the length of one walk.  Steps of one grid
// with 4, 8, 16 and 32 rows, us: 256^2 17.5, 20.7, 27.3, 40.8; 777^2 27.2, 28.8, 32.6, 42.9; 1024^2 36.2, 33.3, 36.8,
// 47.6; 1536^2 62.7, 57.2, 56.5, 65.9; 2048^2 99.3, 85.7, 84.1, 84.6, and 81.3 with 16 for E_z and 32 for H.  In a
// batch the next shorter blocks begin to pay at fewer warps, 1216: 64 cavities of 256 cells, 1536 warps for E_z with 32
// rows, take 137.8 us per step so and 140.6 with 16 (r = 0.65: 158.7, 163.9).
template <typename Warps>
int solve_rows(Warps warps, int most) {
  int rows = 32;
  while (rows > 8 && warps(rows) < most) rows /= 2;
  if (rows == 8 && warps(8) < 608) rows = 4;
  return rows;
}

}  // namespace

SArgs make_s(const ms_grid* g, int f, const float* p1, const float* p2, int nfields) {
  SArgs a{};
  const int N = g->N;
  const int mc = f == HY ? 0 : 1;  // column of m = 0
  a.ld = g->ld32;
  a.hi = g->hi[f] + mc;
  a.lo = g->lo[f] + mc;
  a.p1 = p1 + mc;
  a.p2 = p2 ? p2 + mc : nullptr;
  a.M = f == HY ? N : N - 1;
  a.u0 = f == HX ? 0 : 1;
  a.u1 = N;
  a.kind = f == EZ ? KIND_E : (f == HX ? KIND_HX : KIND_HY);
  const Cheb& p = g->walk.cheb;
  for (int l = 0; l < p.m - 2; ++l) a.q[l] = (float)p.q[p.m - 1 - l];
  const double s = (f == EZ ? 12.0 * g->Z / g->desc.r : 12.0 / (g->desc.r * g->Z)) * p.p0 * plane_rhs_scale(g);
  const Split sp = split(s), lp = split(s * p.q[1]);
  a.s_hi = sp.hi;
  a.s_lo = sp.lo;
  a.l_hi = lp.hi;
  a.l_lo = lp.lo;
  a.nstrip = (a.M + SOUT - 1) / SOUT;
  const int nr = a.u1 - a.u0;
  const int rows = solve_rows([&](int q) { return nfields * a.nstrip * ((nr + q - 1) / q); }, 2000);
  a.nblk = (nr + rows - 1) / rows;
  a.rows = (nr + a.nblk - 1) / a.nblk;
  return a;
}

namespace {

int blocks_of(int items) { return (items + WPB - 1) / WPB; }

}  // namespace

void line_segments(int M, int rows, int* nseg, int* chunk, int* rb) {
  int K = (M + rows - 1) / rows;
  if (K < 2) K = 2;
  const int lastr = std::max(8, M / (8 * K) * 8);
  *rb = M - lastr;
  *chunk = std::max(8, ((*rb + K - 2) / (K - 1) + 7) / 8 * 8);
  *nseg = (*rb + *chunk - 1) / *chunk + 1;
}

double walk_rhs_scale() { return (1.0 - (double)kRhoF) * (1.0 - (double)kRhoF); }
double plane_rhs_scale(const ms_grid* g) { return g->N <= kTinyN ? 1.0 : walk_rhs_scale(); }

int walk_ld(int N) { return (N + 8 + 31) / 32 * 32; }
size_t plane_floats(int N) { return (size_t)(N + 1) * walk_ld(N) + 64; }
size_t plane_origin(int f) { return 32 + (f == HY ? 4 : 3); }

ms_status walk_setup(ms_grid* g) {
  g->ld32 = walk_ld(g->N);
  line_ends(g->desc.closure, HALF_TO_NODE, false, &g->walk.ends[HALF_TO_NODE]);
  line_ends(g->desc.closure, NODE_TO_HALF, false, &g->walk.ends[NODE_TO_HALF]);
  // D as in k_rec64.cu; at least two levels, at most four (every stable r needs m <= 5)
  if (!cheb_coefs(6.0 * g->c1 * g->h * g->h + 36.0, 20.0, 16.0, 1e-10, &g->walk.cheb, 3) || g->walk.cheb.m > 5)
    return MS_ENOTCONV;
  return MS_OK;
}

void walk_d(ms_grid* g, int step, const float* src_hi, const float* src_lo) {
  // Step 1: along y into s32[4], along x into s32[1]; Step 2: s32[2] (H_x), s32[3] (H_y)
  const YArgs y = make_y(g, step, step == 0 ? g->s32[4] : g->s32[2], step == 0 ? g->s32[1] : g->s32[3], src_hi, src_lo);
  const XArgs x = make_x(g, step, step == 0 ? g->s32[1] : g->s32[3], src_hi, src_lo);
  const int nyb = blocks_of(y.nstrip * y.nseg);
  const dim3 grd(nyb + blocks_of(x.nstrip * x.nblk)), blk(32 * WPB);
  if (step == 0) launch_pdl(k_walk_d<false, true>, grd, blk, 0, g->stream, y, x, nyb);
  else if (src_hi) launch_pdl(k_walk_d<true, false>, grd, blk, 0, g->stream, y, x, nyb);
  else launch_pdl(k_walk_d<true, true>, grd, blk, 0, g->stream, y, x, nyb);
}

void walk_s(ms_grid* g, int step) {
  const int P = g->walk.cheb.m - 1;
  SArgs a, b;
  int na, nb = 0;
  if (step == 0) {
    a = b = make_s(g, EZ, g->s32[4], g->s32[1], 1);
    na = blocks_of(a.nstrip * a.nblk);
  } else {
    a = make_s(g, HX, g->s32[2], nullptr, 2);
    b = make_s(g, HY, g->s32[3], nullptr, 2);
    na = blocks_of(a.nstrip * a.nblk);
    nb = blocks_of(b.nstrip * b.nblk);
  }
  const dim3 grd(na + nb), blk(32 * WPB);
  if (P == 2) launch_pdl(k_walk_s<2>, grd, blk, 0, g->stream, a, b, na);
  else if (P == 3) launch_pdl(k_walk_s<3>, grd, blk, 0, g->stream, a, b, na);
  else launch_pdl(k_walk_s<4>, grd, blk, 0, g->stream, a, b, na);
}

int walk_batch_build(ms_grid* const* cav, int count, int order, WalkBatch* wb, std::string* err) {
  std::vector<YArgs> ya(2 * (size_t)count);
  std::vector<XArgs> xa(2 * (size_t)count);
  std::vector<SArgs> sa(3 * (size_t)count);
  std::vector<int> seq(count);
  for (int c = 0; c < count; ++c) seq[c] = c;
  if (order == 2) std::stable_sort(seq.begin(), seq.end(), [&](int a, int b) { return cav[a]->N > cav[b]->N; });
  wb->P = cav[0]->walk.cheb.m - 1;
  wb->ny = 2 * count;
  for (int c = 0; c < count; ++c) {
    const ms_grid* g = cav[c];
    ya[c] = make_y(g, 0, g->s32[4], g->s32[1], nullptr, nullptr);
    ya[count + c] = make_y(g, 1, g->s32[2], g->s32[3], nullptr, nullptr);
    xa[c] = make_x(g, 0, g->s32[1], nullptr, nullptr);
    xa[count + c] = make_x(g, 1, g->s32[3], nullptr, nullptr);
    sa[c] = make_s(g, EZ, g->s32[4], g->s32[1], 1);
    sa[count + c] = make_s(g, HX, g->s32[2], nullptr, 2);
    sa[2 * count + c] = make_s(g, HY, g->s32[3], nullptr, 2);
  }
  // row blocks by the warps of a whole launch, all cavities together (us per step, chosen so and with 32 rows
  // whatever the cavities: four of 64 to 256 cells 21 and 46, a hundred of 32 cells 24 and 44, 16 of 256 cells 45 and 60)
  for (int l = 0; l < 2; ++l) {
    SArgs *first = sa.data() + (size_t)l * count, *last = sa.data() + (size_t)(l ? 3 : 1) * count;
    const int rows = solve_rows([&](int q) {
      int n = 0;
      for (const SArgs* a = first; a != last; ++a) n += a->nstrip * ((a->u1 - a->u0 + q - 1) / q);
      return n;
    }, 1216);
    for (SArgs* a = first; a != last; ++a) {
      const int nr = a->u1 - a->u0;
      a->nblk = (nr + rows - 1) / rows;
      a->rows = (nr + a->nblk - 1) / a->nblk;
    }
  }
  std::vector<int> list[4];
  auto add = [&](std::vector<int>& l, int arg, int items) {
    for (int i = 0; i < items; i += WPB) l.insert(l.end(), {arg, i});
  };
  // order 1: the cavities one strip wide (nothing but walls) ahead of the others
  for (int pass = 0; pass < (order == 1 ? 2 : 1); ++pass)
    for (int c : seq) {
      if (order == 1 && (sa[c].nstrip == 1) != (pass == 0)) continue;
      for (int k = 0; k < 2; ++k) {
        const YArgs& y = ya[(size_t)k * count + c];
        const XArgs& x = xa[(size_t)k * count + c];
        add(list[2 * k], k * count + c, y.nstrip * y.nseg);
        add(list[2 * k], wb->ny + k * count + c, x.nstrip * x.nblk);
      }
      add(list[1], c, sa[c].nstrip * sa[c].nblk);
      for (int k = 1; k < 3; ++k) add(list[3], k * count + c, sa[(size_t)k * count + c].nstrip * sa[(size_t)k * count + c].nblk);
    }
  std::vector<int> work;
  for (int k = 0; k < 4; ++k) {
    wb->off[k] = work.size();
    wb->n[k] = (int)(list[k].size() / 2);
    work.insert(work.end(), list[k].begin(), list[k].end());
  }
  if (dev_malloc(&wb->d_y, ya.size() * sizeof(YArgs)) != cudaSuccess ||
      dev_malloc(&wb->d_x, xa.size() * sizeof(XArgs)) != cudaSuccess ||
      dev_malloc(&wb->d_s, sa.size() * sizeof(SArgs)) != cudaSuccess ||
      dev_malloc(&wb->d_work, work.size() * sizeof(int)) != cudaSuccess) {
    *err = "cudaMalloc of the batch work lists failed";
    return -1;
  }
  if (cudaMemcpy(wb->d_y, ya.data(), ya.size() * sizeof(YArgs), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(wb->d_x, xa.data(), xa.size() * sizeof(XArgs), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(wb->d_s, sa.data(), sa.size() * sizeof(SArgs), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(wb->d_work, work.data(), work.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) {
    *err = "copy of the batch work lists failed";
    return -1;
  }
  // blocks resident on the device at once (persistent launches)
  int dev = 0, sms = 0, pd = 0, ps = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pd, k_batch_d<true>, 32 * WPB, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, wb->P == 2 ? k_batch_s<2> : (wb->P == 3 ? k_batch_s<3> : k_batch_s<4>),
                                                32 * WPB, 0);
  wb->resident_d = sms * pd;
  wb->resident_s = sms * ps;
  return 0;
}

void walk_batch_step(const WalkBatch& wb, cudaStream_t st, int persistent) {
  const dim3 blk(32 * WPB);
  auto blocks = [&](int n, int resident) { return dim3((persistent && resident > 0 && resident < n) ? resident : n); };
  const YArgs* y = wb.d_y;
  const XArgs* x = wb.d_x;
  const SArgs* s = wb.d_s;
  for (int k = 0; k < 4; ++k) {
    const int* w = wb.d_work + wb.off[k];
    const int n = wb.n[k];
    const dim3 gd = blocks(n, wb.resident_d), gs = blocks(n, wb.resident_s);
    if (k == 0) launch_pdl(k_batch_d<false>, gd, blk, 0, st, y, x, wb.ny, w, n);
    else if (k == 2) launch_pdl(k_batch_d<true>, gd, blk, 0, st, y, x, wb.ny, w, n);
    else if (wb.P == 2) launch_pdl(k_batch_s<2>, gs, blk, 0, st, s, w, n);
    else if (wb.P == 3) launch_pdl(k_batch_s<3>, gs, blk, 0, st, s, w, n);
    else launch_pdl(k_batch_s<4>, gs, blk, 0, st, s, w, n);
  }
}

void walk_batch_free(WalkBatch* wb) {
  dev_free(wb->d_y);
  dev_free(wb->d_x);
  dev_free(wb->d_s);
  dev_free(wb->d_work);
  *wb = WalkBatch{};
}

}  // namespace ms
