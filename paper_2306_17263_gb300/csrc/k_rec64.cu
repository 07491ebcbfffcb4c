// FP64 Pade derivatives by recurrences and P1 solves by a Chebyshev polynomial.
//
// GB300 issues one FP64 warp instruction per SM every 16 clocks, so these kernels are bound by the
// number of FP64 operations; loads, index arithmetic and shared memory hide behind them.
//
// Pade derivative.  A = (1/24) tridiag(1, 22, 1) = (1 - rho E^-1)(1 - rho E) / (1 - rho)^2 away from the
// line ends, so A^{-1} d is a forward and a backward first-order recurrence (one FMA per row each)
// instead of a band of 34 taps; a segment of L rows starts its recurrences kRecWarm rows outside itself
// (rho^14 = 1.65e-19).  The closure's end rows change the solution by a multiple of a decaying vector
// (LineEnds), so a line end costs 18 FMAs, not 16 explicit band rows.  A step at 1024 x 1024 takes 399 us with
// these kernels, 1023 us with the band and Richardson sweeps; 3D, 96^3: 1.09 and 2.97 ms.
//
// P1 solve.  6 h^2 P1 = D - T with T = (L_x + 6)(L_y + 6), D = 6 c1 h^2 + 36, and T has its spectrum in
// [4, 36] on every field, Dirichlet or Neumann.  The Chebyshev polynomial p(T) ~ 1 / (D - T) in Horner
// form costs five FP64 operations per point and level (two for w = (L_x + 6) y, two for (L_y + 6) w, one
// FMA with b) where a Richardson sweep with its residual took 21.  Small grids are bound by launches: a
// block runs every level of its tile with b, y and w in shared memory and a halo of one cell per level.
#include <cmath>

#include "k_fp64.cuh"
#include "k_pdl.cuh"
#include "k_rec64.cuh"

namespace ms {

static long double rho_l() { return -11.0L + std::sqrt(120.0L); }

void line_ends(int closure, int kind, bool transposed, LineEnds* e) {
  const long double rho = rho_l();
  long double pw[kRecWarm + 8];
  pw[0] = 1.0L;
  for (int k = 1; k < kRecWarm + 8; ++k) pw[k] = pw[k - 1] * rho;
  const bool paper = closure == MS_CLOSURE_PAPER;
  if (!transposed) {
    // the end row applied to Y + phi rho^i equals 24 d_0 = Y_{-1} + 22 Y_0 + Y_1, Y_{-1} = rho Y_0
    long double den, g[4] = {0, 0, 0, 0};
    if (paper) {
      den = 26.0L - 5.0L * pw[1] + 4.0L * pw[2] - pw[3];
      g[0] = rho - 4.0L;
      g[1] = 6.0L;
      g[2] = -4.0L;
      g[3] = 1.0L;
    } else if (kind == NODE_TO_HALF) {
      den = 23.0L + rho;
      g[0] = rho - 1.0L;
    } else {
      den = 22.0L + rho;
      g[0] = rho;
    }
    for (int k = 0; k < 4; ++k) e->g[k] = (double)(g[k] / den);
    for (int i = 0; i < kRecWarm; ++i) e->v[i] = (double)pw[i];
    return;
  }
  // A^T = (1/24)(T + r0 e_0^T + ..), T the truncated Toeplitz matrix, r0 the end row minus T's:
  // v = T^{-1} 24 u - T^{-1} r0 v_0, and T^{-1} x = G x - rho^{i+2} (G x)_0 with G the infinite inverse
  long double r0[4] = {0, 0, 0, 0};
  if (paper) {
    r0[0] = 4.0L;
    r0[1] = -6.0L;
    r0[2] = 4.0L;
    r0[3] = -1.0L;
  } else if (kind == NODE_TO_HALF) {
    r0[0] = 1.0L;
  }
  const long double kap = 1.0L / (22.0L + 2.0L * rho);
  long double gr[kRecWarm] = {};  // (G r0)_i
  for (int i = 0; i < kRecWarm; ++i)
    for (int k = 0; k < 4; ++k) gr[i] += kap * pw[i > k ? i - k : k - i] * r0[k];
  const long double f = (1.0L - pw[2]) / (1.0L + gr[0] * (1.0L - pw[2]));
  for (int i = 0; i < kRecWarm; ++i) e->v[i] = (double)(-pw[i + 2] - (gr[i] - pw[i + 2] * gr[0]) * f);
  e->g[0] = 1.0;
  e->g[1] = e->g[2] = e->g[3] = 0.0;
}

bool cheb_coefs(double D, double c, double s, double tol, Cheb* p, int mmin) {
  // T_m((t - c) / s) as a polynomial in t, and its value at D
  const int n = kChebMax + 1;
  long double a[kChebMax + 2] = {1.0L}, b[kChebMax + 2] = {-(long double)c / s, 1.0L / (long double)s};
  const long double x = ((long double)D - c) / s;
  long double va = 1.0L, vb = x;
  int m = 1;
  while (m < mmin || 1.0L / vb > tol) {
    if (++m > kChebMax) return false;
    long double t[kChebMax + 2] = {};
    for (int k = 0; k < n; ++k) t[k] = 2.0L * (-(long double)c / s * b[k] + (k ? b[k - 1] / s : 0.0L)) - a[k];
    const long double vt = 2.0L * x * vb - va;
    for (int k = 0; k <= n; ++k) {
      a[k] = b[k];
      b[k] = k < n ? t[k] : 0.0L;
    }
    va = vb;
    vb = vt;
  }
  // (D - t) p(t) = 1 - e(t), e = T_m / T_m(D): coefficients of p by synthetic division
  p->m = m;
  long double pk[kChebMax + 1];
  pk[0] = (1.0L - b[0] / vb) / D;
  for (int k = 1; k < m; ++k) pk[k] = (pk[k - 1] - b[k] / vb) / D;
  p->p0 = (double)pk[0];
  for (int k = 1; k < m; ++k) p->q[k] = (double)(pk[k] / pk[k - 1]);
  return true;
}

namespace {

constexpr double kRho = -0.045548849896677730860604;  // -11 + sqrt(120)

// The two recurrences over rows s .. s + NR - 1 of a line: ys[t] = (A^{-1} d)_{s+t} / (1 - rho)^2 before
// the end corrections; get(m) is d_m, called for m = s - kRecWarm .. s + NR + kRecWarm - 1 in order.
template <int NR, typename Get>
__device__ __forceinline__ void rec_rows64(int s, double (&ys)[NR + kRecWarm], Get get) {
  double z = 0.0;
#pragma unroll
  for (int t = -kRecWarm; t < NR + kRecWarm; ++t) {
    z = fma(kRho, z, get(s + t));
    if (t >= 0) ys[t] = z;
  }
  double y = 0.0;
#pragma unroll
  for (int t = NR + kRecWarm - 1; t >= 0; --t) {
    y = fma(kRho, y, ys[t]);
    ys[t] = y;
  }
}

// Corrections of a segment whose row r0 is ys[0] (first end at row 0, last end at row M - 1); the first
// row of a line is row 0 of its first segment, the last row of a line the last of its last segment.
// O: rows of ys before row 0 of the line (1 in the transposed form's first segment).
template <int NR, int O0, int O1>
__device__ __forceinline__ void end_rows64(double (&ys)[NR + kRecWarm], const LineEnds& e, bool first, bool last) {
  if (first) {
    const double phi = fma(e.g[0], ys[O0], fma(e.g[1], ys[O0 + 1], fma(e.g[2], ys[O0 + 2], e.g[3] * ys[O0 + 3])));
#pragma unroll
    for (int t = 0; t < kRecWarm; ++t) ys[O0 + t] = fma(e.v[t], phi, ys[O0 + t]);
  }
  if (last) {
    constexpr int Z = NR - 1 - O1;
    const double phi = fma(e.g[0], ys[Z], fma(e.g[1], ys[Z - 1], fma(e.g[2], ys[Z - 2], e.g[3] * ys[Z - 3])));
#pragma unroll
    for (int t = 0; t < kRecWarm; ++t) ys[Z - t] = fma(e.v[t], phi, ys[Z - t]);
  }
}

// Outputs s .. s + L - 1 of one line, from d_m = in_{m+1} - in_m (get_in(m): input m of the line, called
// in order).  Transposed: input rows are u_m, output k = v_{k-1} - v_k with v = A^{-T} u, v_{-1} = v_M = 0,
// on k = 0 .. M.  res(t, value) receives output s + t over (1 - rho)^2.
template <int L, bool TRANS, typename GetIn, typename Res>
__device__ __forceinline__ void line_segment64(int s, int M, const LineEnds& e, GetIn get_in, Res res) {
  if (!TRANS) {
    double ys[L + kRecWarm];
    // inputs m and m + 1 of row m; beyond the line d = 0
    double prev = get_in(s - kRecWarm);
    rec_rows64<L>(s, ys, [&](int m) {
      const double nx = get_in(m + 1);
      const double d = (m >= 0 && m < M) ? nx - prev : 0.0;
      prev = nx;
      return d;
    });
    end_rows64<L, 0, 0>(ys, e, s == 0, s + L == M);
#pragma unroll
    for (int t = 0; t < L; ++t) res(t, ys[t]);
  } else {
    double ys[L + 1 + kRecWarm];  // rows s - 1 .. s + L - 1 of v
    rec_rows64<L + 1>(s - 1, ys, [&](int m) { return get_in(m); });
    end_rows64<L + 1, 1, 1>(ys, e, s == 0, s + L == M + 1);
    if (s == 0) ys[0] = 0.0;
    if (s + L == M + 1) ys[L] = 0.0;
#pragma unroll
    for (int t = 0; t < L; ++t) res(t, ys[t] - ys[t + 1]);
  }
}

struct LineBatch {
  LineArgs a[kLineBatch];
  LineEnds e;
  int n1;  // largest n1 of the batch
};

constexpr int LW = 4;  // warps per block of the row form (LS <= LW segments per tile)
constexpr int kShortLS = 1;  // segments of 16 rows per block
constexpr double kOneMinusRhoSq = 1.093172397520265540654504;  // (1 - rho)^2 = -24 rho

// Lines across a strided axis, lanes across the contiguous one: a thread walks its segment of a line,
// every load coalesced.  The last segment of a line is aligned to its end and writes all its rows (the
// one before it stops there), so both ends and the rows they correct sit at fixed places of a segment.
template <int L, bool TRANS>
__device__ __forceinline__ void line_walk64(const LineArgs& a, const LineEnds& e, int l0, int l1, int seg) {
  const int R = TRANS ? a.M + 1 : a.M;
  const int nseg = (R + L - 1) / L;
  if (l0 >= a.n0 || seg >= nseg) return;
  double* o = a.out + l0 * a.out_s0 + l1 * a.out_s1;
  const bool live = l0 >= a.lo && l0 < a.hi;
  const bool lastseg = seg == nseg - 1;
  const int s = lastseg ? R - L : seg * L;
  const int cnt = lastseg ? L : min(L, R - L - s);  // rows it writes
  if (!a.accumulate) {  // points of the line beyond its outputs
    if (seg == 0)
      for (int q = 0; q < a.out_off; ++q) o[q * a.out_sa] = 0.0;
    if (lastseg)
      for (int q = R + a.out_off; q < a.out_len; ++q) o[q * a.out_sa] = 0.0;
  }
  double* op = o + (size_t)(s + a.out_off) * a.out_sa;
  if (!live) {
    if (!a.accumulate)
      for (int t = 0; t < cnt; ++t) op[t * a.out_sa] = 0.0;
    return;
  }
  const double* ip = a.in + l0 * a.in_s0 + l1 * a.in_s1;
  const double scale = a.scale * kOneMinusRhoSq;
  const int n_in = TRANS ? a.M : a.M + 1;
  double ys[L];
  line_segment64<L, TRANS>(
      s, a.M, e, [&](int m) { return (m >= 0 && m < n_in) ? ip[m * (ptrdiff_t)a.in_sa] : 0.0; },
      [&](int t, double v) { ys[t] = v; });
#pragma unroll
  for (int t0 = 0; t0 < L; t0 += 8) {  // eight loads in flight
    double old[8] = {};
    if (a.accumulate) {
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t0 + t < cnt) old[t] = op[(t0 + t) * a.out_sa];
    }
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (t0 + t < cnt) op[(t0 + t) * a.out_sa] = a.accumulate ? fma(scale, ys[t0 + t], old[t]) : scale * ys[t0 + t];
  }
}

template <int L, int LS, bool TRANS>
__global__ void __launch_bounds__(32 * LS) k_line_walk64(LineBatch b) {
  pdl_wait();
  const int which = blockIdx.z / b.n1, l1 = blockIdx.z - which * b.n1;
  if (l1 >= b.a[which].n1) return;
  line_walk64<L, TRANS>(b.a[which], b.e, blockIdx.x * 32 + threadIdx.x, l1, blockIdx.y * LS + threadIdx.y);
}

// Lines along the contiguous axis: a block takes LS segments of 32 lines.  Whole warps read the lines
// into shared memory (odd pitch: lanes across the lines are conflict-free), a thread takes one
// segment of one line, and the results go back through shared memory.
template <int L, int LS>
struct RowsTile {
  static constexpr int OUTS = LS * L, PW = OUTS + 2 * kRecWarm + 3;  // odd
  static_assert(PW % 2 == 1, "odd row pitch");
};
template <int L, int LS, bool TRANS>
__device__ __forceinline__ void line_rows64(const LineArgs& a, const LineEnds& e, int bx, int by, int l1, double* sm) {
  constexpr int OUTS = RowsTile<L, LS>::OUTS, PW = RowsTile<L, LS>::PW;
  const int lane = threadIdx.x, warp = threadIdx.y;
  const int R = TRANS ? a.M + 1 : a.M;
  const int nseg = (R + L - 1) / L;
  const int t0 = bx * OUTS;
  const int b0 = min(t0, R - L);           // first output of the tile
  const int base = b0 - kRecWarm - 1;      // input index of column 0
  const int n_in = TRANS ? a.M : a.M + 1;
  const int la = by * 32;
  const double* in = a.in + l1 * a.in_s1;
  double* out = a.out + l1 * a.out_s1;
#pragma unroll 4
  for (int q = warp; q < 32; q += LW) {
    const int l0 = la + q;
    const bool live = l0 >= a.lo && l0 < a.hi;
    const double* ip = in + (live ? l0 : 0) * a.in_s0;
#pragma unroll
    for (int c = 0; c < (PW + 31) / 32; ++c) {
      const int col = 32 * c + lane, m = base + col;
      if (col < PW) sm[q * PW + col] = (live && m >= 0 && m < n_in) ? ip[m] : 0.0;
    }
  }
  __syncthreads();
  const int seg = bx * LS + warp;
  const bool lastseg = seg == nseg - 1, has = warp < LS && seg < nseg;
  const int s = lastseg ? R - L : seg * L;
  double ys[L];
  if (has) {
    const double* row = sm + lane * PW - base;  // row[m]: input m of the line
    line_segment64<L, TRANS>(s, a.M, e, [&](int m) { return row[m]; },
                             [&](int t, double v) { ys[t] = v; });
  }
  __syncthreads();
  if (has) {
    const int cnt = lastseg ? L : min(L, R - L - s);
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (t < cnt) sm[lane * PW + s - b0 + t] = ys[t];
  }
  __syncthreads();
  const bool last_tile = (bx + 1) * LS >= nseg;
  const double scale = a.scale * kOneMinusRhoSq;
  const int nout = (last_tile ? R : min(t0 + OUTS, R - L)) - b0;
  constexpr int NC = (OUTS + 31) / 32;  // nout <= OUTS: the last tile, aligned to the end, starts earlier
#pragma unroll
  for (int q0 = 0; q0 < 32; q0 += 4 * LW) {
    double old[4][NC] = {};
    if (a.accumulate) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int l0 = la + q0 + u * LW + warp;
        const double* op = out + l0 * a.out_s0 + b0 + a.out_off;
#pragma unroll
        for (int c = 0; c < NC; ++c)
          if (l0 >= a.lo && l0 < a.hi && 32 * c + lane < nout) old[u][c] = op[32 * c + lane];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = q0 + u * LW + warp, l0 = la + q;
      if (l0 >= a.n0) continue;
      const bool live = l0 >= a.lo && l0 < a.hi;
      double* o = out + l0 * a.out_s0;
      double* op = o + b0 + a.out_off;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int col = 32 * c + lane;
        if (col < nout) {
          if (live) op[col] = a.accumulate ? fma(scale, sm[q * PW + col], old[u][c]) : scale * sm[q * PW + col];
          else if (!a.accumulate) op[col] = 0.0;
        }
      }
      if (!a.accumulate) {
        if (t0 == 0 && lane < a.out_off) o[lane] = 0.0;
        if (last_tile && R + a.out_off + lane < a.out_len) o[R + a.out_off + lane] = 0.0;
      }
    }
  }
}

template <int L, int LS, bool TRANS>
__global__ void __launch_bounds__(32 * LW) k_line_rows64(LineBatch b) {
  __shared__ double sm[32 * RowsTile<L, LS>::PW];
  pdl_wait();
  const int which = blockIdx.z / b.n1, l1 = blockIdx.z - which * b.n1;
  if (l1 >= b.a[which].n1) return;
  line_rows64<L, LS, TRANS>(b.a[which], b.e, blockIdx.x, blockIdx.y, l1, sm);
}

// One derivative along each axis (a[0] along the contiguous one), independent of one another, in one
// launch: on small grids a launch takes the latency of one chain of recurrences whatever it holds.  With both
// half-steps' pairs joined, 64^2 went 58.3 -> 39.9 us per step, 321^2 101 -> 83 us.
template <int L, bool TRANS>
__global__ void __launch_bounds__(32 * LW) k_line_pair64(LineBatch b, int rows_x, int rows_n, int walk_x) {
  __shared__ double sm[32 * RowsTile<L, 1>::PW];
  pdl_wait();
  const int q = blockIdx.x - rows_n;
  if (q < 0) line_rows64<L, 1, TRANS>(b.a[0], b.e, blockIdx.x % rows_x, blockIdx.x / rows_x, 0, sm);
  else if (threadIdx.y == 0) line_walk64<L, TRANS>(b.a[1], b.e, (q % walk_x) * 32 + threadIdx.x, 0, q / walk_x);
}

}  // namespace

// Segments of 32 rows do 3.3 FMAs per output, of 16 rows 4.6; the shorter ones win while the longer
// ones would leave FP64 pipes (4 per SM) without a warp.  A block takes one short segment: warps of one
// SM share its FP64 rate (64^2: 64.0 us per step with four, 56.7 us with one; 321^2: 110.4 and 102.1 us).
static bool lines64_short(int n0, int R, int n1) {
  return R < 64 || (double)((n0 + 31) / 32) * ((R + 31) / 32) * n1 < 600.0;
}

void launch_line64(const LineArgs* args, int count, const LineEnds& e, bool transposed, cudaStream_t st) {
  LineBatch b;
  b.e = e;
  b.n1 = 0;
  int n0 = 0;
  const int M = args[0].M, R = transposed ? M + 1 : M;
  for (int k = 0; k < kLineBatch; ++k) {
    b.a[k] = args[k < count ? k : 0];
    b.n1 = b.a[k].n1 > b.n1 ? b.a[k].n1 : b.n1;
    n0 = b.a[k].n0 > n0 ? b.a[k].n0 : n0;
  }
  const bool rows = args[0].in_sa == 1;
  const bool l32 = !lines64_short(n0, R, b.n1 * count);
  const int L = l32 ? 32 : 16, LS = l32 ? 4 : kShortLS;
  const int nseg = (R + L - 1) / L;
  const dim3 blk(32, rows ? LW : LS);
  const dim3 grd = rows ? dim3((nseg + LS - 1) / LS, (n0 + 31) / 32, b.n1 * count)
                        : dim3((n0 + 31) / 32, (nseg + LS - 1) / LS, b.n1 * count);
#define MS_LINE(K)                                                                 \
  do {                                                                             \
    if (l32 && transposed) launch_pdl(K<32, 4, true>, grd, blk, 0, st, b);         \
    else if (l32) launch_pdl(K<32, 4, false>, grd, blk, 0, st, b);                 \
    else if (transposed) launch_pdl(K<16, kShortLS, true>, grd, blk, 0, st, b);    \
    else launch_pdl(K<16, kShortLS, false>, grd, blk, 0, st, b);                   \
  } while (0)
  if (rows) MS_LINE(k_line_rows64);
  else MS_LINE(k_line_walk64);
#undef MS_LINE
}

bool launch_line64_pair(const LineArgs& x, const LineArgs& y, const LineEnds& e, bool transposed, cudaStream_t st) {
  const int R = transposed ? x.M + 1 : x.M;
  if (!lines64_short(x.n0, R, 1)) return false;
  LineBatch b;
  b.e = e;
  b.n1 = 1;
  for (int k = 0; k < kLineBatch; ++k) b.a[k] = k == 1 ? y : x;
  const int nseg = (R + 15) / 16, nl = (x.n0 + 31) / 32, nw = (y.n0 + 31) / 32;
  const dim3 grd(nseg * (nl + nw)), blk(32, LW);
  if (transposed) launch_pdl(k_line_pair64<16, true>, grd, blk, 0, st, b, nseg, nseg * nl, nw);
  else launch_pdl(k_line_pair64<16, false>, grd, blk, 0, st, b, nseg, nseg * nl, nw);
  return true;
}

// ---------------------------------------------------------------------------------------
// The 2D solve.
namespace {

struct Cheb2dArgs {
  Cheb2dField f[2];
  Cheb p;
  double out_scale, upd_scale;  // x = out_scale y, upd += upd_scale y
  int TS;                       // output tile edge
};

constexpr int C2T = 256;  // threads per block
static_assert(3 * 8 * (16 + 2 * (kChebMax - 1)) * (16 + 2 * (kChebMax - 1)) <= 48 * 1024, "default shared memory");

// A block solves a TS x TS tile: b on the tile plus a halo of m - 1 cells in shared memory, then one
// level after another on a region that shrinks by a cell, each in two passes over it (w = 4 y + y_left +
// y_right, then y = b + q (w_up + w_down + 4 w)).  Points off the unknowns hold 0 (Dirichlet); across a
// Neumann wall the ghost equals its mirror, the point itself.
__global__ void __launch_bounds__(C2T) k_cheb2d64(Cheb2dArgs A) {
  extern __shared__ double sm64[];
  pdl_wait();
  const Cheb2dField& F = A.f[blockIdx.z];
  const int nx = F.s.nx, ny = F.s.ny;
  const int TS = A.TS, H = A.p.m - 1, W = TS + 2 * H;
  // tiles cover the unknowns; the first and the last of a row or column write the walls of `out` too
  const int dx = F.s.bcx == DIR, dy = F.s.bcy == DIR;
  const int tx0 = dx + blockIdx.x * TS, ty0 = dy + blockIdx.y * TS;
  if (tx0 >= nx - dx || ty0 >= ny - dy) return;
  const int gx0 = tx0 - H, gy0 = ty0 - H;
  double* bs = sm64;
  double* ys = bs + W * W;
  double* ws = ys + W * W;
  auto unknown = [&](int gx, int gy) {
    return gx >= 0 && gx < nx && gy >= 0 && gy < ny && interior(F.s.bcx, gx, nx) && interior(F.s.bcy, gy, ny);
  };
  for (int t = threadIdx.x; t < W * W; t += C2T) {
    const int r = t / W, c = t - r * W;
    const int gx = gx0 + c, gy = gy0 + r;
    double v = 0.0;
    if (unknown(gx, gy)) {
      v = F.b[(size_t)gy * nx + gx];
      if (F.b2) v += F.b2[(size_t)gy * nx + gx];
    }
    bs[t] = v;
    ys[t] = v;
  }
  const bool neu_x = F.s.bcx == NEU, neu_y = F.s.bcy == NEU;
  for (int k = 1; k <= H; ++k) {
    const double q = A.p.q[A.p.m - k];
    const int wd = W - 2 * k;  // columns of this level
    __syncthreads();
    for (int t = threadIdx.x; t < wd * (wd + 2); t += C2T) {
      const int r = t / wd, c = k + t - r * wd;
      const int gx = gx0 + c, p = (r + k - 1) * W + c;
      const double y = ys[p];
      const double l = (neu_x && gx == 0) ? y : ys[p - 1], u = (neu_x && gx == nx - 1) ? y : ys[p + 1];
      ws[p] = fma(4.0, y, l + u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < wd * wd; t += C2T) {
      const int r = t / wd, c = k + t - r * wd;
      const int gx = gx0 + c, gy = gy0 + r + k, p = (r + k) * W + c;
      const double w = ws[p];
      const double u = (neu_y && gy == 0) ? w : ws[p - W], d = (neu_y && gy == ny - 1) ? w : ws[p + W];
      if (unknown(gx, gy)) ys[p] = fma(q, fma(4.0, w, u + d), bs[p]);
    }
  }
  __syncthreads();
  const int c0 = tx0 == dx ? -dx : 0, r0 = ty0 == dy ? -dy : 0, wd = TS + 1 + dx;
  for (int t = threadIdx.x; t < wd * (TS + 1 + dy); t += C2T) {
    const int rr = t / wd, r = r0 + rr, c = c0 + t - rr * wd;
    const int gx = tx0 + c, gy = ty0 + r;
    // own points, and a wall next to the last unknown
    if (gx >= nx || gy >= ny || (c >= TS && !(dx && gx == nx - 1 && c == TS)) ||
        (r >= TS && !(dy && gy == ny - 1 && r == TS)))
      continue;
    const double y = ys[(r + H) * W + c + H];
    const size_t g = (size_t)gy * nx + gx;
    if (F.out) F.out[g] = A.out_scale * y;
    if (F.upd && unknown(gx, gy)) F.upd[g] = fma(A.upd_scale, y, F.upd[g]);
  }
}

// Large grids: one level per launch, nothing recomputed.  A thread takes C2R rows of one column, w of
// each row formed once and shared by the three rows it enters (5.5 FP64 operations per point).
constexpr int C2R = 8;
struct Cheb2dLevel {
  const double* y[2];
  const double* b[2];
  double* yout[2];
  Cheb2dField f[2];
  double q, out_scale, upd_scale;
};
template <bool LAST>
__global__ void __launch_bounds__(128) k_cheb2d64_level(Cheb2dLevel A) {
  pdl_wait();
  const int fi = blockIdx.z;
  const Cheb2dField& F = A.f[fi];
  const int nx = F.s.nx, ny = F.s.ny, dx = F.s.bcx == DIR, dy = F.s.bcy == DIR;
  const int i = dx + blockIdx.x * 32 + threadIdx.x;
  const int j0 = dy + (blockIdx.y * 4 + threadIdx.y) * C2R, j1 = min(j0 + C2R, ny - dy);
  if (i >= nx - dx || j0 >= j1) return;
  const double* __restrict__ y = A.y[fi];
  // walls of a Dirichlet axis count as 0 (b may hold anything there); ghosts of a Neumann axis mirror
  const int il = clampi(i - 1, nx), ir = clampi(i + 1, nx);
  const bool wl = dx && i == 1, wr = dx && i == nx - 2;
  auto w = [&](int j) {
    j = clampi(j, ny);
    if (dy && (j == 0 || j == ny - 1)) return 0.0;
    const double* r = y + (size_t)j * nx;
    return fma(4.0, r[i], (wl ? 0.0 : r[il]) + (wr ? 0.0 : r[ir]));
  };
  double wu = w(j0 - 1), w0 = w(j0);
#pragma unroll
  for (int t = 0; t < C2R; ++t) {
    const int j = j0 + t;
    if (j >= j1) break;
    const double wd = w(j + 1);
    const size_t g = (size_t)j * nx + i;
    const double v = fma(A.q, fma(4.0, w0, wu + wd), A.b[fi][g]);
    if (LAST) {
      if (F.out) F.out[g] = A.out_scale * v;
      if (F.upd) F.upd[g] = fma(A.upd_scale, v, F.upd[g]);
    } else {
      A.yout[fi][g] = v;
    }
    wu = w0;
    w0 = wd;
  }
  if (LAST && F.out) {  // walls
    const bool fx = dx && i == 1, lx = dx && i == nx - 2;
    for (int j = j0; j < j1; ++j) {
      if (fx) F.out[(size_t)j * nx] = 0.0;
      if (lx) F.out[(size_t)j * nx + nx - 1] = 0.0;
    }
    auto wall_row = [&](int j) {
      F.out[(size_t)j * nx + i] = 0.0;
      if (fx) F.out[(size_t)j * nx] = 0.0;
      if (lx) F.out[(size_t)j * nx + nx - 1] = 0.0;
    };
    if (dy && j0 == 1) wall_row(0);
    if (dy && j1 == ny - 1) wall_row(ny - 1);
  }
}

}  // namespace

// Planes a launch of the solve must touch: b, and y apart from it after the first level, read; the iterate, or
// the solution and the updated field (read and written), written.
static double level_planes(bool first, bool last, bool b2, bool out, bool upd) {
  return 1.0 + !first + b2 + (last ? (out ? 1.0 : 0.0) + (upd ? 2.0 : 0.0) : 1.0);
}

int launch_cheb2d64(ms_grid* g, int kind, const Cheb2dField* f, int nf, double* const (*buf)[2], const Cheb& p,
                    double bscale, double upd_scale) {
  const cudaStream_t st = g->stream;
  auto mark = [&](bool first, bool last) {
    double bytes = 0.0;
    for (int q = 0; q < nf; ++q)
      bytes += 8.0 * (double)f[q].s.size() * level_planes(first, last, f[q].b2, f[q].out, f[q].upd);
    prof_mark(g, kind, bytes);
  };
  const double out_scale = p.p0 * bscale;
  const int nx = f[0].s.nx > f[nf - 1].s.nx ? f[0].s.nx : f[nf - 1].s.nx;
  const int ny = f[0].s.ny > f[nf - 1].s.ny ? f[0].s.ny : f[nf - 1].s.ny;
  const long pts = (long)nx * ny * nf;
  if (!cheb2d64_tiles(pts)) {
    // the tiles' halo would cost 1.4 to 1.9 times the operations; a launch per level costs about 1 us
    const dim3 grd((nx + 31) / 32, (ny + 4 * C2R - 1) / (4 * C2R), nf);
    for (int k = p.m - 1; k >= 1; --k) {
      const int step = p.m - 1 - k;
      Cheb2dLevel A;
      for (int q = 0; q < 2; ++q) {
        const int c = q < nf ? q : 0;
        A.f[q] = f[c];
        A.b[q] = f[c].b;
        A.y[q] = step == 0 ? f[c].b : buf[c][(step + 1) & 1];
        A.yout[q] = buf[c][step & 1];
      }
      A.q = p.q[k];
      A.out_scale = out_scale;
      A.upd_scale = upd_scale * out_scale;
      if (k == 1) launch_pdl(k_cheb2d64_level<true>, grd, dim3(32, 4), 0, st, A);
      else launch_pdl(k_cheb2d64_level<false>, grd, dim3(32, 4), 0, st, A);
      mark(step == 0, k == 1);
    }
    return p.m - 1;
  }
  Cheb2dArgs A;
  A.f[0] = f[0];
  A.f[1] = f[nf - 1];
  A.p = p;
  A.out_scale = out_scale;
  A.upd_scale = upd_scale * out_scale;
  // Tile edge: a small tile recomputes more of its halo, a large one leaves SMs without a block.
  A.TS = pts <= 40000 ? 8 : 16;
  const int W = A.TS + 2 * (p.m - 1);
  const size_t smem = 3 * sizeof(double) * (size_t)W * W;  // at most 35 KB
  launch_pdl(k_cheb2d64, dim3((nx + A.TS - 1) / A.TS, (ny + A.TS - 1) / A.TS, nf), dim3(C2T), smem, st, A);
  mark(true, true);
  return 1;
}

// ---------------------------------------------------------------------------------------
// The 3D solve: 6 h^2 P1 = D - T with D = 6 c1 h^2 + 24 and, from the 19-point stencil,
// T y = 2 e + c + (2 y + e)_{z-1} + (2 y + e)_{z+1}, e and c the sums over the four edge and the four
// corner neighbours in the plane; its spectrum lies in [-8, 24].  One level of the Horner form per
// launch for up to three components: a thread marches CZ planes of one column along z, keeping
// q = 2 y + e of the planes below and above in registers (11 FP64 operations per point and level, 34
// by a Richardson sweep with its residual; 96^3: 61 us per sweep).  Threads are laid along the flattened
// unknowns of a plane, so no lane idles at the end of a row.
namespace {

constexpr int C3Z = 8;
constexpr int C3T = 128;

struct Cheb3dArgs {
  Cheb3dField f[kCheb3dBatch];
  double q, out_scale, upd_scale;
  int nz;  // blocks along z of the largest component
};

template <bool LAST>
__global__ void __launch_bounds__(C3T) k_cheb3d64(Cheb3dArgs A) {
  pdl_wait();
  const int which = blockIdx.y / A.nz, kz = blockIdx.y - which * A.nz;
  const Cheb3dField& F = A.f[which];
  const int n0 = F.n[0], n1 = F.n[1], n2 = F.n[2];
  const int d0 = F.bc[0] == DIR, d1 = F.bc[1] == DIR, d2 = F.bc[2] == DIR;
  const int u0 = n0 - 2 * d0, u1 = n1 - 2 * d1, u2 = n2 - 2 * d2;  // unknowns per axis
  const int t = blockIdx.x * C3T + threadIdx.x;
  const int k0 = d2 + kz * C3Z, k1 = min(k0 + C3Z, d2 + u2);
  if (t >= u0 * u1 || k0 >= k1) return;
  const int jy = t / u0, i = d0 + t - jy * u0, j = d1 + jy;
  const size_t sz = (size_t)n0 * n1;
  // neighbours: stored wall zeros on a Dirichlet axis (b has none there: masked), even ghosts clamped
  const int im = clampi(i - 1, n0), ip = clampi(i + 1, n0), jm = clampi(j - 1, n1), jp = clampi(j + 1, n1);
  const bool wm = d0 && im == 0, wp = d0 && ip == n0 - 1, vm = d1 && jm == 0, vp = d1 && jp == n1 - 1;
  const size_t om = (size_t)jm * n0, o0 = (size_t)j * n0, op = (size_t)jp * n0;
  auto plane = [&](int k, double& y, double& e, double& c) {
    k = clampi(k, n2);
    if (d2 && (k == 0 || k == n2 - 1)) {
      y = e = c = 0.0;
      return;
    }
    const double* p = F.y + k * sz;
    auto row = [&](size_t o, bool off, double& m, double& s) {
      m = off ? 0.0 : p[o + i];
      s = ((off || wm) ? 0.0 : p[o + im]) + ((off || wp) ? 0.0 : p[o + ip]);
    };
    double ym, sm, yp, sp, s0;
    row(o0, false, y, s0);
    row(om, vm, ym, sm);
    row(op, vp, yp, sp);
    e = s0 + (ym + yp);
    c = sm + sp;
  };
  double y, e, c, qm, q0;
  plane(k0 - 1, y, e, c);
  qm = fma(2.0, y, e);
  plane(k0, y, e, c);
  q0 = fma(2.0, y, e);
  for (int k = k0; k < k1; ++k) {
    double yn, en, cn;
    plane(k + 1, yn, en, cn);
    const double qn = fma(2.0, yn, en);
    const size_t g = k * sz + o0 + i;
    const double v = fma(A.q, fma(2.0, e, c) + (qm + qn), F.b[g]);
    if (LAST) {
      if (F.out) F.out[g] = A.out_scale * v;
      if (F.upd) F.upd[g] = fma(A.upd_scale, v, F.upd[g]);
    } else {
      F.out[g] = v;
    }
    qm = q0;
    q0 = qn;
    e = en;
    c = cn;
  }
}

}  // namespace

int launch_cheb3d64(ms_grid* g, int kind, const Cheb3dField* f, double* const (*buf)[2], int count, const Cheb& p,
                    double bscale, double upd_scale) {
  const cudaStream_t st = g->stream;
  Cheb3dArgs A;
  size_t plane = 0;
  int nz = 0;
  for (int k = 0; k < count; ++k) {
    const Cheb3dField& F = f[k];
    const size_t pl = (size_t)(F.n[0] - 2 * (F.bc[0] == DIR)) * (F.n[1] - 2 * (F.bc[1] == DIR));
    plane = pl > plane ? pl : plane;
    const int z = (F.n[2] - 2 * (F.bc[2] == DIR) + C3Z - 1) / C3Z;
    nz = z > nz ? z : nz;
  }
  A.nz = nz;
  A.out_scale = p.p0 * bscale;
  A.upd_scale = upd_scale * A.out_scale;
  const dim3 grd((unsigned)((plane + C3T - 1) / C3T), nz * count);
  for (int k = p.m - 1; k >= 1; --k) {
    A.q = p.q[k];
    const int step = p.m - 1 - k;
    for (int c = 0; c < kCheb3dBatch; ++c) {
      const int cc = c < count ? c : 0;
      A.f[c] = f[cc];
      A.f[c].y = step == 0 ? f[cc].b : buf[cc][(step + 1) & 1];
      if (k > 1) A.f[c].out = buf[cc][step & 1];
    }
    if (k == 1) launch_pdl(k_cheb3d64<true>, grd, dim3(C3T), 0, st, A);
    else launch_pdl(k_cheb3d64<false>, grd, dim3(C3T), 0, st, A);
    double bytes = 0.0;
    for (int c = 0; c < count; ++c)
      bytes += 8.0 * (double)f[c].n[0] * f[c].n[1] * f[c].n[2] * level_planes(step == 0, k == 1, false, f[c].out, f[c].upd);
    prof_mark(g, kind, bytes);
  }
  return p.m - 1;
}

}  // namespace ms
