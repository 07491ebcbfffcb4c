// Device code shared by the FP32 walks of the 2D step (k_tiled.cu), of the reverse pass (adjoint32.cu) and of the
// 3D step (grid3d.cu): constants, paired arithmetic, line ends, the row ring and the 2D solve.
#pragma once

#include "k_fp64.cuh"
#include "k_pdl.cuh"

namespace ms {

// Arguments of walk_s for one field; pointers at the first unknown column of row 0.
struct SArgs {
  const float* p1;  // right-hand side; of E_z the sum of two planes
  const float* p2;
  float* hi;
  float* lo;
  float* out;       // reverse pass: low part of the solution
  int ld, M;        // unknown columns 0 .. M-1
  int u0, u1;       // unknown rows u0 .. u1-1
  int kind;         // KIND_*
  float q[4];          // levels of the solve but for the last
  float s_hi, s_lo;    // increment scale s
  float l_hi, l_lo;    // last level: s q (reverse pass: its coefficient alone)
  int nstrip, nblk, rows;
};

namespace {

constexpr float kRhoF = -0.045548850f;  // rounds to the FP32 root
constexpr float kR2 = kRhoF * kRhoF, kR4 = kR2 * kR2;
constexpr int WPB = 4;      // warps per block
constexpr int YOUT = 30;    // columns a walk_y warp writes
constexpr int XOUT = 112;   // columns a warp writes along x
constexpr int XHALO = 8;
constexpr int SOUT = 120;   // columns a walk_s warp writes
constexpr int SHALO = 4;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kEnd = 8;     // rows of a line the end correction reaches

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// Paired FP32 instructions (two correctly rounded operations each, bitwise those of the scalar ones): the
// walks are bound by instruction issue.  a - b as one FMA with -1, which rounds the same.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }

// phi = g_0 y_0 + .. + g_3 y_3 of the end correction (y counted from the line's end).
template <typename Args>
__device__ __forceinline__ float end_phi(const Args& A, float y0, float y1, float y2, float y3) {
  const float lo = fmaf(A.gl[0], y0, fmaf(A.gl[1], y1, fmaf(A.gl[2], y2, A.gl[3] * y3)));
  return fmaf(A.g[0], y0, fmaf(A.g[1], y1, fmaf(A.g[2], y2, fmaf(A.g[3], y3, lo))));
}

// The eight rows at an end of a line with their correction, y_t = z_t + (rho y_{t+1} + v phi).  It joins rho y, a
// twentieth of y: added to y itself it would round away from the fifth row on, always the same way (frequencies of
// small grids off by 1e-9 to 3e-9; 1e-10 to 4e-10 this way).  v is one FP32 number each, an error of 6e-11 y.
template <bool LAST>
__device__ __forceinline__ void end_rows(float (&y)[8], const float (&z)[8], float ynext, float phi,
                                         const float (&v)[kEnd]) {
#pragma unroll
  for (int t = 0; t < kEnd; ++t)
    y[t] = z[t] + fmaf(v[LAST ? kEnd - 1 - t : t], phi, kRhoF * (t < kEnd - 1 ? y[t + 1 < kEnd ? t + 1 : t] : ynext));
}

// Host: a coefficient as a pair, and the end corrections of a kind of line.
struct Split {
  float hi, lo;
};
inline Split split(double v) {
  Split s;
  s.hi = (float)v;
  s.lo = (float)(v - (double)s.hi);
  return s;
}
template <typename Args>
void set_ends(const LineEnds& e, Args* a) {
  for (int k = 0; k < 4; ++k) {
    const Split g = split(e.g[k]);
    a->g[k] = g.hi;
    a->gl[k] = g.lo;
  }
  for (int k = 0; k < kEnd; ++k) a->v[k] = (float)e.v[k];
}

// Rows come through a ring in shared memory that each warp fills for itself with cp.async, kAhead rows
// ahead: the walk of a row is shorter than a memory round trip, and the registers are taken.  A slot is
// refilled one row after it was read.
constexpr int kAhead = 3, kRing = kAhead + 1;
__device__ __forceinline__ void cp16(float4* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- solve and update ----------------------------------------------------------------------

// (hi, lo) += s b + l t, s and l hi + lo pairs, |l t| <= 36 / D |s b| over a field (2.2e-2 at the stability
// limit): an exact two-product of s_hi b with the other products in its error term, and a two-sum into the
// pair.  One FP32 number each for the last level's q and for s on it were coherent errors of up to 1e-9 of the
// increment; an earlier level's q is off by (36 / D)^2 2^-25 of it, 1.4e-11 at most.
__device__ __forceinline__ void ff_add_scaled(float2& hi, float2& lo, float2 b, float2 t, float2 s_hi, float2 n_hi,
                                              float2 s_lo, float2 l_hi, float2 l_lo) {
  const float2 np = mul2(n_hi, b);  // -p, p = fl(s_hi b)
  float2 e = fma2(s_hi, b, np);
  e = fma2(s_lo, b, e);
  e = fma2(l_lo, t, e);
  e = fma2(l_hi, t, e);
  const float2 u = sub2(hi, np);
  const float2 bb = sub2(u, hi);
  const float2 err = sub2(sub2(hi, sub2(u, bb)), add2(np, bb));
  const float2 l = add2(lo, add2(err, e));
  const float2 h2 = add2(u, l);
  lo = sub2(l, sub2(h2, u));
  hi = h2;
}

// The kinds of field: right-hand side in two planes (E_z), Neumann along y (H_x), along x (H_y).
enum { KIND_E = 0, KIND_HX = 1, KIND_HY = 2 };

// One block of rows of one 128-column strip; P levels.  EDGE: lanes beyond the field hold zeros.  PAIR (the
// reverse pass): the right-hand side is the float-float field (p1, lo) and the solution over its value at T = 36 is
// left as the pair (p1, out), out = lo + l (T - 36) y (adjoint32.cu), the last level on first differences of y.
template <int P, int KIND, bool EDGE, bool PAIR>
__device__ __forceinline__ void s_block(const SArgs& A, float4* ring, int strip, int blk) {
  constexpr bool TWO = KIND == KIND_E && !PAIR;
  const int lane = threadIdx.x & 31;
  const int m0 = SOUT * strip - SHALO + 4 * lane;
  const int M = A.M, u0 = A.u0, u1 = A.u1;
  const int j0 = u0 + blk * A.rows, j1 = min(j0 + A.rows, u1);
  const size_t ld = A.ld;
  const bool ok = !EDGE || (m0 >= 0 && m0 < M);
  const bool out = lane >= SHALO / 4 && lane < (SHALO + SOUT) / 4 && ok;
  bool in[4] = {true, true, true, true}, first = false, lastc[4] = {};
  if (EDGE) {
    first = KIND == KIND_HY && m0 == 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      in[k] = m0 + k >= 0 && m0 + k < M;
      lastc[k] = KIND == KIND_HY && m0 + k == M - 1;
    }
  }
  auto mask = [&](float2(&y)[2]) {
    if (EDGE) {
      y[0].x = in[0] ? y[0].x : 0.0f;
      y[0].y = in[1] ? y[0].y : 0.0f;
      y[1].x = in[2] ? y[1].x : 0.0f;
      y[1].y = in[3] ? y[1].y : 0.0f;
    }
  };
  const float2 four = bc2(4.0f);
  // w = 4 y + left + right
  auto wsum = [&](const float2(&y)[2], float2(&w)[2]) {
    float a = __shfl_up_sync(kFull, y[1].y, 1), b = __shfl_down_sync(kFull, y[0].x, 1);
    float r0 = y[0].y, r1 = y[1].x, r2 = y[1].y;
    if (EDGE && KIND == KIND_HY) {
      a = first ? y[0].x : a;
      r0 = lastc[0] ? y[0].x : r0;
      r1 = lastc[1] ? y[0].y : r1;
      r2 = lastc[2] ? y[1].x : r2;
      b = lastc[3] ? y[1].y : b;
    }
    w[0] = fma2(four, y[0], make_float2(a + r0, y[0].x + r1));
    w[1] = fma2(four, y[1], make_float2(y[0].y + r2, y[1].x + b));
  };
  // l = (left - y) + (right - y)
  auto lapx = [&](const float2(&y)[2], float2(&l)[2]) {
    float a = __shfl_up_sync(kFull, y[1].y, 1), b = __shfl_down_sync(kFull, y[0].x, 1);
    float r0 = y[0].y, r1 = y[1].x, r2 = y[1].y;
    if (EDGE && KIND == KIND_HY) {
      a = first ? y[0].x : a;
      r0 = lastc[0] ? y[0].x : r0;
      r1 = lastc[1] ? y[0].y : r1;
      r2 = lastc[2] ? y[1].x : r2;
      b = lastc[3] ? y[1].y : b;
    }
    l[0] = add2(sub2(make_float2(a, y[0].x), y[0]), sub2(make_float2(r0, r1), y[0]));
    l[1] = add2(sub2(make_float2(y[0].y, y[1].x), y[1]), sub2(make_float2(r2, b), y[1]));
  };
  const int js = max(j0 - P, u0);
  // ring: [slot][p1, p2 of row jj, hi, lo of row jj - P][lane]
  const size_t off = ok ? m0 : 0;
  const float* f1 = A.p1 + (size_t)js * ld + off;  // row jj of the planes, row jj - P of the state
  const float* f2 = TWO ? A.p2 + (size_t)js * ld + off : nullptr;
  const float* fh = A.hi + off + ((ptrdiff_t)js - P) * (ptrdiff_t)ld;
  const float* fl = A.lo + off + ((ptrdiff_t)js - P) * (ptrdiff_t)ld;
  const int jb = min(j1 + P, u1);  // rows of b
  int jf = js;                     // next row to fetch
  auto fetch = [&](int slot) {
    float4* r = ring + 4 * slot * 32 + lane;
    if (jf < jb) {
      cp16(r, f1, ok);
      if (TWO) cp16(r + 32, f2, ok);
    }
    if (out && jf >= j0 + P && jf < j1 + P) {
      if (!PAIR) cp16(r + 64, fh, true);
      cp16(r + 96, fl, true);
    }
    cp_commit();
    f1 += ld;
    if (TWO) f2 += ld;
    fh += ld;
    fl += ld;
    ++jf;
  };
#pragma unroll
  for (int t = 0; t < kAhead; ++t) fetch(t);
  int rd = 0, wr = kAhead;
  const float2 z2 = bc2(0.0f);
  float2 b[P + 1][2], w[P][2][2];  // b[l]: row jj - l; w[l][1]: level l at row jj - l - 1, w[l][0] above it
#pragma unroll
  for (int l = 0; l <= P; ++l) b[l][0] = b[l][1] = z2;
#pragma unroll
  for (int l = 0; l < P; ++l) w[l][0][0] = w[l][0][1] = w[l][1][0] = w[l][1][1] = z2;
  float2 x[2][2], yn[2], xr[2], rn[2];  // PAIR: w[P - 1] holds l of the last level's y, x that y, xr what it rounded away
  x[0][0] = x[0][1] = x[1][0] = x[1][1] = yn[0] = yn[1] = xr[0] = xr[1] = rn[0] = rn[1] = z2;
  float2 ql[P];  // (a batch's arguments sit in shared memory, read again after every asynchronous copy)
#pragma unroll
  for (int l = 0; l < P - 1; ++l) ql[l] = bc2(A.q[l]);
  const float2 s_hi = bc2(A.s_hi), n_hi = bc2(-A.s_hi), s_lo = bc2(A.s_lo), l_hi = bc2(A.l_hi), l_lo = bc2(A.l_lo);
  float* ph = (PAIR ? A.out : A.hi) + off + (size_t)j0 * ld;
  float* pl = A.lo + off + (size_t)j0 * ld;
  const int jend = j1 + P;
#pragma unroll 1
  for (int jj = js; jj < jend; ++jj) {
    cp_wait<kAhead - 1>();
    const float4* r = ring + 4 * rd * 32 + lane;
    fetch(wr);
    rd = rd == kRing - 1 ? 0 : rd + 1;
    wr = wr == kRing - 1 ? 0 : wr + 1;
    float2 wn[2];
#pragma unroll
    for (int l = P; l > 0; --l)
#pragma unroll
      for (int k = 0; k < 2; ++k) b[l][k] = b[l - 1][k];
    if (jj < u1) {  // b of row jj
      const float4 c = r[0];
      b[0][0] = make_float2(c.x, c.y);
      b[0][1] = make_float2(c.z, c.w);
      if (TWO) {
        const float4 e = r[32];
        b[0][0] = add2(b[0][0], make_float2(e.x, e.y));
        b[0][1] = add2(b[0][1], make_float2(e.z, e.w));
      }
      mask(b[0]);
      wsum(b[0], wn);
    } else {
      b[0][0] = b[0][1] = wn[0] = wn[1] = z2;
    }
    // level l + 1 at row t = jj - l - 1 from w of level l at rows t - 1, t, t + 1
#pragma unroll
    for (int l = 0; l < P; ++l) {
      const int t = jj - l - 1;
      float2 tt[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (PAIR && l == P - 1) {  // (T - 36) y = 6 (L_x + L_y) y + L_y L_x y
          float2 yu = x[0][k], yd = yn[k], lu = w[l][0][k], ld = wn[k];
          if (KIND == KIND_HX && (t == u0 || t == u1 - 1)) {  // the ghost row equals the wall row
            yu = t == u0 ? x[1][k] : yu;
            lu = t == u0 ? w[l][1][k] : lu;
            yd = t == u1 - 1 ? x[1][k] : yd;
            ld = t == u1 - 1 ? w[l][1][k] : ld;
          }
          const float2 ly = add2(sub2(yu, x[1][k]), sub2(yd, x[1][k]));
          tt[k] = fma2(bc2(6.0f), add2(w[l][1][k], ly), add2(sub2(lu, w[l][1][k]), sub2(ld, w[l][1][k])));
          x[0][k] = x[1][k];
          x[1][k] = yn[k];
        } else {
          float2 ud = add2(w[l][0][k], wn[k]);
          if (KIND == KIND_HX && (t == u0 || t == u1 - 1))  // the ghost row equals the wall row
            ud = add2(w[l][1][k], t == u0 ? wn[k] : w[l][0][k]);
          tt[k] = fma2(four, w[l][1][k], ud);
        }
        w[l][0][k] = w[l][1][k];
        w[l][1][k] = wn[k];
      }
      if (l < P - 1) {
        if ((unsigned)(t - u0) < (unsigned)(u1 - u0)) {
          float2 y[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            y[k] = fma2(ql[l], tt[k], b[l + 1][k]);
            if (PAIR && l == P - 2) rn[k] = fma2(ql[l], tt[k], sub2(b[l + 1][k], y[k]));
          }
          mask(y);
          if (PAIR && l == P - 2) {
            yn[0] = y[0];
            yn[1] = y[1];
            lapx(y, wn);
          } else {
            wsum(y, wn);
          }
        } else {
          wn[0] = wn[1] = yn[0] = yn[1] = rn[0] = rn[1] = z2;
        }
      } else if (t >= j0) {
        if (out) {
          const float4 sl = r[96];
          float2 o[2] = {make_float2(sl.x, sl.y), make_float2(sl.z, sl.w)};
          if (PAIR) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              // with what y rounded away and the field's low part, of which the point itself is most of the sum
              const float2 T = fma2(bc2(-20.0f), add2(xr[k], o[k]), tt[k]);
              o[k] = fma2(l_hi, T, fma2(l_lo, T, o[k]));
            }
            if (!EDGE || m0 + 4 <= M) {
              *reinterpret_cast<float4*>(ph) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
            } else {
              const float ov[3] = {o[0].x, o[0].y, o[1].x};
#pragma unroll
              for (int k = 0; k < 3; ++k)
                if (in[k]) ph[k] = ov[k];
            }
          } else {
            const float4 sh = r[64];
            float2 h[2] = {make_float2(sh.x, sh.y), make_float2(sh.z, sh.w)};
#pragma unroll
            for (int k = 0; k < 2; ++k) ff_add_scaled(h[k], o[k], b[P][k], tt[k], s_hi, n_hi, s_lo, l_hi, l_lo);
            if (!EDGE || m0 + 4 <= M) {
              *reinterpret_cast<float4*>(ph) = make_float4(h[0].x, h[0].y, h[1].x, h[1].y);
              *reinterpret_cast<float4*>(pl) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
            } else {
              const float hv[3] = {h[0].x, h[0].y, h[1].x}, ov[3] = {o[0].x, o[0].y, o[1].x};
#pragma unroll
              for (int k = 0; k < 3; ++k)
                if (in[k]) {
                  ph[k] = hv[k];
                  pl[k] = ov[k];
                }
            }
          }
        }
        ph += ld;
        pl += ld;
      }
    }
    xr[0] = rn[0];
    xr[1] = rn[1];
  }
}

template <int P, bool PAIR = false>
__device__ __forceinline__ void s_item(const SArgs& A, float4* ring, int item) {
  if (item >= A.nstrip * A.nblk) return;
  const int blk = item / A.nstrip, strip = item - blk * A.nstrip;
  const bool edge = strip == 0 || A.M - 1 < SOUT * strip - SHALO + 127;
  if (A.kind == KIND_E) {
    if (edge) s_block<P, KIND_E, true, PAIR>(A, ring, strip, blk);
    else s_block<P, KIND_E, false, PAIR>(A, ring, strip, blk);
  } else if (A.kind == KIND_HX) {
    if (edge) s_block<P, KIND_HX, true, PAIR>(A, ring, strip, blk);
    else s_block<P, KIND_HX, false, PAIR>(A, ring, strip, blk);
  } else {
    if (edge) s_block<P, KIND_HY, true, PAIR>(A, ring, strip, blk);
    else s_block<P, KIND_HY, false, PAIR>(A, ring, strip, blk);
  }
}

}  // namespace

}  // namespace ms
