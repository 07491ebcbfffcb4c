// FP32_REFINED step of 2D grids (k_tiled.cu): warps that walk along y, two launches per half-step; and constants
// shared with the other FP32 paths.
#pragma once

#include <string>

#include "ms_internal.h"

namespace ms {

constexpr int kBand32Max = 12;   // largest half-width of the FP32 band tables
constexpr int kMaxSweeps32 = 6;  // largest Richardson sweep count ms_solver_sweeps grants in 2D

// Coefficients of the FP32 step of a grid (k_mixed.cu), split hi + lo: 12 beta, 6 c1 h^2, the Richardson
// relaxation of the sweeps after a transform solve, and the increment scales 12 Z / r and 12 / (r Z).
struct MixedConsts {
  float cb_hi, cb_lo, d_hi, d_lo, omega, sE_hi, sE_lo, sH_hi, sH_lo;
};
MixedConsts mixed_consts(const ms_grid* g);

// The right-hand sides of the walk kernels are those of 6 h^2 P1 x = b over this factor, (1 - rho)^2
// with rho the FP32 root: the recurrences give A^{-1} d up to it, and the increment scales carry it.
double walk_rhs_scale();
// The factor of a 2D grid's planes: that one, or 1 on grids of at most kTinyN cells (explicit rows of A^{-1}).
// One FP32 number 1 / (1 - rho)^2 on every right-hand side would shift every frequency of those grids by 8e-8.
double plane_rhs_scale(const ms_grid* g);

// Segments of a line of M >= 16 rows that warps walk along: about `rows` rows each, `chunk` rows (a multiple
// of 8) but for the last one, which is [rb, M), a multiple of 8 rows; every other one ends at least 8
// rows before the line's end, and the first holds the first 8 rows.
void line_segments(int M, int rows, int* nseg, int* chunk, int* rb);

// FP32 planes of 2D grids: rows of ld floats (a multiple of 32), with the first unknown column of every
// field on a 16-byte boundary.  plane_floats: floats of one plane; plane_origin: offset of point (0, 0)
// of field f in it.
int walk_ld(int N);
size_t plane_floats(int N);
size_t plane_origin(int f);

// The FP32 Pade end corrections and the solve polynomial of a grid; MS_ENOTCONV if none is held.
ms_status walk_setup(ms_grid* g);

// step 0 (Step 1): the derivatives into the E_z planes s32[4] (along y) and s32[1] (along x); step 1
// (Step 2): into s32[2] (H_x, along y) and s32[3] (H_y, along x).  src_hi, src_lo != NULL: Step 2 from that
// already filtered E_z-shaped field.
void walk_d(ms_grid* g, int step, const float* src_hi = nullptr, const float* src_lo = nullptr);
// The solve and the state update of the half-step's fields from those planes.
void walk_s(ms_grid* g, int step);
constexpr int kTinyN = 16;

// Arguments of the solve of field f on its own (k_walk_dev.cuh), with the row blocks of a launch over
// nfields fields.
struct SArgs;
SArgs make_s(const ms_grid* g, int f, const float* p1, const float* p2, int nfields);

// One launch per kernel for many cavities: per-cavity arguments and (cavity, item) work lists.
struct YArgs;
struct XArgs;
struct WalkBatch {
  YArgs* d_y = nullptr;    // [Step 1 of every cavity][Step 2]
  XArgs* d_x = nullptr;    // the same
  SArgs* d_s = nullptr;    // [E_z of every cavity][H_x][H_y]
  int* d_work = nullptr;   // (argument, first item) pairs of the step's four launches
  int ny = 0;              // arguments of derivatives along x are numbered from ny
  int n[4] = {};
  size_t off[4] = {};
  int P = 0;  // solve levels
  int resident_d = 0, resident_s = 0;
};
// order: 0 cavity by cavity, 1 the strips at a wall of every cavity first, 2 largest cavities first.
// persistent: launch only as many blocks as are resident at once, each striding over the work list.
int walk_batch_build(ms_grid* const* cav, int count, int order, WalkBatch* wb, std::string* err);
void walk_batch_step(const WalkBatch& wb, cudaStream_t st, int persistent);
void walk_batch_free(WalkBatch* wb);

}  // namespace ms
