// stream.cu -- temporal blocking in the register file: the STREAM schedule.
//
// The paper's deep temporal blocking (Zhang et al., GPGPU'23, Sections 3.1 and
// 3.3, Figure 1) keeps a tile on chip for several time steps so that one trip
// through HBM carries many steps.  On GB300 the register file (256 KB per SM)
// is larger than shared memory (228 KB), so this schedule keeps the time steps
// of a tile in registers; shared memory only stages the input rows on their
// way in (a ring of a few rows per warp, filled by asynchronous copies).
//
// Each warp owns one column band of the grid, 32 lanes x one 16-byte vector
// (128 FP32 / 64 FP64 columns), and a run of rows, and sweeps the run from top
// to bottom once per pass.  A pass advances M time steps as a pipeline: when
// row i of the pass's input arrives, the warp evaluates step 1 of row i-1,
// step 2 of row i-2, ..., step M of row i-M, each from the two rows of the step
// below that it keeps in registers and the row that step has just produced
// (the update of row r at step t reads rows r-1, r and r+1 of step t-1).  Row
// i-M at step M leaves for HBM.  The x +- 1 neighbours come from the adjacent
// lanes by shuffles; beyond the warp's two edges the missing neighbours spoil
// one more column per step, so a band evaluates 32V columns and stores the
// middle 32V - 2G (G >= M, a multiple of V): an overlapped halo in x, as the
// paper's tiles have.  In y, a run starts M rows above its first stored row
// and ends M rows below its last, so the runs of a band overlap by 2M rows.
// The ring (one cell deep, held constant) is kept by holding a ring cell's
// value at every step: ring columns in the bands that contain one (a select
// per cell), ring rows in the few iterations of a run where a step reaches row
// 0 or row ny+1 (a uniform test).  Cells outside the logical array never
// reach a stored cell: the held ring separates them.
//
// Every cell is evaluated exactly as the one-step kernel evaluates it: FP32 by
// the chain of stencil() in common.cuh (here two cells per paired FP32 multiply
// and fused multiply-add, each element rounded as the scalar instruction
// rounds it), FP64 by stencil_cell() with the integer path on the same cells, or the
// same values in windowed fixed point where a unit's values allow it (window.cuh).
// So the results are bit-identical to every other kernel of the library.
//
// One launch per pass (a pass waits for the one before it; a run of S steps is
// ceil(S / M) passes, the first one taking the remainder, which at two FP64 steps a
// pass the one-step kernel takes), with several waves of (band, run) units so that
// the block scheduler balances the SMs.  Per cell update HBM carries 2 * sizeof(T) * (1 + overlap) / M bytes.
// The same pipeline serves the 3x3 box (j2d9pt) and, for state-keeping runs,
// stores every step's rows instead of the last step's only.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "window.cuh"

namespace j2d {

// Warps per block (each warp is independent): FP32 one, so that registers
// are granted warp by warp (FP32 16384^2, k = 8: 3808 against 3228 GCells/s
// with four-warp blocks); FP64 four (155.6 against 161.2 with one).
template <typename T> struct WarpsOf { static constexpr int W = 1; };
template <> struct WarpsOf<double> { static constexpr int W = 4; };
inline int stream_warps(j2d_dtype dt) { return dt == J2D_F64 ? WarpsOf<double>::W : WarpsOf<float>::W; }

struct StreamParams {
  const void *in;
  void *out;
  long pitch;   // elements per row
  int off;      // element offset of logical column 0
  int nx, ny;
  int G;        // halo columns on each side of a band (a multiple of V, >= the pass's steps)
  int vw;       // stored (valid) columns per band: 32V - 2G
  int bands;    // column bands
  int H;        // rows stored per unit
  int runs;     // units per band
  int meff;     // steps of this pass (<= M: steps t > meff leave rows unchanged)
  void *keep;   // keeping every state: step t's rows go to keep + (t - 1) * keep_stride
  long keep_stride;
  int ipath;    // FP64: integer path on
  long nelem;   // elements of each buffer ((ny + 2) * pitch), for the checked build
  int *status;  // checked build: J2D_ERR_BOUNDS is recorded here
  double w[9];  // five-point: W, E, S, C, N; box: the nine weights, rows y-1, y, y+1, columns x-1, x, x+1
  WindowWeights win;       // FP64: the weights in windowed fixed point (window.cuh), five-point
  WindowWeightsN<9> win9;  // and box
};

// ---- one lane's 16-byte vector of a row, in registers -------------------------

// FP32: four columns v0..v3 held as two pairs a = (v0, v2), b = (v1, v3), so
// that the x - 1 and x + 1 operands of each pair are pairs too (mostly the
// other pair), and one paired instruction evaluates two cells.
struct RowF {
  float2 a, b;
};
struct WeightsF {
  float2 w, e, s, c, n;  // each weight in both halves
};

__device__ __forceinline__ RowF row_zero(RowF *) { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ void row_store(float *p, const RowF &r) {
  *reinterpret_cast<float4 *>(p) = make_float4(r.a.x, r.b.x, r.a.y, r.b.y);
}
// Keep the cells whose bit is set in m (bit v: column v of the vector) at c.
__device__ __forceinline__ RowF row_hold(RowF n, const RowF &c, unsigned m) {
  if (m & 1u) n.a.x = c.a.x;
  if (m & 2u) n.b.x = c.b.x;
  if (m & 4u) n.a.y = c.a.y;
  if (m & 8u) n.b.y = c.b.y;
  return n;
}

// One step of the four cells of row c (ym: the row above at the same step,
// yp: the row below), in the order of stencil(): y-1, centre, x-1, x+1, y+1.
// The two operand pairs that would mix registers of both pairs (x-1 of
// (v0, v2) is (L, v1); x+1 of (v1, v3) is (v2, R)) take two scalar FMAs each
// instead of a move into a register pair and one paired FMA.
__device__ __forceinline__ RowF row_step(const WeightsF &k, const RowF &ym, const RowF &c, const RowF &yp) {
  const float L = __shfl_up_sync(0xffffffffu, c.b.y, 1);    // column x0 - 1: the left lane's v3
  const float R = __shfl_down_sync(0xffffffffu, c.a.x, 1);  // column x0 + 4: the right lane's v0
  float2 ra = __fmul2_rn(k.s, ym.a);
  ra = __ffma2_rn(k.c, c.a, ra);
  ra.x = __fmaf_rn(k.w.x, L, ra.x);      // x-1 of v0
  ra.y = __fmaf_rn(k.w.x, c.b.x, ra.y);  // x-1 of v2
  ra = __ffma2_rn(k.e, c.b, ra);         // x+1 of (v0, v2)
  ra = __ffma2_rn(k.n, yp.a, ra);
  float2 rb = __fmul2_rn(k.s, ym.b);
  rb = __ffma2_rn(k.c, c.b, rb);
  rb = __ffma2_rn(k.w, c.a, rb);         // x-1 of (v1, v3)
  rb.x = __fmaf_rn(k.e.x, c.a.y, rb.x);  // x+1 of v1
  rb.y = __fmaf_rn(k.e.x, R, rb.y);      // x+1 of v3
  rb = __ffma2_rn(k.n, yp.b, rb);
  return {ra, rb};
}

// FP64: two columns.
struct RowD {
  double a, b;
};
struct WeightsD {
  Links<double> l;
  ExactW u;
};

__device__ __forceinline__ RowD row_zero(RowD *) { return {0.0, 0.0}; }
__device__ __forceinline__ void row_store(double *p, const RowD &r) {
  *reinterpret_cast<double2 *>(p) = make_double2(r.a, r.b);
}
__device__ __forceinline__ RowD row_hold(RowD n, const RowD &c, unsigned m) {
  if (m & 1u) n.a = c.a;
  if (m & 2u) n.b = c.b;
  return n;
}
// ea, eb: the row's two cells take the integer path (exact_cell(): the same
// cells as in every other kernel).
__device__ __forceinline__ RowD row_step(const WeightsD &k, const RowD &ym, const RowD &c, const RowD &yp,
                                         bool ea, bool eb) {
  const double L = __shfl_up_sync(0xffffffffu, c.b, 1);
  const double R = __shfl_down_sync(0xffffffffu, c.a, 1);
  return {stencil_cell(k.l, k.u, ea, L, c.b, ym.a, c.a, yp.a), stencil_cell(k.l, k.u, eb, c.a, R, ym.b, c.b, yp.b)};
}

// ---- the 3x3 box (j2d9pt): every row also carries its outer neighbours ---------
// A box cell reads the x - 1 and x + 1 columns of all three rows, so a row's
// two values beyond the lane (L: column x0 - 1, R: the column after the
// lane's last) are taken by shuffles once, when the row is produced, and
// travel with it through the three steps that read it.  The chain order is
// that of stencil_box() in common.cuh.
struct RowF9 {
  float2 a, b;  // (v0, v2), (v1, v3) as in RowF
  float L, R;
};
struct WeightsF9 {
  float2 w[9];  // Box9 chain order, each weight in both halves
};
struct RowD9 {
  double a, b, L, R;
};
struct WeightsD9 {
  Box9<double> b;
  ExactWN<9> u;
};

__device__ __forceinline__ RowF9 row_zero(RowF9 *) { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f), 0.f, 0.f}; }
__device__ __forceinline__ RowD9 row_zero(RowD9 *) { return {0.0, 0.0, 0.0, 0.0}; }
__device__ __forceinline__ void row_nbrs(RowF9 &r) {
  r.L = __shfl_up_sync(0xffffffffu, r.b.y, 1);
  r.R = __shfl_down_sync(0xffffffffu, r.a.x, 1);
}
__device__ __forceinline__ void row_nbrs(RowD9 &r) {
  r.L = __shfl_up_sync(0xffffffffu, r.b, 1);
  r.R = __shfl_down_sync(0xffffffffu, r.a, 1);
}
__device__ __forceinline__ void row_store(float *p, const RowF9 &r) {
  *reinterpret_cast<float4 *>(p) = make_float4(r.a.x, r.b.x, r.a.y, r.b.y);
}
__device__ __forceinline__ void row_store(double *p, const RowD9 &r) {
  *reinterpret_cast<double2 *>(p) = make_double2(r.a, r.b);
}
__device__ __forceinline__ RowF9 row_hold(RowF9 n, const RowF9 &c, unsigned m) {
  if (m & 1u) n.a.x = c.a.x;
  if (m & 2u) n.b.x = c.b.x;
  if (m & 4u) n.a.y = c.a.y;
  if (m & 8u) n.b.y = c.b.y;
  return n;
}
__device__ __forceinline__ RowD9 row_hold(RowD9 n, const RowD9 &c, unsigned m) {
  if (m & 1u) n.a = c.a;
  if (m & 2u) n.b = c.b;
  return n;
}

// Terms in chain order: (y-1, x), (y-1, x-1), (y-1, x+1), (y, x), (y, x-1),
// (y, x+1), (y+1, x), (y+1, x-1), (y+1, x+1).  For the pair (v0, v2) the
// x - 1 operands (L, v1) mix the pairs and take scalar FMAs, the x + 1
// operands are the pair (v1, v3); for (v1, v3) the x - 1 operands are
// (v0, v2) and the x + 1 operands (v2, R) take scalar FMAs.
__device__ __forceinline__ RowF9 row_step9(const WeightsF9 &k, const RowF9 &ym, const RowF9 &c, const RowF9 &yp) {
  float2 ra = __fmul2_rn(k.w[0], ym.a);
  ra.x = __fmaf_rn(k.w[1].x, ym.L, ra.x);
  ra.y = __fmaf_rn(k.w[1].x, ym.b.x, ra.y);
  ra = __ffma2_rn(k.w[2], ym.b, ra);
  ra = __ffma2_rn(k.w[3], c.a, ra);
  ra.x = __fmaf_rn(k.w[4].x, c.L, ra.x);
  ra.y = __fmaf_rn(k.w[4].x, c.b.x, ra.y);
  ra = __ffma2_rn(k.w[5], c.b, ra);
  ra = __ffma2_rn(k.w[6], yp.a, ra);
  ra.x = __fmaf_rn(k.w[7].x, yp.L, ra.x);
  ra.y = __fmaf_rn(k.w[7].x, yp.b.x, ra.y);
  ra = __ffma2_rn(k.w[8], yp.b, ra);
  float2 rb = __fmul2_rn(k.w[0], ym.b);
  rb = __ffma2_rn(k.w[1], ym.a, rb);
  rb.x = __fmaf_rn(k.w[2].x, ym.a.y, rb.x);
  rb.y = __fmaf_rn(k.w[2].x, ym.R, rb.y);
  rb = __ffma2_rn(k.w[3], c.b, rb);
  rb = __ffma2_rn(k.w[4], c.a, rb);
  rb.x = __fmaf_rn(k.w[5].x, c.a.y, rb.x);
  rb.y = __fmaf_rn(k.w[5].x, c.R, rb.y);
  rb = __ffma2_rn(k.w[6], yp.b, rb);
  rb = __ffma2_rn(k.w[7], yp.a, rb);
  rb.x = __fmaf_rn(k.w[8].x, yp.a.y, rb.x);
  rb.y = __fmaf_rn(k.w[8].x, yp.R, rb.y);
  return {ra, rb, 0.f, 0.f};
}
// SKIP (windowed kernels, whose general sweep is for fields of both signs first of all):
// the integer path wants nine positive normal values, which few of a row's 64 cells then
// have, and a row without any skips the attempt (300 instructions a cell).  The test
// also takes the two cells one after the other: deeper pipelines lose by it (k = 4,
// 9000x8000 x 4 of both signs 7617 -> 9903 us).
template <bool SKIP>
__device__ __forceinline__ RowD9 row_step9(const WeightsD9 &k, const RowD9 &ym, const RowD9 &c, const RowD9 &yp,
                                           bool ea, bool eb) {
  if (SKIP && (ea || eb)) {
    const int lo = min(min(__double2hiint(ym.a), __double2hiint(ym.b)),
                       min(min(__double2hiint(c.a), __double2hiint(c.b)), min(__double2hiint(yp.a), __double2hiint(yp.b))));
    const int la = min(lo, min(__double2hiint(ym.L), min(__double2hiint(c.L), __double2hiint(yp.L))));
    const int lb = min(lo, min(__double2hiint(ym.R), min(__double2hiint(c.R), __double2hiint(yp.R))));
    if (!__any_sync(0xffffffffu, max(la, lb) >= 0x100000)) ea = eb = false;
  }
  return {stencil_box_cell(k.b, k.u, ea, ym.L, ym.a, ym.b, c.L, c.a, c.b, yp.L, yp.a, yp.b),
          stencil_box_cell(k.b, k.u, eb, ym.a, ym.b, ym.R, c.a, c.b, c.R, yp.a, yp.b, yp.R), 0.0, 0.0};
}

template <typename T, int SH> struct RowOf;
template <> struct RowOf<float, 5> { using R = RowF; using W = WeightsF; };
template <> struct RowOf<double, 5> { using R = RowD; using W = WeightsD; };
template <> struct RowOf<float, 9> { using R = RowF9; using W = WeightsF9; };
template <> struct RowOf<double, 9> { using R = RowD9; using W = WeightsD9; };

// Five-point rows take their neighbours when they are read.
__device__ __forceinline__ void row_nbrs(RowF &) {}
__device__ __forceinline__ void row_nbrs(RowD &) {}

// ea, eb: the lane's first / second cell takes the integer path (FP64; known
// at compile time where the trip's row phases are: the column parities of a
// lane's two cells are fixed, its first column being odd).
template <bool SKIP>
__device__ __forceinline__ RowF step_any(const WeightsF &k, const RowF &ym, const RowF &c, const RowF &yp, bool,
                                         bool) {
  return row_step(k, ym, c, yp);
}
template <bool SKIP>
__device__ __forceinline__ RowD step_any(const WeightsD &k, const RowD &ym, const RowD &c, const RowD &yp, bool ea,
                                         bool eb) {
  return row_step(k, ym, c, yp, ea, eb);
}
template <bool SKIP>
__device__ __forceinline__ RowF9 step_any(const WeightsF9 &k, const RowF9 &ym, const RowF9 &c, const RowF9 &yp, bool,
                                          bool) {
  return row_step9(k, ym, c, yp);
}
template <bool SKIP>
__device__ __forceinline__ RowD9 step_any(const WeightsD9 &k, const RowD9 &ym, const RowD9 &c, const RowD9 &yp,
                                          bool ea, bool eb) {
  return row_step9<SKIP>(k, ym, c, yp, ea, eb);
}

// In the checked build, is [e, e + V) inside the buffer of nelem elements?
__device__ __forceinline__ bool stream_ok(long e, int V, const StreamParams &p) {
  if (!kChecked) return true;
  const bool ok = e >= 0 && e + V <= p.nelem;
  if (!ok) set_error(p.status, DEV_BOUNDS);
  return ok;
}

// Kernels whose units run in windowed fixed point.
template <typename T, int M, bool IP, bool KEEP, int SH>
constexpr bool kWindowed = std::is_same<T, double>::value && M <= (SH == 5 ? 4 : 2) && IP;

// The pipeline of one warp: for each step t = 0..M-1 the two most recent rows
// of step t (A: the older, B: the newer).
// KEEP: every step's rows are stored (to p.keep), not only the last step's.
template <typename T, int M, bool EDGE, bool IP, bool KEEP, int SH> struct Pipe {
  using R = typename RowOf<T, SH>::R;
  using W = typename RowOf<T, SH>::W;
  R A[M], B[M];
  const W &k;
  const StreamParams &p;
  T *out;
  long e0;        // element offset of this lane's vector within a row
  int x0;         // logical column of the vector's first element
  unsigned hold;  // ring columns in this lane's vector
  bool st;        // this lane's vector is stored
  int y0, y1;     // stored rows [y0, y1)
  T *dst;         // FP32: this lane's vector of the row an iteration finishes (set by the sweep, advanced a row each time)

  __device__ __forceinline__ Pipe(const W &k_, const StreamParams &p_, T *out_, long e0_, int x0_, unsigned hold_,
                                  bool st_, int y0_, int y1_)
      : k(k_), p(p_), out(out_), e0(e0_), x0(x0_), hold(hold_), st(st_), y0(y0_), y1(y1_) {
#pragma unroll
    for (int t = 0; t < M; ++t) {
      A[t] = row_zero((R *)nullptr);
      B[t] = row_zero((R *)nullptr);
    }
  }

  // Iteration i: row i of step 0 arrives; steps 1..M advance one row each.
  // CHK: some step reaches ring row 0 or ny + 1 in this iteration, the row it
  // finishes may not be one to store, or the pass has fewer than M steps (steps
  // beyond meff pass their rows through).
  // ph: i mod 4 when the caller knows it at compile time (FP64 trips), so
  // that each step's integer-path choice (exact_cell(): rows y mod 4 in
  // {0, 1}) is a constant; -1 otherwise.
  template <bool CHK> __device__ __forceinline__ void iter(int i, R cur, int ph) {
#pragma unroll
    for (int t = 1; t <= M; ++t) {
      const int r = i - t;  // the row step t evaluates
      const int yy = ph >= 0 ? ph - t + 4 * M : r;  // the row, or a row of the same phase mod 4
      R n = step_any<kWindowed<T, M, IP, KEEP, SH>>(k, A[t - 1], B[t - 1], cur, IP && exact_cell(1, yy, true), IP && exact_cell(0, yy, true));
      if (EDGE) n = row_hold(n, B[t - 1], hold);
      if (CHK && (r == 0 || r == p.ny + 1 || t > p.meff)) n = B[t - 1];
      if (SH == 9 && t < M) row_nbrs(n);  // read with its neighbours by steps t + 1 (three times)
      A[t - 1] = B[t - 1];
      B[t - 1] = cur;
      cur = n;
      if (KEEP && t <= p.meff && st && r >= y0 && r < y1) {
        const long e = (long)r * p.pitch + e0;
        if (stream_ok(e, VecOf<T>::V, p)) row_store(static_cast<T *>(p.keep) + (t - 1) * p.keep_stride + e, n);
      }
    }
    const int r = i - M;
    if constexpr (sizeof(T) == 8) {
      if (!KEEP && st && r >= y0 && r < y1) {
        const long e = (long)r * p.pitch + e0;
        if (stream_ok(e, VecOf<T>::V, p)) row_store(out + e, cur);
      }
    } else if (!KEEP) {
      if (st && (!CHK || (r >= y0 && r < y1)) && stream_ok(dst - out, VecOf<T>::V, p)) row_store(dst, cur);
      dst += p.pitch;
    }
  }
};

// Input rows reach the warp through a ring of shared-memory slots of one row
// each (16 bytes per lane), filled by asynchronous copies kAhead rows ahead of
// use: the copies wait in the memory system instead of in registers.  Each
// lane copies and reads back only its own 16 bytes, so the ring needs no
// synchronisation beyond the lane's own copy groups.  The ring has two trips'
// worth of slots (2U >= kAhead + 2), so a slot is refilled at least two
// iterations after it was read.
constexpr int kAhead = 4;

// Iterations per trip of the sweep loop.  FP32: 3, the period of a step's
// three-row window, so the unrolled trip rotates its registers without moves.
// FP64: 4, the period of the integer-path row pattern (trips start on rows 0
// mod 4, so each step's choice between the integer path and the FMA chain is
// known at compile time and the trip is straight-line code).
template <typename T> struct TripOf { static constexpr int U = 3; };
template <> struct TripOf<double> { static constexpr int U = 4; };
constexpr int kStageMax = 8;  // slots per warp, the largest 2U

__device__ __forceinline__ void stage_copy(uint32_t dst, const void *src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory"); }
__device__ __forceinline__ void stage_drain() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Start the copy of input row i into the slot at shared address dst (rows
// past the ring row ny + 1, and vectors outside the row, read as zero).
template <typename T>
__device__ __forceinline__ void issue_row(const T *in, const StreamParams &p, int i, long e0, bool live, uint32_t dst) {
  bool on = live && i >= 0 && i <= p.ny + 1;
  const long e = on ? (long)i * p.pitch + e0 : 0;
  if (on) on = stream_ok(e, VecOf<T>::V, p);
  stage_copy(dst, in + (on ? e : 0), on);
}

__device__ __forceinline__ RowF read_slot(const float4 *q, RowF *) {
  const float4 v = *q;
  return {make_float2(v.x, v.z), make_float2(v.y, v.w)};
}
__device__ __forceinline__ RowF9 read_slot(const float4 *q, RowF9 *) {
  const float4 v = *q;
  RowF9 r = {make_float2(v.x, v.z), make_float2(v.y, v.w), 0.f, 0.f};
  row_nbrs(r);
  return r;
}
__device__ __forceinline__ RowD9 read_slot(const float4 *q, RowD9 *) {
  const double2 v = *reinterpret_cast<const double2 *>(q);
  RowD9 r = {v.x, v.y, 0.0, 0.0};
  row_nbrs(r);
  return r;
}
__device__ __forceinline__ RowD read_slot(const float4 *q, RowD *) {
  const double2 v = *reinterpret_cast<const double2 *>(q);
  return {v.x, v.y};
}

template <typename T, int M, bool EDGE, bool IP, bool KEEP, int SH>
__device__ __forceinline__ void stream_sweep(const StreamParams &p, const typename RowOf<T, SH>::W &k, long e0, int x0,
                                             unsigned hold, bool live, bool st, int y0, int y1, float4 *ring) {
  using R = typename RowOf<T, SH>::R;
  constexpr int U = TripOf<T>::U;
  constexpr int S = 2 * U;  // slots
  static_assert(S >= kAhead + 2 && S <= kStageMax, "ring too small");
  const T *in = static_cast<const T *>(p.in);
  T *out = static_cast<T *>(p.out);
  Pipe<T, M, EDGE, IP, KEEP, SH> pipe(k, p, out, e0, x0, hold, st, y0, y1);
  // the first row the last stored row's pipeline needs; FP64 trips start on rows
  // congruent to PH mod 4, where a unit of whole trips (y0 = 1 + a multiple of 4)
  // needs its first
  constexpr int PH = (1 - M) & 3;
  int a = max(y0 - M, 0);
  if (U == 4) a = y0 - M - ((y0 - M - PH) & 3);
  const int iend = y1 + M;  // the last iteration stores row y1 - 1
  const bool short_pass = p.meff < M;
  // this lane's slot j is ring[32 * j]; row a + n sits in slot n mod S
  const uint32_t base = smem_u32(ring);
#pragma unroll
  for (int j = 0; j < kAhead; ++j) issue_row(in, p, a + j, e0, live, base + 512u * j);
  int s = 0;  // slot of row i: 0 or U
  if constexpr (sizeof(T) == 8) {
    // FP64: addresses from the row number (running ones cost registers these
    // kernels do not have: box k = 2, 16384^2, 92 -> 86 GCells/s)
    for (int i = a; i < iend; i += U) {
      if (short_pass || i <= M || i + U - 1 >= p.ny + 2) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          stage_wait();
          const R c = read_slot(ring + 32 * (s + u), (R *)nullptr);
          const int sn = s + u + kAhead;
          issue_row(in, p, i + u + kAhead, e0, live, base + 512u * (sn >= S ? sn - S : sn));
          pipe.template iter<true>(i + u, c, (u + PH) & 3);
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          stage_wait();
          const R c = read_slot(ring + 32 * (s + u), (R *)nullptr);
          const int sn = s + u + kAhead;
          issue_row(in, p, i + u + kAhead, e0, live, base + 512u * (sn >= S ? sn - S : sn));
          pipe.template iter<false>(i + u, c, (u + PH) & 3);
        }
      }
      s = s == 0 ? U : 0;
    }
  } else {
    // FP32: the copies' source (row i + kAhead) and the stored row's address
    // advance a row per iteration, and steady trips (every finished row stored, all
    // copied rows inside the grid, no step at a ring row) test nothing; a run's
    // first and last trips and short passes do (k = 8, 16384^2: 4260 -> 4670
    // GCells/s, of an issue-bound sweep)
    const long step = live ? p.pitch : 0;
    const T *src = in + (live ? (long)(a + kAhead) * p.pitch + e0 : 0);
    pipe.dst = out + ((long)(a - M) * p.pitch + e0);
    const int lo = max(y0 + M, M + 1), hi = short_pass ? -1 : min(y1 + M, p.ny + 2 - kAhead) - U;
    for (int i = a; i < iend; i += U) {
      if (i < lo || i > hi) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          stage_wait();
          const R c = read_slot(ring + 32 * (s + u), (R *)nullptr);
          const int sn = s + u + kAhead;
          bool on = live && i + u + kAhead <= p.ny + 1;
          if (on) on = stream_ok(src - in, VecOf<T>::V, p);
          stage_copy(base + 512u * (sn >= S ? sn - S : sn), on ? src : in, on);
          src += step;
          pipe.template iter<true>(i + u, c, -1);
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          stage_wait();
          const R c = read_slot(ring + 32 * (s + u), (R *)nullptr);
          const int sn = s + u + kAhead;
          const bool on = kChecked ? live && stream_ok(src - in, VecOf<T>::V, p) : live;
          stage_copy(base + 512u * (sn >= S ? sn - S : sn), kChecked && !on ? in : src, on);
          src += step;
          pipe.template iter<false>(i + u, c, -1);
        }
      }
      s = s == 0 ? U : 0;
    }
  }
  stage_drain();
}

// ---- FP64 in windowed fixed point (window.cuh) -----------------------------------
// The same pipeline with every row also in fixed point: rows y mod 4 in {0, 1} take
// the exact sum, the others the chain with its first two operations, on the
// integer pipes.  A sweep picks its window from the first interior rows it reads
// and stops before the first row that depends on an interior value outside it; the
// caller takes the next rows through stream_sweep() and comes back.  Ring values
// never change, so a sweep does not stop for them: a row beside a ring value
// outside the window takes its affected cells through the general evaluation.
struct RowX {
  double a, b;
  Fx xa, xb;
  bool ring_out;  // this lane's ring cell in the row is outside the window
};

// The chain's weights and the window of a shape.
template <int SH> struct WindowCoef {
  using L = Links<double>;
  static __device__ __forceinline__ const WindowWeights &window(const StreamParams &p) { return p.win; }
};
template <> struct WindowCoef<9> {
  using L = Box9<double>;
  static __device__ __forceinline__ const WindowWeightsN<9> &window(const StreamParams &p) { return p.win9; }
};
// Operations of the box's nine-term chain on the integer pipes: the y - 1 row's, so
// that its doubles are not needed again.
constexpr int kBoxHead = 3;

// Rows [y0, y1) of the unit; returns the first row not stored (y1: all are).
template <int M, bool EDGE, bool KEEP, int SH>
__device__ __forceinline__ int stream_sweep_window(const StreamParams &p, const typename WindowCoef<SH>::L &lk, long e0, int x0,
                                                   unsigned hold, bool live, bool st, int y0, int y1, float4 *ring) {
  constexpr int U = 4, S = 2 * U;
  const double *in = static_cast<const double *>(p.in);
  double *out = static_cast<double *>(p.out);
  const auto &w = WindowCoef<SH>::window(p);
  // trips start on rows congruent to 1 - M mod 4: where a run of whole trips
  // (y0 = 1 + run * H, H a multiple of 4) needs its first row
  constexpr int PH = (1 - M) & 3;
  const int a = y0 - M - ((y0 - M - PH) & 3);
  const int iend = y1 + M;
  const bool short_pass = p.meff < M;
  const uint32_t base = smem_u32(ring);
#pragma unroll
  for (int j = 0; j < kAhead; ++j) issue_row(in, p, a + j, e0, live && a + j >= 0, base + 512u * j);
  // columns of this lane outside the logical array hold a value of the window
  const bool oa = EDGE && (x0 < 0 || x0 > p.nx + 1), ob = EDGE && (x0 + 1 < 0 || x0 + 1 > p.nx + 1);
  if (EDGE) hold |= (oa ? 1u : 0u) | (ob ? 2u : 0u);
  // window: its top one binade above the largest value of the rows probed, the first
  // four interior ones and four spread over the unit, read here beside the copies
  // (whose first rows may lie above the grid: M = 4, the first unit of a band).  A value
  // of theirs below the window ends the attempt before its pipeline is filled.  With
  // the first rows alone, fields that rise down a unit ran out of its window, and steep ones
  // out of every other (64 steps of the box, 4096^2: a field growing by 2% a cell 24.0
  // -> 14.8 ms, where the skewed tiles take 15.0; 1 + sin / 2 with weights that leave four
  // binades 13.3 -> 9.5).
  const int r0 = max(a, 1);
  const bool ka = live && !(EDGE && (hold & 1u)), kb = live && !(EDGE && (hold & 2u));  // interior columns
  int top = 0, low = 0x7fffffff;  // high words: negative for negative values
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    double2 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = min(part == 0 ? r0 + j : y0 + (j + 1) * (y1 - 1 - y0) / 4, p.ny);
      const long e = (long)r * p.pitch + e0;
      v[j] = live && stream_ok(e, 2, p) ? __ldcg(reinterpret_cast<const double2 *>(in + e)) : make_double2(1.0, 1.0);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (ka) top = max(top, __double2hiint(v[j].x)), low = min(low, __double2hiint(v[j].x));
      if (kb) top = max(top, __double2hiint(v[j].y)), low = min(low, __double2hiint(v[j].y));
    }
  }
  Window q;
  if (!window_set(q, w, __reduce_max_sync(0xffffffffu, top) >> 20) || __any_sync(0xffffffffu, low < (int)q.cref)) {
    stage_drain();
    return y0;
  }
  const double dummy = window_dummy(q);
  RowX A[M], B[M];
  {
    uint32_t d = 0;
    const Fx x = window_conv(dummy, q, d);
#pragma unroll
    for (int t = 0; t < M; ++t) A[t] = B[t] = RowX{dummy, dummy, x, x, false};
  }
  // a row's fixed-point form; d collects the distances of its interior values
  // (none in the ring rows and beyond)
  auto conv = [&](RowX &r, bool ring_row, uint32_t &d) {
    uint32_t da = 0, db = 0;
    r.xa = window_conv(r.a, q, da);
    r.xb = window_conv(r.b, q, db);
    if (EDGE) {
      r.ring_out = ((hold & 1u) && da >= w.lim) || ((hold & 2u) && db >= w.lim);
      if (hold & 1u) da = 0;
      if (hold & 2u) db = 0;
    }
    if (!ring_row) d |= da | db;
  };
  // the asynchronous copies' source (row i + kAhead) and the stored row's
  // address, advanced a row per iteration
  const long step = live ? p.pitch : 0;
  const double *src = in + (live ? (long)(a + kAhead) * p.pitch + e0 : 0);
  double *dst = out + ((long)(a - M) * p.pitch + e0);
  // Iteration i: row i of step 0 arrives (ph = i mod 4); false: some interior
  // value is outside the window.  chk: a trip with rows that are not stored, near
  // the ring rows or past the grid, or a pass of fewer than M steps.
  auto iter = [&](int i, const float4 *slot, uint32_t fill, int ph, bool chk) -> bool {
    stage_wait();
    const double2 v = *reinterpret_cast<const double2 *>(slot);
    {
      bool on = live && (!chk || i + kAhead <= p.ny + 1);
      if (on) on = stream_ok(src - in, 2, p);
      stage_copy(fill, chk || kChecked ? (on ? src : in) : src, on);
      src += step;
    }
    RowX cur{v.x, v.y, {}, {}, false};
    if (EDGE && oa) cur.a = dummy;
    if (EDGE && ob) cur.b = dummy;
    if (chk && i > p.ny + 1) cur.a = cur.b = dummy;
    uint32_t d = 0;
    conv(cur, chk && (i < 1 || i > p.ny), d);
#pragma unroll
    for (int t = 1; t <= M; ++t) {
      const RowX &c = B[t - 1], &ym = A[t - 1];
      const int r = i - t;
      RowX n;
      n.ring_out = false;
      // a row beside the ring rows, or beside a ring column's value outside the window
      const bool beside = (chk && (r == 1 || r == p.ny)) ||
                          (EDGE && __any_sync(0xffffffffu, c.ring_out || (SH == 9 && (ym.ring_out || cur.ring_out))));
      const bool exact = ((ph - t + 4 * M) & 3) < 2;
      if constexpr (SH == 9) {
        // the nine neighbours' columns: L, a, b, R of each row
        if (exact) {
          const Fx mL = shfl_up_fx(ym.xb), mR = shfl_down_fx(ym.xa), cL = shfl_up_fx(c.xb), cR = shfl_down_fx(c.xa),
                   pL = shfl_up_fx(cur.xb), pR = shfl_down_fx(cur.xa);
          n.a = window_sum<9>(w, q, {ym.xa, mL, ym.xb, c.xa, cL, c.xb, cur.xa, pL, cur.xb});
          n.b = window_sum<9>(w, q, {ym.xb, ym.xa, mR, c.xb, c.xa, cR, cur.xb, cur.xa, pR});
        }
        const bool plain = (EDGE || chk) && beside;
        if (!exact || plain) {
          const double cL = __shfl_up_sync(0xffffffffu, c.b, 1), cR = __shfl_down_sync(0xffffffffu, c.a, 1);
          const double pL = __shfl_up_sync(0xffffffffu, cur.b, 1), pR = __shfl_down_sync(0xffffffffu, cur.a, 1);
          if (plain) {
            const double mL = __shfl_up_sync(0xffffffffu, ym.b, 1), mR = __shfl_down_sync(0xffffffffu, ym.a, 1);
            if (!exact) {
              n.a = stencil_box(lk, mL, ym.a, ym.b, cL, c.a, c.b, pL, cur.a, cur.b);
              n.b = stencil_box(lk, ym.a, ym.b, mR, c.a, c.b, cR, cur.a, cur.b, pR);
            } else {
              uint32_t da = 0, db = 0;
              for (double u : {mL, ym.a, ym.b, cL, c.a, c.b, pL, cur.a, cur.b}) da |= (uint32_t)__double2hiint(u) - q.cref;
              for (double u : {ym.a, ym.b, mR, c.a, c.b, cR, cur.a, cur.b, pR}) db |= (uint32_t)__double2hiint(u) - q.cref;
              if (da >= w.lim) n.a = general_box_cell(lk, mL, ym.a, ym.b, cL, c.a, c.b, pL, cur.a, cur.b);
              if (db >= w.lim) n.b = general_box_cell(lk, ym.a, ym.b, mR, c.a, c.b, cR, cur.a, cur.b, pR);
              __syncwarp();
            }
          } else {
            const Fx mL = shfl_up_fx(ym.xb), mR = shfl_down_fx(ym.xa);
            const double ca[6] = {c.a, cL, c.b, cur.a, pL, cur.b}, cb[6] = {c.b, c.a, cR, cur.b, cur.a, pR};
            n.a = window_head<kBoxHead>(w, q, {0, 1, 2}, {ym.xa, mL, ym.xb});
            n.b = window_head<kBoxHead>(w, q, {0, 1, 2}, {ym.xb, ym.xa, mR});
#pragma unroll
            for (int u = 0; u < 6; ++u) {
              n.a = fma_rn(lk.w[3 + u], ca[u], n.a);
              n.b = fma_rn(lk.w[3 + u], cb[u], n.b);
            }
          }
        }
      } else if (exact) {
        const Fx L = shfl_up_fx(c.xb), R = shfl_down_fx(c.xa);
        n.a = window_exact(w, q, L, c.xb, ym.xa, c.xa, cur.xa);
        n.b = window_exact(w, q, c.xa, R, ym.xb, c.xb, cur.xb);
        if ((EDGE || chk) && beside) {
          const double l = __shfl_up_sync(0xffffffffu, c.b, 1), rr = __shfl_down_sync(0xffffffffu, c.a, 1);
          uint32_t da = 0, db = 0;
          for (double u : {l, c.b, ym.a, c.a, cur.a}) window_conv(u, q, da);
          for (double u : {c.a, rr, ym.b, c.b, cur.b}) window_conv(u, q, db);
          if (da >= w.lim) n.a = general_exact_cell(p.w[0], p.w[1], p.w[2], p.w[3], p.w[4], l, c.b, ym.a, c.a, cur.a);
          if (db >= w.lim) n.b = general_exact_cell(p.w[0], p.w[1], p.w[2], p.w[3], p.w[4], c.a, rr, ym.b, c.b, cur.b);
          __syncwarp();
        }
      } else {
        const double L = __shfl_up_sync(0xffffffffu, c.b, 1), R = __shfl_down_sync(0xffffffffu, c.a, 1);
        if ((EDGE || chk) && beside) {
          n.a = stencil(lk, L, c.b, ym.a, c.a, cur.a);
          n.b = stencil(lk, c.a, R, ym.b, c.b, cur.b);
        } else {
          n.a = window_head<2>(w, q, {2, 3}, {ym.xa, c.xa});
          n.b = window_head<2>(w, q, {2, 3}, {ym.xb, c.xb});
          n.a = fma_rn(lk.yp, cur.a, fma_rn(lk.xp, c.b, fma_rn(lk.xm, L, n.a)));
          n.b = fma_rn(lk.yp, cur.b, fma_rn(lk.xp, R, fma_rn(lk.xm, c.a, n.b)));
        }
      }
      if (EDGE && (hold & 1u)) n.a = c.a;
      if (EDGE && (hold & 2u)) n.b = c.b;
      if (chk && (r == 0 || r == p.ny + 1 || t > p.meff)) {
        n.a = c.a;
        n.b = c.b;
      }
      if (t < M) conv(n, chk && (r < 1 || r > p.ny), d);
      A[t - 1] = B[t - 1];
      B[t - 1] = cur;
      cur = n;
    }
    if (__any_sync(0xffffffffu, d >= w.lim)) return false;
    const int r = i - M;
    if (KEEP) {
      // every step's finished row (B[t] holds step t's until the next iteration)
#pragma unroll
      for (int t = 1; t <= M; ++t) {
        const RowX &n = t < M ? B[t < M ? t : 0] : cur;
        if (st && t <= p.meff && i - t >= y0 && i - t < y1 && stream_ok(dst - out + (M - t) * p.pitch, 2, p))
          row_store(static_cast<double *>(p.keep) + (t - 1) * p.keep_stride + (dst - out) + (M - t) * p.pitch,
                    RowD{n.a, n.b});
      }
    } else if (st && (!chk || (r >= y0 && r < y1)) && stream_ok(dst - out, 2, p)) {
      row_store(dst, RowD{cur.a, cur.b});
    }
    dst += p.pitch;
    return true;
  };
  int s = 0;
  auto trip = [&](int i, bool chk) -> int {  // U iterations; U, or the one that found a value outside the window
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int sn = s + u + kAhead;
      if (!iter(i + u, ring + 32 * (s + u), base + 512u * (sn >= S ? sn - S : sn), (u + PH) & 3, chk)) return u;
    }
    s = s == 0 ? U : 0;
    return U;
  };
  // steady trips: every row stored, all copied rows inside the grid
  const int lo = max(y0 + M, M + 2), hi = short_pass ? 0 : min(y1 + M, p.ny + 2 - kAhead) - U;  // [lo, hi]: first rows
  for (int i = a; i < iend; i += U) {
    const int n = EDGE || i < lo || i > hi ? trip(i, true) : trip(i, false);
    if (n != U) {
      stage_drain();
      return max(y0, i + n - M);
    }
  }
  stage_drain();
  return y1;
}

__device__ __forceinline__ const Links<double> &chain_of(const WeightsD &k) { return k.l; }
__device__ __forceinline__ const Box9<double> &chain_of(const WeightsD9 &k) { return k.b; }

// A unit in windowed fixed point; from the first row that depends on a value outside
// the window, or at once when its first rows hold one, kWindowRetry rows by the
// general sweep before the next attempt.  Units are seldom taller, so most try one
// window a pass: a value that fits none has others near it, and each further attempt
// costs its probe and two pipelines' filling (noise, three attempts a unit and one:
// FP64 8192^2 x 4 1792 -> 1440 us, where the kernel without windows took 1620; box
// 2048x1536 x 6 416 -> 320 us, 397 without).
constexpr int kWindowRetry = 256;
template <int M, bool EDGE, bool KEEP, int SH>
__device__ __forceinline__ void stream_unit_window(const StreamParams &p, const typename RowOf<double, SH>::W &k, long e0, int x0,
                                                   unsigned hold, bool live, bool st, int y0, int y1, float4 *ring) {
  const bool window = WindowCoef<SH>::window(p).lim != 0;  // the weights have one
  while (y0 < y1) {
    if (window) y0 = stream_sweep_window<M, EDGE, KEEP, SH>(p, chain_of(k), e0, x0, hold, live, st, y0, y1, ring);
    if (y0 < y1) {
      const int ye = window ? min(y0 + kWindowRetry, y1) : y1;
      stream_sweep<double, M, EDGE, true, KEEP, SH>(p, k, e0, x0, hold, live, st, y0, ye, ring);
      y0 = ye;
    }
  }
}

__device__ __forceinline__ void make_weights(const StreamParams &p, WeightsF *k) {
  const float w = (float)p.w[0], e = (float)p.w[1], s = (float)p.w[2], c = (float)p.w[3], n = (float)p.w[4];
  k->w = make_float2(w, w);
  k->e = make_float2(e, e);
  k->s = make_float2(s, s);
  k->c = make_float2(c, c);
  k->n = make_float2(n, n);
}
__device__ __forceinline__ void make_weights(const StreamParams &p, WeightsF9 *k) {
  const Box9<float> b = box_chain<float>(p.w);
#pragma unroll
  for (int i = 0; i < 9; ++i) k->w[i] = make_float2(b.w[i], b.w[i]);
}
__device__ __forceinline__ void make_weights(const StreamParams &p, WeightsD9 *k) {
  k->b = box_chain<double>(p.w);
  k->u = box_exact_weights(k->b);
}
__device__ __forceinline__ void make_weights(const StreamParams &p, WeightsD *k) {
  const Links<double> l{p.w[0], p.w[1], p.w[2], p.w[3], p.w[4]};
  k->l = vreg_links(l);
  k->u = exact_weights(l);
}

// Resident blocks per SM asked of the compiler (0: its own choice).  Windowed, M = 2:
// five blocks of four warps (96 registers, some spilled in the rare branches)
// measured faster than four or six (FP64 16384^2: 259, 252 and 255 GCells/s); box:
// four (144 at 16384^2; three 137, five 144; without the window 92).
// Deep FP32 pipelines: the warps they had without steady-trip registers on top
// (k = 12, 16384^2: 4126 GCells/s at 12 warps, 3872 at 10; box k = 8, 9000x8000 x 48:
// 1587 us at 11, 1650 with the compiler's own choice of 196 registers).
template <typename T, int M, bool IP, bool KEEP, int SH> constexpr int stream_blocks() {
  if (kWindowed<T, M, IP, KEEP, SH>) return SH == 9 ? 4 : 7 - M;
  if (KEEP) return 0;
  if (std::is_same<T, float>::value && SH == 5) return M == 10 ? 13 : M == 12 ? 12 : 0;
  if (std::is_same<T, float>::value) return M == 8 ? 11 : 0;
  return 0;
}

template <typename T, int M, bool IP, bool KEEP, int SH>
__global__ void __launch_bounds__(32 * WarpsOf<T>::W, stream_blocks<T, M, IP, KEEP, SH>())
    stream_kernel(StreamParams p) {
  constexpr int V = VecOf<T>::V;
  const int lane = threadIdx.x & 31;
  const int unit = blockIdx.x * WarpsOf<T>::W + (threadIdx.x >> 5);
  if (unit >= p.bands * p.runs) return;  // whole warps
  // units in band-fastest order: the warps running at the same time cover
  // neighbouring bands of the same rows, so the overlapped halo columns two
  // bands read are found in L2 the second time
  const int band = unit % p.bands, run = unit / p.bands;
  const int xb = 1 + band * p.vw - p.G;  // logical column of lane 0's first element
  const int x0 = xb + V * lane;
  const long e0 = p.off + x0;
  const bool live = e0 >= 0 && e0 + V <= p.pitch;
  const bool st = live && x0 >= xb + p.G && x0 < xb + 32 * V - p.G && x0 <= p.nx;
  unsigned hold = 0;
#pragma unroll
  for (int v = 0; v < V; ++v)
    if (x0 + v == 0 || x0 + v == p.nx + 1) hold |= 1u << v;
  const bool edge = __any_sync(0xffffffffu, hold != 0);
  const int y0 = 1 + run * p.H, y1 = min(y0 + p.H, p.ny + 1);
  typename RowOf<T, SH>::W k;
  make_weights(p, &k);
  __shared__ float4 ring[WarpsOf<T>::W][2 * TripOf<T>::U * 32];
  float4 *mine = &ring[threadIdx.x >> 5][lane];
  grid_dependency_wait();  // the pass before this one has finished and its rows are visible
  if constexpr (kWindowed<T, M, IP, KEEP, SH>) {
    if (edge)
      stream_unit_window<M, true, KEEP, SH>(p, k, e0, x0, hold, live, st, y0, y1, mine);
    else
      stream_unit_window<M, false, KEEP, SH>(p, k, e0, x0, hold, live, st, y0, y1, mine);
  } else if (edge)
    stream_sweep<T, M, true, IP, KEEP, SH>(p, k, e0, x0, hold, live, st, y0, y1, mine);
  else
    stream_sweep<T, M, false, IP, KEEP, SH>(p, k, e0, x0, hold, live, st, y0, y1, mine);
  grid_launch_dependents();  // this warp's rows are written: the next pass may be launched (it waits above for them)
}

// ---- host side ------------------------------------------------------------------

using StreamFn = void (*)(StreamParams);

template <typename T, bool IP, bool KEEP, int SH, int... Ms> struct StreamTable;
template <typename T, bool IP, bool KEEP, int SH> struct StreamTable<T, IP, KEEP, SH> {
  static StreamFn get(int) { return nullptr; }
};
template <typename T, bool IP, bool KEEP, int SH, int M0, int... Ms> struct StreamTable<T, IP, KEEP, SH, M0, Ms...> {
  static StreamFn get(int m) {
    return m == M0 ? stream_kernel<T, M0, IP, KEEP, SH> : StreamTable<T, IP, KEEP, SH, Ms...>::get(m);
  }
};

int stream_max_depth(j2d_dtype dt) { return dt == J2D_F64 ? kStreamMaxF64 : kStreamMaxF32; }

// Steps per pass with a kernel of their own; a run's shorter pass runs the
// kernel of the run's depth with fewer steps.  Runs that keep every state
// have kernels for fewer depths.
static StreamFn stream_fn(j2d_dtype dt, int m, int ipath, bool keep = false, int shape = 5) {
  if (shape == 9) {  // the box: no state-keeping runs
    if (keep) return nullptr;
    if (dt == J2D_F64)
      return ipath ? StreamTable<double, true, false, 9, 2, 3, 4>::get(m)
                   : StreamTable<double, false, false, 9, 2, 3, 4>::get(m);
    return StreamTable<float, false, false, 9, 4, 6, 8>::get(m);
  }
  if (dt == J2D_F64) {
    if (keep)
      return ipath ? StreamTable<double, true, true, 5, 2, 3, 4>::get(m)
                   : StreamTable<double, false, true, 5, 2, 3, 4>::get(m);
    return ipath ? StreamTable<double, true, false, 5, 2, 3, 4, 6>::get(m)
                 : StreamTable<double, false, false, 5, 2, 3, 4, 6>::get(m);
  }
  if (keep) return StreamTable<float, false, true, 5, 4, 8>::get(m);
  return StreamTable<float, false, false, 5, 4, 6, 8, 10, 12>::get(m);
}

bool stream_depth_ok(j2d_dtype dt, int m, int shape) { return stream_fn(dt, m, 1, false, shape) != nullptr; }
bool stream_keep_ok(j2d_dtype dt, int m) { return stream_fn(dt, m, 1, true) != nullptr; }

// Resident blocks per SM of one instantiation (cached).
static int stream_occupancy(j2d_dtype dt, int m, int shape) {
  static std::mutex mu;
  static int cache[2][2][16] = {};
  std::lock_guard<std::mutex> lk(mu);
  int &c = cache[shape == 9 ? 1 : 0][dt == J2D_F64 ? 1 : 0][m];
  if (c == 0) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, stream_fn(dt, m, 1, false, shape), 32 * stream_warps(dt), 0) != cudaSuccess ||
        nb < 1) {
      cudaGetLastError();
      nb = 1;
    }
    c = nb;
  }
  return c;
}

StreamGeom stream_geometry(j2d_dtype dt, const GridDesc &g, int depth, int sms) {
  const int d = std::max(1, std::min(depth, stream_max_depth(dt)));
  const long warps = (long)stream_occupancy(dt, d, g.shape) * stream_warps(dt) * std::max(sms, 1);
  return stream_geometry_warps(dt, g.nx, g.ny, depth, warps);
}

StreamGeom stream_geometry_warps(j2d_dtype dt, int nx, int ny, int depth, long warps) {
  StreamGeom q;
  const int V = dt == J2D_F64 ? 2 : 4;
  q.depth = std::max(1, std::min(depth, stream_max_depth(dt)));
  q.G = (q.depth + V - 1) / V * V;
  q.vw = 32 * V - 2 * q.G;
  q.bands = (nx + q.vw - 1) / q.vw;
  // Several waves of units per pass, so that the block scheduler balances
  // the SMs as units finish, each run at least 32M (FP64) or 16M (FP32) rows tall,
  // its 2M-row overlap then costing at most 6% or 12% (FP32 k = 8, 16384^2: 3958
  // GCells/s with one wave, 4254 with 2 or 3, 4235 with 4, 4090 with 8; FP32
  // 4096^2: 2764 against 2175 with 32M).
  warps = std::max(warps, 1L);
  const int hmin = (dt == J2D_F64 ? 32 : 16) * q.depth;
  if (dt == J2D_F64) {
    // Whole waves of units, up to eight with runs of at least 44M rows (k = 2,
    // 8192^2: 212, 233, 236, 238, 239 and 235 GCells/s with 1, 2, 3, 4, 6 and 8
    // waves, 16384^2: 258 with 6, 259 with 8, 258 with 16); one wave for
    // smaller grids (4096^2: 193 with one, 185 with one and a half, 187 with
    // three).  A run has a whole number of the sweep's four-row trips.
    const long r1 = std::max<long>(1, warps / q.bands);
    const long waves = std::min<long>(8, std::max<long>(1, ny / (r1 * 44 * q.depth)));
    const long hu = ((ny + waves * r1 - 1) / (waves * r1) + 3) / 4 * 4;
    q.H = (int)std::min<long>(ny, std::max<long>(hu, hmin));
    // too few units of that height for one wave: the warps share the runs
    q.hu = (int)std::min<long>(q.H, std::max<long>(hu, 8));
  } else {
    int runs = (int)std::max<long>(1, 3 * warps / q.bands);
    runs = std::min(runs, std::max(1, ny / hmin));
    q.H = (ny + runs - 1) / runs;
    // smaller grids: one wave of shorter units, at least 3.5M rows (FP32 2048x1536,
    // k = 6: 2.4, 2.1 and 2.8 us a step with a quarter, half and one wave of
    // units, before passes overlapped; 3.3 on chip; 3000^2: 3.8 and 3.5 with half
    // and one)
    const long r1 = std::max<long>(1, warps / q.bands);
    q.hu = (int)std::min<long>(q.H, std::max<long>((ny + r1 - 1) / r1, 7 * q.depth / 2));
  }
  q.H = (q.H + q.hu - 1) / q.hu * q.hu;  // a run is a whole number of its warps' units
  q.runs = (ny + q.H - 1) / q.H;
  q.units = (ny + q.hu - 1) / q.hu;
  return q;
}

// A pass of m <= q.depth steps, in -> out (distinct buffers whose rings
// agree); with keep set, step t's state goes to keep + (t - 1) * keep_stride
// elements instead (out unused).  The one step that a run of an odd number of steps
// has over at two steps a pass is the one-step kernel's: a pass for it takes as long as
// for two (4096^2 x 7, noise 810 -> 645 us, both signs 1433 -> 1248; box 1481 -> 1094 and
// 2712 -> 2329; 100^2 x 7 box 125 -> 96).
cudaError_t launch_stream_pass(j2d_dtype dt, const void *in, void *out, const GridDesc &g, const StreamGeom &q, int m,
                               int ipath, int *status, cudaStream_t s, void *keep, long keep_stride) {
  if (dt == J2D_F64 && q.depth == 2 && m == 1) return launch_onestep(dt, false, in, keep ? keep : out, g, ipath, s);
  StreamParams p;
  p.in = in;
  p.out = out;
  p.pitch = g.pitch;
  p.off = (int)g.off;
  p.nx = g.nx;
  p.ny = g.ny;
  p.G = q.G;
  p.vw = q.vw;
  p.bands = q.bands;
  p.H = q.hu;
  p.runs = q.units;
  p.meff = m;
  p.keep = keep;
  p.keep_stride = keep_stride;
  p.ipath = ipath;
  p.nelem = (long)(g.ny + 2) * g.pitch;
  p.status = status;
  for (int i = 0; i < 9; ++i) p.w[i] = g.w[i];
  p.win = WindowWeights{};
  p.win9 = WindowWeightsN<9>{};
  if (dt == J2D_F64 && g.shape == 9) p.win9 = window_weights(box_chain<double>(g.w).w);
  if (dt == J2D_F64 && g.shape == 5) p.win = window_weights({g.w[0], g.w[1], g.w[2], g.w[3], g.w[4]});
  StreamFn fn = stream_fn(dt, q.depth, ipath, keep != nullptr, g.shape);
  if (!fn || m < 1 || m > q.depth) return cudaErrorInvalidValue;
  const long units = (long)q.bands * p.runs;
  const int W = stream_warps(dt);
  const unsigned blocks = (unsigned)((units + W - 1) / W);
  // Programmatic dependent launch: the next pass is launched when every warp of
  // this one has stored its rows, and waits in the kernel for the end of this
  // one (FP32, 1024^2, k = 6: 1.74 -> 1.45 us a step; released at a kernel's
  // start instead, its waiting blocks take slots from the running pass: 1.87).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(32 * W);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, fn, p);
}

}  // namespace j2d
