// Launchers of the transfer-block preparation and the SGS sweep kernels (kernels_sweep.cu).
#pragma once
#include "fasw_fp64.cuh"
#include "fasw_internal.cuh"

namespace fasw {

// SWEEP_HP: hyperplane-staged FP32 sweep with the default ring depth; SWEEP_HP4 / SWEEP_HP8: with a
// ring of 4 / 8 steps (where 8 does not fit in shared memory, 4).  SWEEP_STRIPS / STRIPS16 /
// STRIPS4: pipelined strips of 8 / 16 / 4 rows.
// SWEEP_WS: warp strips of 8 rows, operands staged by bulk copies, FP32 recurrence; in FP64
// contexts followed by one FP64 defect correction (a second FP32 sweep on the FP64 residual of
// the first), which brings the result to FP64 accuracy.
enum SweepKind {
  SWEEP_AUTO = 0, SWEEP_LEGACY = 1, SWEEP_CTA = 2, SWEEP_STRIPS = 3, SWEEP_STRIPS16 = 4,
  SWEEP_HP = 5, SWEEP_HP4 = 6, SWEEP_HP8 = 7, SWEEP_STRIPS4 = 8, SWEEP_WS = 9, SWEEP_WS8 = 10
};
inline bool is_hp(int kind) { return kind == SWEEP_HP || kind == SWEEP_HP4 || kind == SWEEP_HP8; }
// SWEEP_WS8: the warp strips with a ring of three stages instead of five (less shared memory, so
// that strips of different cases of a batch can share an SM)
inline bool is_ws(int kind) { return kind == SWEEP_WS || kind == SWEEP_WS8; }

// the level's sweep is the warp strips'
inline bool ws_level(int kind, const LevelDev& L) { return is_ws(kind) && L.wsF; }
// FP64 levels up to this many cells take the half rows of k_ws_prep64, and a block row per thread in the right-hand
// side's and the defect's kernels; larger ones two kernels and a cell per thread.  A smoothing step (RANS), split
// against not: preparation 18,432 cells 482 / 496 us, 20,736 475 / 480, 25,600 516 / 516, 36,864 643 / 637,
// 65,536 881 / 885; right-hand side and defect 18,432 477 / 496, 25,600 513 / 516, 36,864 632 / 637, 50,176
// 747 / 748, 65,536 885 / 885.  So the lines could lie at about 24,000 and 45,000 cells, for 1 to 4 % of a step
// between; up to 16,384 cells the split forms win by more (256x64 preparation 32 -> 25 us, defect 7.1 -> 6.4).
constexpr int PREP_SPLIT_CELLS = 16384;
constexpr int WS_SPLIT_CELLS = 16384;
// launch_sgs_prep forms the diagonal blocks itself (aw, eta as in launch_diag_blocks, which is left out)
inline bool prep_forms_diag(int kind, const LevelDev& L, int mixed) {
  return ws_level(kind, L) && (mixed || L.n <= PREP_SPLIT_CELLS);
}
// kind: the resolved sweep kind of this level (SWEEP_HP writes the hyperplane-major blocks,
// SWEEP_WS also the skewed FP32 blocks of the warp strips).
void launch_sgs_prep(const LevelDev& L, int mixed, int kind, cudaStream_t st, int aw = 0, double eta = 0.0);
// Forward and backward sweep of one stage: y = (D+L)^-1 rhs, z = (D+U)^-1 D y into L.yz64 /
// L.yz32, with the stage update u = u0 - alpha z (AW) or u0 - alpha dt* z (ARK) when
// do_update.  prog: 2 * sweep_strips(L) flags, err: device error word.  Returns the number of
// kernels launched.  Warp strips only: rhs null when D^-1 rhs is in place already (ResArgs::wsC);
// pending non-null: the stage update is left to it.
int launch_sweep(const LevelDev& L, int mixed, int kind, int do_update, int aw, double alpha, const double* rhs,
                 long long* prog, int* err, long long limit, cudaStream_t st, int exact_iters = 0,
                 struct WsPending* pending = nullptr);
int sweep_strips(const LevelDev& L);
// Warp-strip sweep (kernels_sweep_ws.cu): whether a level can use it, the sizes of its arrays
// (floats of wsF / wsB; of wsC / wsY), its strips, and one application (refine: FP64 defect
// correction in FP64 contexts; the skewed blocks come from launch_sgs_prep).  Returns the
// kernels launched.
// Warp-strip layout: strips of WS_ROWS rows, a strip's operands stored step by step (row r of the
// strip at step s holds cell i = s - r), the steps padded to whole stages of WS_U; per step
// WS_F4_STEP float4 of blocks: for each of the two blocks, the 4 block rows of each row's cell.
constexpr int WS_ROWS = 8;
constexpr int WS_U = 8;  // steps per stage of the operand ring
constexpr int WS_F4_STEP = 8 * WS_ROWS;
// steps stored per strip: the ni + R - 1 steps that hold a cell (R = min(nj, WS_ROWS)), padded
__host__ __device__ __forceinline__ int ws_steps(int ni, int nj) {
  const int R = nj < WS_ROWS ? nj : WS_ROWS;
  return (ni + R - 1 + WS_U - 1) / WS_U * WS_U;
}
// Skewed index of cell (i, j) in the forward order: strip j / WS_ROWS, step i + r, row r.
__device__ __forceinline__ size_t ws_fpos(int i, int j, int Mp) {
  const int jl = j & (WS_ROWS - 1);
  return ((size_t)(j / WS_ROWS) * Mp + (i + jl)) * WS_ROWS + jl;
}

// Skewed index of cell (i, j) in the backward order (the layout of y as the backward pass reads
// it and of its result z): strip j / WS_ROWS, step Mp - 1 - i - r, row r.
__device__ __forceinline__ size_t ws_bpos(int i, int j, int Mp) {
  const int jl = j & (WS_ROWS - 1);
  return ((size_t)(j / WS_ROWS) * Mp + (Mp - 1 - i - jl)) * WS_ROWS + jl;
}

__device__ __forceinline__ void ws_load64(const float4* z, size_t pos, double x[4]) {
  const float4 v = z[pos];
  x[0] = f2d(v.x);
  x[1] = f2d(v.y);
  x[2] = f2d(v.z);
  x[3] = f2d(v.w);
}

// A stage update u = u0 - alpha z (AW) or u0 - alpha dt* z (ARK), z = z0 (+ dz), that the sweep left to
// the kernel that next reads the state, the cell auxiliaries' (launch_bc_aux).  z0 null: none.  dz2: the
// second correction (adjoint).
struct WsPending {
  const float4 *z0, *dz, *dz2;
  double alpha;
  int aw;
};

// the updated state of interior cell (i, j)
__device__ __forceinline__ void ws_updated(const LevelDev& L, const WsPending& p, int i, int j, double w[4]) {
  const int c = j * L.ni + i;
  const size_t zp = ws_bpos(i, j, ws_steps(L.ni, L.nj));
  double z[4];
  ws_load64(p.z0, zp, z);
  if (p.dz) {
    double d[4];
    ws_load64(p.dz, zp, d);
#pragma unroll
    for (int q = 0; q < 4; ++q) z[q] += d[q];
  }
  const double sc = p.aw ? p.alpha : p.alpha * L.dts[c];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = fma(-sc, z[q], L.u0[q * (size_t)L.n + c]);
}

// L.tb (FP64) into the warp-strip layout: L.wsF, L.wsB, L.wsCut
void launch_ws_skew(const LevelDev& L, cudaStream_t st);
// The form of the sweep (operand ring, edge buffers) for a level: the first, in order of speed, that the
// device can launch, -1: none (another sweep).  deep: kind 9.  cluster_bytes: 0 asks the current device whether
// it holds a cluster of more than eight CTAs; else only with up to that much shared memory a CTA.
int ws_form(int ni, int nj, int nw, bool deep, long long cluster_bytes = 0);
void ws_form_shape(int ni, int nj, int nw, int form, int* stages, int* edges, long long* bytes);
size_t ws_floats(int ni, int nj);
size_t ws_vec_floats(int ni, int nj);
int ws_strips(int nj);
// refine: FP64 defect corrections of the FP32 sweep (FP64 levels; L.wsZ holds one vector more than that);
// exact_iters > 0: that many block Gauss-Seidel corrections toward the exact (D + L + U)^-1;
// deep: the deeper operand ring (false for SWEEP_WS8)
int launch_ws_sweep(const LevelDev& L, int mixed, int refine, int do_update, int aw, double alpha, const double* rhs,
                    int* err, long long limit, cudaStream_t st, int exact_iters = 0, bool deep = true,
                    WsPending* pending = nullptr);
// Hyperplane-staged FP32 sweep: whether a level fits (rows, shared memory), and the entries
// (ni + nj - 1) * nj of its hyperplane-major arrays (hpF, hpB: 32 floats each; hpC, hpY: 4).
bool hp_fits(int ni, int nj, int nw);
size_t hp_floats(int ni, int nj);

}  // namespace fasw
