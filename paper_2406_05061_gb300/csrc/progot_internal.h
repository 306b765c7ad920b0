// Internal (C++) interfaces between the host orchestration and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "progot_common.cuh"

namespace progot {

// Parameters of the barycentric-projection sweep (map step of Alg. 2 / Alg. 3).
struct MapParams {
  const float* A;      // nA x d current points (may alias out)
  const float* B;      // nB x d target points
  const float* Bn;     // |b_j|^2
  const float* potB;   // g
  const float* L;      // per-row log2-sum-exp of t_ij (from an LSE sweep)
  float* out;          // nA x d: x + alpha (T(x) - x)
  float* Opart;        // [splits][nA][d] partial numerators
  float* Rpart;        // [splits][nA] partial row sums of P
  unsigned int* cnt;   // [row blocks] arrival counters (zero between launches)
  int64_t nA, nB;
  int32_t d;
  int32_t splits, tiles_per_split, dchunks;
  float scale, bscale;
  float alpha;
  int32_t cost;        // CostKind (the p-norm map moves x by grad h*(sum_j Q_ij grad h(x - y_j)))
  float cost_p;
  const float* C;      // p-norm: stored cost sums (SweepParams::C), or nullptr
  int64_t ldc;
};

void count_launch();
// Text returned by progot_last_error_string() on the calling thread.
void set_last_error_message(const char* msg);

// float32 CUDA-core sweeps (sweep_fp32.cu)
cudaError_t launch_lse_sweep_fp32(const SweepParams& p, cudaStream_t stream);
cudaError_t launch_map_sweep_fp32(const MapParams& p, cudaStream_t stream);
// p-norm cost: barycentric displacement x <- x - alpha grad h*(sum_j Q_ij grad h(x_i - y_j))
cudaError_t launch_map_sweep_pnorm(const MapParams& p, cudaStream_t stream);
// out[0] = sum_ij h(x_i - y_j) for the p-norm cost (float64, fixed order; partial holds
// reduce_parts() doubles)
cudaError_t launch_pairwise_cost_sum(const float* X, int64_t n, const float* Y, int64_t m, int32_t d, int32_t cost,
                                     float cost_p, double* partial, double* out, cudaStream_t s);
// C[i ld + j] = sum_k |x_ik - y_jk|^p, zeros for m <= j < 128 ceil(m / 128) <= ld
cudaError_t launch_pnorm_cost(const float* X, int64_t n, const float* Y, int64_t m, int32_t d, int32_t cost, float cost_p,
                              float* C, int64_t ld, cudaStream_t s);
int fp32_tile_rows();
int fp32_tile_cols();
int map_dchunk();

// small kernels (prep.cu)
cudaError_t launch_row_sqnorm(const float* X, int64_t n, int32_t d, float* out, cudaStream_t s);
cudaError_t launch_lse_uncenter(float* L, const float* X, int64_t n, int32_t d, const float* mu, float bscale,
                                cudaStream_t s);
cudaError_t launch_init_state(SolverState* st, cudaStream_t s);
// out[0] = sum_i |x_i|^2, out[1 + k] = sum_i x_ik (float64; partial buffer of
// `parts` x (d + 1) doubles, deterministic two-pass reduction)
cudaError_t launch_moments(const float* X, int64_t n, int32_t d, double* partial, int parts, double* out,
                           cudaStream_t s);
// out[0] = sum_i ||a_i - b_i||^2 (float64, deterministic)
cudaError_t launch_sq_error(const float* A, const float* B, int64_t n, int32_t d, double* partial, int parts,
                            double* out, cudaStream_t s);
int reduce_parts();
// out[0] = sum_i P_ii, out[1] = sum_i log P_ii for n = m, log P_ii = (f_i + g_i - |x_i - y_i|^2)/eps;
// logd (optional) receives log P_ii in float32; partial holds parts x 2 doubles
cudaError_t launch_diag(const float* X, const float* Y, const float* f, const float* g, int64_t n, int32_t d, double eps,
                        float* logd, double* partial, int parts, double* out, cudaStream_t s);
// *out = mean_ij |x_i - y_j|^2 from launch_moments outputs mx (of X, n rows) and my (of Y, m rows)
cudaError_t launch_mean_cost_closed(const double* mx, const double* my, int64_t n, int64_t m, int32_t d, double* out,
                                    cudaStream_t s);
// out[k] = sum_b partial[b * width + k], b = 0..parts-1 in order
cudaError_t launch_sum_parts(const double* partial, int parts, int width, double* out, cudaStream_t s);

// tcgen05 sweeps (sweep_tc.cu) on the operands of operands.cu; maps point at CUtensorMap objects.
// bias map: (nB padded to 128) x 16 bf16 rows [beta_hi, beta_mid, beta_lo, 0...] of the
// B side; bias_out (optional): the same rows for the A side, written from the updated
// potential in potential mode (the next sweep's B bias).
struct TcMaps {
  const void* a[3];   // operand maps of the rows' side (128-row boxes): hi, lo, (grid split) third part
  const void* b[3];   // of the columns' side (bn-row boxes)
  const void* bias;   // bias rows of the columns' side (bn-row boxes)
  const void* a_part[2];  // the rows' side bf16 hi, lo operand rows (NULL: grid operands)
};
// parts: operand parts in use (1 bf16, 2 bf16x3); words non-NULL: the integer-grid split
// (grid_split.cuh; three parts, bn = 128) with its device words.
cudaError_t launch_lse_sweep_tc(const SweepParams& p, const TcMaps& maps, int nkb, int parts, const GridWords* words,
                                int bn, int G, int maxseg, int32_t* fault, void* bias_out, cudaStream_t stream,
                                const float* lrow = nullptr, void* prob = nullptr, int64_t a_row0 = 0);
// x <- x + alpha (T(x) - x) for rows [row0, row0 + rows) from the P tiles and row sums a
// kModeProb sweep left (pv_tc.cu); mapY: the parts of the y operand in 64-row boxes.
struct PvLaunch {
  const float* X;      // row row0 of the points (may alias out)
  float* out;
  const float* rsum;   // [rows]
  const void* prob;
  const void* mapY[kGridParts];
  const GridWords* words;
  const float* mu;
  int64_t rows, m;
  int32_t d;
  float alpha, inv_sc; // inv_sc = 1 / sqrt(c)
  int32_t* fault;
};
int64_t pv_prob_bytes_per_block(int64_t m);  // P bytes of one 128-row block
cudaError_t launch_pv_tc(const PvLaunch& p, int sms, cudaStream_t stream);
// The steps of a map that the grid's kernels left alone or gave up, in one launch (sweep_fp32.cu);
// nothing to do when words->bad and *fault are zero. eps, alpha: host, K values, read by the call.
struct MapRedo {
  const float* src;     // the points before step 0 (a fault starts again from them), NULL: only words->bad counts
  float* x;             // n x d, in place
  const float* y;
  const float* g;       // K x m
  float* T;             // n x d of scratch
  const GridWords* words;
  const int32_t* fault;
  int64_t n, m;
  int32_t d, K;
  const double* eps;
  const double* alpha;
  bool alpha_last_one;  // the last step's alpha is 1 whatever alpha says (Alg. 3)
};
cudaError_t launch_map_redo(const MapRedo& q, cudaStream_t stream);
// Tensor-core operands (operands.cu).
// mu = (mean of the rows of X + mean of the rows of Y) / 2, the sums carried beyond float64
// rounding of their order; partial: reduce_parts() * d doubles of scratch; ticket: a zero
// word, zero again afterwards; words (or NULL): their norms and counts zeroed for launch_operands.
cudaError_t launch_center(const float* X, int64_t n, const float* Y, int64_t m, int32_t d, double* partial,
                          unsigned* ticket, float* mu, GridWords* words, cudaStream_t s);
// Both clouds: parts of sqrt(c) (x - mu), rows of dp 16-bit elements (zeros past d): bf16
// hi, lo, or the integer grid's three half-precision parts (grid_split.cuh); unused
// parts are NULL. Centred squared norms, and bias rows of both sides from the potentials f
// (x side) and g (y side) where given, into one or two buffers each, rows padded to a
// multiple of 256. Grid: the words of the split; step is what words->bad becomes (when zero)
// if the clouds are out of its range.
struct OperandPrep {
  const float* x;
  const float* y;
  int64_t n, m;
  int32_t d, dp;
  float sc, sc_lo;          // sqrt(c) = sc + sc_lo (bf16: sc alone)
  const float* mu;
  float* xnc;
  float* ync;
  GridWords* words;
  int32_t step;
  int32_t min_exp;          // least ex + ey within range
  void* xp[3];
  void* yp[3];
  const float* f;           // NULL: no x-side bias rows
  const float* g;
  float bscale, bscale_lo;  // log2(e) / eps = bscale + bscale_lo
  void* xb[2];
  void* yb[2];
};
// What a persistent loop finds when it starts: its work-split tables, ready flags, counters
// and state.
struct LoopSetupSide {
  void* segs;               // int4 [G * maxseg]
  int32_t* nseg;            // [G]
  int2* crow;               // [R] (offset, count) into cslot
  int32_t* cslot;
  uint32_t* flag;           // [R]
  unsigned long long* cnt;  // [R]
  unsigned long long* done;
  int32_t R, T;
  uint32_t flag_init;
};
struct LoopSetup {
  LoopSetupSide side[2];
  SolverState* state;       // [2]
  int32_t G, maxseg;
  int32_t aligned;          // every CTA on one row block (tc::aligned_segment)
};
// kGridHull: the integer grid for clouds inside the hull of the two that the last kGrid call
// on this workspace saw (same mu and words).
enum class OperandKind { kBf16, kGrid, kGridHull };
cudaError_t launch_operands(const OperandPrep& op, OperandKind kind, const LoopSetup* loop, cudaStream_t s);
cudaError_t launch_loop_finish(const float* f_new, const float* an, const float* w, double log_w_uniform, double eps,
                               int64_t n, float* L, const float* f_cur, float* f_out, cudaStream_t s);
cudaError_t launch_warm_start(float* g, const float* g_prev, int64_t m, float* f, int64_t n, float c, cudaStream_t s);
void tc_plan(int64_t nA, int64_t nB, int bn, int sms, int* G, int* maxseg);
// Barycentric displacement on the tensor cores for d <= 64 (map_tc.cu): x <- x + alpha
// (T(x) - x) in place (out may alias X), L from a log-sum-exp pass of the same t; the
// A / B / bias maps use 128-row boxes; the B operand sqrt(c) (y - mu) also serves the
// P Y product, whose result is mapped back with inv_sc = 1 / sqrt(c) and mu (d floats).
cudaError_t launch_map_sweep_tc(const float* X, float* out, const float* L, int64_t nA, int64_t nB, int32_t d,
                                float alpha, const void* mapAh, const void* mapAl, const void* mapBh,
                                const void* mapBl, const void* mapBbias, float inv_sc, const float* mu,
                                float* Opart, float* Rpart, unsigned* cnt, int G, int maxseg, int32_t split3,
                                int32_t* fault, cudaStream_t stream);
size_t map_sweep_tc_smem();
// The same for 64 < d <= 256 in one pass (map_tc_onepass.cu): tiles of 64 columns (B maps
// and bias rows in 64-row boxes) whose K blocks all stay in one stage, S formed once per
// tile and every chunk of 64 output coordinates accumulated in TMEM; Opart slots hold
// 128 rows x 64 nkb floats. xh is the bf16 hi operand of X (nA x 64 nkb, the buffer the
// A maps describe), read directly into TMEM.
bool map_tc_onepass_supported(int nkb);
int map_tc_onepass_tile_cols();
cudaError_t launch_map_sweep_tc_onepass(const float* X, float* out, const float* L, int64_t nA, int64_t nB,
                                        int32_t d, int32_t nkb, float alpha, const void* mapAl,
                                        const void* mapBh, const void* mapBl, const void* mapBbias, float inv_sc,
                                        const float* mu, const void* xh, float* Opart, float* Rpart, unsigned* cnt,
                                        int G, int maxseg, int32_t split3, int32_t* fault, cudaStream_t stream);
int tc_stages(int nkb, int split3);
int tc_tile_cols(int nkb, int split3);  // 128 or 256

// Persistent tensor-core Sinkhorn loop (loop_tc.cu). Side 0 is the f-update (rows of X
// against Y), side 1 the g-update. A finisher publishes its row block's bias rows, then
// the row block's ready flag (the index of the sweep that wrote it, plus one).
struct LoopSideLaunch {
  SweepParams p;             // potential mode; An / Bn the centred norms; role 1 (f) or 2 (g)
  float* out0;               // f-update: f buffers 0 and 1 (the state's fcur selects); g-update: g
  float* out1;
  void* bias_out[2];         // bias rows (rows x 16 bf16) of this side's rows, by iteration parity
  uint32_t* flag_out;        // [row blocks] ready flags of this side, zero at the loop's start
  const uint32_t* flag_in;   // the other side's flags
  unsigned long long* cnt;   // [row blocks] arrival counters, zero at the loop's start
  unsigned long long* done;  // finished row blocks, zero at the loop's start
  float2* partial;           // (max, sum) slots of this side's sweeps
  const void* a_part[2];     // operand rows of this side, hi and lo (read where A sits in TMEM)
  // the work split's tables (LoopSetupSide)
  const void* segs;
  const int32_t* nseg;
  const int2* crow;
  const int32_t* cslot;
};
struct LoopLaunch {
  LoopSideLaunch side[2];
  // CUtensorMap: X hi, X lo, Y hi, Y lo (128-row boxes); X hi, X lo, Y hi, Y lo (bn-row
  // boxes); third parts of the grid split: X, Y (128-row), X, Y (bn-row; any map without
  // the grid split); bias rows X[0], X[1], Y[0], Y[1] (bn-row boxes)
  const void* maps[16];
  const GridWords* words;    // grid split: its device words (NULL: bf16 operands)
  double* errpart;           // [2][row blocks of X]
  SolverState* state;
  int32_t* fault;
  unsigned long long wait_ns;
  int nkb, split3, bn, G, maxseg, seq0, niter;
};
cudaError_t launch_sinkhorn_loop_tc(const LoopLaunch& L, cudaStream_t stream);

// Library settings and helpers shared with the batched engine (progot_api.cu).
// encode_operand_map: 2-D bf16 tensor map (CUtensorMap*) over a rows x dp row-major
// buffer, 64-wide 128-byte-swizzled boxes (dp a multiple of 64) or 16-wide 32-byte
// swizzled bias boxes (dp = 16), box_rows rows per box.
int encode_operand_map(void* map, void* base, int64_t rows, int32_t dp, int box_rows);
int32_t stall_window_setting();
unsigned long long wait_limit_setting();
int device_sm_count();
// Workspace that progot_solve makes use of (float32 solves beyond d = 64 run on CUDA cores).
size_t solve_workspace_size(int64_t n, int64_t m, int32_t d, int32_t precision);
int fail_message(int code, const char* msg);  // sets the last-error text, returns code
bool loop_tc_supported(int bn, int nkb, int split3, bool grid);

void loop_tc_plan(int64_t n, int64_t m, int bn, int sms, int* G, int* maxseg, int* aligned);

}  // namespace progot
