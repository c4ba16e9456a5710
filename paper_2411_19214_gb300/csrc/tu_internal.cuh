// tu_internal.cuh -- internal declarations shared by the translation units of
// libtu_ipfp.so: the market object, the per-row scaling update, and the inline
// PTX wrappers (mbarrier, TMA, tcgen05) used by the sm_103a kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <string>
#include <utility>
#include <vector>

#include "../../include/tu_ipfp.h"

// ---------------------------------------------------------------------------
// Sizes shared by host and device code
// ---------------------------------------------------------------------------
namespace tu {

constexpr int kFusedOwnRows = 256;      // own-side rows per CTA tile (two 128-row MMAs)
constexpr int kFusedPartnerRows = 128;  // partner rows per pipeline stage (MMA N)
constexpr int kKBlock = 64;             // bf16 elements per 128-byte swizzle row
constexpr int kRowPad = 256;            // every per-side vector is padded to this multiple
constexpr int kMaxPartials = 4096;      // per-CTA FP64 partials per half-sweep

// results[] slots (FP64, device), written by the finalize kernels
enum : int {
  kResXInf = 0,   // max_x |r_x| / n_x of the state entering the X half-sweep
  kResXL1 = 1,    // sum_x |r_x|
  kResXSq = 2,    // sum_x u_x^2 after the X half-sweep
  kResYSq = 3,    // sum_y v_y^2 after the Y half-sweep
  kResNonfin = 4, // count of non-finite potentials written
  kResSlots = 8
};

// Per-market FP64 scalars on the device (tu_market::st), kept up to date by
// the preparation and finalize kernels of every half-sweep, so that no O(N)
// pass is needed to prepare a half-sweep or to take the translation step.
// Side s: 0 = X, 1 = Y.
enum : int {
  kStLmax = 0,     // [2] max over the side of its stored ell
  kStLogS = 2,     // [2] log sum e^{2 log u} over the side's true potentials
  kStOff = 4,      // [2] true log u = stored log u + offset (a translation not yet written to the arrays)
  kStTauNext = 6,  // the translation step for the next half-sweep of a sweep
  kStTauUsed = 7,  // the translation step the current half-sweep's preparation applied
  kStShift = 8,    // the current half-sweep's partner shift: lmax + offset + tau (natural log)
  kStOwnOff = 9,   // the current half-sweep's own-side offset: offset - tau
  kStCount = 10,   // a counter (int) of the flush's finished blocks
  kStSlots = 16
};

// Per-32-row group of a side (Side::grp, a float4): max 2 log u, sum of
// e^{2 log u - max}, max ell; written by the side's own half-sweep.
constexpr int kGroupRows = 32;
constexpr int kMaxSplit = 8;  // partner ranges per own tile (tu_market_set_split)

// Residual of the state entering an X half-sweep (the pass's `residual`):
// none, an estimate with FP32 terms (inside sweeps) or exact FP64 terms
// (certifying passes).
enum : int { kResidualNone = 0, kResidualEstimate = 1, kResidualExact = 2 };

// device error word codes (first error wins)
enum : int { kErrNone = 0, kErrTimeout = 1, kErrNonfinite = 2 };

// Where the rows' sums of a fused half-sweep are cut (cut_plan, fused.cu). Own
// tiles (256 rows; pair: 512) from t0 on, taken as one line of (tile, partner tile)
// pairs, are cut after every `span` pairs; a row's sum is formed range by range
// and the ranges are added in order. span = 0: nothing is cut. The cuts belong
// to the market's shape, not to a launch: a launch that gives each range to
// another CTA and one that runs a row's ranges in turn give the same bits.
// `pair`: the half-sweep runs on pairs of CTAs, and the tiles are 512 rows.
struct CutPlan {
  int t0 = 0, span = 0, spans = 0;
  bool pair = false;
};

struct Side {
  int64_t rows = 0;      // users on this side
  int64_t rows_pad = 0;  // rows rounded up to kRowPad
  double* log_u = nullptr;  // log u (side X) or log v (side Y), rows_pad (FP64 state)
  double* ell = nullptr;    // log u + b / (2 sigma), rows_pad (FP64 state)
  float* b2s = nullptr;     // b / (2 sigma), rows_pad, or nullptr without bias
  double* mass = nullptr;   // capacities, rows_pad (padding 1)
  float* pvec = nullptr;    // this side's potentials prepared for the other side's half-sweep, rows_pad
  float4* grp = nullptr;    // per-32-row groups {max 2 log u, scaled sum, max ell, 0}, rows_pad / 32 + 2 kMaxPartials
  double sum_mass = 0.0;    // host copy of sum of capacities
  __nv_bfloat16* fac16 = nullptr;  // packed [F | K] (or [G | L]) rows x kp, bf16, zero padded
  uint8_t* fac8 = nullptr;         // FP8 markets: packed rows x kp e4m3 of [F | K] / fs (zero padded)
  float* fs = nullptr;             // FP8 markets: per-row scales, rows_pad (padding 1)
  uint8_t* fold = nullptr;         // packed rows of one or two 128-byte blocks, BF16 or e4m3 with one scale per
                                   // side: this side's g / c as the K = 16 operand of the partner tiles' extra
                                   // MMA (rows_pad x 32 bytes, tcgen05 layout; unused while the market is wide)
  int fp8_exp = 0;                 // FP8 markets with one scale per side: its exponent (fs = 2^fp8_exp)
  float* fac32 = nullptr;          // packed rows x kp, fp32 (dense path), zero padded
  CUtensorMap tm_own;       // TMA map, box kKBlock x kFusedOwnRows
  CUtensorMap tm_partner;   // TMA map, box kKBlock x kFusedPartnerRows
  CUtensorMap tm_half;      // TMA map, box kKBlock x kFusedPartnerRows / 2 (pairs of CTAs)
  CUtensorMap tm_fold;      // TMA map of `fold` (pairs of CTAs)
  CutPlan cut;              // fused path: the cuts of the half-sweep that updates this side
};

// Over-relaxation controller of the solve loops (host side, one per market).
// Plain sweeps until the residual is below 0.1 and (in automatic mode) the
// per-sweep decay q of the plain iteration has settled, then the fixed factor,
// or in automatic mode omega = 2 / (1 + sqrt(1 - q)) (successive
// over-relaxation) tapered towards 1 over the last decade above tol (the
// relaxed sweep amplifies the FP32 rounding of the row sums by about
// omega / (2 - omega)). In both modes the excess over 1 is halved whenever the
// residual grows tenfold over the best seen.
struct RelaxControl {
  static constexpr int kProbe = 10;  // sweeps between convergence-rate estimates
  double cfg = 1.0;                  // 1: plain; (1, 2): fixed; 0: automatic
  double omega = 1.0, target = 1.0, best = 1.0 / 0.0, q_prev = -1.0;
  int last_est = 0;
  std::vector<std::pair<int, double>> hist;

  explicit RelaxControl(double c = 1.0) : cfg(c) {}
  bool enabled() const { return cfg != 1.0; }

  // r: residual of the state entering the last sweep of a block that ended
  // after `done` sweeps (r > tol). Returns the omega of the next block.
  double observe(int done, double r, double tol);
};

// log |dm| of the translation step (0 for dm = 0, where it is not used)
inline double log_abs(double dm) { return dm == 0.0 ? 0.0 : std::log(std::fabs(dm)); }

// e4m3 markets (per-row or per-side scales)
inline bool is_fp8(int dtype) { return dtype == TU_DTYPE_FP8E4M3 || dtype == TU_DTYPE_FP8E4M3_SIDE; }

// The library's kernels are built for sm_103a only (compute capability 10.3):
// any other device would fail at the first launch ("no kernel image").
inline bool device_supported(int dev) {
  int major = 0, minor = 0;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return major == 10 && minor == 3;
}

// Sweeps in the next block of a solve loop (the residual is read back between
// blocks). The first block is one sweep; each later one is at most twice the
// previous block, cut to the sweeps the per-sweep decay measured over the last
// block needs to take the residual to tol, and at most `cap`. r_prev and r are
// the residuals read after the last two blocks (r_prev < 0: none yet), last_k
// the sweeps of the last block (0: none yet).
inline int plan_block(int last_k, double r_prev, double r, double tol, int cap) {
  int k = last_k <= 0 ? 1 : 2 * last_k;
  if (last_k > 0 && r_prev > 0.0 && r > tol && r < r_prev && tol > 0.0) {
    const double log_q = std::log(r / r_prev) / (double)last_k;
    const double need = std::ceil(std::log(tol / r) / log_q);
    if (need >= 1.0 && need < (double)k) k = (int)need;
  }
  if (k > cap) k = cap;
  return k < 1 ? 1 : k;
}

// How a dense sweep in one pass over A-hat is laid out (dense.cu); cl = 0: the
// market takes two passes.
struct DensePlan {
  int cl = 0;        // CTAs of a cluster, each with a slice of every row's columns
  int width = 0;     // columns of a slice (multiple of 4)
  int rows = 1;      // rows of a pipeline unit
  int slots = 0;     // units in the ring
  int clusters = 0;  // clusters of the launch
};

}  // namespace tu

struct tu_market {
  int64_t N = 0, M = 0, d = 0;
  int64_t kp = 0;           // packed row length in elements: fused BF16 64, 128 or 256, FP8 128, 256
                            // or 512 bytes (fused_row_length); dense FP32 2d rounded up to 64
  bool fp8_caller_scales = false;  // FP8 created from caller e4m3 bytes and per-row scales
  float cmul = 0.0f;        // fused path: log2(e) / (2 sigma), times 2^(k_X + k_Y) for FP8 markets
  int dtype = 0, path = 0;
  double sigma = 1.0;
  int64_t partition = 0;
  cudaStream_t stream = nullptr;
  int device = 0;
  int num_sms = 0;
  tu::Side X, Y;
  float* Ahat = nullptr;     // dense path: N x ldA fp32
  int64_t ldA = 0;
  double* partials = nullptr;   // kMaxPartials x 4 doubles
  double* st = nullptr;          // device scalars (kSt*): shifts, sums, offsets and steps of both sides
  float* AhatT = nullptr;       // dense path: transpose of A-hat, M x ldN fp32
  tu::DensePlan dplan;          // dense path: the one-pass sweep's layout
  float* colsum = nullptr;      // its scratch: clusters x ldA column sums, then the clusters' scales (int)
  int64_t ldN = 0;
  double* results = nullptr;       // device, kResSlots, then the error word
  double* results_host = nullptr;  // pinned, likewise
  int* err_dev = nullptr;          // device error word (behind results)
  int* err_host = nullptr;         // pinned (behind results_host)
  char* arena = nullptr;           // one block that holds the buffers made at creation
  size_t arena_bytes = 0, arena_used = 0;
  bool measuring = false;          // dev_alloc only adds up arena_bytes
  float* scratch = nullptr;        // kScratch floats: maxima read back after factor and bias loads
  void* staging = nullptr;         // device staging buffer for host-memory arguments
  size_t staging_bytes = 0;
  void* aux = nullptr;             // ranked-list hand-over scratch (grow-only)
  size_t aux_bytes = 0;
  cudaGraphExec_t graph = nullptr; // captured block of sweeps
  int graph_sweeps = 0;
  int last_block = 0;              // sweeps of the last block
  bool use_graphs = true;          // tu_market_use_graphs
  int small_mode = 1;              // tu_market_set_small_tiles: 0 256-row own tiles, 1 128-row when they
                                   // fit one wave, 2 always 128-row
  int split = 1;                   // tu_market_set_split: partner ranges per own tile (fused sweeps)
  bool split_blocks = false;       // tu_market_set_partner_blocks: the ranges run one after another
  int64_t l2_bytes = 0;            // the device's L2 size (partner tiles: evict-last / evict-first policy)
  float4* split_part = nullptr;    // split > 1: partial row sums, split x max(N, M)
  int* split_cnt = nullptr;        // split > 1: arrivals per (own tile, 32-row block), zeroed
  int split_cap = 0;               // the split the buffers were sized for
  float4* cut_part = nullptr;      // cut half-sweeps: the ranges' sums, 2 x 256 per span of the larger plan
  float2* cut_m = nullptr;         // and their shifts (wide markets)
  int* cut_cnt = nullptr;          // arrivals per (own tile, 32-row block), zeroed
  bool translate = true;           // tu_market_set_translation: translation step before every half-sweep
  bool wide = false;               // factor range beyond one shift per half-sweep: per-row running maxima
  bool poisoned = false;
  std::string last_error;
  // benchmark timing (tu_profile_enable / tu_profile_read)
  // over-relaxation: device scalar read by every pass (graphs stay valid when it changes)
  double* omega_dev = nullptr;
  double* omega_host = nullptr;  // pinned staging for updates of omega_dev
  double omega_cfg = 1.0;        // 1: plain IPFP; (1, 2): fixed; 0: automatic in tu_ipfp_solve
  // serving: completion of the last asynchronous tu_ipfp_sweep (tu_market_query)
  cudaEvent_t done_ev = nullptr;
  double* query_host = nullptr;  // pinned: kResSlots doubles + the error word
  int64_t sweeps_enqueued = 0;
  int64_t query_sweeps = 0;
  // automatic relaxation of asynchronous sweeps (tu_market_relax_update)
  tu::RelaxControl relax;
  int64_t relax_base = 0;   // sweeps_enqueued when the controller was last reset
  int64_t relax_seen = -1;  // query_sweeps last fed to the controller
  bool profiling = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_pool;
  size_t ev_used = 0;
};

// ---------------------------------------------------------------------------
// Launchers (one translation unit each); all return cudaGetLastError().
// ---------------------------------------------------------------------------
namespace tu {

// reduce.cu
// Prepare the partner's FP32 vector for a half-sweep of the other side and the
// pass's scalars (with translate, the translation step taken before it).
// (offset: where in pvec the vector starts, 0 to 3)
cudaError_t launch_prep(tu_market* m, Side& partner, int fused_mode, int translate, int offset = 0);
// Reduce a pass's partials; after an update, also the own side's groups into
// the market scalars (ngroups: groups the pass wrote).
// prep_next: also set the scalars of the half-sweep that follows, which updates
// the other side (1: without, 2: with the translation step).
cudaError_t launch_finalize(tu_market* m, int nparts, int is_x, int residual, int update, int64_t ngroups,
                            int prep_next = 0);
// Groups and scalars of both sides from their stored potentials (after the
// potentials were set from outside a sweep).
cudaError_t launch_rescan(tu_market* m);
// Finalize a pass that updated a side (is_x: X) and prepare the half-sweep of the
// other side against it.
cudaError_t launch_between(tu_market* m, int nparts, int is_x, int residual, int64_t ngroups, int fused_mode,
                           int translate);
// Write the sides' pending offsets into their arrays (end of a block of sweeps).
cudaError_t launch_flush(tu_market* m);
cudaError_t launch_pack_factors(tu_market* m, Side& s, const void* A, const void* B, int src_dtype);
cudaError_t launch_init_side(tu_market* m, Side& s, const float* bias_dev, int has_bias);  // and the mass padding
cudaError_t launch_reset(tu_market* m);  // u = v = 1 on both sides, with their groups and scalars
cudaError_t launch_set_potentials(tu_market* m, Side& s, const float* log_u_dev);
cudaError_t launch_set_potentials64(tu_market* m, Side& s, const double* log_u_dev);
// FP64 state -> FP32 (either may be null)
cudaError_t launch_get_potentials(tu_market* m, float* out_x, float* out_y);
// the largest row norm into *out_max (zeroed by the caller)
cudaError_t launch_row_norms(tu_market* m, Side& s, float* out_max);
// FP8 markets: max |entry| of the FP32 factor pair (A, B: rows x d each) into *out_max
cudaError_t launch_max_abs(tu_market* m, const float* A, const float* B, int64_t count, float* out_max);
// FP8 markets: pack [A | B | 0] * 2^-k into s.fac8 (rows x 128 e4m3, round to nearest even, saturating)
constexpr int kPerRowScale = -1000000;  // launch_pack_fp8_rows: each row its own scale
cudaError_t launch_pack_fp8_rows(tu_market* m, Side& s, const float* A, const float* B, int side_k,
                                 unsigned int* bad);
cudaError_t launch_pack_fp8_bytes(tu_market* m, Side& s, const uint8_t* A, const uint8_t* B, const float* sc,
                                  unsigned int* bad);
cudaError_t launch_sum_sq(tu_market* m, Side& s, int is_x);  // results[kResXSq or kResYSq] = sum exp(2 log u)

// dense.cu
cudaError_t launch_dense_build(tu_market* m);
cudaError_t launch_dense_rowpass(tu_market* m, int residual, int update, int* nparts_out, int64_t* ngroups_out);
cudaError_t launch_dense_colpass(tu_market* m, int update, int* nparts_out, int64_t* ngroups_out);
// A whole sweep with one pass over A-hat (markets with a DensePlan): the X
// half-sweep and the column sums of the new u, then (after the X half-sweep's
// finalize has set the Y half-sweep's scalars) the Y update from them.
cudaError_t launch_dense_sweep(tu_market* m, int residual, int* nparts_out, int64_t* ngroups_out);
cudaError_t launch_dense_cols(tu_market* m, int* nparts_out, int64_t* ngroups_out);
DensePlan dense_plan(const tu_market* m);
size_t dense_plan_floats(const DensePlan& p);  // scratch of a plan, in floats

// fused.cu
cudaError_t fused_prepare(tu_market* m);  // tensor maps + kernel attributes
// The whole own side (nrows < 0), or own users [row0, row0 + nrows) only (no groups written).
cudaError_t launch_fused_halfsweep(tu_market* m, int side, int residual, int update, int* nparts_out,
                                   int64_t row0 = 0, int64_t nrows = -1);

// The cuts of a half-sweep of own_rows against partner_rows on sms SMs; kblocks:
// 128-byte k blocks of a packed row.
CutPlan cut_plan(int64_t own_rows, int64_t partner_rows, int kblocks, int sms);
// Scratch of cut launches, in ranges' slots of kFusedOwnRows rows (0: none).
int64_t cut_slots(const CutPlan& p);

// The fused half-sweep on caller-described device buffers (no market object).
struct FusedRaw {
  const __nv_bfloat16* own16;  // rows x kp packed own factors
  int64_t rows;
  const __nv_bfloat16* par16;  // cols x kp packed partner factors
  int64_t cols;
  int64_t kp;                  // 64 or 128
  double sigma;
  const float* g;              // prepared partner vector, >= ceil(cols / 128) * 128, -inf padded
  const double* lmax;          // partner shift
  const float* b2s;            // own bias / (2 sigma) or nullptr
  const double* mass;          // own capacities
  double* log_u;               // own log u (in: old, out: new)
  double* ell;                 // own ell (out)
  double* partials;            // >= min(ceil(rows / 256), num_sms) x 4
  int* err;
  int residual;
};
cudaError_t launch_fused_halfsweep_raw(const FusedRaw& r, cudaStream_t stream, int num_sms, int* nparts_out);

// One market of a batched launch, for the half-sweep that updates its "own"
// side against its "partner" side (device copy; the tensor maps keep their
// 128-byte alignment, so an array of these is a valid TMA operand array).
// Two per market: X against Y and Y against X.
struct BatchDesc {
  CUtensorMap tm_own;          // own packed factors, box kKBlock x kFusedOwnRows
  CUtensorMap tm_partner;      // partner packed factors, box kKBlock x kFusedPartnerRows
  const float* b2s;            // own bias / (2 sigma) or nullptr
  const double* mass;          // own capacities
  double* log_u;               // own potentials (in: old, out: new)
  double* ell;                 // own ell (out)
  const double* partner_ell;   // partner ell (read by the preparation kernel)
  float* g;                    // partner prepared vector (written by the preparation kernel)
  uint8_t* gfold;              // the partner's g / c operand of the extra MMA (Side::fold, written by the
                               // preparation kernel), or nullptr
  double* st;                  // the market's scalars (kSt*; shift and own offset of the pass)
  const float* fs_own;         // e4m3 markets: own per-row scales, else nullptr
  const float* fs_par;         // e4m3 markets: partner per-row scales, else nullptr
  float4* grp;                 // own-side groups (written by the pass, reduced by the finalize)
  const double* omega;         // over-relaxation factor of this market (device scalar)
  double dm_next;              // sum of own capacities - sum of partner capacities (the next step's tau)
  double log_dm;               // log |dm_next|
  int own_side;                // 0: X is own, 1: Y is own
  int translate;               // the market's translation-step setting at batch creation
  int64_t rows;                // own users
  int64_t partner_rows;        // partner users
  int64_t partner_rows_pad;    // partner vector length (multiple of kRowPad)
  int num_own_tiles;           // ceil(rows / kFusedOwnRows)
  int num_partner_tiles;       // ceil(partner_rows / kFusedPartnerRows)
  int cut_t0, cut_span;        // CutPlan of this half-sweep
  int cut_rows;                // rows of its tiles
  int slot0;                   // first own-tile slot of this market in the partials array
  float c;                     // log2(e) / (2 sigma)
};

// Epilogue warps that write per-tile partials in a batched launch (the warps
// that own the row updates); each own tile has kBatchSlotWarps x 4 doubles.
constexpr int kBatchSlotWarps = 8;

// A batched half-sweep: the CTA b processes items[cta_start[b] .. cta_start[b + 1])
// in order, an item being (market, own tile).
struct BatchLaunch {
  const BatchDesc* desc;   // device, indexed by market
  const int2* items;       // device
  const int* cta_start;    // device, grid + 1 entries
  double* partials;        // device, [slot][kBatchSlotWarps][4]
  int* err;
  int grid;
  int64_t kp;              // 64 or 128 (BF16), the same for every market
  int ksteps;              // the most of any member (FusedParams::ksteps)
  int dtype;               // the members' dtype (e4m3 markets: kp = 128 bytes per row, the same format)
  int residual;
  int update;
};
cudaError_t launch_fused_batch(const BatchLaunch& b, cudaStream_t stream);
// The steps of a packed row [F | K | 0] that the MMAs take: one is 32 bytes of it.
inline int k_steps(const tu_market* m) { return (int)((2 * m->d * (is_fp8(m->dtype) ? 1 : 2) + 31) / 32); }
// ranked lists / mu block through the tensor-core pipeline (partner vector prepared in log2 mode)
cudaError_t launch_fused_topk(tu_market* m, int side, int k, int64_t row0, int64_t nrows, int32_t* idx, float* logmu,
                              float* hand_v, int32_t* hand_i);
int mu_vector_offset(const tu_market* m, int64_t y0);
cudaError_t launch_fused_mu(tu_market* m, int64_t x0, int64_t nx, int64_t y0, int64_t ny, float* out, int64_t ld);

// topk.cu (dense-path outputs, read from A-hat)
cudaError_t launch_mu_block(tu_market* m, int64_t x0, int64_t nx, int64_t y0, int64_t ny, float* out,
                            int64_t ld);
cudaError_t launch_topk(tu_market* m, int side, int k, int64_t row0, int64_t nrows, int32_t* idx,
                        float* logmu);



}  // namespace tu

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------
#ifdef __CUDACC__
namespace tu {

constexpr double kLnHalf = -0.69314718055994530942;
constexpr float kLog2e = 1.4426950408889634f;

struct RowResult {
  double log_u, ell;
  double r_rel, r_abs;  // residual of the entering state (0 without)
  float u2;             // u^2
  bool finite;          // the new potentials
};

// ln (a + b + c) of a positive row sum given as three FP32 parts, to an
// absolute error of about 6e-8 whatever the size of the sum. The parts are
// added in FP32 with the rounding error of each addition kept (Knuth's
// two-sum), x = hi + lo; hi = m 2^e with m in [0.5, 1), so
// ln x = e ln 2 + ln m + lo / hi, and |ln m| < 0.7 keeps logf's rounding small.
// (logf(x) itself rounds to half an FP32 ulp of ln x: 4.8e-7 for the sums of
// ~1e6 terms of a large market, ln x ~ 14, which would put a floor of ~1e-6
// under the residual.)
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
// The logarithm as e ln 2 + the returned float, e an integer.
__device__ __forceinline__ float log_row_sum_parts(float a, float b, float c, int& e) {
  float e1, e2;
  const float s1 = two_sum(a, b, e1);
  const float hi = two_sum(s1, c, e2);
  const float lo = __fadd_rn(e1, e2);
  const float m = frexpf(hi, &e);
  return __fadd_rn(logf(m), __fdividef(lo, hi));
}
__device__ __forceinline__ double log_row_sum(float a, float b, float c) {
  int ex;
  const float lm = log_row_sum_parts(a, b, c, ex);
  return __dadd_rn((double)ex * 0.69314718055994530942, (double)lm);
}

__device__ __forceinline__ bool finite64(double v) {
  return ((uint32_t)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

// The closed-form update of Eq. iteration for one user, in logs.
//   ex, lm   : ex ln 2 + lm = log of sum_y exp(phi_hat_xy / (2 sigma) + ell_y - shift)
//   shift    : the partner-side shift (max_y ell_y) taken out of the sum
//   b2s      : this user's bias / (2 sigma)
//   log_s    = log(1/2) + b2s + shift + ex ln 2 + lm    (s = 1/2 sum_y A_xy v_y)
//   log u    = 1/2 log n - asinh(exp(log s - 1/2 log n)) (= sqrt(n + s^2) - s)
// With residual, r = u_old^2 + 2 u_old s - n is the row equation of Eq. IPFP
// evaluated at the state entering the half-sweep.
//
// Precision: the sums are FP32, so the transcendentals of the update are
// evaluated in FP32 (FP64 transcendentals are slow on this part) while the
// additions whose operands may be large and cancel (log s, log u, ell: |.| up
// to ~100 with popularity biases) stay in FP64. For z = log s - 1/2 log n > 0,
// asinh(e^z) = z + c(z) with c(z) = log1p(sqrt(1 + e^{-2z})) in (ln 2, 0.89],
// so only the bounded correction c is rounded to FP32 (absolute error ~1e-7).
// The residual r = u^2 + 2 u s - n (residual = kResidualExact) is formed from
// FP64 exponentials of the FP64 state, so a certified residual carries no FP32
// rounding; inside sweeps (kResidualEstimate), where it only decides when to
// certify, its terms are FP32 exponentials (absolute error ~2e-7 of n), which
// keeps two FP64 exponentials per row out of the half-sweep (FP64 throughput
// is a small fraction of FP32 on this part). The u^2 summed for the match
// count (sum n - sum u^2, where sum u^2 is a small part) is FP32.
//
// omega != 1 over-relaxes the update in the log domain:
// log u <- log u_old + omega * (update - log u_old) (same fixed point).
// An FP64 operation has a latency of about 80 cycles here and issues at 2 per
// clock and SM, conversions included, so the chain keeps to the additions that
// need it: doublings, comparisons and tests of finiteness are FP32 or integer,
// and the estimate's quotient r / n is FP32. (45 FP64 instructions per row and
// FP64 butterflies over all epilogue warps ended a tile in 15,000 cycles: half
// of the time of a 1,000 x 1,000 half-sweep. See row_partials.)
__device__ __forceinline__ RowResult row_update(int ex, float lm, double shift, float b2s, double mass,
                                                double log_u_old, int residual, double omega = 1.0) {
  RowResult o;
  const double b = (double)b2s;
  const float nf = (float)mass;
  const double ln = (double)logf(nf);  // log n
  const double ls = fma((double)ex, 0.69314718055994530942, __dadd_rn(__dadd_rn(shift, kLnHalf), b));  // log s - lm
  o.r_rel = 0.0;
  o.r_abs = 0.0;
  if (residual == kResidualExact) {
    // r = u^2 + 2 u s - n with u^2 = e^{2 log u}, 2 u s = e^{log u + log s + ln 2}
    const double r = exp(2.0 * log_u_old) + exp(log_u_old + (ls + (double)lm) + 0.69314718055994530942) - mass;
    o.r_abs = fabs(r);
    o.r_rel = fabs(r) / mass;
  } else if (residual == kResidualEstimate) {
    const float e2 = expf((float)__dadd_rn(__dadd_rn(__dadd_rn(log_u_old, 0.69314718055994530942), ls), (double)lm));
    const double r = __dadd_rn(__dadd_rn((double)expf(2.0f * (float)log_u_old), -mass), (double)e2);
    o.r_abs = fabs(r);
    o.r_rel = (double)__fdiv_rn(fabsf((float)r), nf);
  }
  // (rounded once: without lm the sum is the same for like rows, and so would be
  // the error of rounding it first, up to 2e-8 of their log u)
  const float z = (float)__dadd_rn(fma(-0.5, ln, ls), (double)lm);
  double lu;
  if (z > 0.0f) {
    const float c = log1pf(sqrtf(1.0f + expf(-2.0f * z)));
    lu = __dadd_rn(__dadd_rn(__dadd_rn(ln, -ls), -(double)lm), -(double)c);
  } else {
    lu = fma(0.5, ln, -(double)asinhf(expf(z)));
  }
  if (omega != 1.0) lu = log_u_old + omega * (lu - log_u_old);
  o.log_u = lu;
  o.ell = __dadd_rn(lu, b);
  o.u2 = expf(2.0f * (float)lu);
  o.finite = finite64(o.log_u) && finite64(o.ell);
  return o;
}

// Partials of one warp's rows (one per lane; lanes with valid = false
// contribute nothing), on lane 0: max r / n, sum |r|, sum u^2, non-finite
// count. The sums of u^2 (and of an estimate's |r|) add FP32 terms with their
// roundings kept; a certifying pass's |r| is summed in FP64.
struct RowPartials {
  double r_max, r_sum, sq, nf;
};
__device__ __forceinline__ RowPartials row_partials(const RowResult& rr, bool valid, int residual) {
  RowPartials p;
  float hi = valid ? rr.u2 : 0.0f, lo = 0.0f;
  for (int o = 16; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    float e;
    hi = two_sum(hi, h2, e);
    lo = __fadd_rn(__fadd_rn(lo, l2), e);
  }
  // (an infinite u^2 makes the error term NaN; the sum itself says what it is)
  p.sq = isfinite(lo) ? (double)hi + (double)lo : (double)hi;
  p.nf = (double)__popc(__ballot_sync(0xffffffffu, valid && !rr.finite));
  p.r_max = p.r_sum = 0.0;
  if (residual == kResidualNone) return p;
  // non-negative floating-point numbers order like their bits; a NaN is left out
  const double rel = valid && rr.r_rel == rr.r_rel ? rr.r_rel : 0.0;
  if (residual == kResidualExact) {
    const unsigned h = (unsigned)__double2hiint(rel), top = __reduce_max_sync(0xffffffffu, h);
    const unsigned l = __reduce_max_sync(0xffffffffu, h == top ? (unsigned)__double2loint(rel) : 0u);
    p.r_max = __hiloint2double((int)top, (int)l);
    double a = valid ? rr.r_abs : 0.0;
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    p.r_sum = a;
  } else {
    p.r_max = (double)__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint((float)rel)));
    float ah = valid ? (float)rr.r_abs : 0.0f, al = 0.0f;
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_xor_sync(0xffffffffu, ah, o), l2 = __shfl_xor_sync(0xffffffffu, al, o);
      float e;
      ah = two_sum(ah, h2, e);
      al = __fadd_rn(__fadd_rn(al, l2), e);
    }
    p.r_sum = isfinite(al) ? (double)ah + (double)al : (double)ah;
  }
  return p;
}
// p += q (one thread)
__device__ __forceinline__ void add_partials(RowPartials& p, const RowPartials& q) {
  p.r_max = q.r_max > p.r_max ? q.r_max : p.r_max;
  p.r_sum += q.r_sum;
  p.sq += q.sq;
  p.nf += q.nf;
}

// ---- translation step and the per-side scalars -------------------------------
// The translation step moves the log potentials of the side updated last by
// +tau and those of the side about to be updated by -tau. Everything it needs
// is kept in the per-market scalars (kSt*): the sums sum e^{2 log u} of both
// sides and the sides' shifts. The half-sweep that updates a side writes one
// (max 2 log u, scaled sum, max ell) group per 32 rows; a single-block
// finalize reduces the groups in a fixed order (the single-market and the
// batched finalize run the same routine with the same block size, so the
// batch's potentials stay bit-identical to the market's own sweeps) and
// computes tau for the next half-sweep; the move itself is recorded as a
// per-side offset and written to the arrays only when a side is next updated
// (for the updated side) or at the end of a block of sweeps.

// Order-preserving float <-> uint mapping for max on floats of any sign.
__device__ __forceinline__ unsigned int float_to_ordered(float f) {
  unsigned int u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ordered_to_float(unsigned int u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Block-wide maxima of two floats (every thread returns them).
// (red: 2 * blockDim.x / 32 floats; a NaN does not take part)
__device__ __forceinline__ void block_reduce_max2(float& a, float& b, float* red) {
  a = ordered_to_float(__reduce_max_sync(0xffffffffu, float_to_ordered(a)));
  b = ordered_to_float(__reduce_max_sync(0xffffffffu, float_to_ordered(b)));
  if (threadIdx.x % 32 == 0) {
    red[2 * (threadIdx.x / 32)] = a;
    red[2 * (threadIdx.x / 32) + 1] = b;
  }
  __syncthreads();
  for (int w = 0; w < (int)blockDim.x / 32; ++w) {
    a = fmaxf(a, red[2 * w]);
    b = fmaxf(b, red[2 * w + 1]);
  }
  __syncthreads();
}

// The group of one warp's 32 rows (lanes with valid = false contribute
// nothing), as {m, s, e, 0}: a reference m near the max of 2 log u (the max of
// the FP32-rounded values), the sum s of e^{2 log u - m} (the argument formed
// in FP64, the terms in FP32, summed by an FP32 butterfly whose result every
// lane shares), and e, a max of ell (of the FP32-rounded values; it serves as
// a shift, and e^{ell - shift} may exceed 1 by a rounding). Warp-collective;
// every lane returns the same group. A NaN potential makes s NaN (the
// translation step then falls back to tau = 0). One FP64 operation per row:
// FP64 throughput is a small fraction of FP32 on this part.
__device__ __forceinline__ float4 warp_group(double lu, double ell, bool valid) {
  const float m2 = 2.0f * (float)lu, e1 = (float)ell;
  const bool mok = valid && m2 == m2, eok = valid && e1 == e1;
  // (a NaN does not take part in the maxima)
  const float m = ordered_to_float(__reduce_max_sync(0xffffffffu, float_to_ordered(mok ? m2 : -INFINITY)));
  const float e = ordered_to_float(__reduce_max_sync(0xffffffffu, float_to_ordered(eok ? e1 : -INFINITY)));
  float t = (valid && m > -INFINITY) ? expf((float)fma(2.0, lu, -(double)m)) : 0.0f;
  if (valid && !mok) t = NAN;
  for (int o = 16; o > 0; o >>= 1) t = __fadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
  return make_float4(m, t, e, 0.0f);
}

// The empty group (no rows).
__device__ __forceinline__ float4 empty_group() { return make_float4(-INFINITY, 0.0f, -INFINITY, 0.0f); }

// (hi, lo) += (h2, l2): an FP32 sum carried with its rounding error. The
// two-sum is error-free and symmetric in its operands, so butterfly partners
// end with the same pair.
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h2, float l2) {
  float e;
  hi = two_sum(hi, h2, e);
  lo = __fadd_rn(__fadd_rn(lo, l2), e);
}

// Reduce `ng` groups in a fixed order (every thread returns the results):
// lmax = max e (the side's shift), and log sum e^{2 log u} = top + ln(hi + lo),
// where top = max m and hi + lo = sum s e^{m - top} (FP32 terms summed with
// their rounding errors kept; the logarithm is taken by the caller, once).
struct GroupTotal {
  float lmax, top, hi, lo;
};
__device__ __forceinline__ GroupTotal block_reduce_groups(const float4* grp, int64_t ng, float* red) {
  float mm = -INFINITY, me = -INFINITY;
  const float4 q0 = (int64_t)threadIdx.x < ng ? __ldcg(grp + threadIdx.x) : make_float4(-INFINITY, 0.0f, -INFINITY, 0.0f);
  mm = fmaxf(mm, q0.x);
  me = fmaxf(me, q0.z);
  for (int64_t i = threadIdx.x + blockDim.x; i < ng; i += blockDim.x) {
    const float4 q = __ldcg(grp + i);
    mm = fmaxf(mm, q.x);
    me = fmaxf(me, q.z);
  }
  GroupTotal r;
  block_reduce_max2(mm, me, red);
  r.top = mm;
  r.lmax = me;
  float hi = 0.0f, lo = 0.0f;
  if (q0.x > -INFINITY || isnan(q0.y)) pair_add(hi, lo, q0.y * expf(q0.x - r.top), 0.0f);
  for (int64_t i = threadIdx.x + blockDim.x; i < ng; i += blockDim.x) {
    const float4 q = __ldcg(grp + i);
    if (q.x > -INFINITY || isnan(q.y)) pair_add(hi, lo, q.y * expf(q.x - r.top), 0.0f);
  }
  for (int o = 16; o > 0; o >>= 1)
    pair_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o));
  if (threadIdx.x % 32 == 0) {
    red[2 * (threadIdx.x / 32)] = hi;
    red[2 * (threadIdx.x / 32) + 1] = lo;
  }
  __syncthreads();
  hi = 0.0f;
  lo = 0.0f;
  for (int w = 0; w < (int)blockDim.x / 32; ++w) pair_add(hi, lo, red[2 * w], red[2 * w + 1]);
  __syncthreads();
  r.hi = hi;
  r.lo = lo;
  return r;
}

// log sum e^{2 log u} of a reduced side (one thread).
__device__ __forceinline__ double group_log_sum(const GroupTotal& t) {
  return (double)t.top + log_row_sum(t.hi, t.lo, 0.0f);
}

// The translation step (an extension; Sec. 5 names acceleration from optimal
// transport as future work). IPFP is block coordinate ascent on the concave
// dual whose stationarity conditions are Eq. IPFP. Moving the partner side's
// log potentials up by tau and the own side's down by tau leaves every pair
// term A_xy u_x v_y unchanged, so along that line the dual reads
//   const + tau (sum mass_P - sum mass_O) - 1/2 e^{2 tau} P - 1/2 e^{-2 tau} O,
// P = sum_P e^{2 log p}, O = sum_O e^{2 log o}, and its maximiser is
// tau = 1/2 log z with z the positive root of P z^2 - dm z - O = 0,
// dm = sum mass_P - sum mass_O, given log_p = log P and log_o = log O.
// dm = 0: z = sqrt(O / P). Otherwise, with L = log |dm|,
// w = log(4 P O / dm^2) and q = log(1 + sqrt(1 + e^w)), the root
// z = (dm + R) / (2 P) for dm > 0 and 2 O / (R - dm) for dm < 0,
// R = sqrt(dm^2 + 4 P O) = |dm| sqrt(1 + e^w), is
// log z = L + q - log 2 - log P (dm > 0) or log 2 + log O - L - q (dm < 0),
// with no cancellation; for |w| > 60, q = w / 2 or log 2 to double precision.
// Non-finite inputs (non-finite potentials, which the half-sweep reports)
// give tau = 0.
// (L, of the two sides' capacities alone, comes from the host.)
__device__ __forceinline__ double translation_tau(double log_p, double log_o, double dm, double L) {
  const double ln2 = 0.69314718055994530942;
  double log_z;
  if (dm == 0.0) {
    log_z = 0.5 * __dadd_rn(log_o, -log_p);
  } else {
    const double w = __dadd_rn(__dadd_rn(__dadd_rn(2.0 * ln2, log_p), log_o), -2.0 * L);
    const double q = w > 60.0 ? 0.5 * w : (w < -60.0 ? ln2 : log1p(sqrt(1.0 + exp(w))));
    log_z = dm > 0.0 ? __dadd_rn(__dadd_rn(__dadd_rn(L, q), -ln2), -log_p)
                     : __dadd_rn(__dadd_rn(__dadd_rn(ln2, log_o), -L), -q);
  }
  const double tau = 0.5 * log_z;
  return isfinite(tau) ? tau : 0.0;
}

// Scalars of a half-sweep that updates side `own` (one thread, before the
// pass): the translation step it takes (tau = 0 unless `translate`), the
// partner shift the pass adds back (natural log) and the own offset under
// which it reads the entering potentials.
__device__ __forceinline__ void prep_scalars(double* st, int own, int translate) {
  const int par = 1 - own;
  const double tau = translate ? st[kStTauNext] : 0.0;
  st[kStTauUsed] = tau;
  st[kStShift] = st[kStLmax + par] + st[kStOff + par] + tau;
  st[kStOwnOff] = st[kStOff + own] - tau;
}

// Scalars after a half-sweep that updated side `own` (one thread): the own
// side's shift and sum from its groups (its arrays now hold true values), the
// step taken before the pass recorded on the partner, and tau for the next
// half-sweep, which updates the partner against this side
// (dm_next = sum mass_own - sum mass_partner).
__device__ __forceinline__ double finite_or_zero(double v) { return (v > -INFINITY && v < INFINITY) ? v : 0.0; }
__device__ __forceinline__ void finish_scalars(double* st, int own, const GroupTotal& g, double dm_next,
                                               double log_dm) {
  const int par = 1 - own;
  const double tau = st[kStTauUsed];
  const double log_s_own = group_log_sum(g);
  // non-finite potentials are reported by the pass (its non-finite count)
  st[kStLmax + own] = finite_or_zero((double)g.lmax);
  st[kStLogS + own] = log_s_own;
  st[kStOff + own] = 0.0;
  st[kStOff + par] += tau;
  st[kStLogS + par] += 2.0 * tau;
  st[kStTauUsed] = 0.0;
  st[kStTauNext] = translation_tau(log_s_own, st[kStLogS + par], dm_next, log_dm);
}

// Scalars of both sides from their reduced groups (one thread; potentials set
// from outside a sweep): shifts, sums, no offsets, and tau for the next
// half-sweep, which updates X against Y (dm = sum m - sum n).
__device__ __forceinline__ void rescan_scalars(double* st, const GroupTotal& x, const GroupTotal& y,
                                               double dm_y_minus_x, double log_dm) {
  const double sx = group_log_sum(x), sy = group_log_sum(y);
  st[kStLmax + 0] = finite_or_zero((double)x.lmax);
  st[kStLmax + 1] = finite_or_zero((double)y.lmax);
  st[kStLogS + 0] = sx;
  st[kStLogS + 1] = sy;
  st[kStOff + 0] = 0.0;
  st[kStOff + 1] = 0.0;
  st[kStTauUsed] = 0.0;
  st[kStTauNext] = translation_tau(sy, sx, dm_y_minus_x, log_dm);
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Time limit of every device-side wait. No legitimate wait in these kernels
// lasts more than microseconds; a wait that runs out sets an error word.
constexpr uint64_t kWaitLimitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---- mbarrier --------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase with the given parity. Returns false when the
// time limit runs out or another role of the CTA has raised the abort flag.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > limit_ns) return false;
  }
}

// The address of a shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
// Store to the shared memory of a CTA of the cluster, counted in bytes on an
// mbarrier of that CTA (which orders it as it does a bulk copy's writes).
__device__ __forceinline__ void cluster_store_async(uint32_t a, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a), "f"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cluster_store_async2(uint32_t a, float v0, float v1, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a), "f"(v0),
               "f"(v1), "r"(bar)
               : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Arrive on an mbarrier of a CTA of the cluster, ordering no memory of other
// proxies or CTAs (what it announces here are TMEM reads, which
// tcgen05.fence::before_thread_sync orders).
__device__ __forceinline__ void cluster_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Every thread of every CTA of the cluster.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Bounded wait that ignores the abort flag: used while draining after an abort,
// so that copies and MMAs already issued complete before shared memory or TMEM
// is released.
__device__ __forceinline__ bool mbar_wait_drain(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > limit_ns) return false;
  }
  return true;
}

// ---- TMA -------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
// The same with an L2 cache policy (createpolicy) for the loaded lines.
__device__ __forceinline__ void tma_load_2d_hint(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int x, int y,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, "
      "%4}], [%2], %5;" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
// L2 policy: the given fraction of the accessed lines evict last, the rest
// with their priority unchanged (evict-first would drop a line before the
// other CTAs of the same wave read it).
__device__ __forceinline__ uint64_t l2_policy_keep_fraction(float fraction) {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.L2::evict_unchanged.b64 %0, %1;" : "=l"(pol) : "f"(fraction));
  return pol;
}
__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// Order earlier writes of a tensor map held in global memory before its use by TMA.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}

// A load by one CTA of a pair, counted on an mbarrier of the pair's first CTA
// (bar: its cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(void* smem_dst, const CUtensorMap* map, uint32_t bar, int x,
                                                      int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}

// ---- tcgen05 ---------------------------------------------------------------
// Pairs of CTAs (cta_group::2): both CTAs of the pair allocate and free; the
// first one issues. D's rows 0-127 (A's, from the first CTA's shared memory)
// are in the first CTA's TMEM, rows 128-255 in the second's; each CTA's shared
// memory holds half of B's rows, at the same offset.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_e4m3_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the mbarrier at this offset in both CTAs.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((unsigned short)3)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, both K-major, BF16 in, FP32 accumulate.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, both K-major, e4m3 in (32 per 32-byte K step), FP32 accumulate.
__device__ __forceinline__ void umma_e4m3(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on an mbarrier once every tcgen05 operation issued so far by this thread completes.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t is;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(is));
  return is != 0;
}

// The folded operand of partner row i (Side::fold): v = g_i * (1 / c) split into
// three BF16 values hi + mid + lo (24 significant bits; -inf padding gives
// hi = -inf, the others 0), written as the row's K = 16 operand of the fused
// kernel's extra MMA (columns 0-2, the rest zero) in the unswizzled K-major
// tcgen05 layout of 128-row tiles:
// byte (i / 128) * 4096 + ((i % 128) / 8) * 256 + (k / 8) * 128 + (i % 8) * 16 + (k % 8) * 2.
// With c, the rounding of 1 / c, which moves every g alike, is made good in lo
// and a fourth value (e4m3 with one scale per side, two k blocks: rms error of
// log u, d = 100, sigma = 0.35, 7.9e-8 without, 4.1e-8 with; 6.7e-8 with g added
// in FP32).
__device__ __forceinline__ void write_fold_row(uint4* fold, int64_t i, float g, float inv_c, float c = 0.0f) {
  unsigned short b[4] = {0, 0, 0, 0};
  if (isinf(g)) {
    b[0] = __bfloat16_as_ushort(__float2bfloat16_rn(g));
  } else {
    const float v = g * inv_c;
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    float r2 = r1 - __bfloat162float(mid);
    if (c != 0.0f) r2 += fmaf(-v, c, g) * inv_c;  // what v misses of g / c
    const __nv_bfloat16 lo = __float2bfloat16_rn(r2);
    if (c != 0.0f) b[3] = __bfloat16_as_ushort(__float2bfloat16_rn(r2 - __bfloat162float(lo)));
    b[0] = __bfloat16_as_ushort(hi);
    b[1] = __bfloat16_as_ushort(mid);
    b[2] = __bfloat16_as_ushort(lo);
  }
  const int64_t t = i / 128, r = i % 128;
  const int64_t q = t * 256 + (r / 8) * 16 + (r % 8);  // 16-byte chunk of columns 0-7
  fold[q] = make_uint4((uint32_t)b[0] | ((uint32_t)b[1] << 16), (uint32_t)b[2] | ((uint32_t)b[3] << 16), 0u, 0u);
  fold[q + 8] = make_uint4(0u, 0u, 0u, 0u);  // columns 8-15
}

// Shared-memory descriptor of an unswizzled K-major operand: core matrices of
// 8 rows x 16 bytes, `lbo` bytes apart along K and `sbo` bytes apart along
// M / N (version 1, layout type 0).
__device__ __forceinline__ uint64_t sdesc_none(uint32_t smem_addr, uint32_t lbo, uint32_t sbo) {
  uint64_t desc = 0;
  desc |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  desc |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  desc |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  desc |= (uint64_t)1u << 46;
  return desc;
}

// Shared-memory matrix descriptor for a K-major tile written by TMA with
// 128-byte swizzle: rows of 128 bytes, 8-row atoms 1024 bytes apart.
//   bits  0-13 start address >> 4     bits 16-29 leading byte offset >> 4 (unused here: 1)
//   bits 32-45 stride byte offset >> 4 (1024 B)   bits 46-47 descriptor version (1)
//   bits 61-63 layout: 2 = 128-byte swizzle
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t smem_addr) {
  uint64_t desc = 0;
  desc |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  desc |= (uint64_t)1u << 16;
  desc |= (uint64_t)(1024u >> 4) << 32;
  desc |= (uint64_t)1u << 46;
  desc |= (uint64_t)2u << 61;
  return desc;
}

// Instruction descriptor of tcgen05.mma kind::f16: D FP32 (bits 4-5 = 1),
// A and B BF16 (bits 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// Instruction descriptor of tcgen05.mma kind::f8f6f4: D FP32 (bits 4-5 = 1),
// A and B e4m3 (format 0 in bits 7-9 and 10-12), both K-major, N >> 3, M >> 4.
__host__ __device__ constexpr uint32_t idesc_e4m3_f32(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// 32 lanes x 32 columns of FP32 from TMEM (lane quadrant fixed by the warp), then wait.
__device__ __forceinline__ void tmem_ld32x32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

}  // namespace tu
#endif  // __CUDACC__
