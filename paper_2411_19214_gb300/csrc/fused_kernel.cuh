// fused_kernel.cuh -- the kernel of the mini-batch IPFP half-sweep (Alg. 2, Eq. iteration_minibatch) on
// sm_103a tensor cores. Phi is formed tile by tile and never written to HBM.
//
// For the half-sweep that updates side "own" against side "partner":
//   S_r = sum_c exp2( c * <a_r, b_c> + g_c ),   c = log2(e) / (2 sigma),
//   g_c = (ell_c - max ell) * log2(e)  (partner potential incl. bias, shifted <= 0),
// then log s_r = log(1/2) + bias_r/(2 sigma) + max ell + log S_r and the
// closed-form update of Eq. iteration gives the new log u_r.
//
// Because the partner biases are folded into g and the shift is the maximum of
// g, every exponent is bounded by c * |a_r| * |b_c| (checked on the host), so
// no per-pair running maximum is needed: the running-max rescale of
// flash-attention collapses to one shift per half-sweep.
//
// CTA layout (576 threads, one CTA per SM, persistent over own tiles; a
// half-sweep of rows of two or more k blocks runs on pairs of CTAs (PAIR): a
// cluster of two takes two own tiles, each CTA holds half of every partner
// tile, and the leader's MMA warp issues cta_group::2 MMAs for both):
//   warp 0     : producer (one elected lane): TMA loads of the own tile
//                [F|K]_j (256 rows x kp) once per own tile (double-buffered
//                when kp = 64) and of partner tiles (128 rows x kp) through a
//                STAGES-deep shared-memory ring (a stage is a whole partner
//                tile, or with four 128-byte k blocks per row one k block of
//                it, in a pair two), plus each partner tile's g: folded (see
//                fold_for), 4 KB of MMA operand in the stage, else 128 floats
//                (e4m3 with row scales: and the 128 scales) into an 8-slot
//                ring that the epilogue reads with broadcast loads.
//   warp 1     : MMA issuer: two tcgen05.mma M=128 N=128 chains
//                (own rows 0-127 and 128-255; a pair: M=256 over both CTAs)
//                per partner tile into one of two TMEM accumulator buffers
//                (2 x 256 columns = all 512).
//   warps 2-17 : epilogue: epilogue warp e reads TMEM lane quadrant (e+2)%4
//                of own sub-tile (e/4)%2 and column half e/8 of every partner
//                tile, i.e. one own row and 64 columns per thread, so the row
//                reduction stays inside the thread; the two column halves of
//                a row meet through shared memory at the end of the own tile.
//                TMEM loads run one 32-column chunk ahead of the arithmetic;
//                per pair of columns one packed FMA (f32x2; a multiply where
//                g is folded), two ex2.approx and one packed add; per-tile partials go into a compensated
//                (Kahan) sum.
// In a batched launch the own tiles of a CTA come from a list of
// (market, own tile) items of many independent markets.
// Every wait is bounded (kWaitLimitNs); a wait that runs out raises the
// abort flag and the error word, the roles drain, TMEM is freed, and the
// kernel returns.
#pragma once

#include "tu_internal.cuh"

namespace tu {

// Epilogue modes of the one fused kernel: the same TMA / MMA pipeline forms
// the tiles of c * phi_hat + g; the epilogue either reduces them (a half-sweep),
// keeps the k best columns of every row (ranked lists) or writes mu.
// Markets whose factor range is too wide for one shift per half-sweep (see
// market.cu) take kModeSweepWide: a half-sweep that keeps a running maximum
// per row and rescales the row's sum whenever it grows (the log-domain
// rescale of an online softmax), so that no term's exponent exceeds 0.
enum : int { kModeSweep = 0, kModeTopK = 1, kModeMu = 2, kModeTopKShared = 3, kModeSweepWide = 4 };

// Operand formats: BF16, e4m3 with one scale per side, e4m3 with one per row.
enum : int { kFmtBF16 = 0, kFmtE4M3Side = 1, kFmtE4M3Rows = 2 };

struct FusedParams {
  int64_t rows;            // own users of this launch: [row0, row0 + rows)
  int64_t row0;            // first own user
  int64_t col0;            // first partner column streamed (multiple of 4)
  int64_t ncols;           // partner columns streamed: [col0, col0 + ncols)
  int num_own_tiles;       // ceil(rows / 256)
  int num_partner_tiles;   // ceil(ncols / 128)
  int ksteps;              // 32-byte steps of a packed row that hold factors (the rest is zeros)  (sweep)
  float c;                 // log2(e) / (2 sigma)
  const float* g;          // partner prepared potentials (index = partner user), -inf padded
  const double* lmax;      // partner shift (natural log)
  const double* own_off;   // offset added to the stored own potentials, or nullptr for 0   (sweep)
  float4* grp;             // own-side groups written by an updating pass, or nullptr        (sweep)
  const float* b2s;        // own bias / (2 sigma), or nullptr          (sweep)
  const double* mass;      // own capacities                             (sweep)
  double* log_u;           // own potentials (in: old, out: new)          (sweep)
  double* ell;             // own ell: out (sweep), in (ranked lists, mu)
  double* partials;        // [gridDim.x][4]                              (sweep)
  int* err;                // device error word
  int residual;
  int update;
  const double* omega;     // over-relaxation factor (device scalar) or nullptr for 1  (sweep)
  // batched launches: per-market descriptors and this launch's item lists
  const BatchDesc* bdesc;
  const int2* items;
  const int* cta_start;
  // ranked lists: for own user row0 + r, idx[r * k + i], logmu[r * k + i], best first
  int k;
  int32_t* idx;
  float* logmu;
  float* hand_v;           // rows x k scratch: second column half's list
  int32_t* hand_i;
  // mu block: out[(r) * ld + (col - y0)] for partner col in [y0, y0 + ny)
  float* out;
  int64_t ld;
  int64_t y0;
  int64_t ny;
  int vec;                 // out, ld and the columns allow 16-byte stores
  // e4m3 factors: per-row scales of the own side (index row0 + r) and of the
  // partner side (index = partner user); the product of row r and partner
  // column j is fs_own[r] * fs_par[j] * <e4m3 row r, e4m3 row j>
  const float* fs_own;
  const float* fs_par;
  // partner split (single-market half-sweeps, 1 = off): an item is an own
  // tile and one of `split` contiguous ranges of its partner tiles; each
  // epilogue warp writes its rows' partial sums to part[s * rows + r], and the
  // warp that completes a (tile, 32-row block), counted in split_cnt, sums
  // the partials in range order and updates the rows
  int split;
  int range_major;         // items ordered range by range (every own tile against range 0 first)
  // L2 residency of the partner matrix (single-market launches): this
  // fraction of its lines is loaded evict-last, so that a partner matrix
  // larger than L2 keeps a fixed part resident across the waves of own tiles
  // (0: no hint)
  float l2_keep;
  float4* part;
  float2* part_m;          // wide markets: the partials' shifts
  int* split_cnt;
  // the market's cuts (CutPlan; cut_span = 0: none). A SPLIT launch with
  // split = 1 gives tiles [0, cut_t0) to CTAs whole and every span of the rest
  // to one CTA; other launches add a row's ranges in turn
  int cut_t0;
  int cut_span;
  int cut_spans;
  int cut_ptiles;          // partner tiles of the market
  int cut_rows;            // rows of the tiles that are cut
  // folded g (see fold_for): the partner side's g / c as the
  // K = 16 operand of one extra MMA per chain and partner tile, 4 KB per
  // partner tile of 128 rows in the unswizzled K-major layout (written by the
  // preparation kernel)
  const uint8_t* gfold;
};

namespace {

constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + kEpiWarps * 32;  // producer warp, MMA warp, epilogue warps
constexpr int kOwnBytesPerKB = kFusedOwnRows * 128;          // 32 KB per 64-wide k block
constexpr int kPartnerBytesPerKB = kFusedPartnerRows * 128;  // 16 KB per 64-wide k block
constexpr int kGSlots = 8;                                   // g ring depth
constexpr int kGBytes = kFusedPartnerRows * 4;               // one partner tile of g (512 B)
constexpr uint32_t kTmemCols = 512;



// Own-tile buffers: with one 128-byte k block per row the next own tile is
// loaded while the current one is still in use (short items of batched
// launches); with two or four there is room for one only.
template <int KB>
constexpr int kABufs = KB == 1 ? 2 : 1;

// k blocks per partner stage: with four k blocks per row (d up to 128 in
// BF16, 256 in e4m3) a whole 64 KB partner tile would leave room for one
// stage beside the 128 KB own tile, so a stage then carries one k block and a
// partner tile takes four stages.
// A pair's CTAs hold half of a partner tile each, so two k blocks fit there.
constexpr int kbs_for(int KB, bool pair = false) { return KB == 4 ? (pair ? 2 : 1) : KB; }


// shared memory: [A: ABUFS x KB x 32 KB][B: STAGES x KBS x 16 KB][g ring: 8 x 512 B]
//                [per-row scales: scale ring 8 x 512 B][barriers and flags: 512 B]
//                [reduction: 512 B][row hand-over: 2 x 256 floats]
constexpr int kTailBytes = 512 + 512 + 2 * kFusedOwnRows * 4;
// folded g: the partner tile's K = 16 operand rides in its (last) stage, the
// own side's constant operand (ones in columns 0-3) is one tile of its own.
// Taken for rows of one and two k blocks (d <= 64 in BF16, d <= 128 in e4m3 with
// one scale per side), where the tensor pipe has room for one more MMA per
// chain and the epilogue, which bounds these kernels, sheds its g loads.
// One block: batched d = 32 half-sweep 5.44 -> 5.12 ms, a 1e5 d = 32 sweep
// 3.54 -> 3.37 ms. Two blocks, on pairs of CTAs: a 100,003 x 79,999 d = 64 sweep
// 2.74 -> 2.60 ms. Without pairs, where shared memory is short, two blocks lose a
// little (own-tile mode 0, d = 64: 100,003 x 79,999 3.31 ms unfolded, 3.45 folded,
// 20,000 x 15,001 0.249 and 0.254; a row range of 50,000 1.03 and 1.07; batches of
// 56 markets 2.71 and 2.81, of 512 small ones 0.487 and 0.483) and fold all the
// same: a market has the same bits in every launch shape. With four blocks the
// tensor pipe is the bound. e4m3: the fold MMA is a separate
// kind::f16 MMA (BF16 ones x BF16 g / c) into the same FP32 accumulator. e4m3
// rows with per-row scales do not fold: the accumulator holds phi over the own
// row's scale, so a per-column constant is not g in every row. Wide half-sweeps
// do not either: c phi and g may be hundreds and cancel, and g * (1 / c) through
// the accumulator and back rounds three times at that size where a fused
// multiply-add rounds once (rms error of log u at sigma = 0.01, d = 32, 6,001 x
// 9,001: 4.6e-6 folded, 3.5e-6 not; 80,000 x 100,001, d = 64: 3.10 ms per sweep
// folded, 3.45 not). In narrow markets the error is smaller folded for most sigma
// (6,001 x 9,001, d = 64, rms of log u folded / not: 0.53 at sigma = 0.5 and 1, 0.9
// at 0.35 and 0.7, 0.6 at 0.25, 1.0 at 0.1; below, where exponents reach tens, up
// to 1.2 of 1e-7 to 3e-7).
constexpr int kFoldBytes = kFusedPartnerRows * 32;
constexpr bool fold_for(int KB, int MODE, bool BATCH, int fmt, bool nofold) {
  return MODE == kModeSweep && (fmt == kFmtBF16 || fmt == kFmtE4M3Side) && KB <= 2 && !nofold;
}
constexpr int stage_bytes(int KB, bool fold, bool pair = false) {
  return (kbs_for(KB, pair) * kPartnerBytesPerKB + (fold ? kFoldBytes : 0)) / (pair ? 2 : 1);
}
constexpr int smem_bytes(int KB, int fmt, int stages, bool fold = false, bool pair = false) {
  return 1024 /*alignment slack*/ + (KB == 1 ? 2 : 1) * KB * kOwnBytesPerKB + stages * stage_bytes(KB, fold, pair) +
         (fold ? kFoldBytes : 0) + kGSlots * kGBytes * (fmt == kFmtE4M3Rows ? 2 : 1) + kTailBytes;
}

__device__ __forceinline__ void raise_error(int* err, volatile int* abort_flag, int code) {
  atomicCAS(err, kErrNone, code);
  *abort_flag = 1;
}

// 1D bulk copy global -> shared, completion counted on an mbarrier (16-byte aligned, size % 16 == 0).
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(gsrc)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Issue a 32-lane x 32-column FP32 TMEM load without waiting for it.
__device__ __forceinline__ void tmem_ld_issue(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// Wait for the outstanding TMEM loads; the registers are passed through so
// that no use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}

// acc(2 lanes) += (ex2(phi0 * c + g0), ex2(phi1 * c + g1)) with packed FP32x2 FMA and add.
__device__ __forceinline__ void pair_step(uint64_t& acc, uint32_t phi0, uint32_t phi1, float g0, float g1,
                                          uint64_t cc) {
  asm("{\n\t.reg .b64 a, gg, t, e;\n\t.reg .f32 t0, t1, e0, e1;\n\t"
      "mov.b64 a, {%1, %2};\n\t"
      "mov.b64 gg, {%3, %4};\n\t"
      "fma.rn.f32x2 t, a, %5, gg;\n\t"
      "mov.b64 {t0, t1}, t;\n\t"
      "ex2.approx.ftz.f32 e0, t0;\n\t"
      "ex2.approx.ftz.f32 e1, t1;\n\t"
      "mov.b64 e, {e0, e1};\n\t"
      "add.rn.f32x2 %0, %0, e;\n\t}"
      : "+l"(acc)
      : "r"(phi0), "r"(phi1), "f"(g0), "f"(g1), "l"(cc));
}

// e4m3 factors: acc += (ex2(phi0 f0 c + g0), ex2(phi1 f1 c + g1)), f the
// partner rows' scales (the own row's scale is folded into c).
__device__ __forceinline__ void pair_step_scaled(uint64_t& acc, uint32_t phi0, uint32_t phi1, float g0, float g1,
                                                 float f0, float f1, uint64_t cc) {
  asm("{\n\t.reg .b64 a, gg, ff, t, e;\n\t.reg .f32 t0, t1, e0, e1;\n\t"
      "mov.b64 a, {%1, %2};\n\t"
      "mov.b64 gg, {%3, %4};\n\t"
      "mov.b64 ff, {%5, %6};\n\t"
      "mul.rn.f32x2 t, a, ff;\n\t"
      "fma.rn.f32x2 t, t, %7, gg;\n\t"
      "mov.b64 {t0, t1}, t;\n\t"
      "ex2.approx.ftz.f32 e0, t0;\n\t"
      "ex2.approx.ftz.f32 e1, t1;\n\t"
      "mov.b64 e, {e0, e1};\n\t"
      "add.rn.f32x2 %0, %0, e;\n\t}"
      : "+l"(acc)
      : "r"(phi0), "r"(phi1), "f"(g0), "f"(g1), "f"(f0), "f"(f1), "l"(cc));
}

// Folded g: acc += (ex2(D0 * c), ex2(D1 * c)), D = phi + g / c from the MMA.
__device__ __forceinline__ void pair_step_fold(uint64_t& acc, uint32_t d0, uint32_t d1, uint64_t cc) {
  asm("{\n\t.reg .b64 a, t, e;\n\t.reg .f32 t0, t1, e0, e1;\n\t"
      "mov.b64 a, {%1, %2};\n\t"
      "mul.rn.f32x2 t, a, %3;\n\t"
      "mov.b64 {t0, t1}, t;\n\t"
      "ex2.approx.ftz.f32 e0, t0;\n\t"
      "ex2.approx.ftz.f32 e1, t1;\n\t"
      "mov.b64 e, {e0, e1};\n\t"
      "add.rn.f32x2 %0, %0, e;\n\t}"
      : "+l"(acc)
      : "r"(d0), "r"(d1), "l"(cc));
}

__device__ __forceinline__ void chunk_sum_fold(const uint32_t (&v)[32], uint64_t cc, uint64_t (&acc)[4]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) pair_step_fold(acc[i & 3], v[2 * i], v[2 * i + 1], cc);
}

// phi of column i of a chunk, times the partner row's scale (e4m3 factors
// with per-row scales)
template <bool RS>
__device__ __forceinline__ float scaled_phi(uint32_t v, const float* fs, int i) {
  if constexpr (RS) return __uint_as_float(v) * fs[i];
  return __uint_as_float(v);
}

__device__ __forceinline__ float unpack_sum(uint64_t a) {
  return __uint_as_float((uint32_t)a) + __uint_as_float((uint32_t)(a >> 32));
}

// Sum over one 32-column chunk: 16 packed pairs into four packed accumulators.
template <bool RS>
__device__ __forceinline__ void chunk_sum(const uint32_t (&v)[32], const float4* gs4, const float4* fs4, uint64_t cc,
                                          uint64_t (&acc)[4]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 gg = gs4[i];
    if constexpr (RS) {
      const float4 ff = fs4[i];
      pair_step_scaled(acc[(2 * i) & 3], v[4 * i + 0], v[4 * i + 1], gg.x, gg.y, ff.x, ff.y, cc);
      pair_step_scaled(acc[(2 * i + 1) & 3], v[4 * i + 2], v[4 * i + 3], gg.z, gg.w, ff.z, ff.w, cc);
    } else {
      pair_step(acc[(2 * i) & 3], v[4 * i + 0], v[4 * i + 1], gg.x, gg.y, cc);
      pair_step(acc[(2 * i + 1) & 3], v[4 * i + 2], v[4 * i + 3], gg.z, gg.w, cc);
    }
  }
}

// ---- wide markets: one pass with a running maximum per row -----------------

// t = (phi0, phi1) * c + (g0, g1); e4m3 per-row scales: (phi0 f0, phi1 f1) * c + (g0, g1)
template <bool RS>
__device__ __forceinline__ uint64_t pair_exponents(uint32_t phi0, uint32_t phi1, float g0, float g1, float f0,
                                                   float f1, uint64_t cc) {
  uint64_t t;
  if constexpr (RS) {
    asm("{\n\t.reg .b64 a, gg, ff, x;\n\t"
        "mov.b64 a, {%1, %2};\n\t"
        "mov.b64 gg, {%3, %4};\n\t"
        "mov.b64 ff, {%5, %6};\n\t"
        "mul.rn.f32x2 x, a, ff;\n\t"
        "fma.rn.f32x2 %0, x, %7, gg;\n\t}"
        : "=l"(t)
        : "r"(phi0), "r"(phi1), "f"(g0), "f"(g1), "f"(f0), "f"(f1), "l"(cc));
  } else {
    asm("{\n\t.reg .b64 a, gg;\n\t"
        "mov.b64 a, {%1, %2};\n\t"
        "mov.b64 gg, {%3, %4};\n\t"
        "fma.rn.f32x2 %0, a, %5, gg;\n\t}"
        : "=l"(t)
        : "r"(phi0), "r"(phi1), "f"(g0), "f"(g1), "l"(cc));
  }
  return t;
}

// acc(2 lanes) += (ex2(t0 + m), ex2(t1 + m)), mm = (m, m)
__device__ __forceinline__ void ex2_add_shifted(uint64_t& acc, uint64_t t, uint64_t mm) {
  asm("{\n\t.reg .b64 x, e;\n\t.reg .f32 x0, x1, e0, e1;\n\t"
      "add.rn.f32x2 x, %1, %2;\n\t"
      "mov.b64 {x0, x1}, x;\n\t"
      "ex2.approx.ftz.f32 e0, x0;\n\t"
      "ex2.approx.ftz.f32 e1, x1;\n\t"
      "mov.b64 e, {e0, e1};\n\t"
      "add.rn.f32x2 %0, %0, e;\n\t}"
      : "+l"(acc)
      : "l"(t), "l"(mm));
}

// acc(2 lanes) *= (s, s)
__device__ __forceinline__ void scale2(uint64_t& acc, float s) {
  const uint64_t ss = ((uint64_t)__float_as_uint(s) << 32) | __float_as_uint(s);
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(ss));
}

// The larger of a, b and c; NaN if any of them is NaN.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// 2^d for an integer-valued d <= 0, as an exact power of two; 0 for d below
// -126 (FP32's normal range), for -inf and for NaN.
__device__ __forceinline__ float exp2_int(float d) {
  return d >= -126.0f ? __int_as_float((127 + (int)d) << 23) : 0.0f;
}

// One 32-column chunk of a wide market's row: the exponents t = c * phi + g,
// their largest; when that exceeds the row's running shift M (an integer,
// -inf before the first term) the shift becomes M' = ceil(max) and all the
// row has summed so far (this tile's packed partials acc, the compensated
// sum over the earlier tiles) is multiplied by 2^(M - M'), a power of two,
// so exactly; then acc += 2^(t - M). Every term is at most 1, and the row's
// log-sum is log(sum) + M ln 2.
template <bool RS>
__device__ __forceinline__ void chunk_sum_wide(uint32_t (&v)[32], const float4* gs4, const float4* fs4, uint64_t cc,
                                               uint64_t (&acc)[4], float& M, float& sum, float& comp) {
  // the exponents replace the loaded values in place
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 gg = gs4[i];
    float4 ff = make_float4(1.f, 1.f, 1.f, 1.f);
    if constexpr (RS) ff = fs4[i];
    const uint64_t t0 = pair_exponents<RS>(v[4 * i + 0], v[4 * i + 1], gg.x, gg.y, ff.x, ff.y, cc);
    const uint64_t t1 = pair_exponents<RS>(v[4 * i + 2], v[4 * i + 3], gg.z, gg.w, ff.z, ff.w, cc);
    v[4 * i + 0] = (uint32_t)t0;
    v[4 * i + 1] = (uint32_t)(t0 >> 32);
    v[4 * i + 2] = (uint32_t)t1;
    v[4 * i + 3] = (uint32_t)(t1 >> 32);
  }
  float mx = -INFINITY;
#pragma unroll
  for (int k = 0; k < 16; ++k) mx = max3_nan(mx, __uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1]));
  if (!(mx <= M)) {  // a larger maximum (or NaN, which then reaches the sum)
    const float Mn = ceilf(mx);
    const float sc = exp2_int(M - Mn);
    sum *= sc;
    comp *= sc;
#pragma unroll
    for (int k = 0; k < 4; ++k) scale2(acc[k], sc);
    M = Mn;
  }
  if (M == -INFINITY) return;  // every exponent so far is -inf: no terms
  const uint64_t mm = ((uint64_t)__float_as_uint(-M) << 32) | __float_as_uint(-M);
#pragma unroll
  for (int k = 0; k < 16; ++k)
    ex2_add_shifted(acc[k & 3], ((uint64_t)v[2 * k + 1] << 32) | v[2 * k], mm);
}

constexpr int kMaxTopK = 64;

// Insert score s of partner col into a thread's list, sorted by decreasing
// score; equal scores keep the earlier (lower) column first. Returns the new
// threshold (the k-th best score, -inf while the list is not full). Kept out
// of line: it runs rarely, and one copy keeps the hot loop small.
__device__ __noinline__ float top_insert(float* tv, int32_t* ti, int* cnt, int k, float s, int32_t col) {
  int c = *cnt;
  int pos = c < k ? c : k - 1;
  while (pos > 0 && s > tv[pos - 1]) {
    tv[pos] = tv[pos - 1];
    ti[pos] = ti[pos - 1];
    --pos;
  }
  tv[pos] = s;
  ti[pos] = col;
  if (c < k) *cnt = ++c;
  return c == k ? tv[k - 1] : -INFINITY;
}

// Ranked lists: score = c * phi_hat + g (log2 units, shifted; same order as
// log mu within a row). The chunk's maximum is compared with the running k-th
// best first, so most chunks cost one FFMA and one max per column.
template <bool RS>
__device__ __forceinline__ void chunk_topk(const uint32_t (&v)[32], const float* g, const float* fs, float c,
                                           int64_t colbase, int k, float* tv, int32_t* ti, int* cnt, float& thr) {
  const float4* g4 = reinterpret_cast<const float4*>(g);
  float s[32];
  float mx = -INFINITY;
#pragma unroll
  for (int i4 = 0; i4 < 8; ++i4) {
    const float4 gg = g4[i4];
    s[4 * i4 + 0] = fmaf(scaled_phi<RS>(v[4 * i4 + 0], fs, 4 * i4 + 0), c, gg.x);
    s[4 * i4 + 1] = fmaf(scaled_phi<RS>(v[4 * i4 + 1], fs, 4 * i4 + 1), c, gg.y);
    s[4 * i4 + 2] = fmaf(scaled_phi<RS>(v[4 * i4 + 2], fs, 4 * i4 + 2), c, gg.z);
    s[4 * i4 + 3] = fmaf(scaled_phi<RS>(v[4 * i4 + 3], fs, 4 * i4 + 3), c, gg.w);
    mx = fmaxf(mx, fmaxf(fmaxf(s[4 * i4 + 0], s[4 * i4 + 1]), fmaxf(s[4 * i4 + 2], s[4 * i4 + 3])));
  }
  if (mx > thr) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (s[e] > thr) thr = top_insert(tv, ti, cnt, k, s[e], (int32_t)(colbase + e));
  }
}

// Ranked lists in shared memory (kModeTopKShared): every epilogue thread
// has list_slots (score, column) slots in shared memory, slot i of thread t
// at [i * list_threads + t] (a warp's accesses to one slot are conflict-free).
// The first k hold the k best of its row and column half, sorted by
// decreasing score, equal scores in increasing column order (the order in
// which a column half's columns arrive); they start as (-inf, INT32_MAX)
// pairs, so the k-th score is the threshold from the first column on. The
// other slots buffer candidates: columns that beat the threshold as of the
// last merge, appended in column order. When a lane's buffer could overflow,
// the whole warp merges: all 32 lanes insert their candidates side by side.
// Rows whose rankings differ (a converged market, where the potentials cancel
// the popularity terms) meet their candidates at different columns; inserting
// each at once ran the lanes' insertions one after another (3 of 32 lanes per
// chunk and more), which cost several times the pass itself.
// (Top-10 lists of 100,000 users over 60,000 partners, d = 64, at solved
// potentials: 4.23 ms with every candidate inserted at once, 2.93 with
// buffers, 2.74 with the shared bound below, 2.71 without the scores kept
// across the vote, 2.16 with the merges of all warps at the same tiles; a
// half-sweep of that size takes 1.4.)
// With own tiles of 128 rows (SMALL) half of the epilogue threads have rows, and
// twice the slots each: lists longer than kSharedTopK, up to kSharedTopKSmall,
// run on such tiles. (Half of the epilogue is idle then, and every partner tile
// is read by twice as many own tiles; the lists of kModeTopK, in local memory
// and entered one lane at a time, cost far more. 60,000 x 50,000, kModeTopK ->
// here: k = 20, d = 64 34.8 -> 2.80 ms; k = 32, d = 32 74.1 -> 5.53; 5,000 x
// 7,000, d = 32, k = 20 1.39 -> 0.31. Longer ones would need more than the
// 41 slots: kModeTopK.)
constexpr int kSharedTopK = 14;
constexpr int kSharedTopKSmall = 32;
constexpr int kTopKSlots = 20;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int list_threads(bool small) { return small ? kEpiThreads / 2 : kEpiThreads; }
constexpr int list_slots(bool small) { return small ? 2 * kTopKSlots + 1 : kTopKSlots; }
// (the slots, then one 8-byte word per thread: the bound that the two threads
// of a row share, see chunk_topk_shared)
constexpr int kTopKListBytes = (kTopKSlots + 1) * kEpiThreads * 8;
// A group of kTopKGroup columns adds at most that many candidates, so a buffer
// of list_slots - k >= kTopKGroup + 1 slots is merged whenever fewer than
// kTopKGroup are free.
constexpr int kTopKGroup = 4;
static_assert(kTopKSlots - kSharedTopK > kTopKGroup && list_slots(true) - kSharedTopKSmall > kTopKGroup,
              "candidate slots");
constexpr int kWideShiftBytes = 2 * kFusedOwnRows * 4;  // kModeSweepWide: the row hand-over's shifts
// kModeMu: each epilogue warp turns its 32 rows x mu_width columns through
// shared memory, so that its stores run along the rows of the output (rows of
// mu_width + 4 floats: 16-byte accesses along and across them are free of bank
// conflicts). Half the width where a four-block own tile leaves no room for more.
constexpr int mu_width(int KB) { return KB == 4 ? 16 : 32; }
constexpr int mu_stage_floats(int KB) { return 32 * (mu_width(KB) + 4); }
// shared memory a mode needs after the tail area
constexpr int mode_extra_bytes(int mode, int KB, bool split, bool ranges) {
  return mode == kModeTopKShared ? kTopKListBytes
         : mode == kModeMu       ? kEpiWarps * mu_stage_floats(KB) * 4
         : mode == kModeSweep || mode == kModeSweepWide
             ? (mode == kModeSweepWide ? kWideShiftBytes : 0) + (split ? kWideShiftBytes : 0) +
                   (ranges ? kEpiThreads * 12 : 0)
             : 0;
}

__device__ __forceinline__ void sts_u64(uint32_t a, uint64_t v) {
  asm volatile("st.volatile.shared.b64 [%0], %1;" ::"r"(a), "l"(v));
}
__device__ __forceinline__ uint64_t lds_u64(uint32_t a) {
  uint64_t v;
  asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(v) : "r"(a));
  return v;
}

// A slot: the score in the low word, the column in the high one.
__device__ __forceinline__ uint64_t slot_of(float s, int32_t col) {
  return ((uint64_t)(uint32_t)col << 32) | __float_as_uint(s);
}
__device__ __forceinline__ float slot_score(uint64_t w) { return __uint_as_float((uint32_t)w); }
__device__ __forceinline__ int32_t slot_col(uint64_t w) { return (int32_t)(w >> 32); }

// Merge a warp's candidate buffers (cnt candidates of this lane) into its
// lists at shared address lv: round j inserts every lane's candidate j, where
// it beats the lane's current k-th score. An insertion reads the entries above
// it four at a time (independent loads: one shared-memory latency per four
// shifts). Returns the new k-th score. Kept out of line: one copy serves every
// call site.
template <uint32_t kSlotStride>
__device__ __noinline__ float list_merge(uint32_t lv, int k, int cnt) {
  const uint32_t last = lv + (uint32_t)(k - 1) * kSlotStride;
  float thr = slot_score(lds_u64(last));
  const int rounds = __reduce_max_sync(0xffffffffu, cnt);
  for (int j = 0; j < rounds; ++j) {
    const uint64_t w = j < cnt ? lds_u64(last + (uint32_t)(j + 1) * kSlotStride) : slot_of(-INFINITY, 0);
    const float s = slot_score(w);
    if (s > thr) {
      uint32_t pos = last;
      bool go = pos != lv;
      while (go) {
        uint64_t e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t a = pos - (uint32_t)(i + 1) * kSlotStride;
          e[i] = (int32_t)(a - lv) >= 0 ? lds_u64(a) : slot_of(INFINITY, 0);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          go = go && s > slot_score(e[i]);
          if (go) {
            sts_u64(pos, e[i]);
            pos -= kSlotStride;
          }
        }
        go = go && pos != lv;
      }
      sts_u64(pos, w);
      thr = slot_score(lds_u64(last));
    }
    __syncwarp();
  }
  return thr;
}

// A row's columns are split over two threads (column halves), each with its own
// list. If both lists hold ceil(k / 2) scores of at least b, the row's k-th
// best is at least b: a column below b cannot be listed. So each thread
// publishes, after every merge, the value just below its list's
// ceil(k / 2)-th score (so that equal scores still pass), tagged with its own
// tile, and takes as threshold the larger of its k-th score and the smaller
// of the two published values: about the k-th best of both halves together,
// which halves the candidates. A word of an older tile (or one read while the
// other thread is a merge behind) only makes the bound weaker, never wrong, so
// the lists do not depend on timing.
struct SharedBound {
  uint32_t mine, other;  // shared addresses of the two threads' words
  uint32_t tag;          // the own tile, counted per CTA
  float pub;             // this thread's published value
  __device__ __forceinline__ void publish(uint32_t lv, int k, uint32_t kSlotStride) {
    pub = nextafterf(slot_score(lds_u64(lv + (uint32_t)((k - 1) / 2) * kSlotStride)), -INFINITY);
    sts_u64(mine, ((uint64_t)tag << 32) | __float_as_uint(pub));
  }
  __device__ __forceinline__ float bound() const {
    const uint64_t w = lds_u64(other);
    return (uint32_t)(w >> 32) == tag ? fminf(pub, __uint_as_float((uint32_t)w)) : -INFINITY;
  }
};

// One 32-column chunk: the scores' maximum in every group of four columns; the
// groups in which some lane beats its threshold form their scores again and
// append them (keeping all 32 beside the next chunk's TMEM load in flight
// would spill).
template <bool RS, bool SMALL>
__device__ __forceinline__ void chunk_topk_shared(const uint32_t (&v)[32], const float* g, const float* fs,
                                                  uint64_t cc, int64_t colbase, int k, uint32_t lv, int& cnt,
                                                  float& thr, SharedBound& sb) {
  constexpr int kGroups = 32 / kTopKGroup;
  constexpr uint32_t kSlotStride = list_threads(SMALL) * 8;
  static_assert(kTopKGroup == 4, "a group is one float4 of g");
  const float4* g4 = reinterpret_cast<const float4*>(g);
  const float4* fs4 = reinterpret_cast<const float4*>(fs);
  auto scores = [&](int i, float (&s)[4]) {
    const float4 gg = g4[i];
    float4 ff = make_float4(1.f, 1.f, 1.f, 1.f);
    if constexpr (RS) ff = fs4[i];
    const uint64_t t0 = pair_exponents<RS>(v[4 * i + 0], v[4 * i + 1], gg.x, gg.y, ff.x, ff.y, cc);
    const uint64_t t1 = pair_exponents<RS>(v[4 * i + 2], v[4 * i + 3], gg.z, gg.w, ff.z, ff.w, cc);
    s[0] = __uint_as_float((uint32_t)t0);
    s[1] = __uint_as_float((uint32_t)(t0 >> 32));
    s[2] = __uint_as_float((uint32_t)t1);
    s[3] = __uint_as_float((uint32_t)(t1 >> 32));
  };
  thr = fmaxf(thr, sb.bound());
  uint32_t hit = 0;
#pragma unroll
  for (int i = 0; i < kGroups; ++i) {
    float s[4];
    scores(i, s);
    if (fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])) > thr) hit |= 1u << i;
  }
  hit = __reduce_or_sync(0xffffffffu, hit);
  if (hit == 0) return;
#pragma unroll
  for (int i = 0; i < kGroups; ++i) {
    if ((hit & (1u << i)) == 0) continue;
    float s[4];
    scores(i, s);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (s[e] > thr) {
        sts_u64(lv + (uint32_t)(k + cnt) * kSlotStride, slot_of(s[e], (int32_t)(colbase + 4 * i + e)));
        ++cnt;
      }
    }
    if (__any_sync(0xffffffffu, cnt > list_slots(SMALL) - k - kTopKGroup)) {
      thr = list_merge<kSlotStride>(lv, k, cnt);
      sb.publish(lv, k, kSlotStride);
      cnt = 0;
    }
  }
}

// mu block: mu = 2^(c * phi_hat + g + lo) * 2^hi, where hi + lo = (shift + ell_row) log2 e;
// 2^hi as the two factors s1, s2 (hi clamped to +-252: beyond, the product is
// 0 or infinite all the same). The warp's 32 rows x 32 columns go through
// `st` in shared memory, W columns at a time, so that the warp's stores run along
// the output's rows: four floats per lane and store (p.vec), or one. nrow: the
// warp's rows inside the block, orow: its first row there.
template <bool RS, int W>
__device__ __forceinline__ void chunk_mu(const uint32_t (&v)[32], const float* g, const float* fs, float c,
                                         int64_t colbase, float lo, int hi, float s1, float s2, int lane, int nrow,
                                         int64_t orow, float* st, const FusedParams& p) {
  const float4* g4 = reinterpret_cast<const float4*>(g);
  float t[32];
  float far = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 gg = g4[i];
    t[4 * i + 0] = fmaf(scaled_phi<RS>(v[4 * i + 0], fs, 4 * i + 0), c, gg.x) + lo;
    t[4 * i + 1] = fmaf(scaled_phi<RS>(v[4 * i + 1], fs, 4 * i + 1), c, gg.y) + lo;
    t[4 * i + 2] = fmaf(scaled_phi<RS>(v[4 * i + 2], fs, 4 * i + 2), c, gg.z) + lo;
    t[4 * i + 3] = fmaf(scaled_phi<RS>(v[4 * i + 3], fs, 4 * i + 3), c, gg.w) + lo;
    far = fmaxf(far, fmaxf(fmaxf(fabsf(t[4 * i + 0]), fabsf(t[4 * i + 1])),
                           fmaxf(fabsf(t[4 * i + 2]), fabsf(t[4 * i + 3]))));
  }
  const bool near = !__any_sync(0xffffffffu, far > 100.0f);
#pragma unroll
  for (int c0 = 0; c0 < 32; c0 += W) {
    float4* mine = reinterpret_cast<float4*>(st + lane * (W + 4));
    if (near) {
#pragma unroll
      for (int i = 0; i < W; i += 4)
        mine[i / 4] = make_float4(ex2_approx(t[c0 + i]) * s1 * s2, ex2_approx(t[c0 + i + 1]) * s1 * s2,
                                  ex2_approx(t[c0 + i + 2]) * s1 * s2, ex2_approx(t[c0 + i + 3]) * s1 * s2);
    } else {
      // (an exponent beyond the FP32 range is brought back by hi first)
      float* m = reinterpret_cast<float*>(mine);
#pragma unroll
      for (int i = 0; i < W; ++i)
        m[i] = fabsf(t[c0 + i]) <= 100.0f ? ex2_approx(t[c0 + i]) * s1 * s2 : ex2_approx(t[c0 + i] + (float)hi);
    }
    __syncwarp();
    const int64_t ocol = colbase + c0 - p.y0;  // (the chunk's first column of the output)
    float* o = p.out + orow * p.ld + ocol;
    if (p.vec && ocol >= 0 && ocol + W <= p.ny) {
      constexpr int kLanes = W / 4, kRows = 32 / kLanes;  // lanes along a row, rows per store
      const int rr = lane / kLanes, cq = lane % kLanes;
#pragma unroll
      for (int i = 0; i < W / 4; ++i) {
        const int row = i * kRows + rr;
        const float4 v4 = *reinterpret_cast<const float4*>(st + row * (W + 4) + 4 * cq);
        if (row < nrow) *reinterpret_cast<float4*>(o + row * p.ld + 4 * cq) = v4;
      }
    } else {
      const int64_t col = ocol + lane % W;
      if (col >= 0 && col < p.ny)
        for (int i = lane / W; i < nrow; i += 32 / W) o[i * p.ld + lane % W] = st[i * (W + 4) + lane % W];
    }
    __syncwarp();
  }
}

// The items of a batched launch are (market, own tile) pairs.
struct ItemRef {
  const BatchDesc* d;
  int t;
};
__device__ __forceinline__ ItemRef batch_item(const FusedParams& p, int it) {
  const int2 v = p.items[it];
  return {p.bdesc + v.x, v.y};
}

// An item of a launch: own tile t against its partner tiles [jb, je), range
// `me` of the n into which the tile is cut.
struct Seg {
  int t, jb, je, me, n;
};

// Contribution c of a cut tile (u: its number among the cut tiles): the slot
// in the partials of the span that formed it. A span has at most two slots, as
// it is no longer than a tile.
__device__ __forceinline__ int cut_first(const FusedParams& p, int u) { return u * p.cut_ptiles / p.cut_span; }
__device__ __forceinline__ int cut_slot(const FusedParams& p, int u, int k) {
  return 2 * k + (u - k * p.cut_span / p.cut_ptiles);
}

// This CTA's i-th item (all roles walk the same sequence): of the batched
// item list; of a single market, own tiles blockIdx.x, blockIdx.x + gridDim.x,
// ...; SPLIT with p.split > 1, (own tile, range) pairs, tile by tile (the
// ranges of one own tile on neighbouring CTAs) or with range_major range by
// range, so that all CTAs stream one range of the partner matrix (small enough
// to stay in L2) against every own tile before the next; SPLIT with p.split =
// 1, the whole tiles and then the CTA's span of the cut ones. False past the
// last one. (Batched: the market's descriptor comes from batch_item.)
// PAIR: the same for both CTAs of a pair, in tiles of 512 rows.
template <bool BATCH, bool SPLIT, bool PAIR>
__device__ __forceinline__ bool item_at(const FusedParams& p, int i, Seg& sg) {
  const int npt = p.num_partner_tiles;
  const int tiles = PAIR ? (p.num_own_tiles + 1) / 2 : p.num_own_tiles;
  const int cta = PAIR ? (int)blockIdx.x / 2 : (int)blockIdx.x, ctas = PAIR ? (int)gridDim.x / 2 : (int)gridDim.x;
  if constexpr (BATCH) {
    sg.t = p.cta_start[blockIdx.x] + i;  // the index in the item list
    return sg.t < p.cta_start[blockIdx.x + 1];
  }
  const int it = cta + i * ctas;
  if constexpr (!SPLIT) {
    sg = {it, 0, npt, 0, 1};
    return it < tiles;
  }
  if (p.split > 1) {
    const int S = p.split;
    if (it >= p.num_own_tiles * S) return false;
    int t, s;
    if (p.range_major) {
      s = it / p.num_own_tiles;
      t = it - s * p.num_own_tiles;
    } else {
      t = it / S;
      s = it - t * S;
    }
    sg = {t, (int)((int64_t)s * npt / S), (int)((int64_t)(s + 1) * npt / S), s, S};
    return true;
  }
  if (it < p.cut_t0) {
    sg = {it, 0, npt, 0, 1};
    return true;
  }
  // (with whole tiles the grid divides cut_t0, so every CTA has the same number of them)
  const int q = i - p.cut_t0 / ctas, k = cta;
  if (p.cut_span == 0 || k >= p.cut_spans || q > 1) return false;
  const int lo = k * p.cut_span, end = (tiles - p.cut_t0) * npt;
  const int hi = lo + p.cut_span < end ? lo + p.cut_span : end;
  const int u = lo / npt + q, u0 = u * npt;
  if (u0 >= hi) return false;
  const int first = cut_first(p, u), last = (u0 + npt - 1) / p.cut_span;
  sg = {p.cut_t0 + u, lo > u0 ? lo - u0 : 0, (hi < u0 + npt ? hi : u0 + npt) - u0, k - first, last - first + 1};
  return true;
}

// Sums of a row's ranges, added in order: hi + lo at shift m (wide markets).
struct RangeSum {
  float hi = 0.0f, lo = 0.0f, m = -INFINITY;
  template <bool WIDE>
  __device__ __forceinline__ void add(float sum, float comp, float shift) {
    if constexpr (WIDE) {
      // both onto the larger shift (exact powers of two)
      const float top = fmaxf(m, shift), a = exp2_int(m - top), b = exp2_int(shift - top);
      hi *= a;
      lo *= a;
      sum *= b;
      comp *= b;
      m = top;
    }
    float e;
    hi = two_sum(hi, sum, e);
    lo = __fadd_rn(lo, __fsub_rn(e, comp));
  }
};

// The partner tile before which a row's sum is next cut at or after `from`
// (none: a number that no tile has).
constexpr int kNoCut = 0x7fffffff;
__device__ __forceinline__ int next_cut(int64_t row, int rows, int t0, int span, int ptiles) {
  const int64_t t = row / rows;
  if (span == 0 || t < t0) return kNoCut;
  const int u0 = (int)(t - t0) * ptiles, c = (u0 / span + 1) * span - u0;
  return c < ptiles ? c : kNoCut;
}

// BATCH: the CTA's own tiles come from the launch's item list and may belong
// to different markets (tensor maps, vectors and sizes from BatchDesc); the
// residual partials are then written per own tile and epilogue warp instead
// of per CTA.
// KB: 128-byte k blocks per packed row (1, 2 or 4: BF16 kp = 64, 128, 256;
// e4m3 kp = 128, 256, 512).
// FMT: kFmtBF16, or e4m3 factors on tcgen05.mma kind::f8f6f4 with one scale
// per side (kFmtE4M3Side: both folded into p.c) or per row (kFmtE4M3Rows: the
// own row's scale is folded into the row's exponent multiplier, the partner
// rows' scales multiply the accumulator entries in the epilogue).
// SMALL: own tiles of 128 rows (one MMA chain; the epilogue warps of the
// second sub-tile take part in every barrier but load and compute nothing),
// for markets whose 256-row tiles would leave SMs idle: twice the CTAs, each
// finishing its rows in about half the time. Every row's arithmetic is the
// same as with 256-row tiles.
// CUTS (and BATCH): launches that run a cut row's ranges in turn.
// PAIR: the CTAs of a cluster of two share every partner tile. The first one's
// MMA warp issues M = 256 MMAs (cta_group::2) over both CTAs' own rows; each
// CTA loads and holds half of the tile's rows, so the tensor core's reads of
// shared memory per tile and SM fall from 128 KB to 96 (A's 128 rows and B's
// 64 per instruction instead of 128 and 128) and the copies from 32 KB to 16.
// That pays where the operands are long (d = 100, 50,001 x 70,000: 2.18 -> 1.75
// ms per sweep) and makes room for the folded g at d = 64 (100,003 x 79,999:
// 2.73 -> 2.60, 300,000 x 300,000: 31.3 -> 29.4). The epilogue warps of the
// second CTA announce a read buffer by a plain remote arrival; a releasing one at
// cluster scope stalled them (300,000 x 300,000: 41.7 ms). Handing each sub-tile
// over by itself was slower (33.2 -> 35.4), releasing a buffer before its
// arithmetic and eight stages instead of six made no difference.
template <int KB, int STAGES, int MODE, bool BATCH, int FMT, bool SMALL = false, bool SPLIT = false,
          bool NOFOLD = false, bool CUTS = false, bool PAIR = false>
__global__ void __launch_bounds__(kThreads, 1)
    k_fused_halfsweep(const __grid_constant__ CUtensorMap tm_own, const __grid_constant__ CUtensorMap tm_partner,
                      const __grid_constant__ CUtensorMap tm_fold, const FusedParams p) {
  static_assert(!BATCH || MODE == kModeSweep, "batched launches run half-sweeps only");
  constexpr bool WIDE = MODE == kModeSweepWide;
  constexpr bool kSweepLike = MODE == kModeSweep || WIDE;
  constexpr bool RANGES = CUTS || BATCH;
  static_assert(!SPLIT || ((kSweepLike || MODE == kModeMu) && !BATCH),
                "partner splits are single-market half-sweeps and mu blocks");
  static_assert(!CUTS || (kSweepLike && !SPLIT && !BATCH), "ranges in turn: unsplit half-sweeps");
  static_assert(!(BATCH && SMALL), "batched launches use 256-row own tiles");
  static_assert(!PAIR || (kSweepLike && KB > 1 && !BATCH && !SMALL && !NOFOLD && !CUTS), "pairs: half-sweeps");
  constexpr int kOwn = SMALL ? kFusedOwnRows / 2 : kFusedOwnRows;  // rows of an own tile
  static_assert(KB == 1 || KB == 2 || KB == 4, "128-byte k blocks per row");
  constexpr bool F8 = FMT != kFmtBF16;      // e4m3 operands
  constexpr bool RS = FMT == kFmtE4M3Rows;  // per-row scales
  constexpr int ABUF = kABufs<KB>;
  constexpr int KBS = kbs_for(KB, PAIR);  // k blocks per partner stage
  constexpr int SPT = KB / KBS;      // stages per partner tile
  constexpr int XB = F8 ? 128 : kKBlock;  // elements per 128-byte k block (TMA x coordinate step)
  constexpr bool FOLD = fold_for(KB, MODE, BATCH, FMT, NOFOLD);  // g added by an extra MMA
  constexpr int SB = stage_bytes(KB, FOLD, PAIR);                        // bytes per partner stage
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_u32 = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_u32 + 1023u) & ~1023u) - raw_u32);
  uint8_t* sA = smem;
  uint8_t* sB = smem + ABUF * KB * kOwnBytesPerKB;
  uint8_t* sOnes = sB + STAGES * SB;  // folded g: the own side's constant operand
  float* sG = reinterpret_cast<float*>(sOnes + (FOLD ? kFoldBytes : 0));
  float* sF = sG + kGSlots * kFusedPartnerRows;  // per-row scales: partner scale ring
  uint64_t* bars =
      reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(sG) + kGSlots * kGBytes * (RS ? 2 : 1));
  uint64_t* full = bars;
  uint64_t* empty = bars + STAGES;
  uint64_t* gfull = bars + 2 * STAGES;
  uint64_t* gempty = gfull + kGSlots;
  uint64_t* a_full = gempty + kGSlots;  // [2]
  uint64_t* a_empty = a_full + 2;       // [2]
  uint64_t* tfull = a_full + 4;         // [2]
  uint64_t* tempty = a_full + 6;        // [2]
  uint64_t* mma_done = a_full + 8;
  uint64_t* rowfull = a_full + 9;   // [2] second column half of the rows written
  uint64_t* rowfree = a_full + 11;  // [2] row hand-over buffer read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(a_full + 13);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  double* red = reinterpret_cast<double*>(reinterpret_cast<uint8_t*>(bars) + 512);      // kEpiWarps x 4 doubles
  float* rowbuf = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + 1024);   // 2 x 256 floats
  // ranked lists in shared memory (kModeTopKShared only): after the tail area
  float* topk_list = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kTailBytes);
  // half-sweeps, in the same place: the second column half's shifts (wide
  // markets) and compensations (SPLIT), 2 x 256 floats each, and the sums over
  // a row's earlier ranges (CUTS, BATCH)
  float* wide_shift = topk_list;
  float* row_comp = wide_shift + (WIDE ? 2 * kFusedOwnRows : 0);
  RangeSum* range_sum = reinterpret_cast<RangeSum*>(row_comp + (SPLIT ? 2 * kFusedOwnRows : 0));
  static_assert(4 * kEpiWarps * 8 <= 512, "reduction area");
  static_assert((2 * STAGES + 2 * kGSlots + 13) * 8 + 8 <= 512, "barrier area");

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = PAIR ? (int)cluster_rank() : 0;
  constexpr int kParBytes = PAIR ? kPartnerBytesPerKB / 2 : kPartnerBytesPerKB;  // of a partner tile's k block here

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < kGSlots; ++s) {
      mbar_init(&gfull[s], 1);
      mbar_init(&gempty[s], kEpiWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&a_full[b], 1);
      mbar_init(&a_empty[b], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], PAIR ? 2 * kEpiWarps : kEpiWarps);
    }
    mbar_init(mma_done, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&rowfull[b], kEpiWarps / 2);
      mbar_init(&rowfree[b], kEpiWarps / 2);
    }
    *abort_flag = 0;
    fence_mbar_init();
    if constexpr (!BATCH) {
      tma_prefetch_map(&tm_own);
      tma_prefetch_map(&tm_partner);
    }
  }
  if (warp == 0) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, kTmemCols);
      tmem_relinquish();
    }
  }
  if constexpr (FOLD) {
    // the own side's operand of the extra MMA: BF16 ones in columns 0-3 of
    // every row (16-byte chunk q holds columns 0-7 when (q / 8) is even),
    // made visible to the tensor core's (async) proxy
    if (threadIdx.x < kFoldBytes / 16) {
      const bool cols0_7 = ((threadIdx.x / 8) % 2) == 0;
      reinterpret_cast<uint4*>(sOnes)[threadIdx.x] =
          cols0_7 ? make_uint4(0x3F803F80u, 0x3F803F80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if constexpr (MODE == kModeTopKShared) {
    // no published bound yet (tags start at 1; shared memory may hold another launch's words)
    if ((int)threadIdx.x >= 64 && (int)threadIdx.x < 64 + list_threads(SMALL))
      sts_u64(smem_u32(topk_list) + (uint32_t)(list_slots(SMALL) * list_threads(SMALL) + (int)threadIdx.x - 64) * 8u,
              0ull);
  }
  tc_fence_before();
  if constexpr (PAIR) {
    cluster_sync();  // (the other CTA's barriers are initialised, too)
  } else {
    __syncthreads();
  }
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int stage = 0, gs = 0, ab = 0;
      uint32_t phase = 0, gphase = 0, a_phase = 0;
      const bool hint = !BATCH && p.l2_keep > 0.0f;
      const uint64_t keep_policy = hint ? l2_policy_keep_fraction(p.l2_keep) : 0ull;
      uint32_t armed[STAGES], garmed[kGSlots], a_armed[2] = {0u, 0u};
      for (int s = 0; s < STAGES; ++s) armed[s] = 0;
      for (int s = 0; s < kGSlots; ++s) garmed[s] = 0;
      const BatchDesc* prev = nullptr;
      bool ok = true;
      Seg sg;
      for (int i = 0; ok && item_at<BATCH, SPLIT, PAIR>(p, i, sg); ++i) {
        const BatchDesc* bd = nullptr;
        int t, jb = 0, je;
        if constexpr (BATCH) {
          const ItemRef w = batch_item(p, sg.t);
          bd = w.d;
          t = w.t;
          je = bd->num_partner_tiles;
          if (bd != prev) {
            tensormap_acquire(&bd->tm_own);
            tensormap_acquire(&bd->tm_partner);
            prev = bd;
          }
        } else {
          t = PAIR ? 2 * sg.t + rank : sg.t;
          jb = sg.jb;
          je = sg.je;
        }
        const CUtensorMap* map_own = BATCH ? &bd->tm_own : &tm_own;
        const CUtensorMap* map_partner = BATCH ? &bd->tm_partner : &tm_partner;
        const float* gsrc = BATCH ? bd->g : p.g + p.col0;
        const float* fsrc = BATCH ? bd->fs_par : p.fs_par + p.col0;
        // (SMALL: the 256-row box also brings the next tile's rows, unused)
        const int64_t arow = BATCH ? (int64_t)t * kFusedOwnRows : p.row0 + (int64_t)t * kOwn;
        if (!mbar_wait(&a_empty[ab], a_phase ^ 1u, abort_flag)) {
          ok = false;
          break;
        }
        if (rank == 0) mbar_arrive_expect_tx(&a_full[ab], (PAIR ? 2 : 1) * KB * kOwnBytesPerKB);
        for (int kb = 0; kb < KB; ++kb) {
          if constexpr (PAIR) {
            tma_load_2d_pair(sA + (ab * KB + kb) * kOwnBytesPerKB, map_own, cluster_addr(&a_full[ab], 0), kb * XB,
                             (int)arow);
          } else {
            tma_load_2d(sA + (ab * KB + kb) * kOwnBytesPerKB, map_own, &a_full[ab], kb * XB, (int)arow);
          }
        }
        ++a_armed[ab];
        if (++ab == ABUF) {
          ab = 0;
          a_phase ^= 1u;
        }
        for (int j = jb; j < je && ok; ++j) {
          for (int sp = 0; sp < SPT; ++sp) {
            if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag)) {
              ok = false;
              break;
            }
            const bool fold_here = FOLD && sp == SPT - 1;  // the tile's g operand rides in its last stage
            if (rank == 0) mbar_arrive_expect_tx(&full[stage], KBS * kPartnerBytesPerKB + (fold_here ? kFoldBytes : 0));
            for (int kb = 0; kb < KBS; ++kb) {
              const int px = (sp * KBS + kb) * XB, py = (int)(p.col0 + (int64_t)j * kFusedPartnerRows);
              uint8_t* dst = sB + stage * SB + kb * kParBytes;
              if constexpr (PAIR) {
                const uint32_t bar = cluster_addr(&full[stage], 0);
                const int y = py + rank * (kFusedPartnerRows / 2);
                if (hint) {
                  tma_load_2d_pair_hint(dst, map_partner, bar, px, y, keep_policy);
                } else {
                  tma_load_2d_pair(dst, map_partner, bar, px, y);
                }
              } else if (hint) {
                tma_load_2d_hint(dst, map_partner, &full[stage], px, py, keep_policy);
              } else {
                tma_load_2d(dst, map_partner, &full[stage], px, py);
              }
            }
            if (PAIR && fold_here) {
              // (a plain bulk copy cannot be counted in the other CTA: through a tensor map, in rows of 256 bytes)
              tma_load_2d_pair(sB + stage * SB + KBS * kParBytes, &tm_fold, cluster_addr(&full[stage], 0), 0,
                               (j * 2 + rank) * (kFoldBytes / 512));
            } else if (fold_here)
              bulk_load(sB + stage * SB + KBS * kPartnerBytesPerKB,
                        (BATCH ? bd->gfold : p.gfold) + (int64_t)j * kFoldBytes, kFoldBytes, &full[stage]);
            ++armed[stage];
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          if constexpr (FOLD) continue;  // g rides in the MMA
          if (!mbar_wait(&gempty[gs], gphase ^ 1u, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&gfull[gs], RS ? 2 * kGBytes : kGBytes);
          bulk_load(sG + gs * kFusedPartnerRows, gsrc + (int64_t)j * kFusedPartnerRows, kGBytes, &gfull[gs]);
          if constexpr (RS)
            bulk_load(sF + gs * kFusedPartnerRows, fsrc + (int64_t)j * kFusedPartnerRows, kGBytes, &gfull[gs]);
          ++garmed[gs];
          if (++gs == kGSlots) {
            gs = 0;
            gphase ^= 1u;
          }
        }
      }
      if constexpr (PAIR) {
        // The first CTA's commits arrive on the barriers of both CTAs, and the
        // cluster barrier at the end orders threads, not these asynchronous
        // arrivals: each CTA stays until the last one on each of its barriers has
        // been seen (those on tfull are the epilogue's), so that none lands in
        // shared memory that another CTA has taken over. At most the ring's
        // stages of MMAs are left here, while the epilogue still works.
        for (int s = 0; s < STAGES && ok; ++s)
          if (armed[s]) ok = mbar_wait(&empty[s], (armed[s] - 1u) & 1u, abort_flag);
        for (int b = 0; b < ABUF && ok; ++b)
          if (a_armed[b]) ok = mbar_wait(&a_empty[b], (a_armed[b] - 1u) & 1u, abort_flag);
        if (ok) ok = mbar_wait(mma_done, 0, abort_flag);
      }
      if (!ok) {
        if (!*abort_flag) raise_error(p.err, abort_flag, kErrTimeout);
        // (the first CTA commits mma_done on every path, at the latest when its
        // own waits have run out)
        if constexpr (PAIR) mbar_wait_drain(mma_done, 0, 2 * kWaitLimitNs);
        // let the copies already issued land before the CTA's shared memory goes
        // away (a pair's second CTA cannot see the barriers they are counted on:
        // it waits for longer than any copy or arrival takes)
        if (PAIR && rank != 0) {
          const uint64_t t0 = global_timer_ns();
          while (global_timer_ns() - t0 < 10000000ull) {
          }
        }
        for (int s = 0; s < STAGES && rank == 0; ++s)
          if (armed[s]) mbar_wait_drain(&full[s], (armed[s] - 1u) & 1u, 10000000ull);
        for (int s = 0; s < kGSlots; ++s)
          if (garmed[s]) mbar_wait_drain(&gfull[s], (garmed[s] - 1u) & 1u, 10000000ull);
        for (int b = 0; b < ABUF && rank == 0; ++b)
          if (a_armed[b]) mbar_wait_drain(&a_full[b], (a_armed[b] - 1u) & 1u, 10000000ull);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (a pair's: in its first CTA)
    // The whole warp runs the loop, and one elected lane the tensor-core
    // instructions: what they are given (descriptors as a base per operand and
    // constants added to it, addresses) then stays in uniform registers. With the
    // loop on one lane each of them was moved there before every MMA, and issuing
    // was the bound: about 100 cycles per MMA that takes 64.
    if (rank == 0) {
      constexpr int M = PAIR ? 256 : 128;
      constexpr uint32_t idesc = F8 ? idesc_e4m3_f32(M, kFusedPartnerRows) : idesc_bf16_f32(M, kFusedPartnerRows);
      constexpr uint32_t idesc_fold = idesc_bf16_f32(M, kFusedPartnerRows);  // (BF16 in every format)
      auto commit = [](uint64_t* bar) {
        if constexpr (PAIR) {
          umma_commit_pair(bar);
        } else {
          umma_commit(bar);
        }
      };
      auto ready = [&](uint64_t* bar, uint32_t ph) {
        const bool got = __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag));
        tc_fence_after();
        return got;
      };
      const uint64_t a_base = sdesc_sw128(smem_u32(sA)), b_base = sdesc_sw128(smem_u32(sB));
      const uint64_t ones = sdesc_none(smem_u32(sOnes), 128, 256), gc_base = sdesc_none(smem_u32(sB), 128, 256);
      int stage = 0, buf = 0, ab = 0;
      uint32_t phase = 0, tphase = 0, a_phase = 0;
      bool ok = true;
      Seg sg;
      for (int i = 0; ok && item_at<BATCH, SPLIT, PAIR>(p, i, sg); ++i) {
        int jb = 0, je;
        if constexpr (BATCH) {
          je = batch_item(p, sg.t).d->num_partner_tiles;
        } else {
          jb = sg.jb;
          je = sg.je;
        }
        if (!ready(&a_full[ab], a_phase)) {
          ok = false;
          break;
        }
        // (descriptors hold shared addresses in units of 16 bytes in their low bits)
        const uint64_t a0 = a_base + (uint32_t)(ab * KB * (kOwnBytesPerKB >> 4));
        uint64_t* a_release = &a_empty[ab];
        if (++ab == ABUF) {
          ab = 0;
          a_phase ^= 1u;
        }
        for (int j = jb; j < je && ok; ++j) {
          if (!ready(&tempty[buf], tphase ^ 1u)) {
            ok = false;
            break;
          }
          for (int sp = 0; sp < SPT; ++sp) {
            if (!ready(&full[stage], phase)) {
              ok = false;
              break;
            }
            if (elect_one()) {
              const uint64_t b0 = b_base + (uint32_t)(stage * (SB >> 4));
#pragma unroll
              for (int h = 0; h < (SMALL ? 1 : 2); ++h) {
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256 + h * 128);
#pragma unroll
                for (int k = 0; k < KBS * 4; ++k) {
                  // Steps of padding add zeros: half-sweeps leave them out, to
                  // the same bits (d = 100 in rows of 128, 13 of 16 steps: 50,001
                  // x 70,000 1.77 -> 1.57 ms per sweep; d = 50, 10,000 x 10,000
                  // 81.7 -> 80.6 us). Ranked lists gain nothing from it and the
                  // test costs them 0.5 %.
                  if constexpr (kSweepLike) {
                    if (sp * KBS * 4 + k >= p.ksteps) break;
                  }
                  const int kbl = k >> 2, kk = k & 3;
                  const uint64_t adesc =
                      a0 + (uint32_t)(sp * KBS * (kOwnBytesPerKB >> 4)) +
                      (uint32_t)((kbl * kOwnBytesPerKB + h * 128 * 128 + kk * 32) >> 4);
                  const uint64_t bdesc = b0 + (uint32_t)((kbl * kParBytes + kk * 32) >> 4);
                  const uint32_t accum = (sp > 0 || k > 0) ? 1u : 0u;
                  if constexpr (PAIR && F8) {
                    umma_e4m3_pair(d_tmem, adesc, bdesc, idesc, accum);
                  } else if constexpr (PAIR) {
                    umma_bf16_pair(d_tmem, adesc, bdesc, idesc, accum);
                  } else if constexpr (F8) {
                    umma_e4m3(d_tmem, adesc, bdesc, idesc, accum);
                  } else {
                    umma_bf16(d_tmem, adesc, bdesc, idesc, accum);
                  }
                }
                if constexpr (FOLD) {
                  // D += ones x (g / c): every row gets the partner column's g / c
                  if (sp == SPT - 1) {
                    const uint64_t gc = gc_base + (uint32_t)((stage * SB + KBS * kParBytes) >> 4);
                    if constexpr (PAIR) {
                      umma_bf16_pair(d_tmem, ones, gc, idesc_fold, 1u);
                    } else {
                      umma_bf16(d_tmem, ones, gc, idesc_fold, 1u);
                    }
                  }
                }
              }
              commit(&empty[stage]);
              if (sp == SPT - 1) {
                commit(&tfull[buf]);
                if (j == je - 1) commit(a_release);
              }
            }
            __syncwarp();
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          buf ^= 1;
          if (buf == 0) tphase ^= 1u;
        }
      }
      if (!ok && lane == 0 && !*abort_flag) raise_error(p.err, abort_flag, kErrTimeout);
      // all MMAs issued by this warp complete before TMEM is released
      if (elect_one()) commit(mma_done);
      __syncwarp();
      mbar_wait_drain(mma_done, 0, 100000000ull);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 2;          // 0..15
    const int q = warp & 3;           // TMEM lane quadrant this warp may access
    const int h = (ew >> 2) & 1;      // own sub-tile: rows [h*128, h*128+128)
    const int half = ew >> 3;         // columns [half*64, half*64+64) of every partner tile
    uint64_t cc = 0ull;
    float crow = p.c;  // this thread's row's exponent multiplier (e4m3: times the row's scale)
    // single market: the shift, own offset and omega of the launch (batched: per item)
    const double shift0 = BATCH ? 0.0 : __ldg(p.lmax);
    // (ranked lists and mu blocks run on potentials without pending offsets:
    // every block of sweeps ends by writing them into the arrays)
    const double own_off0 = (kSweepLike && !BATCH && p.own_off != nullptr) ? *p.own_off : 0.0;
    const double omega0 = (!BATCH && p.omega != nullptr && p.update) ? *p.omega : 1.0;
    int buf = 0, gs = 0;
    uint32_t tphase = 0, gphase = 0;
    bool ok = true;
    if constexpr (kSweepLike && !BATCH) {
      // this warp's partials over its own tiles, in shared memory: carried in
      // registers they would stay live across the tile loop
      if (lane == 0) *reinterpret_cast<RowPartials*>(red + 4 * ew) = RowPartials{0.0, 0.0, 0.0, 0.0};
    }
    uint32_t va[32], vb[32];
    // ranked lists: this thread's sorted candidates for its row and column half
    float tv[MODE == kModeTopK ? kMaxTopK : 1];
    int32_t ti[MODE == kModeTopK ? kMaxTopK : 1];
    // shared-memory lists: this thread's entry 0 (128-row tiles: warps 0-3
    // and 8-11 have rows; the others share their addresses and touch none)
    constexpr uint32_t kSlotStride = list_threads(SMALL) * 8;
    const int lt = (SMALL ? (ew >> 3) * 4 + (ew & 3) : ew) * 32 + lane;
    const uint32_t lv = smem_u32(topk_list) + (uint32_t)lt * 8u;
    SharedBound sb{};
    {
      // (a row's other column half: epilogue warp ew ^ 8)
      const uint32_t words = smem_u32(topk_list) + (uint32_t)(list_slots(SMALL) * list_threads(SMALL)) * 8u;
      sb.mine = words + (uint32_t)lt * 8u;
      sb.other = words + (uint32_t)(lt ^ (list_threads(SMALL) / 2)) * 8u;
    }
    int tcnt = 0;
    int merge_at = 0;  // the partner tile before which every warp merges its candidates
    float thr = -INFINITY;
    int tile_iter = 0;
    Seg sg;
    for (; ok && item_at<BATCH, SPLIT, PAIR>(p, tile_iter, sg); ++tile_iter) {
      const BatchDesc* bd = nullptr;
      int t, jb = 0, je;
      if constexpr (BATCH) {
        const ItemRef w = batch_item(p, sg.t);
        bd = w.d;
        t = w.t;
        je = bd->num_partner_tiles;
      } else {
        t = PAIR ? 2 * sg.t + rank : sg.t;
        jb = sg.jb;
        je = sg.je;
      }
      const double shift = BATCH ? bd->st[kStShift] : shift0;
      const int rloc = h * 128 + q * 32 + lane;          // row within the own tile
      const int64_t r = (int64_t)t * kOwn + rloc;         // row within the launch
      const bool row_ok = rloc < kOwn && r < (BATCH ? bd->rows : p.rows);
      crow = BATCH ? bd->c : p.c;
      if constexpr (RS) {
        const float* fso = BATCH ? bd->fs_own : p.fs_own;
        if (row_ok) crow *= fso[(BATCH ? 0 : p.row0) + r];
      }
      {
        const uint32_t cb = __float_as_uint(crow);
        cc = ((uint64_t)cb << 32) | cb;
      }
      float sum = 0.0f, comp = 0.0f;
      float mu_lo = 0.0f;
      int mu_hi = 0;
      float mu_s1 = 1.0f, mu_s2 = 1.0f;
      // mu blocks: this warp's first row of the block, and how many it has there
      const int64_t mu_row = (int64_t)t * kOwn + h * 128 + q * 32;
      const int mu_nrow = MODE == kModeMu ? (int)(p.rows - mu_row < 32 ? p.rows - mu_row : 32) : 0;
      float wide_m = -INFINITY;  // wide markets: the row's running shift (an integer, log2 units)
      // the partner tile before which this row's sum is cut next, and whether it was cut at all
      int cut_at = kNoCut;
      bool was_cut = false;
      if constexpr (RANGES) {
        cut_at = BATCH ? next_cut((int64_t)t * kFusedOwnRows, bd->cut_rows, bd->cut_t0, bd->cut_span, je)
                       : next_cut(p.row0 + r, p.cut_rows, p.cut_t0, p.cut_span, p.cut_ptiles);
      }
      if constexpr (MODE == kModeMu) {
        if (row_ok) {
          const double off = (shift + p.ell[p.row0 + r]) * 1.4426950408889634;
          const double fl = floor(off);
          mu_hi = (int)fl;
          mu_lo = (float)(off - fl);
          const int e = mu_hi < -252 ? -252 : (mu_hi > 252 ? 252 : mu_hi);
          mu_s1 = __int_as_float((127 + e / 2) << 23);
          mu_s2 = __int_as_float((127 + e - e / 2) << 23);
        }
      }
      if constexpr (MODE == kModeTopK) {
        tcnt = 0;
        thr = -INFINITY;
      }
      if constexpr (MODE == kModeTopKShared) {
        if (!(SMALL && h == 1))
          for (int i = 0; i < p.k; ++i) sts_u64(lv + (uint32_t)i * kSlotStride, slot_of(-INFINITY, 0x7fffffff));
        thr = -INFINITY;
        tcnt = 0;
        merge_at = jb + 1;
        sb.tag = (uint32_t)tile_iter + 1u;
        sb.pub = -INFINITY;
        if (!(SMALL && h == 1)) sts_u64(sb.mine, ((uint64_t)sb.tag << 32) | __float_as_uint(-INFINITY));
      }
      for (int j = jb; j < je; ++j) {
        // every lane waits; the outcome is made warp-uniform so that the
        // .sync.aligned TMEM loads below never run with a partial warp
        bool got = mbar_wait(&tfull[buf], tphase, abort_flag);
        if constexpr (!FOLD) got = got && mbar_wait(&gfull[gs], gphase, abort_flag);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr =
            tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + h * 128 + half * 64);
        const float* gsf = sG + gs * kFusedPartnerRows + half * 64;
        const float4* gs4 = reinterpret_cast<const float4*>(gsf);
        const float* fsf = sF + gs * kFusedPartnerRows + half * 64;  // (per-row scales only)
        const float4* fs4 = reinterpret_cast<const float4*>(fsf);
        const int64_t colbase = p.col0 + (int64_t)j * kFusedPartnerRows + half * 64;
        uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
        // SMALL: the second sub-tile's warps keep step with the barriers only
        const bool idle = SMALL && h == 1;
        if (!idle) {
          // the second 32-column chunk is loaded while the first is processed
          tmem_ld_issue(taddr, va);
          tmem_ld_wait(va);
          tmem_ld_issue(taddr + 32, vb);
          if constexpr (FOLD) chunk_sum_fold(va, cc, acc);
          if constexpr (MODE == kModeSweep && !FOLD) chunk_sum<RS>(va, gs4, fs4, cc, acc);
          if constexpr (MODE == kModeSweepWide) chunk_sum_wide<RS>(va, gs4, fs4, cc, acc, wide_m, sum, comp);
          if constexpr (MODE == kModeTopK) chunk_topk<RS>(va, gsf, fsf, crow, colbase, p.k, tv, ti, &tcnt, thr);
          if constexpr (MODE == kModeTopKShared)
            chunk_topk_shared<RS, SMALL>(va, gsf, fsf, cc, colbase, p.k, lv, tcnt, thr, sb);
          if constexpr (MODE == kModeMu)
            chunk_mu<RS, mu_width(KB)>(va, gsf, fsf, crow, colbase, mu_lo, mu_hi, mu_s1, mu_s2, lane, mu_nrow, mu_row,
                         topk_list + ew * mu_stage_floats(KB), p);
          tmem_ld_wait(vb);
        }
        // this warp's part of the accumulator buffer has been read: hand it back to the MMA warp
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) {
            cluster_arrive(cluster_addr(&tempty[buf], 0));
          } else {
            mbar_arrive(&tempty[buf]);
          }
        }
        if (!idle) {
          if constexpr (FOLD) chunk_sum_fold(vb, cc, acc);
          if constexpr (MODE == kModeSweep && !FOLD) chunk_sum<RS>(vb, gs4 + 8, fs4 + 8, cc, acc);
          if constexpr (MODE == kModeSweepWide) chunk_sum_wide<RS>(vb, gs4 + 8, fs4 + 8, cc, acc, wide_m, sum, comp);
          if constexpr (MODE == kModeTopK)
            chunk_topk<RS>(vb, gsf + 32, fsf + 32, crow, colbase + 32, p.k, tv, ti, &tcnt, thr);
          if constexpr (MODE == kModeTopKShared)
            chunk_topk_shared<RS, SMALL>(vb, gsf + 32, fsf + 32, cc, colbase + 32, p.k, lv, tcnt, thr, sb);
          if constexpr (MODE == kModeMu)
            chunk_mu<RS, mu_width(KB)>(vb, gsf + 32, fsf + 32, crow, colbase + 32, mu_lo, mu_hi, mu_s1, mu_s2, lane, mu_nrow,
                         mu_row, topk_list + ew * mu_stage_floats(KB), p);
        }
        if constexpr (!FOLD) {
          // the g slot has been read by this warp
          __syncwarp();
          if (lane == 0) mbar_arrive(&gempty[gs]);
        }
        if constexpr (kSweepLike) {
          // compensated (Kahan) accumulation of the per-tile partial sums
          const float tile =
              (unpack_sum(acc[0]) + unpack_sum(acc[1])) + (unpack_sum(acc[2]) + unpack_sum(acc[3]));
          const float y = tile - comp;
          const float tsum = sum + y;
          comp = (tsum - sum) - y;
          sum = tsum;
        }
        if constexpr (RANGES) {
          if (j + 1 == cut_at) {
            RangeSum rs = was_cut ? range_sum[ew * 32 + lane] : RangeSum();
            rs.add<WIDE>(sum, comp, wide_m);
            range_sum[ew * 32 + lane] = rs;
            sum = comp = 0.0f;
            wide_m = -INFINITY;
            was_cut = true;
            cut_at += BATCH ? bd->cut_span : p.cut_span;
            if (cut_at >= (BATCH ? je : p.cut_ptiles)) cut_at = kNoCut;
          }
        }
        if constexpr (MODE == kModeTopKShared) {
          // All warps merge after the same tiles, each a quarter further into
          // the row: a merge takes some thousand cycles, and the accumulator
          // buffers let a warp run two tiles ahead of the slowest, so merges
          // at different tiles would hold up the whole CTA one after another.
          if (j + 1 == merge_at) {
            merge_at += 1 + (merge_at - jb) / 4;
            if (!idle) {
              thr = list_merge<kSlotStride>(lv, p.k, tcnt);
              sb.publish(lv, p.k, kSlotStride);
              tcnt = 0;
            }
          }
        }
        buf ^= 1;
        if (buf == 0) tphase ^= 1u;
        if (++gs == kGSlots) {
          gs = 0;
          gphase ^= 1u;
        }
      }
      if (!ok) break;
      if constexpr (MODE == kModeMu) continue;
      if constexpr (RANGES) {
        if (was_cut) {  // the last range; the row's sum as hi + lo in the place of sum - comp
          RangeSum rs = range_sum[ew * 32 + lane];
          rs.add<WIDE>(sum, comp, wide_m);
          sum = rs.hi;
          comp = -rs.lo;
          wide_m = rs.m;
        }
      }
      if constexpr (MODE == kModeTopKShared) {
        if (!(SMALL && h == 1)) list_merge<kSlotStride>(lv, p.k, tcnt);
      }
      // the two column halves of a row meet (double-buffered by own-tile
      // parity, handed over through bounded mbarrier waits)
      const int pb = tile_iter & 1;
      const uint32_t rphase = (uint32_t)(tile_iter >> 1) & 1u;
      float* rb = rowbuf + pb * kFusedOwnRows;
      if (half == 1) {
        if (!__all_sync(0xffffffffu, mbar_wait(&rowfree[pb], rphase ^ 1u, abort_flag))) {
          ok = false;
          break;
        }
        if constexpr (kSweepLike) rb[rloc] = SPLIT ? sum : sum - comp;
        if constexpr (kSweepLike && SPLIT) row_comp[pb * kFusedOwnRows + rloc] = comp;
        if constexpr (MODE == kModeSweepWide) wide_shift[pb * kFusedOwnRows + rloc] = wide_m;
        if constexpr (MODE == kModeTopK) {
          if (row_ok)
            for (int i = 0; i < p.k; ++i) {
              p.hand_v[r * p.k + i] = i < tcnt ? tv[i] : -INFINITY;
              p.hand_i[r * p.k + i] = i < tcnt ? ti[i] : 0x7fffffff;
            }
        }
        if constexpr (MODE == kModeTopKShared) {
          if (row_ok)
            for (int i = 0; i < p.k; ++i) {
              const uint64_t w = lds_u64(lv + (uint32_t)i * kSlotStride);
              p.hand_v[r * p.k + i] = slot_score(w);
              p.hand_i[r * p.k + i] = slot_col(w);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfull[pb]);
        continue;
      }
      if (!__all_sync(0xffffffffu, mbar_wait(&rowfull[pb], rphase, abort_flag))) {
        ok = false;
        break;
      }
      if constexpr (MODE == kModeTopK) {
        if (row_ok) {
          // merge the two sorted halves: higher score first, lower index on ties
          const double base = shift + p.ell[p.row0 + r];
          int a = 0, b = 0;
          for (int i = 0; i < p.k; ++i) {
            const float bv = p.hand_v[r * p.k + b];
            const int32_t bi = p.hand_i[r * p.k + b];
            const bool take_a = a < tcnt && (b >= p.k || tv[a] > bv || (tv[a] == bv && ti[a] < bi));
            const float sv = take_a ? tv[a] : bv;
            p.idx[r * p.k + i] = take_a ? ti[a] : bi;
            if (p.logmu != nullptr) p.logmu[r * p.k + i] = (float)((double)sv * 0.69314718055994530942 + base);
            if (take_a) ++a; else ++b;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfree[pb]);
      }
      if constexpr (MODE == kModeTopKShared) {
        if (row_ok) {
          // merge the two sorted halves (both exactly k entries, padded with
          // (-inf, INT32_MAX)): higher score first, lower index on ties
          const double base = shift + p.ell[p.row0 + r];
          int a = 0, b = 0;
          for (int i = 0; i < p.k; ++i) {
            const uint64_t w = lds_u64(lv + (uint32_t)a * kSlotStride);
            const float av = slot_score(w);
            const int32_t ai = slot_col(w);
            const float bv = p.hand_v[r * p.k + b];
            const int32_t bi = p.hand_i[r * p.k + b];
            const bool take_a = av > bv || (av == bv && ai < bi);
            const float sv = take_a ? av : bv;
            p.idx[r * p.k + i] = take_a ? ai : bi;
            if (p.logmu != nullptr) p.logmu[r * p.k + i] = (float)((double)sv * 0.69314718055994530942 + base);
            if (take_a) ++a; else ++b;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfree[pb]);
      }
      if constexpr (kSweepLike) {
        float other = rb[rloc];
        float other_m = 0.0f, other_comp = 0.0f;
        if constexpr (WIDE) other_m = wide_shift[pb * kFusedOwnRows + rloc];
        if constexpr (SPLIT) other_comp = row_comp[pb * kFusedOwnRows + rloc];
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfree[pb]);
        const int64_t row = p.row0 + r;
        if constexpr (SPLIT) {
          if (sg.n > 1) {
            // this range's partial; the warp that completes the (tile, 32-row
            // block) sums all ranges in order and updates the rows (no wait:
            // the other warps of this block move on)
            const int64_t blk = (int64_t)t * (kFusedOwnRows / 32) + (h * 128 + q * 32) / 32;
            const bool cuts = p.split == 1;
            const int u = sg.t - p.cut_t0, k0 = cuts ? cut_first(p, u) : 0;
            auto slot = [&](int c) -> int64_t {
              return cuts ? ((int64_t)cut_slot(p, u, k0 + c) * (PAIR ? 2 : 1) + rank) * kFusedOwnRows + rloc
                          : (int64_t)c * p.rows + r;
            };
            if (row_ok) {
              p.part[slot(sg.me)] = make_float4(sum, comp, other, other_comp);
              if constexpr (WIDE) p.part_m[slot(sg.me)] = make_float2(wide_m, other_m);
            }
            __threadfence();
            __syncwarp();
            int prev = 0;
            if (lane == 0) prev = atomicAdd(p.split_cnt + blk, 1);
            prev = __shfl_sync(0xffffffffu, prev, 0);
            if (prev != sg.n - 1) continue;
            if (lane == 0) p.split_cnt[blk] = 0;  // ready for the next launch
            __threadfence();
            if (row_ok) {
              RangeSum a, b;
              for (int c0 = 0; c0 < sg.n; c0 += 4) {  // four loads in flight
                float4 v[4];
                float2 m[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const int64_t at = slot(c0 + c < sg.n ? c0 + c : c0);
                  v[c] = __ldcg(p.part + at);
                  if constexpr (WIDE) m[c] = __ldcg(p.part_m + at);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  if (c0 + c >= sg.n) break;
                  a.add<WIDE>(v[c].x, v[c].y, WIDE ? m[c].x : 0.0f);
                  b.add<WIDE>(v[c].z, v[c].w, WIDE ? m[c].y : 0.0f);
                }
              }
              sum = a.hi;
              comp = -a.lo;
              wide_m = a.m;
              other = b.hi;
              other_comp = -b.lo;
              other_m = b.m;
            }
          }
          other -= other_comp;
        }
        float row_m = 0.0f;  // wide markets: the shift of the row's sum (log2 units)
        if constexpr (WIDE) {
          // the two halves' sums onto the larger of their shifts (exact powers of two)
          row_m = fmaxf(wide_m, other_m);
          const float own_scale = exp2_int(wide_m - row_m);
          sum *= own_scale;
          comp *= own_scale;
          other *= exp2_int(other_m - row_m);
        }
        // the row's sum as three FP32 parts
        const float s_hi = sum, s_lo = -comp, s_o = other;
        RowResult rr{};
        if (row_ok) {
          const float* b2s = BATCH ? bd->b2s : p.b2s;
          double* log_u = BATCH ? bd->log_u : p.log_u;
          double* ell = BATCH ? bd->ell : p.ell;
          const double omega = BATCH ? ((bd->omega != nullptr && p.update) ? *bd->omega : 1.0) : omega0;
          const double own_off = BATCH ? bd->st[kStOwnOff] : own_off0;
          int ex;
          const float lm = log_row_sum_parts(s_hi, s_lo, s_o, ex);
          // wide markets: the row's shift comes back into the sum's logarithm
          // (no finite exponent: the sum is 0 and its logarithm -inf whatever is added)
          if constexpr (MODE == kModeSweepWide) ex += row_m > -1e9f ? (int)row_m : 0;
          rr = row_update(ex, lm, shift, b2s ? b2s[row] : 0.0f, (BATCH ? bd->mass : p.mass)[row],
                          log_u[row] + own_off, p.residual, omega);
          if (p.update) {
            log_u[row] = rr.log_u;
            ell[row] = rr.ell;
          }
        }
        // this warp's 32 rows form one group of the own side (the finalize
        // reduces the groups into the side's shift and sum of u^2)
        float4* grp = BATCH ? bd->grp : p.grp;
        const int64_t g = (int64_t)t * (kOwn / kGroupRows) + (h * 128 + q * 32) / kGroupRows;
        if (SMALL && h == 1) continue;  // (no rows)
        if (p.update && grp != nullptr && g * kGroupRows < (BATCH ? bd->rows : p.rows)) {
          const float4 gv = warp_group(rr.log_u, rr.ell, row_ok);
          if (lane == 0) grp[g] = gv;
        }
        const RowPartials rp = row_partials(rr, row_ok, p.residual);
        if (lane == 0) {
          if constexpr (BATCH) {
            // partials of this own tile and warp (warps ew = 0..7 own the row
            // updates); the batched finalize sums them per market in a fixed order
            *reinterpret_cast<RowPartials*>(p.partials + ((int64_t)(bd->slot0 + t) * kBatchSlotWarps + ew) * 4) = rp;
          } else {
            add_partials(*reinterpret_cast<RowPartials*>(red + 4 * ew), rp);
          }
        }
      }
    }
    if (!ok && !*abort_flag) raise_error(p.err, abort_flag, kErrTimeout);
    if constexpr (kSweepLike && !BATCH) {
      // the CTA's partials: those of the warps that own the row updates
      named_bar_sync(1, kEpiWarps * 32);
      if (ew == 0 && lane < 8) {
        RowPartials v = *reinterpret_cast<const RowPartials*>(red + 4 * lane);
        for (int o = 4; o > 0; o >>= 1) {
          const RowPartials w = {__shfl_xor_sync(0xffu, v.r_max, o), __shfl_xor_sync(0xffu, v.r_sum, o),
                                 __shfl_xor_sync(0xffu, v.sq, o), __shfl_xor_sync(0xffu, v.nf, o)};
          add_partials(v, w);
        }
        if (lane == 0) *reinterpret_cast<RowPartials*>(p.partials + 4 * blockIdx.x) = v;
      }
    }
  }

  tc_fence_before();
  if constexpr (PAIR) {
    cluster_sync();  // the pair's MMAs read and write both CTAs
  } else {
    __syncthreads();
  }
  if (warp == 0) {
    tc_fence_after();
    if constexpr (PAIR) {
      tmem_dealloc_pair(tmem_base, kTmemCols);
    } else {
      tmem_dealloc(tmem_base, kTmemCols);
    }
  }
}

// ---- instantiations and launches

constexpr int kSmemLimit = 232448;  // dynamic shared memory per CTA (227 KB)

// Partner stages per instantiation: as many as fit beside the own tile(s), the
// g (and scale) rings, the tail and (kModeTopKShared) the ranked lists, at
// most 6 whole tiles (one k block per row), 4 (two) or 5 single k blocks
// (four: 1.25 partner tiles in flight).
constexpr int stages_for(int KB, int MODE, int fmt, bool fold, bool split, bool ranges, bool pair) {
  const int fixed = smem_bytes(KB, fmt, 0, fold, pair) + mode_extra_bytes(MODE, KB, split, ranges);
  const int fit = (kSmemLimit - fixed) / stage_bytes(KB, fold, pair);
  const int cap = KB == 1 ? 6 : (KB == 2 ? (pair ? 6 : 4) : 5);
  return fit < cap ? fit : cap;
}

template <int KB, int MODE, int FMT, bool FOLD, bool SPLIT, bool RANGES, bool PAIR = false>
constexpr int kStages = stages_for(KB, MODE, FMT, FOLD, SPLIT, RANGES, PAIR);

template <int KB, int MODE, int FMT, bool FOLD, bool SPLIT, bool RANGES, bool PAIR = false>
constexpr int kSmemTotal =
    smem_bytes(KB, FMT, kStages<KB, MODE, FMT, FOLD, SPLIT, RANGES, PAIR>, FOLD, PAIR) + mode_extra_bytes(MODE, KB, SPLIT, RANGES);

// Instantiations that exist: batched launches take one or two k blocks
// (e4m3: one); the shared-memory ranked lists leave too little room for
// partner stages beside a four-block own tile (those lists use kModeTopK).
// SPLIT: the partner-split instantiation (single-market half-sweeps with
// tu_market_set_split > 1); the default kernel carries none of its code.
// NOFOLD: the BF16 half-sweep with g from the shared ring instead of the
// extra MMA, for callers without the folded operand (the allocation-free
// entry point).
// CUTS: unsplit half-sweeps of a market whose sums are cut (row ranges, the
// fixed own-tile heights).
template <int KB, int MODE, bool BATCH, int FMT, bool SPLIT = false, bool SMALL = false, bool NOFOLD = false,
          bool CUTS = false>
constexpr bool kBuilt = !(CUTS && (BATCH || SPLIT || NOFOLD || (MODE != kModeSweep && MODE != kModeSweepWide))) &&
                        !(BATCH && (KB == 4 || (FMT != kFmtBF16 && KB != 1))) &&
                        !(MODE == kModeTopKShared && KB == 4) && !(SPLIT && MODE != kModeSweep && MODE != kModeSweepWide && MODE != kModeMu) &&
                        !(SPLIT && MODE == kModeSweepWide && SMALL) &&
                        !(SPLIT && BATCH) && !(MODE == kModeMu && (!SPLIT || SMALL)) &&
                        !(NOFOLD && (!fold_for(KB, MODE, BATCH, FMT, false) || SPLIT || SMALL));

template <int KB, int MODE, bool BATCH, int FMT = kFmtBF16, bool SMALL = false, bool SPLIT = false,
          bool NOFOLD = false, bool CUTS = false>
cudaError_t launch_kernel(const CUtensorMap& own, const CUtensorMap& partner, const FusedParams& p, int grid,
                          cudaStream_t stream) {
  if constexpr (!kBuilt<KB, MODE, BATCH, FMT, SPLIT, SMALL, NOFOLD, CUTS>) {
    return cudaErrorNotSupported;
  } else {
    constexpr bool FD = fold_for(KB, MODE, BATCH, FMT, NOFOLD);
    constexpr int kSmem = kSmemTotal<KB, MODE, FMT, FD, SPLIT, CUTS || BATCH>;
    static_assert(kStages<KB, MODE, FMT, FD, SPLIT, CUTS || BATCH> >= 2, "at least two partner stages");
    static_assert(kSmem <= kSmemLimit, "shared memory budget");
    if (FD && !BATCH && p.gfold == nullptr) return cudaErrorInvalidValue;  // the folded operand must be prepared
    k_fused_halfsweep<KB, kStages<KB, MODE, FMT, FD, SPLIT, CUTS || BATCH>, MODE, BATCH, FMT, SMALL, SPLIT, NOFOLD, CUTS>
        <<<grid, kThreads, kSmem, stream>>>(own, partner, partner, p);
    return cudaGetLastError();
  }
}

template <int KB, int MODE, bool BATCH, int FMT, bool SMALL, bool SPLIT = false, bool NOFOLD = false,
          bool CUTS = false>
cudaError_t set_attribute_one() {
  if constexpr (!kBuilt<KB, MODE, BATCH, FMT, SPLIT, SMALL, NOFOLD, CUTS>) {
    return cudaSuccess;
  } else {
    constexpr bool FD = fold_for(KB, MODE, BATCH, FMT, NOFOLD);
    return cudaFuncSetAttribute(
        k_fused_halfsweep<KB, kStages<KB, MODE, FMT, FD, SPLIT, CUTS || BATCH>, MODE, BATCH, FMT, SMALL, SPLIT, NOFOLD, CUTS>,
        cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTotal<KB, MODE, FMT, FD, SPLIT, CUTS || BATCH>);
  }
}

template <int MODE, bool BATCH, bool SMALL, int FMT, bool SPLIT, bool CUTS>
cudaError_t set_attributes_fmt() {
  cudaError_t e = set_attribute_one<1, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>();
  if (e == cudaSuccess) e = set_attribute_one<2, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>();
  if (e == cudaSuccess) e = set_attribute_one<4, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>();
  return e;
}

template <int MODE, bool BATCH, bool SMALL, bool SPLIT = false, bool CUTS = false>
cudaError_t set_attributes_variant() {
  cudaError_t e = set_attributes_fmt<MODE, BATCH, SMALL, kFmtBF16, SPLIT, CUTS>();
  if (e == cudaSuccess) e = set_attributes_fmt<MODE, BATCH, SMALL, kFmtE4M3Side, SPLIT, CUTS>();
  if (e == cudaSuccess) e = set_attributes_fmt<MODE, BATCH, SMALL, kFmtE4M3Rows, SPLIT, CUTS>();
  return e;
}

template <int MODE, bool BATCH>
cudaError_t set_attributes_mode() {
  cudaError_t e = set_attributes_variant<MODE, BATCH, false>();
  if (e == cudaSuccess && !BATCH) e = set_attributes_variant<MODE, false, true>();
  if (MODE == kModeMu) {
    if (e == cudaSuccess) e = set_attributes_variant<MODE, false, false, true>();
  }
  if ((MODE == kModeSweep || MODE == kModeSweepWide) && !BATCH) {
    if (e == cudaSuccess) e = set_attributes_variant<MODE, false, false, true>();
    if (e == cudaSuccess) e = set_attributes_variant<MODE, false, true, true>();
    if (e == cudaSuccess) e = set_attributes_variant<MODE, false, false, false, true>();
    if (e == cudaSuccess) e = set_attributes_variant<MODE, false, true, false, true>();
  }
  return e;
}

// 128-byte k blocks of a packed row: kp elements of 2 bytes (BF16) or 1 (e4m3).
int k_blocks(int64_t kp, int fmt) { return (int)(fmt != kFmtBF16 ? kp / 128 : kp / kKBlock); }

template <int MODE, bool BATCH, bool SMALL, int FMT, bool SPLIT, bool CUTS>
cudaError_t launch_fmt(int kb, const CUtensorMap& own, const CUtensorMap& partner, const FusedParams& p, int grid,
                       cudaStream_t stream) {
  if (kb == 1) return launch_kernel<1, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>(own, partner, p, grid, stream);
  if (kb == 2) return launch_kernel<2, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>(own, partner, p, grid, stream);
  if (kb == 4) return launch_kernel<4, MODE, BATCH, FMT, SMALL, SPLIT, false, CUTS>(own, partner, p, grid, stream);
  return cudaErrorNotSupported;
}

template <int MODE, bool BATCH = false, bool SMALL = false, bool SPLIT = false, bool CUTS = false>
cudaError_t launch_variant(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                           const FusedParams& p, int grid, cudaStream_t stream) {
  const int kb = k_blocks(kp, fmt);
  if (fmt == kFmtE4M3Rows)
    return launch_fmt<MODE, BATCH, SMALL, kFmtE4M3Rows, SPLIT, CUTS>(kb, own, partner, p, grid, stream);
  if (fmt == kFmtE4M3Side)
    return launch_fmt<MODE, BATCH, SMALL, kFmtE4M3Side, SPLIT, CUTS>(kb, own, partner, p, grid, stream);
  return launch_fmt<MODE, BATCH, SMALL, kFmtBF16, SPLIT, CUTS>(kb, own, partner, p, grid, stream);
}

// small: 128-row own tiles (single-market launches only; see use_small_tiles)
template <int MODE, bool BATCH = false>
cudaError_t launch_any(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                       const FusedParams& p, int grid, cudaStream_t stream, bool small = false) {
  if constexpr (!BATCH) {
    if (small) return launch_variant<MODE, false, true>(kp, fmt, own, partner, p, grid, stream);
  }
  return launch_variant<MODE, BATCH, false>(kp, fmt, own, partner, p, grid, stream);
}

// Pairs of CTAs (kb > 1): the pair kernel's attributes and launch.
template <int KB, int MODE, int FMT, bool SPLIT>
cudaError_t pair_kernel(const CUtensorMap* own, const CUtensorMap* half, const CUtensorMap* fold, const FusedParams* p,
                        int grid, cudaStream_t stream) {
  constexpr bool FD = fold_for(KB, MODE, false, FMT, false);
  constexpr int kSt = kStages<KB, MODE, FMT, FD, SPLIT, false, true>;
  constexpr int kSmem = kSmemTotal<KB, MODE, FMT, FD, SPLIT, false, true>;
  static_assert(kSt >= 4 && kSmem <= kSmemLimit, "shared memory budget");
  auto kern = k_fused_halfsweep<KB, kSt, MODE, false, FMT, false, SPLIT, false, false, true>;
  if (p == nullptr) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3(kThreads);
  c.dynamicSmemBytes = kSmem;
  c.stream = stream;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kern, *own, *half, *fold, *p);
}
template <int MODE, int FMT>
cudaError_t pair_fmt(int kb, bool split, const CUtensorMap* own, const CUtensorMap* half, const CUtensorMap* fold,
                     const FusedParams* p, int grid,
                     cudaStream_t stream) {
  if (kb == 2)
    return split ? pair_kernel<2, MODE, FMT, true>(own, half, fold, p, grid, stream)
                 : pair_kernel<2, MODE, FMT, false>(own, half, fold, p, grid, stream);
  if (kb == 4)
    return split ? pair_kernel<4, MODE, FMT, true>(own, half, fold, p, grid, stream)
                 : pair_kernel<4, MODE, FMT, false>(own, half, fold, p, grid, stream);
  return cudaErrorNotSupported;
}
// p == nullptr: set the attributes
template <int MODE>
cudaError_t launch_pair(int kb, int fmt, bool split, const CUtensorMap* own, const CUtensorMap* half,
                        const CUtensorMap* fold, const FusedParams* p, int grid, cudaStream_t stream) {
  if (fmt == kFmtE4M3Rows) return pair_fmt<MODE, kFmtE4M3Rows>(kb, split, own, half, fold, p, grid, stream);
  if (fmt == kFmtE4M3Side) return pair_fmt<MODE, kFmtE4M3Side>(kb, split, own, half, fold, p, grid, stream);
  return pair_fmt<MODE, kFmtBF16>(kb, split, own, half, fold, p, grid, stream);
}
template <int MODE>
cudaError_t set_pair_attributes() {
  for (int kb : {2, 4})
    for (int fmt : {(int)kFmtBF16, (int)kFmtE4M3Side, (int)kFmtE4M3Rows})
      for (bool split : {false, true}) {
        const cudaError_t e = launch_pair<MODE>(kb, fmt, split, nullptr, nullptr, nullptr, nullptr, 0, nullptr);
        if (e != cudaSuccess) return e;
      }
  return cudaSuccess;
}

// Half-sweeps of one market: split over CTAs (by the caller's ranges or the
// market's cuts), a cut row's ranges in turn, or plain.
template <int MODE>
cudaError_t launch_sweep(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                         const FusedParams& p, int grid, cudaStream_t stream, bool small, bool split) {
  if (split && small) return launch_variant<MODE, false, true, true>(kp, fmt, own, partner, p, grid, stream);
  if (split) return launch_variant<MODE, false, false, true>(kp, fmt, own, partner, p, grid, stream);
  if (p.cut_span > 0) {
    if (small) return launch_variant<MODE, false, true, false, true>(kp, fmt, own, partner, p, grid, stream);
    return launch_variant<MODE, false, false, false, true>(kp, fmt, own, partner, p, grid, stream);
  }
  return launch_any<MODE>(kp, fmt, own, partner, p, grid, stream, small);
}

}  // namespace

// fused_out.cu: the instantiations of wide half-sweeps, ranked lists and mu
// blocks (compiled beside fused.cu's narrow and batched half-sweeps).
cudaError_t set_out_attributes();
cudaError_t launch_wide_sweep(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                              const FusedParams& p, int grid, cudaStream_t stream, bool small, bool split);
cudaError_t launch_wide_pair(int kb, int fmt, bool split, const CUtensorMap* own, const CUtensorMap* half,
                             const CUtensorMap* fold, const FusedParams* p, int grid, cudaStream_t stream);
cudaError_t launch_lists(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                         const FusedParams& p, int grid, cudaStream_t stream, bool small);
bool lists_want_small(int k, int64_t kp, int fmt);
cudaError_t launch_mu(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner, const FusedParams& p,
                      int grid, cudaStream_t stream);

}  // namespace tu
