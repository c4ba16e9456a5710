// dense.cu -- batch IPFP (Alg. 1, Eq. iteration_matrix) over a materialised
// FP32 kernel. A-hat_xy = exp((Phi_xy - b^X_x - b^Y_y) / (2 sigma)) is built
// once; the biases live in the potentials (ell = log u + b / (2 sigma)), so
//     s_x = 1/2 exp(b^X_x / 2 sigma) sum_y A-hat_xy exp(ell_y)
// and sweeps are HBM streams over a row-major matrix: one per sweep
// (k_dense_sweep) where the market's shape allows it, else one per half-sweep.
//
// HBM layout: A-hat (N x ldA, ldA = M rounded up to 4) and its transpose
// (M x ldN). With both resident, the v step (s = A^T u / 2) is the same row
// stream as the u step (s = A v / 2): each row is streamed once through a
// shared-memory ring by bulk copies, reduced in a fixed order and updated in
// closed form (k_dense_rowpass). Deterministic; the price is 2 * N * M * 4
// bytes of HBM instead of N * M * 4.
#include "tu_internal.cuh"

#include <type_traits>

namespace tu {

namespace {

// s += x * w with Kahan compensation c (the running error of s, subtracted
// from the next term); the product enters the compensated add unrounded.
__device__ __forceinline__ void kahan_fma(float& s, float& c, float x, float w) {
  const float y = fmaf(x, w, -c);
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

constexpr int kThreads = 256;  // the A-hat build

// A-hat and its transpose from the packed FP32 factors (setup, once per factor
// update). 64 x 64 output tile per CTA; the transposed tile is staged in
// shared memory so both stores are coalesced.
__global__ void __launch_bounds__(256) k_dense_build(const float* __restrict__ AX, const float* __restrict__ AY,
                                                     int64_t N, int64_t M, int64_t kp, float inv2s,
                                                     float* __restrict__ Ahat, int64_t ldA, float* __restrict__ AhatT,
                                                     int64_t ldN) {
  __shared__ float As[16][64 + 4];
  __shared__ float Bs[16][64 + 4];
  __shared__ float Ts[64][64 + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t col0 = (int64_t)blockIdx.x * 64;
  // row tiles in steps of the grid's height (at most 65,535), so that any N
  // fits one launch; the trip count is the same for every thread of a block
  for (int64_t row0 = (int64_t)blockIdx.y * 64; row0 < N; row0 += (int64_t)gridDim.y * 64) {
    float acc[4][4] = {};
    for (int64_t k0 = 0; k0 < kp; k0 += 16) {
      for (int e = threadIdx.x; e < 16 * 64; e += kThreads) {
        const int r = e / 16, kk = e % 16;
        const int64_t gr = row0 + r, gc = col0 + r;
        As[kk][r] = (gr < N) ? AX[gr * kp + k0 + kk] : 0.0f;
        Bs[kk][r] = (gc < M) ? AY[gc * kp + k0 + kk] : 0.0f;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {
        float a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t r = row0 + ty * 4 + i;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t c = col0 + tx * 4 + j;
        const float v = (r < N && c < M) ? expf(acc[i][j] * inv2s) : 0.0f;
        Ts[tx * 4 + j][ty * 4 + i] = v;
        if (r < N && c < ldA) Ahat[r * ldA + c] = v;
      }
    }
    __syncthreads();
    // transposed tile: row c of A-hat^T holds column c of A-hat
    for (int e = threadIdx.x; e < 64 * 64; e += kThreads) {
      const int cl = e / 64, rl = e % 64;
      const int64_t c = col0 + cl, r = row0 + rl;
      if (c < M && r < ldN) AhatT[c * ldN + r] = (r < N) ? Ts[cl][rl] : 0.0f;
    }
    __syncthreads();  // Ts is rewritten by the next row tile
  }
}

// A warp's partials to its CTA's place.
__device__ __forceinline__ void store_partials(double* dst, const RowPartials& p) {
  dst[0] = p.r_max;
  dst[1] = p.r_sum;
  dst[2] = p.sq;
  dst[3] = p.nf;
}

// One half-sweep over a row-major matrix A (rows x ld): for every row r,
// s_r = 1/2 exp(b_r / 2 sigma) exp(shift) sum_c A[r][c] w_c with
// w_c = exp(ell_c - shift) of the partner side (zero-padded to ld), then the
// closed-form update of the row's potential. RELAX: the update is
// over-relaxed by the device scalar *omega_p (markets with relaxation
// enabled); the plain instantiation is Eq. iteration exactly.
//
// Roles of a CTA (rows blockIdx.x, blockIdx.x + gridDim.x, ... in turn):
//   producer warp   one thread streams each row in kChunk-float pieces into a
//                   kStages ring in shared memory with 1D bulk copies
//                   (completion counted on the stage's mbarrier), so the
//                   bytes in flight do not depend on registers or on what
//                   the other warps are doing;
//   consumer warps  every warp takes strided float4s of each piece against
//                   the partner vector, releases the stage, and parks its
//                   share of the row sum; a block of kSlots rows is handed
//                   over once complete (double-buffered);
//   update warp     sums a block's parked shares in a fixed order and runs
//                   the kSlots closed-form updates in parallel (one per lane),
//                   off the stream's critical path, then frees the buffer.
// Every wait is bounded and sets the market's error word when it runs out;
// the producer then waits for its copies in flight before the CTA exits.
constexpr int kStages = 4;
constexpr int kChunk = 4096;  // floats per stage (16 KB)
constexpr int kConsumerWarps = 8;
constexpr int kUpdateWarp = kConsumerWarps;
constexpr int kProducerWarp = kConsumerWarps + 1;
constexpr int kPassThreads = (kConsumerWarps + 2) * 32;
constexpr int kSlots = 32;  // rows per block of updates: one per lane of the update warp

struct PassSmem {
  float ring[kStages][kChunk];
  float part[2][kSlots][kConsumerWarps];
  uint64_t full[kStages];   // a piece has landed (transaction count)
  uint64_t empty[kStages];  // every consumer warp is done with the stage
  uint64_t done[2];         // a block's row shares are parked
  uint64_t freed[2];        // the update warp has read the block
  int abort;
};

__device__ __forceinline__ void bulk_copy(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(gsrc)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void pass_abort(int* err, volatile int* flag) {
  atomicCAS(err, kErrNone, kErrTimeout);
  *flag = 1;
}

template <bool RELAX>
__global__ void __launch_bounds__(kPassThreads) k_dense_rowpass(
    const float* __restrict__ A, int64_t ld, int64_t rows, const float* __restrict__ w,
    const double* __restrict__ st, const float* __restrict__ b2s, const double* __restrict__ mass,
    double* __restrict__ log_u, double* __restrict__ ell, float4* __restrict__ grp, int64_t grp_blocks,
    double* __restrict__ partials, int residual, int update, const double* __restrict__ omega_p,
    int* __restrict__ err) {
  extern __shared__ __align__(128) uint8_t pass_smem_raw[];
  PassSmem& S = *reinterpret_cast<PassSmem*>(pass_smem_raw);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  volatile int* abort_flag = &S.abort;
  if (threadIdx.x == 0) {
    for (int t = 0; t < kStages; ++t) {
      mbar_init(&S.full[t], 1);
      mbar_init(&S.empty[t], kConsumerWarps);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&S.done[t], kConsumerWarps);
      mbar_init(&S.freed[t], 1);
    }
    S.abort = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const int64_t G = gridDim.x;
  const int64_t nchunks = (ld + kChunk - 1) / kChunk;
  // rows of this CTA (the grid never exceeds rows)
  const int64_t nrows = (rows - blockIdx.x + G - 1) / G;

  if (warp == kProducerWarp) {
    if (lane == 0) {
      int t = 0;
      uint32_t ph = 0, issued = 0, issued_ph = 0;
      bool ok = true;
      for (int64_t k = 0; k < nrows && ok; ++k) {
        const float* arow = A + (blockIdx.x + k * G) * ld;
        for (int64_t c = 0; c < nchunks; ++c) {
          if (!mbar_wait(&S.empty[t], ph ^ 1u, abort_flag)) {
            ok = false;
            break;
          }
          const int64_t c0 = c * kChunk;
          const uint32_t n = (uint32_t)(ld - c0 < kChunk ? ld - c0 : kChunk);
          mbar_arrive_expect_tx(&S.full[t], n * 4u);
          bulk_copy(S.ring[t], arow + c0, n * 4u, &S.full[t]);
          issued |= 1u << t;
          issued_ph = (issued_ph & ~(1u << t)) | (ph << t);
          if (++t == kStages) {
            t = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok && !*abort_flag) pass_abort(err, abort_flag);
      // copies in flight complete before the CTA's shared memory is released
      for (int u = 0; u < kStages; ++u)
        if (issued & (1u << u)) mbar_wait_drain(&S.full[u], (issued_ph >> u) & 1u, 100000000ull);
    }
    return;
  }

  if (warp < kConsumerWarps) {
    const float4* w4 = reinterpret_cast<const float4*>(w);
    int t = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int64_t k = 0; k < nrows && ok; ++k) {
      // four compensated (Kahan) sums per lane: a row of a few million terms
      // gives each accumulator thousands of them, where a plain FP32 sum
      // would drift by that many units of 2^-24; the pass is memory-bound,
      // so the three extra operations per term are free
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
      float e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;  // their compensations
      for (int64_t c = 0; c < nchunks; ++c) {
        const bool got = mbar_wait(&S.full[t], ph, abort_flag);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        const int64_t c0 = c * kChunk;
        const int nq = (int)((ld - c0 < kChunk ? ld - c0 : kChunk) / 4);
        const float4* r4 = reinterpret_cast<const float4*>(S.ring[t]);
        const float4* g4 = w4 + c0 / 4;
        for (int q = warp * 32 + lane; q < nq; q += kConsumerWarps * 32) {
          const float4 x = r4[q];
          const float4 y = __ldg(g4 + q);
          kahan_fma(a0, e0, x.x, y.x);
          kahan_fma(a1, e1, x.y, y.y);
          kahan_fma(a2, e2, x.z, y.z);
          kahan_fma(a3, e3, x.w, y.w);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.empty[t]);
        if (++t == kStages) {
          t = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      float sum = ((a0 - e0) + (a1 - e1)) + ((a2 - e2) + (a3 - e3));
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const int slot = (int)(k % kSlots);
      const int64_t blk = k / kSlots;
      const int pb = (int)(blk & 1);
      if (slot == 0 && blk >= 2) {
        // the update warp has read this buffer's previous block
        const bool fr = mbar_wait(&S.freed[pb], (uint32_t)(((blk >> 1) - 1) & 1), abort_flag);
        if (!__all_sync(0xffffffffu, fr)) {
          ok = false;
          break;
        }
      }
      if (lane == 0) {
        S.part[pb][slot][warp] = sum;
        if (slot == kSlots - 1 || k == nrows - 1) mbar_arrive(&S.done[pb]);
      }
    }
    if (!ok && !*abort_flag) pass_abort(err, abort_flag);
    return;
  }

  if (warp != kUpdateWarp) return;
  RowPartials acc = {0.0, 0.0, 0.0, 0.0};
  // the pass's partner shift and own offset (market scalars set by the preparation)
  double shift = 0.0, own_off = 0.0;
  if constexpr (!RELAX) {
    shift = st[kStShift];
    own_off = st[kStOwnOff];
  }
  // a block's shares arrive after kSlots rows are streamed: allow for 1 GB/s per CTA
  const uint64_t block_limit = kWaitLimitNs + (uint64_t)kSlots * (uint64_t)ld * 4ull;
  bool ok = true;
  for (int64_t blk = 0; blk * kSlots < nrows; ++blk) {
    const int pb = (int)(blk & 1);
    const bool got = mbar_wait(&S.done[pb], (uint32_t)((blk >> 1) & 1), abort_flag, block_limit);
    if (!__all_sync(0xffffffffu, got)) {
      ok = false;
      break;
    }
    const int64_t k = blk * kSlots + lane;
    RowResult rr{};
    if (k < nrows) {
      const int64_t row = blockIdx.x + k * G;
      // the eight warps' shares, added with their roundings kept (two-sum)
      float sum = 0.0f, err = 0.0f;
      for (int cw = 0; cw < kConsumerWarps; ++cw) {
        float e;
        sum = two_sum(sum, S.part[pb][lane][cw], e);
        err = __fadd_rn(err, e);
      }
      double omega = 1.0;
      if constexpr (RELAX) {
        shift = __ldg(st + kStShift);
        own_off = __ldg(st + kStOwnOff);
        omega = (update && omega_p != nullptr) ? __ldg(omega_p) : 1.0;
      }
      int ex;
      const float lm = log_row_sum_parts(sum, err, 0.0f, ex);
      rr = row_update(ex, lm, shift, b2s ? b2s[row] : 0.0f, mass[row], log_u[row] + own_off, residual, omega);
      if (update) {
        log_u[row] = rr.log_u;
        ell[row] = rr.ell;
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.freed[pb]);
    if (update) {
      // the block's rows (this CTA's rows blk * 32 .. blk * 32 + 31) form group blk * G + blockIdx.x
      const float4 gv = warp_group(rr.log_u, rr.ell, k < nrows);
      if (lane == 0) grp[blk * G + blockIdx.x] = gv;
    }
    add_partials(acc, row_partials(rr, k < nrows, residual));
  }
  if (update && ok && lane == 0) {
    // groups of the blocks this CTA does not have (the grid's rows are
    // dealt round-robin, so some CTAs have one block fewer) contribute nothing
    for (int64_t blk = (nrows + kSlots - 1) / kSlots; blk < grp_blocks; ++blk) grp[blk * G + blockIdx.x] = empty_group();
  }
  if (!ok && !*abort_flag) pass_abort(err, abort_flag);
  // this warp holds every partial of the CTA
  if (lane == 0) store_partials(partials + 4 * blockIdx.x, acc);
}

// One sweep from one pass over A-hat. The v step needs s_y = 1/2 sum_x A_xy u_x
// with the new u, and row x of A-hat is all that u_x needs: so while a row is
// in shared memory, its dot product with v gives u_x, and the row scaled by u_x
// is added to the column sums. A-hat is read once per sweep instead of A-hat and
// its transpose (at 20,000 x 10,000 two passes of 800 MB took 2 x 120 us).
//
// Roles of a CTA (a cluster of `cl` CTAs shares every row when it is longer
// than kSweepWidth columns; each holds a slice of the columns):
//   producer warp   streams units of `rows` rows (one slice of a row in a
//                   cluster) into a ring in shared memory with bulk copies.
//   dot warps       every thread owns fixed columns, its part of v in registers;
//                   a row's dot product (compensated) is parked per warp.
//   update warp     (the cluster's first CTA) sums a unit's parked shares and
//                   hands the rows' weights 2^(ell log2 e - R) to the sum warps
//                   of the cluster, in FP32.
//   sum warps       every thread owns fixed columns, their sums (compensated) in
//                   registers: a unit is added once its weights are there, and
//                   its slot released.
//   row warp        (the cluster's first CTA) the rows' stored potentials in
//                   FP64, residual and groups, 32 rows at a time, off the path.
// A sweep of 20,000 x 10,000 takes 177 us (two passes: 268); rows in clusters,
// 30,000 x 30,000 649 us (1,101), 3,000 x 40,000 143 (206). With plain dot products
// and FP32 weights 20,000 x 10,000 took 149 (the pass at 6.5 TB/s, 0.96 of the
// measured copy rate): the compensation's three more operations per pair of terms
// are what bounds the pass now. Eight dot warps, of 736 threads with 80 registers: five took 220 us at
// 20,000 x 10,000, six 228, seven 211, ten 183. The shares and weights of a cluster travel
// by asynchronous stores; with plain remote stores and releasing arrivals its
// update warp took 1.5 us per row and the pass was slower than two.
// A row passes through load, dot, update and sum one after another, about
// 5,000 cycles; with one slot of the ring per row in flight the SM still takes
// one 40 KB row per 1,700 cycles, its share of HBM. (One set of warps doing
// both products in turn was the bound: 165 us per 800 MB pass.)
// A row's weight is that of its stored potential, rounded once: the FP32
// logarithms are those of row_update, and what FP32 rounds off their sum is kept
// (weight_pow2). The rms error of log v against float64 is then 0.93 of the two
// passes' over 27 heights and widths (0.64 to 1.32: the FP32 logarithm of a sum
// rounds by where in its binade the sum lies); with exp2f of an FP32 exponent
// its mean was off by up to 3e-8, where the two passes' is by 1e-8.
// R is an integer per cluster, raised when a row's exponent passes it by 40
// (weights up to 2^40 against A-hat up to e^40 stay in the FP32 range); the
// column sums so far are then rescaled by a power of two, exactly. At the end
// each CTA writes its column sums and R; k_dense_cols adds them up.
// A unit is at most 40 KB and the ring takes what shared memory there is.
// 2^d for any integer d, exactly, flushed to 0 below FP32's normal range and to infinity above it
__device__ __forceinline__ float exp2_whole(int d) {
  return d < -126 ? 0.0f : (d > 127 ? INFINITY : __int_as_float((127 + d) << 23));
}

// 2^(f + l), f in [-0.5, 0.5] and l a few units of f's last place, to half a
// unit: the series of e^x - 1 at x = (f + l) ln 2, |x| <= 0.35, up to x^8 / 8!,
// whose first term keeps its rounding.
__device__ __forceinline__ float weight_pow2(float f, float l) {
  const float kLn2 = 0.693147182464599609375f, kLn2Lo = -1.904654323e-9f;
  const float x = f * kLn2;
  const float xl = fmaf(f, kLn2, -x) + fmaf(f, kLn2Lo, l * kLn2);
  // (in pairs of terms: the update warp's chain is what the clusters wait for)
  const float x2 = x * x;
  const float q6 = fmaf(x2, 1.0f / 40320.0f, fmaf(x, 1.0f / 5040.0f, 1.0f / 720.0f));
  const float q0 = fmaf(x2, fmaf(x, 1.0f / 120.0f, 1.0f / 24.0f), fmaf(x, 1.0f / 6.0f, 0.5f));
  return 1.0f + (x + fmaf(x2, fmaf(x2 * x2, q6, q0), xl));
}

constexpr int kSweepWidth = 10240;  // columns of a slice, at most
constexpr int kSweepSums = 12;      // sum warps (28 columns per thread, at most)
constexpr int kSweepDots = 8;       // dot warps (40 columns per thread, at most)
constexpr int kSweepRows = 8;       // rows of a unit, at most
constexpr int kSweepSlots = 24;     // ring slots, at most
constexpr int kSweepCl = 8;         // cluster size, at most
constexpr int kSweepUpdate = kSweepSums + kSweepDots;  // the update warp
constexpr int kSweepProducer = kSweepUpdate + 1;       // the producer warp; then the row warp
constexpr int kSweepThreads = (kSweepUpdate + 3) * 32;
constexpr int kSweepMinCols = 512;  // fewer columns leave most threads without work

// Packed pairs of floats, and four floats as two of them.
struct __align__(16) Quad {
  uint64_t x, y;
};
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  return ((uint64_t)__float_as_uint(b) << 32) | __float_as_uint(a);
}
__device__ __forceinline__ float low2(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float high2(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// s += n; what the addition rounds off stays in n
__device__ __forceinline__ void carry2(uint64_t& s, uint64_t& n) {
  const uint64_t t = add2(s, n);
  n = sub2(n, sub2(t, s));
  s = t;
}
// kahan_fma on pairs; n is the compensation with its sign turned
__device__ __forceinline__ void kahan_fma2(uint64_t& s, uint64_t& n, uint64_t x, uint64_t w) {
  n = fma2(x, w, n);
  carry2(s, n);
}

struct SweepSmem {
  // per slot of the ring: a unit's parked shares (the cluster's first CTA; a
  // cluster's units are one row), its rows' weights, the factor that the column
  // sums so far take before them (in a cluster: beside the one weight)
  float part[kSweepSlots][kSweepRows][kSweepDots];
  float weight[kSweepSlots][kSweepRows];
  float scale[kSweepSlots];
  float4 row[2][32];            // a batch's rows: constants of their updates, see row warp
  float4 frac[2][32];
  float2 sum[2][32];            // and their sums (hi, lo)
  uint64_t full[kSweepSlots];   // a unit has landed
  uint64_t empty[kSweepSlots];  // every sum warp is done with it
  uint64_t done[kSweepSlots];   // its shares are parked
  uint64_t ready[kSweepSlots];  // its weights are here
  uint64_t ahead[2];            // a batch's constants are here
  uint64_t summed[2];           // a batch's sums are here
  int abort;
};
static_assert(kSweepRows >= kSweepCl, "a cluster's shares of one row use the unit's rows");
constexpr size_t kSweepRing = (sizeof(SweepSmem) + 127) / 128 * 128;  // the ring's offset
constexpr size_t kSweepSmemMax = 232448;                              // shared memory of a CTA

struct SweepArgs {
  const float* A;
  int64_t ld, rows;
  const float* w;  // the partner vector exp(ell - shift), zero-padded
  const double* st;
  const float* b2s;
  const double* mass;
  double* log_u;
  double* ell;
  float4* grp;
  int64_t grp_units;  // groups per cluster
  double* partials;
  int residual;
  int* err;
  float* colsum;  // clusters x ld
  int* scale;     // R of each cluster
  DensePlan plan;
};

// NA, ND: groups of four columns per thread of the sum and of the dot warps
template <int NA, int ND, bool CLUSTER>
__global__ void __launch_bounds__(kSweepThreads, 1) k_dense_sweep(const SweepArgs a) {
  extern __shared__ __align__(128) uint8_t sweep_smem_raw[];
  SweepSmem& S = *reinterpret_cast<SweepSmem*>(sweep_smem_raw);
  float* ring = reinterpret_cast<float*>(sweep_smem_raw + kSweepRing);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  volatile int* abort_flag = &S.abort;
  const int cl = CLUSTER ? a.plan.cl : 1;
  const int rank = CLUSTER ? (int)cluster_rank() : 0;
  const int64_t P = a.plan.clusters;
  const int64_t cid = CLUSTER ? blockIdx.x / cl : blockIdx.x;
  const int B = CLUSTER ? 1 : a.plan.rows;
  const int slots = a.plan.slots;
  const int64_t c0 = (int64_t)rank * a.plan.width;
  const int width = (int)(a.ld - c0 < a.plan.width ? a.ld - c0 : a.plan.width);  // (never empty, see dense_plan)
  const int slot_floats = B * a.plan.width;
  const int64_t units = (a.rows + B - 1) / B;
  const int64_t nu = (units - cid + P - 1) / P;  // this cluster's units: cid, cid + P, ...
  if (threadIdx.x == 0) {
    for (int t = 0; t < slots; ++t) {
      mbar_init(&S.full[t], 1);
      mbar_init(&S.empty[t], kSweepSums);
      mbar_init(&S.done[t], CLUSTER ? 1 : kSweepDots);
      mbar_init(&S.ready[t], 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&S.ahead[t], 1);
      mbar_init(&S.summed[t], 1);
    }
    S.abort = 0;
    fence_mbar_init();
  }
  if constexpr (CLUSTER) {
    cluster_sync();
  } else {
    __syncthreads();
  }

  if (warp == kSweepProducer) {
    // ---------------------------------------------------------- producer
    if (lane == 0) {
      int t = 0;
      uint32_t ph = 0, issued = 0, issued_ph = 0;
      bool ok = true;
      for (int64_t k = 0; k < nu; ++k) {
        if (!mbar_wait(&S.empty[t], ph ^ 1u, abort_flag)) {
          ok = false;
          break;
        }
        const int64_t r0 = (cid + k * P) * B;
        const int nb = (int)(a.rows - r0 < B ? a.rows - r0 : B);
        // (outside a cluster a unit's rows are one run of memory)
        const uint32_t bytes = (uint32_t)(CLUSTER ? width : nb * width) * 4u;
        if constexpr (CLUSTER) {
          // what the unit's barriers will count: the weight and scale, and in the
          // first CTA every dot warp's share (both sent by asynchronous stores)
          mbar_arrive_expect_tx(&S.ready[t], 8u);
          if (rank == 0) mbar_arrive_expect_tx(&S.done[t], (uint32_t)(4 * kSweepDots * cl));
        }
        mbar_arrive_expect_tx(&S.full[t], bytes);
        bulk_copy(ring + (size_t)t * slot_floats, a.A + r0 * a.ld + c0, bytes, &S.full[t]);
        issued |= 1u << t;
        issued_ph = (issued_ph & ~(1u << t)) | (ph << t);
        if (++t == slots) {
          t = 0;
          ph ^= 1u;
        }
      }
      if (!ok && !*abort_flag) pass_abort(a.err, abort_flag);
      // copies in flight complete before the CTA's shared memory is released
      for (int u = 0; u < slots; ++u)
        if (issued & (1u << u)) mbar_wait_drain(&S.full[u], (issued_ph >> u) & 1u, 100000000ull);
    }
    __syncwarp();
  } else if (warp < kSweepSums) {
    // ---------------------------------------------------------- sum warps
    constexpr int kStep = kSweepSums * 32;
    const int nq = width / 4;
    Quad s[NA], e[NA];  // the column sums and their compensations
#pragma unroll
    for (int j = 0; j < NA; ++j) s[j] = e[j] = Quad{0ull, 0ull};
    int t = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int64_t k = 0; k < nu; ++k) {
      if (!__all_sync(0xffffffffu, mbar_wait(&S.ready[t], ph, abort_flag))) {
        ok = false;
        break;
      }
      // (the copy's own writes are made visible by its barrier)
      if (!__all_sync(0xffffffffu, mbar_wait(&S.full[t], ph, abort_flag))) {
        ok = false;
        break;
      }
      const float sc = *reinterpret_cast<volatile float*>(CLUSTER ? &S.weight[t][1] : &S.scale[t]);
      if (sc != 1.0f) {
        const uint64_t sc2 = pack2(sc, sc);
#pragma unroll
        for (int j = 0; j < NA; ++j) {
          s[j] = Quad{mul2(s[j].x, sc2), mul2(s[j].y, sc2)};
          e[j] = Quad{mul2(e[j].x, sc2), mul2(e[j].y, sc2)};
        }
      }
      const int64_t r0 = (cid + k * P) * B;
      const int nb = (int)(a.rows - r0 < B ? a.rows - r0 : B);
      const Quad* r4 = reinterpret_cast<const Quad*>(ring + (size_t)t * slot_floats) + threadIdx.x;
      for (int b = 0; b < nb; ++b, r4 += nq) {
        const float u = *reinterpret_cast<volatile float*>(&S.weight[t][b]);
        const uint64_t uu = pack2(u, u);
#pragma unroll
        for (int j = 0; j < NA; ++j) {
          if ((int)threadIdx.x + j * kStep < nq) {
            const Quad x = r4[j * kStep];
            kahan_fma2(s[j].x, e[j].x, x.x, uu);
            kahan_fma2(s[j].y, e[j].y, x.y, uu);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.empty[t]);
      if (++t == slots) {
        t = 0;
        ph ^= 1u;
      }
    }
    if (ok) {
      Quad* out = reinterpret_cast<Quad*>(a.colsum + cid * a.ld + c0) + threadIdx.x;
#pragma unroll
      for (int j = 0; j < NA; ++j)
        if ((int)threadIdx.x + j * kStep < nq) out[j * kStep] = Quad{add2(s[j].x, e[j].x), add2(s[j].y, e[j].y)};
    } else if (!*abort_flag) {
      pass_abort(a.err, abort_flag);
    }
  } else if (warp < kSweepUpdate) {
    // ---------------------------------------------------------- dot warps
    constexpr int kStep = kSweepDots * 32;
    const int dw = warp - kSweepSums, tid = dw * 32 + lane;
    const int nq = width / 4;
    const Quad* w4 = reinterpret_cast<const Quad*>(a.w + c0) + tid;
    Quad w[ND];  // this thread's part of v
#pragma unroll
    for (int j = 0; j < ND; ++j) w[j] = tid + j * kStep < nq ? w4[j * kStep] : Quad{0ull, 0ull};
    int t = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int64_t k = 0; k < nu; ++k) {
      if (!__all_sync(0xffffffffu, mbar_wait(&S.full[t], ph, abort_flag))) {
        ok = false;
        break;
      }
      const int64_t r0 = (cid + k * P) * B;
      const int nb = (int)(a.rows - r0 < B ? a.rows - r0 : B);
      const Quad* r4 = reinterpret_cast<const Quad*>(ring + (size_t)t * slot_floats) + tid;
      for (int b = 0; b < nb; ++b, r4 += nq) {
        // four compensated sums per thread, as in the row pass (carry2 outside the
        // test: without a column it adds the compensation alone)
        uint64_t d0 = 0ull, d1 = 0ull, n0 = 0ull, n1 = 0ull;
#pragma unroll
        for (int j = 0; j < ND; ++j) {
          if (tid + j * kStep < nq) {
            const Quad x = r4[j * kStep];
            n0 = fma2(x.x, w[j].x, n0);
            n1 = fma2(x.y, w[j].y, n1);
          }
          carry2(d0, n0);
          carry2(d1, n1);
        }
        d0 = add2(add2(d0, n0), add2(d1, n1));
        float r = low2(d0) + high2(d0);
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (lane == 0) {
          if constexpr (CLUSTER) {
            cluster_store_async(cluster_addr(&S.part[t][rank][dw], 0), r, cluster_addr(&S.done[t], 0));
          } else {
            S.part[t][b][dw] = r;
          }
        }
      }
      if (!CLUSTER && lane == 0) mbar_arrive(&S.done[t]);
      __syncwarp();
      if (++t == slots) {
        t = 0;
        ph ^= 1u;
      }
    }
    if (!ok && !*abort_flag) pass_abort(a.err, abort_flag);
  } else if (warp == kSweepUpdate) {
    // ---------------------------------------------------------- update warp
    if (rank == 0) {
      // (A cluster's units are single rows, and this warp's chain of about 2,000
      // cycles per turn is what it waits for: with slots to spare the half-warps
      // take a unit each, 30,000 x 30,000 in 7 slots 891 -> 649 us per sweep. With
      // 5 slots two units at a time leave too few loads in flight, 3,000 x 40,000
      // 143 -> 167.)
      int R = 0, pb = 0;
      uint32_t dph = 0;
      bool ok = true;
      auto update = [&](auto units) {
        constexpr int U = decltype(units)::value, L = 32 / U;  // units at a time, lanes per unit
        const int half = lane / L, hl = lane % L;
        for (int64_t k = 0; k < nu; k += U) {
          const bool here = k + half < nu;  // (this half-warp has a unit)
          const int sl = pb + half < slots ? pb + half : pb + half - slots;
          const uint32_t sph = pb + half < slots ? dph : dph ^ 1u;
          const int64_t r0 = (cid + (k + half) * P) * B;
          const int nb = !here ? 0 : (int)(a.rows - r0 < B ? a.rows - r0 : B);
          const bool mine = hl < nb;
          const int64_t batch = k * B / 32;
          const int at = (int)(k * B % 32) + half + (mine ? hl : 0);  // this row in its batch
          const int bb = (int)(batch & 1);
          bool got = k * B % 32 != 0 || mbar_wait(&S.ahead[bb], (uint32_t)(batch >> 1) & 1u, abort_flag);
          if (here) got = got && mbar_wait(&S.done[sl], sph, abort_flag);
          if (!__all_sync(0xffffffffu, got)) {
            ok = false;
            break;
          }
          const float4 cst = S.row[bb][at], frc = S.frac[bb][at];
          // the warps' shares of a row, added with their roundings kept
          float hi = 0.0f, lo = 0.0f;
          if constexpr (CLUSTER) {
            const volatile float* p = S.part[sl][0];
            for (int i = hl; i < kSweepDots * cl; i += L) pair_add(hi, lo, p[i], 0.0f);
            for (int o = L / 2; o > 0; o >>= 1)
              pair_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o));
          } else {
            const volatile float* p = S.part[pb][mine ? lane : 0];
#pragma unroll
            for (int i = 0; i < kSweepDots; ++i) pair_add(hi, lo, p[i], 0.0f);
          }
          // The row's weight u 2^-R in FP32 from row_update's closed form, z = log s -
          // 1/2 log n and the logarithms with its values; log2 u is an integer plus a
          // fraction in two floats, so that no digits go to its size.
          // (log_row_sum_parts without its third part, which is 0)
          int ex;
          float rest;
          const float total = two_sum(hi, lo, rest);
          const float lm = __fadd_rn(logf(frexpf(total, &ex)), __fdividef(rest, total));
          const float z = fmaf((float)(__float_as_int(cst.x) + ex), 0.69314718056f, cst.y + lm);
          int n;
          float v, ve = 0.0f, f, l;  // the logarithm to take off (natural, two floats), and from what (log2)
          if (z > 0.0f) {
            v = two_sum(lm, log1pf(sqrtf(1.0f + expf(-2.0f * z))), ve);
            n = __float_as_int(cst.z) - ex;
            f = frc.x;
            l = frc.y;
          } else {
            v = asinhf(expf(z));
            n = __float_as_int(cst.w);
            f = frc.z;
            l = frc.w;
          }
          const float kLog2eLo = 1.925962989e-8f, pr = v * kLog2e;  // (kLog2e + kLog2eLo is log2 e)
          float fe;
          f = two_sum(f, -pr, fe);
          l += fe - (fmaf(v, kLog2e, -pr) + fmaf(ve, kLog2e, v * kLog2eLo));
          // (a sum that is not finite: 0 for an infinite one, else not a number)
          const bool fin = v < INFINITY;
          const float whole = fin ? rintf(f) : 0.0f;
          n += (int)whole;
          const float frac_u = fin ? weight_pow2(f - whole, l) : (v > 0.0f ? 0.0f : v);
          // what the column sums so far take before each unit, and the units' scale
          float sc = 1.0f;
          int scale_here = R;
          for (int h = 0; h < U && k + h < nu; ++h) {
            const int top = CLUSTER ? __shfl_sync(0xffffffffu, n, h * L) : __reduce_max_sync(0xffffffffu, mine ? n : -0x40000000);
            float s1 = 1.0f;
            if (k + h == 0 || top > R + 40) {
              if (k + h > 0) s1 = exp2_whole(R - top);
              R = top;
            }
            if (half == h) {
              sc = s1;
              scale_here = R;
            }
          }
          const float u = frac_u * exp2_whole(n - scale_here);
          if constexpr (CLUSTER) {
            const float u0 = __shfl_sync(0xffffffffu, u, half * L);
            if (here && hl < cl)
              cluster_store_async2(cluster_addr(&S.weight[sl][0], hl), u0, sc, cluster_addr(&S.ready[sl], hl));
          } else {
            if (mine) S.weight[pb][lane] = u;
            if (lane == 0) S.scale[pb] = sc;
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.ready[pb]);
          }
          if (mine) S.sum[bb][at] = make_float2(hi, lo);
          __syncwarp();
          if (lane == 0 && ((k + U) * B % 32 == 0 || k + U >= nu)) mbar_arrive(&S.summed[bb]);
          pb += U;
          if (pb >= slots) {
            pb -= slots;
            dph ^= 1u;
          }
        }
      };
      if constexpr (CLUSTER) {
        if (slots >= 7) update(std::integral_constant<int, 2>());
        else update(std::integral_constant<int, 1>());
      } else {
        update(std::integral_constant<int, 1>());
      }
      if (ok && lane == 0) a.scale[cid] = R;
      if (!ok && !*abort_flag) pass_abort(a.err, abort_flag);
    }
  } else if (rank == 0) {
    // ---------------------------------------------------------- row warp
    // Batches of 32 of the cluster's rows, one per lane: what the update warp
    // needs of them, a batch ahead; then, from their sums, the FP64 update of
    // the stored potentials, the residual and the batch's group. FP64 runs at a
    // few operations per clock and SM: a row's chain of it takes microseconds,
    // which the update warp cannot wait for.
    RowPartials acc = {0.0, 0.0, 0.0, 0.0};
    const double shift = a.st[kStShift], own_off = a.st[kStOwnOff];
    const int64_t last0 = (cid + (nu - 1) * P) * B;
    const int64_t nr = (nu - 1) * B + (a.rows - last0 < B ? a.rows - last0 : B);  // this cluster's rows
    const int64_t batches = (nr + 31) / 32;
    auto row_of = [&](int64_t i) { return (cid + i / B * P) * B + i % B; };
    auto ahead = [&](int64_t j) {
      const int64_t i = j * 32 + lane;
      if (i < nr) {
        const int64_t row = row_of(i);
        const double b = a.b2s != nullptr ? (double)a.b2s[row] : 0.0;
        const double hl = 0.5 * (double)logf((float)a.mass[row]);
        // z is c2 plus the sum's logarithm; log u + b is d2 less that and log1p's
        // (z > 0), or b2 less asinh's: in log2 units, as an integer and a fraction
        const double c2 = ((kLnHalf + b + shift) - hl) * 1.4426950408889634, b2 = (hl + b) * 1.4426950408889634;
        const double d2 = b2 - c2, cn = rint(c2), bn = rint(b2), dn = rint(d2);
        const float df = (float)(d2 - dn), bf = (float)(b2 - bn);
        S.row[j & 1][lane] = make_float4(__int_as_float((int)cn), (float)((c2 - cn) * 0.69314718055994530942),
                                         __int_as_float((int)dn), __int_as_float((int)bn));
        S.frac[j & 1][lane] = make_float4(df, (float)((d2 - dn) - (double)df), bf, (float)((b2 - bn) - (double)bf));
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.ahead[j & 1]);
    };
    bool ok = true;
    ahead(0);
    for (int64_t j = 0; j < batches; ++j) {
      if (j + 1 < batches) ahead(j + 1);  // (its buffers: batch j - 1 is done)
      const bool got = mbar_wait(&S.summed[j & 1], (uint32_t)(j >> 1) & 1u, abort_flag, 2 * kWaitLimitNs);
      if (!__all_sync(0xffffffffu, got)) {
        ok = false;
        break;
      }
      const int64_t i = j * 32 + lane;
      const bool valid = i < nr;
      RowResult rr{};
      if (valid) {
        const int64_t row = row_of(i);
        const volatile float2* s2 = &S.sum[j & 1][lane];
        int ex;
        const float lm = log_row_sum_parts(s2->x, s2->y, 0.0f, ex);
        rr = row_update(ex, lm, shift, a.b2s != nullptr ? a.b2s[row] : 0.0f, a.mass[row], a.log_u[row] + own_off,
                        a.residual);
        a.log_u[row] = rr.log_u;
        a.ell[row] = rr.ell;
      }
      add_partials(acc, row_partials(rr, valid, a.residual));
      const float4 gv = warp_group(rr.log_u, rr.ell, valid);
      if (lane == 0) a.grp[j * P + cid] = gv;
    }
    if (ok && lane == 0)
      for (int64_t j = batches; j < a.grp_units; ++j) a.grp[j * P + cid] = empty_group();
    if (!ok && !*abort_flag) pass_abort(a.err, abort_flag);
    if (lane == 0) store_partials(a.partials + 4 * cid, acc);
  }
  // no CTA of a cluster leaves while another may still write to its shared memory
  // (the asynchronous stores of a pass that ends as it should have been counted by
  // then; after an abort they get longer than any takes to land)
  if constexpr (CLUSTER) {
    cluster_sync();
    if (*abort_flag) {
      const uint64_t t0 = global_timer_ns();
      while (global_timer_ns() - t0 < 10000000ull) {
      }
    }
  }
}

// The Y update from the clusters' column sums: 32 columns per block, the
// clusters dealt to kColSegs threads per column, each sum kept with its
// roundings and added in a fixed order.
constexpr int kColSegs = 16;

__global__ void __launch_bounds__(32 * kColSegs) k_dense_cols(const float* __restrict__ colsum,
                                                             const int* __restrict__ scale, int64_t ld, int clusters,
                                                             int64_t cols, const double* __restrict__ st,
                                                             const float* __restrict__ b2s,
                                                             const double* __restrict__ mass,
                                                             double* __restrict__ log_u, double* __restrict__ ell,
                                                             float4* __restrict__ grp, double* __restrict__ partials) {
  __shared__ float2 seg[kColSegs][32];
  __shared__ int top[kColSegs];
  const int lane = threadIdx.x % 32, sg = threadIdx.x / 32;
  const int64_t c = (int64_t)blockIdx.x * 32 + lane;
  int R = -0x40000000;
  for (int p = threadIdx.x; p < clusters; p += 32 * kColSegs) R = max(R, __ldg(scale + p));
  R = __reduce_max_sync(0xffffffffu, R);
  if (lane == 0) top[sg] = R;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kColSegs; ++i) R = max(R, top[i]);
  float hi = 0.0f, lo = 0.0f;
  if (c < cols)
#pragma unroll 4
    for (int p = sg; p < clusters; p += kColSegs)
      pair_add(hi, lo, __ldg(colsum + p * ld + c) * exp2_whole(__ldg(scale + p) - R), 0.0f);
  seg[sg][lane] = make_float2(hi, lo);
  __syncthreads();
  if (sg != 0) return;
  for (int i = 1; i < kColSegs; ++i) pair_add(hi, lo, seg[i][lane].x, seg[i][lane].y);
  RowResult rr{};
  if (c < cols) {
    // the rows' weights are relative to R instead of the side's shift: the
    // pass's shift without the shift, plus R ln 2
    const double shift = st[kStShift] - st[kStLmax + 0];
    int ex;
    const float lm = log_row_sum_parts(hi, lo, 0.0f, ex);
    rr = row_update(ex + R, lm, shift, b2s != nullptr ? b2s[c] : 0.0f, mass[c], log_u[c] + st[kStOwnOff],
                    kResidualNone);
    log_u[c] = rr.log_u;
    ell[c] = rr.ell;
  }
  const float4 gv = warp_group(rr.log_u, rr.ell, c < cols);
  const RowPartials p = row_partials(rr, c < cols, kResidualNone);
  if (lane == 0) {
    grp[blockIdx.x] = gv;
    store_partials(partials + 4 * blockIdx.x, p);
  }
}

// The instantiation for a slice width.
typedef void (*SweepKernel)(SweepArgs);
template <bool CLUSTER>
SweepKernel sweep_kernel_for(int width) {
  const int na = (width / 4 + kSweepSums * 32 - 1) / (kSweepSums * 32);
  if (na <= 1) return k_dense_sweep<1, 2, CLUSTER>;
  if (na == 2) return k_dense_sweep<2, 3, CLUSTER>;
  if (na == 3) return k_dense_sweep<3, 5, CLUSTER>;
  if (na == 4) return k_dense_sweep<4, 6, CLUSTER>;
  if (na == 5) return k_dense_sweep<5, 8, CLUSTER>;
  if (na == 6) return k_dense_sweep<6, 9, CLUSTER>;
  return k_dense_sweep<7, 10, CLUSTER>;
}
// (a slice of up to na * 1,536 columns needs na * 1.5 quads per dot thread, the longest 10)
static_assert(7 * kSweepSums * 128 >= kSweepWidth && 10 * kSweepDots * 128 >= kSweepWidth, "columns per thread");
static_assert(kSweepDots * 2 >= kSweepSums && kSweepDots * 3 >= kSweepSums * 2 && kSweepDots * 5 >= kSweepSums * 3 &&
                  kSweepDots * 6 >= kSweepSums * 4 && kSweepDots * 8 >= kSweepSums * 5 &&
                  kSweepDots * 9 >= kSweepSums * 6,
              "columns per thread");
SweepKernel sweep_kernel(const DensePlan& p) {
  return p.cl > 1 ? sweep_kernel_for<true>(p.width) : sweep_kernel_for<false>(p.width);
}
size_t sweep_smem(const DensePlan& p) { return kSweepRing + (size_t)p.slots * p.rows * p.width * 4; }

cudaError_t sweep_attributes(const DensePlan& p) {
  return cudaFuncSetAttribute(sweep_kernel(p), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSweepSmemMax);
}

cudaLaunchConfig_t sweep_config(const DensePlan& p, cudaLaunchAttribute* attr, cudaStream_t stream) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)(p.clusters * p.cl));
  c.blockDim = dim3(kSweepThreads);
  c.dynamicSmemBytes = sweep_smem(p);
  c.stream = stream;
  if (p.cl > 1) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)p.cl;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    c.attrs = attr;
    c.numAttrs = 1;
  }
  return c;
}

// CTAs of a pass: as many as fit on the device at once (the ring's shared
// memory allows a few per SM), at most one per row.
int rowpass_grid(tu_market* m, int64_t rows) {
  static int per_sm = 0;
  if (per_sm == 0) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_dense_rowpass<false>, kPassThreads,
                                                      sizeof(PassSmem)) != cudaSuccess ||
        b < 1) {
      cudaGetLastError();
      b = 1;
    }
    per_sm = b;
  }
  int64_t g = (int64_t)m->num_sms * per_sm;
  if (g > rows) g = rows;
  if (g > kMaxPartials) g = kMaxPartials;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t launch_dense_build(tu_market* m) {
  // the row pass's ring exceeds the default 48 KB of dynamic shared memory
  // (set here, at creation and factor updates, never inside a graph capture)
  cudaError_t e = cudaFuncSetAttribute(k_dense_rowpass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(PassSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_dense_rowpass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(PassSmem));
  if (e == cudaSuccess && m->dplan.cl > 0) e = sweep_attributes(m->dplan);
  if (e != cudaSuccess) return e;
  const int64_t row_tiles = (m->N + 63) / 64;
  dim3 grid((unsigned)((m->M + 63) / 64), (unsigned)(row_tiles < 65535 ? row_tiles : 65535));
  k_dense_build<<<grid, kThreads, 0, m->stream>>>(m->X.fac32, m->Y.fac32, m->N, m->M, m->kp,
                                                  (float)(0.5 / m->sigma), m->Ahat, m->ldA, m->AhatT, m->ldN);
  return cudaGetLastError();
}

cudaError_t launch_dense_rowpass(tu_market* m, int residual, int update, int* nparts_out, int64_t* ngroups_out) {
  const int g = rowpass_grid(m, m->N);
  const int64_t blocks = ((m->N + g - 1) / g + kSlots - 1) / kSlots;  // update blocks of the fullest CTA
  auto kern = m->omega_cfg != 1.0 ? k_dense_rowpass<true> : k_dense_rowpass<false>;
  kern<<<g, kPassThreads, sizeof(PassSmem), m->stream>>>(m->Ahat, m->ldA, m->N, m->Y.pvec, m->st, m->X.b2s,
                                                         m->X.mass, m->X.log_u, m->X.ell, m->X.grp, blocks,
                                                         m->partials, residual, update, m->omega_dev, m->err_dev);
  *nparts_out = g;
  *ngroups_out = blocks * g;
  return cudaGetLastError();
}

cudaError_t launch_dense_colpass(tu_market* m, int update, int* nparts_out, int64_t* ngroups_out) {
  const int g = rowpass_grid(m, m->M);
  const int64_t blocks = ((m->M + g - 1) / g + kSlots - 1) / kSlots;
  auto kern = m->omega_cfg != 1.0 ? k_dense_rowpass<true> : k_dense_rowpass<false>;
  kern<<<g, kPassThreads, sizeof(PassSmem), m->stream>>>(m->AhatT, m->ldN, m->M, m->X.pvec, m->st, m->Y.b2s,
                                                         m->Y.mass, m->Y.log_u, m->Y.ell, m->Y.grp, blocks,
                                                         m->partials, 0, update, m->omega_dev, m->err_dev);
  *nparts_out = g;
  *ngroups_out = blocks * g;
  return cudaGetLastError();
}

// The layout of a market's one-pass sweep. Markets with very short rows, or
// rows longer than a cluster holds, take the two passes.
DensePlan dense_plan(const tu_market* m) {
  DensePlan p;
  if (m->M < kSweepMinCols || m->N < kSweepMinCols || m->ldA > (int64_t)kSweepCl * kSweepWidth) return p;
  int cl = 1;
  while ((int64_t)cl * kSweepWidth < m->ldA) cl *= 2;
  p.width = (int)(((m->ldA + cl - 1) / cl + 3) / 4 * 4);
  p.rows = 1;
  while (cl == 1 && 2 * p.rows <= kSweepRows && 2 * p.rows * p.width <= kSweepWidth) p.rows *= 2;
  const size_t fit = (kSweepSmemMax - kSweepRing) / ((size_t)p.rows * p.width * 4);
  p.slots = (int)(fit < (size_t)kSweepSlots ? fit : (size_t)kSweepSlots);
  p.cl = cl;
  p.clusters = m->num_sms / cl;
  if (cl > 1) {
    // clusters that fit on the device at once
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t c = sweep_config(p, &attr, nullptr);
    int n = 0;
    if (sweep_attributes(p) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, sweep_kernel(p), &c) != cudaSuccess ||
        n < 1) {
      cudaGetLastError();
      return DensePlan();
    }
    if (n < p.clusters) p.clusters = n;
  }
  const int64_t units = (m->N + p.rows - 1) / p.rows;
  if (units < p.clusters) p.clusters = (int)units;
  return p;
}

size_t dense_plan_floats(const DensePlan& p) {
  return (size_t)p.clusters * ((size_t)p.cl * p.width) + (size_t)p.clusters;
}

cudaError_t launch_dense_sweep(tu_market* m, int residual, int* nparts_out, int64_t* ngroups_out) {
  const DensePlan& p = m->dplan;
  SweepArgs a;
  a.A = m->Ahat;
  a.ld = m->ldA;
  a.rows = m->N;
  a.w = m->Y.pvec;
  a.st = m->st;
  a.b2s = m->X.b2s;
  a.mass = m->X.mass;
  a.log_u = m->X.log_u;
  a.ell = m->X.ell;
  a.grp = m->X.grp;
  const int64_t units = (m->N + p.rows - 1) / p.rows;
  const int64_t most = (units + p.clusters - 1) / p.clusters;  // units of the fullest cluster
  a.grp_units = (most * p.rows + kGroupRows - 1) / kGroupRows;
  a.partials = m->partials;
  a.residual = residual;
  a.err = m->err_dev;
  a.colsum = m->colsum;
  a.scale = reinterpret_cast<int*>(m->colsum + (size_t)p.clusters * m->ldA);
  a.plan = p;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t c = sweep_config(p, &attr, m->stream);
  *nparts_out = p.clusters;
  *ngroups_out = a.grp_units * p.clusters;
  return cudaLaunchKernelEx(&c, sweep_kernel(p), a);
}

cudaError_t launch_dense_cols(tu_market* m, int* nparts_out, int64_t* ngroups_out) {
  const DensePlan& p = m->dplan;
  const int blocks = (int)((m->M + 31) / 32);
  k_dense_cols<<<blocks, 32 * kColSegs, 0, m->stream>>>(
      m->colsum, reinterpret_cast<const int*>(m->colsum + (size_t)p.clusters * m->ldA), m->ldA, p.clusters, m->M, m->st,
      m->Y.b2s, m->Y.mass, m->Y.log_u, m->Y.ell, m->Y.grp, m->partials);
  *nparts_out = blocks;
  *ngroups_out = blocks;
  return cudaGetLastError();
}

}  // namespace tu
