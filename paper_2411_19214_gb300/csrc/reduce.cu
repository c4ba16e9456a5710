// reduce.cu -- O(N + M) kernels around the half-sweeps: factor packing, side
// initialisation, the partner-potential preparation that precedes every
// half-sweep, and the FP64 reductions that close it.
#include "tu_internal.cuh"

#include <cuda_fp8.h>

namespace tu {

namespace {

constexpr int kThreads = 256;

__global__ void k_pack_factors(const void* __restrict__ A, const void* __restrict__ B, int src_dtype,
                               int64_t rows, int64_t d, int64_t kp, __nv_bfloat16* __restrict__ out16,
                               float* __restrict__ out32) {
  // [A | B | 0] packed row-major rows x kp: the inner product of two packed rows
  // is <f_x, g_y> + <k_x, l_y> (Sec. 3.3), i.e. Phi = [F | K] [G | L]^T.
  const int64_t total = rows * kp;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / kp;
    const int64_t k = i - r * kp;
    float v = 0.0f;
    const void* src = nullptr;
    int64_t off = 0;
    if (k < d) {
      src = A;
      off = r * d + k;
    } else if (k < 2 * d) {
      src = B;
      off = r * d + (k - d);
    }
    if (src != nullptr) {
      if (src_dtype == TU_DTYPE_BF16) {
        v = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(src)[off]);
      } else {
        v = reinterpret_cast<const float*>(src)[off];
      }
    }
    if (out16 != nullptr) out16[i] = __float2bfloat16_rn(v);
    if (out32 != nullptr) out32[i] = v;
  }
}

// Largest |entry| of two FP32 arrays of `count` entries each (non-negative
// floats order like their bit patterns, so an unsigned atomicMax is exact).
__global__ void k_max_abs(const float* __restrict__ A, const float* __restrict__ B, int64_t count,
                          unsigned int* __restrict__ out) {
  __shared__ float red[kThreads / 32];
  float best = 0.0f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const float a = fmaxf(fabsf(A[i]), fabsf(B[i]));
    // fmaxf drops a NaN operand: a NaN entry counts as +inf, so the host's finiteness check sees it
    best = (isnan(A[i]) || isnan(B[i])) ? INFINITY : fmaxf(best, a);
  }
  for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    float b = 0.0f;
    for (int w = 0; w < kThreads / 32; ++w) b = fmaxf(b, red[w]);
    atomicMax(out, __float_as_uint(b));
  }
}

// FP8 packing with per-row scales (one warp per row): row r of the output is
// [A_r | B_r | 0] * 2^-k_r rounded to the nearest e4m3 value (ties to even,
// saturating at +-448), kp bytes, with k_r the smallest integer such that
// max_i |entry| <= 448 * 2^k_r (exact: 448 = 0.875 * 2^9 and frexpf is exact),
// and fs[r] = 2^k_r the scale that multiplies the row back; an all-zero row
// has k_r = 0. With side_k != kPerRowScale every row takes k_r = side_k (one
// scale per side). Rows [rows, rows_pad) get fs = 1. A NaN or infinite entry
// sets *bad.
__global__ void k_pack_fp8_rows(const float* __restrict__ A, const float* __restrict__ B, int64_t rows,
                                int64_t rows_pad, int64_t d, int64_t kp, int side_k, uint8_t* __restrict__ out,
                                float* __restrict__ fs, unsigned int* __restrict__ bad) {
  const int lane = threadIdx.x % 32;
  const int64_t wpb = blockDim.x / 32;
  for (int64_t r = blockIdx.x * wpb + threadIdx.x / 32; r < rows_pad; r += (int64_t)gridDim.x * wpb) {
    if (r >= rows) {
      if (lane == 0) fs[r] = 1.0f;
      continue;
    }
    float mx = 0.0f;
    bool nonfinite = false;
    for (int64_t i = lane; i < 2 * d; i += 32) {
      const float v = i < d ? A[r * d + i] : B[r * d + (i - d)];
      nonfinite |= !isfinite(v);
      mx = fmaxf(mx, fabsf(v));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (__any_sync(0xffffffffu, nonfinite)) {
      if (lane == 0) atomicOr(bad, 1u);
      continue;
    }
    int k = side_k;
    if (side_k == kPerRowScale && mx > 0.0f) {
      int e = 0;
      frexpf(mx, &e);
      k = mx <= ldexpf(448.0f, e - 9) ? e - 9 : e - 8;
      if (k < -100) k = -100;  // (rows of subnormal size: 2^100 keeps the scaled entries finite)
    } else if (side_k == kPerRowScale) {
      k = 0;
    }
    const float inv = ldexpf(1.0f, -k);
    if (lane == 0) fs[r] = ldexpf(1.0f, k);
    for (int64_t i = lane; i < kp; i += 32) {
      float v = 0.0f;
      if (i < d) {
        v = A[r * d + i];
      } else if (i < 2 * d) {
        v = B[r * d + (i - d)];
      }
      out[r * kp + i] = (uint8_t)__nv_cvt_float_to_fp8(v * inv, __NV_SATFINITE, __NV_E4M3);
    }
  }
}

// FP8 packing of caller-quantized rows: [A_r | B_r | 0] copied as bytes (kp
// per row), fs[r] = sc[r]; rows [rows, rows_pad) get fs = 1. A non-finite
// scale sets *bad.
__global__ void k_pack_fp8_bytes(const uint8_t* __restrict__ A, const uint8_t* __restrict__ B,
                                 const float* __restrict__ sc, int64_t rows, int64_t rows_pad, int64_t d, int64_t kp,
                                 uint8_t* __restrict__ out, float* __restrict__ fs, unsigned int* __restrict__ bad) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows * kp;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / kp;
    const int64_t k = i - r * kp;
    uint8_t v = 0;
    if (k < d) {
      v = A[r * d + k];
    } else if (k < 2 * d) {
      v = B[r * d + (k - d)];
    }
    out[i] = v;
  }
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < rows_pad;
       r += (int64_t)gridDim.x * blockDim.x) {
    const float v = r < rows ? sc[r] : 1.0f;
    if (!isfinite(v)) atomicOr(bad, 1u);
    fs[r] = v;
  }
}

__global__ void k_init_side(const float* __restrict__ bias, int has_bias, float inv2s, int64_t rows,
                            int64_t rows_pad, float* __restrict__ b2s, double* __restrict__ log_u,
                            double* __restrict__ ell, double* __restrict__ mass) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows_pad;
       i += (int64_t)gridDim.x * blockDim.x) {
    float b = 0.0f;
    if (has_bias && i < rows) b = (float)((double)bias[i] * (double)inv2s);
    if (b2s != nullptr) b2s[i] = b;
    log_u[i] = 0.0;  // u = 1 (Alg. 1 / Alg. 2 initialisation)
    ell[i] = (i < rows) ? (double)b : 0.0;
    if (i >= rows) mass[i] = 1.0;  // padding capacities: padded rows never produce log(0)
  }
}

__global__ void k_set_potentials(const float* __restrict__ src, const float* __restrict__ b2s, int64_t rows,
                                 double* __restrict__ log_u, double* __restrict__ ell) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double lu = (double)src[i];
    log_u[i] = lu;
    ell[i] = (b2s != nullptr) ? lu + (double)b2s[i] : lu;
  }
}

__global__ void k_set_potentials64(const double* __restrict__ src, const float* __restrict__ b2s, int64_t rows,
                                   double* __restrict__ log_u, double* __restrict__ ell) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double lu = src[i];
    log_u[i] = lu;
    ell[i] = (b2s != nullptr) ? lu + (double)b2s[i] : lu;
  }
}

// FP32 copies of the potentials (either output may be null)
__global__ void k_get_potentials(const double* __restrict__ lu, int64_t nx, float* __restrict__ out_x,
                                 const double* __restrict__ lv, int64_t ny, float* __restrict__ out_y) {
  const int64_t n = nx > ny ? nx : ny;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (out_x != nullptr && i < nx) out_x[i] = (float)lu[i];
    if (out_y != nullptr && i < ny) out_y[i] = (float)lv[i];
  }
}

__global__ void k_row_norm_max(const float* __restrict__ f32, const __nv_bfloat16* __restrict__ f16,
                               const uint8_t* __restrict__ f8, const float* __restrict__ fs, int64_t rows,
                               int64_t kp, unsigned int* __restrict__ out) {
  __shared__ float red[kThreads / 32];
  float best = 0.0f;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int64_t r = blockIdx.x * (int64_t)(kThreads / 32) + warp; r < rows;
       r += (int64_t)gridDim.x * (kThreads / 32)) {
    float s = 0.0f;
    for (int64_t k = lane; k < kp; k += 32) {
      float v;
      if (f8 != nullptr) {
        const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)f8[r * kp + k], __NV_E4M3);
        v = __half2float(__half(h)) * fs[r];
      } else {
        v = f32 ? f32[r * kp + k] : __bfloat162float(f16[r * kp + k]);
      }
      s = fmaf(v, v, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float nrm = sqrtf(s);
    // fmaxf drops a NaN operand: a row with a NaN entry counts as an infinite norm
    best = isnan(nrm) ? INFINITY : fmaxf(best, nrm);
  }
  if (lane == 0) red[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    float b = 0.0f;
    for (int w = 0; w < kThreads / 32; ++w) b = fmaxf(b, red[w]);
    atomicMax(out, __float_as_uint(b));  // non-negative floats order like their bit patterns
  }
}

// Partner preparation: the vector the half-sweep consumes, from the partner's
// stored ell and its maximum (a per-market scalar kept by the finalize
// kernels): fused_mode 1: (ell - max) * log2(e), padding -inf (exp2 of it is
// 0); fused_mode 0: exp(ell - max), padding 0. The vector depends on
// ell - max ell only, so no translation step or offset changes it; thread 0
// of block 0 records the pass's scalars (prep_scalars: its translation step,
// the partner shift it adds back and the own offset). No other thread reads
// the scalars it writes.
__device__ __forceinline__ void prep_row(int64_t i, int64_t rows, const double* __restrict__ ell, double top,
                                        int fused_mode, float* __restrict__ out, uint4* __restrict__ fold,
                                        float inv_c, float c) {
  float v;
  if (i < rows) {
    // the FP64 state is rounded once, to the FP32 vector the half-sweep streams
    const double z = ell[i] - top;
    v = fused_mode ? (float)(z * 1.4426950408889634) : (float)exp(z);
  } else {
    v = fused_mode ? -INFINITY : 0.0f;
  }
  out[i] = v;
  if (fold != nullptr) write_fold_row(fold, i, v, inv_c, c);
}

__global__ void k_prep(const double* __restrict__ ell, int64_t rows, int64_t rows_pad, double* __restrict__ st,
                       int own, int translate, int fused_mode, float* __restrict__ out, uint4* __restrict__ fold,
                       float inv_c, float c) {
  const double top = st[kStLmax + (1 - own)];
  if (blockIdx.x == 0 && threadIdx.x == 0) prep_scalars(st, own, translate);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows_pad;
       i += (int64_t)gridDim.x * blockDim.x) {
    prep_row(i, rows, ell, top, fused_mode, out, fold, inv_c, c);
  }
}

// Groups of both sides' stored potentials (one warp per 32 rows), as a
// half-sweep writes them for the rows it updates; with reset, of u = v = 1,
// which it stores (Alg. 1 / Alg. 2 initialisation).
struct ScanSide {
  double* log_u;
  double* ell;
  const float* b2s;
  float4* grp;
  int64_t rows;
};
__global__ void k_scan_groups(const ScanSide x, const ScanSide y, int reset) {
  const int64_t nx = (x.rows + kGroupRows - 1) / kGroupRows, ng = nx + (y.rows + kGroupRows - 1) / kGroupRows;
  const int lane = threadIdx.x % 32;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; i < ng;
       i += (int64_t)gridDim.x * blockDim.x / 32) {
    const ScanSide& s = i < nx ? x : y;
    const int64_t g = i < nx ? i : i - nx, r = g * kGroupRows + lane;
    const bool valid = r < s.rows;
    double lu = 0.0, el = 0.0;
    if (valid && reset) {
      el = s.b2s != nullptr ? (double)s.b2s[r] : 0.0;
      s.log_u[r] = lu;
      s.ell[r] = el;
    } else if (valid) {
      lu = s.log_u[r];
      el = s.ell[r];
    }
    const float4 gv = warp_group(lu, el, valid);
    if (lane == 0) s.grp[g] = gv;
  }
}

// Scalars of both sides from their groups (one block): shifts and sums,
// offsets cleared, and tau for the next half-sweep, which updates X against Y.
__global__ void k_rescan_scalars(const float4* __restrict__ grp_x, int64_t ng_x, const float4* __restrict__ grp_y,
                                 int64_t ng_y, double dm_next, double log_dm, double* __restrict__ st) {
  __shared__ float red[2 * kThreads / 32];
  const GroupTotal x = block_reduce_groups(grp_x, ng_x, red);
  const GroupTotal y = block_reduce_groups(grp_y, ng_y, red);
  if (threadIdx.x == 0) rescan_scalars(st, x, y, dm_next, log_dm);
}

// End of a block of sweeps: write the sides' offsets into their arrays and fold
// them into the scalars (by the last block to finish: every block has read the
// offsets by then; the counter, in a spare scalar slot, wraps to 0).
__global__ void k_flush(double* __restrict__ lu_x, double* __restrict__ ell_x, int64_t nx, double* __restrict__ lu_y,
                        double* __restrict__ ell_y, int64_t ny, double* __restrict__ st) {
  const double ox = st[kStOff + 0], oy = st[kStOff + 1];
  const int64_t n = nx > ny ? nx : ny;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (ox != 0.0 && i < nx) {
      lu_x[i] += ox;
      ell_x[i] += ox;
    }
    if (oy != 0.0 && i < ny) {
      lu_y[i] += oy;
      ell_y[i] += oy;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicInc(reinterpret_cast<unsigned*>(st + kStCount), gridDim.x - 1) == gridDim.x - 1) {
      st[kStLmax + 0] += ox;
      st[kStLmax + 1] += oy;
      st[kStOff + 0] = 0.0;
      st[kStOff + 1] = 0.0;
    }
  }
}

// What the finalize of a pass needs.
struct FinalizeArgs {
  const double* partials;
  int nparts, is_x, residual, update;
  const float4* grp;
  int64_t ngroups;
  double dm_next;   // sum of own capacities - sum of partner capacities
  double log_dm;    // log |dm_next|
  double* st;
  double* results;
  int prep_next;    // also the scalars of the half-sweep that follows (2: with the translation step)
};

// FP64 reduction of the per-CTA partials (max r/n, sum |r|, sum u^2, non-finite
// count), by one block. After a pass that updated its side (update), also that
// side's groups into the market scalars (finish_scalars), with the same routine
// and block size as the batched finalize.
__device__ __forceinline__ void finalize_pass(const FinalizeArgs& a) {
  __shared__ double red[4];
  __shared__ float redf[2 * kThreads / 32];
  // one warp per quantity: an FP64 addition takes about 80 cycles, so four
  // short chains side by side, and the groups meanwhile
  const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (w < 4) {
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = lane; i < a.nparts; i += 128) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double x = i + 32 * j < a.nparts ? a.partials[4 * (int64_t)(i + 32 * j) + w] : 0.0;
        v[j] = w == 0 ? (x > v[j] ? x : v[j]) : v[j] + x;
      }
    }
    double t = w == 0 ? fmax(fmax(v[0], v[1]), fmax(v[2], v[3])) : (v[0] + v[1]) + (v[2] + v[3]);
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, t, o);
      t = w == 0 ? (x > t ? x : t) : t + x;
    }
    if (lane == 0) red[w] = t;
  }
  GroupTotal g{};
  if (a.update) g = block_reduce_groups(a.grp, a.ngroups, redf);  // synchronises the block
  else __syncthreads();
  if (threadIdx.x == 0) {
    const double mx = red[0], l1 = red[1], sq = red[2], nf = red[3];
    if (a.is_x) {
      if (a.residual) {
        a.results[kResXInf] = mx;
        a.results[kResXL1] = l1;
      }
      a.results[kResXSq] = sq;
    } else {
      a.results[kResYSq] = sq;
    }
    if (nf != 0.0) a.results[kResNonfin] += nf;
    if (a.update) finish_scalars(a.st, a.is_x ? 0 : 1, g, a.dm_next, a.log_dm);
    if (a.prep_next) prep_scalars(a.st, a.is_x ? 1 : 0, a.prep_next > 1);
  }
}

__global__ void __launch_bounds__(kThreads) k_finalize(const FinalizeArgs a) { finalize_pass(a); }

// Between two half-sweeps: block 0 finalizes the pass before (results,
// scalars, the step and scalars of the next half-sweep); the others form the
// shift of the side just updated from its groups, as block 0 does, and write its
// vector for the pass that follows. The finalize is a chain of FP64 operations
// on one thread (5 us and more, log and exp at about 80 cycles per operation),
// which the pass needs only at its end and the vector not at all, so finalize
// and preparation one after the other took 12 us of a 10,000-user half-sweep.
__global__ void __launch_bounds__(kThreads) k_between(const FinalizeArgs a, const double* __restrict__ ell,
                                                     int64_t rows, int64_t rows_pad, int fused_mode,
                                                     float* __restrict__ out, uint4* __restrict__ fold, float inv_c, float c) {
  if (blockIdx.x == 0) {
    finalize_pass(a);
    return;
  }
  __shared__ float red[2 * kThreads / 32];
  float mm = -INFINITY, me = -INFINITY;
  for (int64_t i = threadIdx.x; i < a.ngroups; i += kThreads) me = fmaxf(me, a.grp[i].z);
  block_reduce_max2(mm, me, red);
  const double top = finite_or_zero((double)me);
  for (int64_t i = (blockIdx.x - 1) * (int64_t)kThreads + threadIdx.x; i < rows_pad;
       i += (int64_t)(gridDim.x - 1) * kThreads)
    prep_row(i, rows, ell, top, fused_mode, out, fold, inv_c, c);
}

// sum_i exp(2 log u_i) in FP64 as per-block partials in the common format.
__global__ void k_sum_sq(const double* __restrict__ log_u, int64_t rows, double* __restrict__ partials) {
  __shared__ double red[kThreads / 32];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x)
    s += exp(2.0 * log_u[i]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) b += red[w];
    partials[4 * blockIdx.x + 0] = 0.0;
    partials[4 * blockIdx.x + 1] = 0.0;
    partials[4 * blockIdx.x + 2] = b;
    partials[4 * blockIdx.x + 3] = 0.0;
  }
}

inline int grid_for(int64_t n, int num_sms, int per_sm = 8) {
  int64_t g = (n + kThreads - 1) / kThreads;
  const int64_t cap = (int64_t)num_sms * per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

cudaError_t launch_pack_factors(tu_market* m, Side& s, const void* A, const void* B, int src_dtype) {
  const int g = grid_for(s.rows * m->kp, m->num_sms, 16);
  k_pack_factors<<<g, kThreads, 0, m->stream>>>(A, B, src_dtype, s.rows, m->d, m->kp, s.fac16, s.fac32);
  return cudaGetLastError();
}

cudaError_t launch_init_side(tu_market* m, Side& s, const float* bias_dev, int has_bias) {
  const int g = grid_for(s.rows_pad, m->num_sms);
  k_init_side<<<g, kThreads, 0, m->stream>>>(bias_dev, has_bias, (float)(0.5 / m->sigma), s.rows,
                                               s.rows_pad, s.b2s, s.log_u, s.ell, s.mass);
  return cudaGetLastError();
}

cudaError_t launch_get_potentials(tu_market* m, float* out_x, float* out_y) {
  const int64_t n = m->X.rows > m->Y.rows ? m->X.rows : m->Y.rows;
  k_get_potentials<<<grid_for(n, m->num_sms), kThreads, 0, m->stream>>>(m->X.log_u, m->X.rows, out_x, m->Y.log_u,
                                                                      m->Y.rows, out_y);
  return cudaGetLastError();
}

cudaError_t launch_set_potentials64(tu_market* m, Side& s, const double* log_u_dev) {
  const int g = grid_for(s.rows, m->num_sms);
  k_set_potentials64<<<g, kThreads, 0, m->stream>>>(log_u_dev, s.b2s, s.rows, s.log_u, s.ell);
  return cudaGetLastError();
}

cudaError_t launch_set_potentials(tu_market* m, Side& s, const float* log_u_dev) {
  const int g = grid_for(s.rows, m->num_sms);
  k_set_potentials<<<g, kThreads, 0, m->stream>>>(log_u_dev, s.b2s, s.rows, s.log_u, s.ell);
  return cudaGetLastError();
}

cudaError_t launch_row_norms(tu_market* m, Side& s, float* out_max) {
  int64_t blocks = (s.rows + (kThreads / 32) - 1) / (kThreads / 32);
  if (blocks > (int64_t)m->num_sms * 8) blocks = (int64_t)m->num_sms * 8;
  k_row_norm_max<<<(int)blocks, kThreads, 0, m->stream>>>(s.fac32, s.fac16, s.fac8, s.fs, s.rows, m->kp,
                                                          reinterpret_cast<unsigned int*>(out_max));
  return cudaGetLastError();
}

cudaError_t launch_max_abs(tu_market* m, const float* A, const float* B, int64_t count, float* out_max) {
  cudaError_t e = cudaMemsetAsync(out_max, 0, sizeof(float), m->stream);
  if (e != cudaSuccess) return e;
  k_max_abs<<<grid_for(count, m->num_sms, 8), kThreads, 0, m->stream>>>(A, B, count,
                                                                       reinterpret_cast<unsigned int*>(out_max));
  return cudaGetLastError();
}

cudaError_t launch_pack_fp8_rows(tu_market* m, Side& s, const float* A, const float* B, int side_k,
                                 unsigned int* bad) {
  const int g = grid_for(s.rows_pad * 32, m->num_sms, 8);  // one warp per row
  k_pack_fp8_rows<<<g, kThreads, 0, m->stream>>>(A, B, s.rows, s.rows_pad, m->d, m->kp, side_k, s.fac8, s.fs, bad);
  return cudaGetLastError();
}

cudaError_t launch_pack_fp8_bytes(tu_market* m, Side& s, const uint8_t* A, const uint8_t* B, const float* sc,
                                  unsigned int* bad) {
  const int g = grid_for(s.rows * m->kp, m->num_sms, 16);
  k_pack_fp8_bytes<<<g, kThreads, 0, m->stream>>>(A, B, sc, s.rows, s.rows_pad, m->d, m->kp, s.fac8, s.fs, bad);
  return cudaGetLastError();
}

// c for write_fold_row, in markets whose folded g makes good the rounding of 1 / c
// (those that never run batched: the batched preparation has the three values)
static float fold_c(const tu_market* m) { return m->dtype == TU_DTYPE_FP8E4M3_SIDE && m->kp == 256 ? m->cmul : 0.0f; }

cudaError_t launch_prep(tu_market* m, Side& partner, int fused_mode, int translate, int offset) {
  const int own = &partner == &m->Y ? 0 : 1;
  const int g = grid_for(partner.rows_pad, m->num_sms, 4);
  k_prep<<<g, kThreads, 0, m->stream>>>(partner.ell, partner.rows, partner.rows_pad, m->st, own, translate, fused_mode,
                                        partner.pvec + offset, fused_mode && !m->wide ? reinterpret_cast<uint4*>(partner.fold) : nullptr,
                                        1.0f / m->cmul, fold_c(m));  // (the batched preparation rounds 1 / c alike)
  return cudaGetLastError();
}

static cudaError_t scan_sides(tu_market* m, int reset) {
  const ScanSide x = {m->X.log_u, m->X.ell, m->X.b2s, m->X.grp, m->X.rows};
  const ScanSide y = {m->Y.log_u, m->Y.ell, m->Y.b2s, m->Y.grp, m->Y.rows};
  const int64_t nx = (x.rows + kGroupRows - 1) / kGroupRows, ny = (y.rows + kGroupRows - 1) / kGroupRows;
  const double dm = m->Y.sum_mass - m->X.sum_mass;
  k_scan_groups<<<grid_for((nx + ny) * 32, m->num_sms, 8), kThreads, 0, m->stream>>>(x, y, reset);
  k_rescan_scalars<<<1, kThreads, 0, m->stream>>>(x.grp, nx, y.grp, ny, dm, log_abs(dm), m->st);
  return cudaGetLastError();
}

cudaError_t launch_rescan(tu_market* m) { return scan_sides(m, 0); }

cudaError_t launch_reset(tu_market* m) { return scan_sides(m, 1); }

cudaError_t launch_flush(tu_market* m) {
  const int64_t n = m->X.rows > m->Y.rows ? m->X.rows : m->Y.rows;
  k_flush<<<grid_for(n, m->num_sms, 4), kThreads, 0, m->stream>>>(m->X.log_u, m->X.ell, m->X.rows, m->Y.log_u,
                                                                   m->Y.ell, m->Y.rows, m->st);
  return cudaGetLastError();
}

cudaError_t launch_sum_sq(tu_market* m, Side& s, int is_x) {
  int g = grid_for(s.rows, m->num_sms, 4);
  if (g > kMaxPartials) g = kMaxPartials;
  k_sum_sq<<<g, kThreads, 0, m->stream>>>(s.log_u, s.rows, m->partials);
  const FinalizeArgs a = {m->partials, g, is_x, 0, 0, nullptr, 0, 0.0, 0.0, m->st, m->results, 0};
  k_finalize<<<1, kThreads, 0, m->stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_finalize(tu_market* m, int nparts, int is_x, int residual, int update, int64_t ngroups,
                            int prep_next) {
  Side& own = is_x ? m->X : m->Y;
  Side& par = is_x ? m->Y : m->X;
  const double dm = own.sum_mass - par.sum_mass;
  const FinalizeArgs a = {m->partials, nparts, is_x, residual, update, own.grp, ngroups, dm, log_abs(dm), m->st,
                          m->results, prep_next};
  k_finalize<<<1, kThreads, 0, m->stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_between(tu_market* m, int nparts, int is_x, int residual, int64_t ngroups, int fused_mode,
                           int translate) {
  // (every block reads the groups: past a few thousand the two kernels are better)
  if (ngroups > 4096) {
    cudaError_t e = launch_finalize(m, nparts, is_x, residual, 1, ngroups);
    return e != cudaSuccess ? e : launch_prep(m, is_x ? m->X : m->Y, fused_mode, translate);
  }
  Side& own = is_x ? m->X : m->Y;
  Side& par = is_x ? m->Y : m->X;
  const double dm = own.sum_mass - par.sum_mass;
  const FinalizeArgs a = {m->partials, nparts, is_x, residual, 1, own.grp, ngroups, dm, log_abs(dm), m->st,
                          m->results, translate ? 2 : 1};
  k_between<<<1 + grid_for(own.rows_pad, m->num_sms, 4), kThreads, 0, m->stream>>>(
      a, own.ell, own.rows, own.rows_pad, fused_mode, own.pvec,
      fused_mode && !m->wide ? reinterpret_cast<uint4*>(own.fold) : nullptr, 1.0f / m->cmul, fold_c(m));
  return cudaGetLastError();
}

}  // namespace tu
