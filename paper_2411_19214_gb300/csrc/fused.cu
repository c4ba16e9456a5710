// fused.cu -- the fused path's host side: tensor maps, launch shapes, and the
// narrow and batched half-sweeps of fused_kernel.cuh (the kernel, its design
// and its instantiations).
#include "fused_kernel.cuh"

#include <cstring>
#include <mutex>

namespace tu {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// Tensor map over packed rows x kp factors (bf16, or e4m3 bytes when fp8);
// the box is one 128-byte swizzle row wide.
cudaError_t make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t kp, int box_rows, bool fp8 = false) {
  EncodeTiledFn enc = get_encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  const size_t esz = fp8 ? 1 : sizeof(__nv_bfloat16);
  const cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)kp * esz};
  const cuuint32_t box[2] = {(cuuint32_t)(128 / esz), (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                         const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Dynamic shared memory opt-in of every instantiation, on the current device.
cudaError_t set_kernel_attributes_now() {
  cudaError_t e = set_attributes_mode<kModeSweep, false>();
  if (e == cudaSuccess) e = set_attributes_mode<kModeSweep, true>();
  if (e == cudaSuccess) e = set_pair_attributes<kModeSweep>();
  if (e == cudaSuccess) e = set_out_attributes();
  // the allocation-free entry point's unfolded half-sweep 
  if (e == cudaSuccess) e = set_attribute_one<1, kModeSweep, false, kFmtBF16, false, false, true>();
  if (e == cudaSuccess) e = set_attribute_one<2, kModeSweep, false, kFmtBF16, false, false, true>();
  return e;
}

// The opt-in is a property of each function in the device's context: made
// once per device (about 130 instantiations, a driver call each), not per
// market, so that creating markets stays cheap for a loop that creates many.
cudaError_t set_kernel_attributes() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return set_kernel_attributes_now();
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  e = set_kernel_attributes_now();
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

// The operand format of a market's dtype.
int fmt_of(int dtype) {
  return dtype == TU_DTYPE_FP8E4M3 ? kFmtE4M3Rows : (dtype == TU_DTYPE_FP8E4M3_SIDE ? kFmtE4M3Side : kFmtBF16);
}

// Tensor map over a side's folded operand (4 KB per 128 users) as rows of 256
// bytes, 8 to a box: the half of a tile that one CTA of a pair loads.
cudaError_t make_fold_map(Side* sd) {
  memset(&sd->tm_fold, 0, sizeof(sd->tm_fold));
  if (sd->fold == nullptr) return cudaSuccess;
  EncodeTiledFn enc = get_encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {64, (cuuint64_t)(sd->rows_pad / 8)};
  const cuuint64_t strides[1] = {256};
  const cuuint32_t box[2] = {64, 8};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(&sd->tm_fold, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, sd->fold, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 128-row own tiles when they all fit one wave (and the market allows them),
// for launches that the cuts leave alone (row ranges, ranked lists, markets of
// four partner tiles and fewer): a CTA with one MMA chain ends its tile in
// about 0.73 of the time of a 256-row tile (measured at 1e4 x 1e4), so the
// small tiles win only while SMs would otherwise stay idle; on a GPU already
// full (other markets' work on other streams) they lose a third of the per-SM
// throughput.
bool use_small_tiles(const tu_market* m, int64_t rows) {
  if (m->small_mode == 0) return false;
  if (m->small_mode == 2) return true;
  const int64_t t256 = (rows + kFusedOwnRows - 1) / kFusedOwnRows;
  const int64_t t128 = (rows + kFusedOwnRows / 2 - 1) / (kFusedOwnRows / 2);
  return t256 < m->num_sms && t128 <= m->num_sms;
}

FusedParams base_params(int64_t rows, int64_t row0, int64_t col0, int64_t ncols, float c, bool small = false) {
  FusedParams p{};
  const int own_rows = small ? kFusedOwnRows / 2 : kFusedOwnRows;
  p.rows = rows;
  p.row0 = row0;
  p.col0 = col0;
  p.ncols = ncols;
  p.num_own_tiles = (int)((rows + own_rows - 1) / own_rows);
  p.num_partner_tiles = (int)((ncols + kFusedPartnerRows - 1) / kFusedPartnerRows);
  p.c = c;
  p.split = 1;
  p.cut_t0 = p.num_own_tiles;
  p.cut_rows = kFusedOwnRows;
  return p;
}

// Partner ranges of a launch of `tiles` own tiles by `ptiles` partner tiles on
// `sms` persistent CTAs, at most `most`: the fewest that minimise the longest
// CTA's work, in partner tiles, where an item costs `overhead` of them besides
// its own (own-tile load, pipeline fill, row updates).
int best_split(int64_t tiles, int64_t ptiles, int sms, int most, double overhead) {
  int best = 1;
  double best_cost = 0.0;
  for (int s = 1; s <= most && s <= ptiles; ++s) {
    const int64_t waves = (tiles * s + sms - 1) / sms;
    const double cost = (double)waves * ((double)((ptiles + s - 1) / s) + overhead);
    if (s == 1 || cost < 0.98 * best_cost) {
      best = s;
      best_cost = cost;
    }
  }
  return best;
}

int grid_for_tiles(int tiles, int num_sms) {
  int grid = tiles < num_sms ? tiles : num_sms;
  if (grid > kMaxPartials) grid = kMaxPartials;
  return grid < 1 ? 1 : grid;
}

}  // namespace

cudaError_t fused_prepare(tu_market* m) {
  const bool f8 = is_fp8(m->dtype);
  const void* x = f8 ? (const void*)m->X.fac8 : (const void*)m->X.fac16;
  const void* y = f8 ? (const void*)m->Y.fac8 : (const void*)m->Y.fac16;
  cudaError_t e;
  if ((e = make_map(&m->X.tm_own, x, m->X.rows, m->kp, kFusedOwnRows, f8)) != cudaSuccess) return e;
  if ((e = make_map(&m->X.tm_partner, x, m->X.rows, m->kp, kFusedPartnerRows, f8)) != cudaSuccess) return e;
  for (Side* sd : {&m->X, &m->Y})
    if ((e = make_fold_map(sd)) != cudaSuccess) return e;
  if ((e = make_map(&m->X.tm_half, x, m->X.rows, m->kp, kFusedPartnerRows / 2, f8)) != cudaSuccess) return e;
  if ((e = make_map(&m->Y.tm_half, y, m->Y.rows, m->kp, kFusedPartnerRows / 2, f8)) != cudaSuccess) return e;
  if ((e = make_map(&m->Y.tm_own, y, m->Y.rows, m->kp, kFusedOwnRows, f8)) != cudaSuccess) return e;
  if ((e = make_map(&m->Y.tm_partner, y, m->Y.rows, m->kp, kFusedPartnerRows, f8)) != cudaSuccess) return e;
  return set_kernel_attributes();
}

// The whole tiles of w full waves run as they are; the rest, one line of (tile,
// partner tile) pairs, is cut into equal spans, one per SM. Without cuts 313
// tiles on 152 SMs take three waves of which the last runs 9 tiles (the
// 100,003-user side of a 79,999-user market), and a market of 40 tiles keeps
// 112 SMs idle. A span costs its partner tiles and about kSpanCost more (two
// pipeline fills, the partials' stores and the sums of the completing warp),
// a tile kTileCost; the cuts are taken when they save 8 % of the longest CTA:
// with eight waves and more the chip runs at its power limit anyway, and idle
// SMs in the last wave give the others clock (300,000 x 300,000, 7.7 waves:
// 33.3 ms per sweep whole, 34.3 cut). Per sweep, whole -> cut: 3,000 x 3,000
// d = 50 58 -> 51 us, 10,000 x 10,000 123 -> 88, 20,000 x 15,001 d = 32 213 ->
// 152, 40,000 x 40,000 1.08 -> 0.67 ms, 100,003 x 79,999 d = 64 3.57 -> 3.05,
// FP8 rows 100,000 x 80,000 3.65 -> 2.96, d = 100 50,001 x 70,000 3.56 -> 2.89;
// spans under four partner tiles lose (1,000 x 1,000: 38 us whole, 45 in spans
// of two).
constexpr int kSpanCost = 8, kTileCost = 4, kMinSpan = 4;

// Own sides of more rows run on pairs of CTAs.
constexpr int kPairRows = 512;

CutPlan cut_plan(int64_t own_rows, int64_t partner_rows, int kblocks, int sms) {
  CutPlan c;
  c.pair = kblocks > 1 && sms % 2 == 0 && own_rows > kPairRows;
  if (c.pair) sms /= 2;
  const int tile = c.pair ? 2 * kFusedOwnRows : kFusedOwnRows;
  const int64_t T = (own_rows + tile - 1) / tile;
  const int64_t P = (partner_rows + kFusedPartnerRows - 1) / kFusedPartnerRows;
  const int64_t w = T / sms, rest = T - w * sms;
  c.t0 = (int)T;
  if (rest == 0 || P <= kMinSpan || rest * P > (1 << 30)) return c;
  int64_t span = (rest * P + sms - 1) / sms;
  if (span < kMinSpan) span = kMinSpan;
  if ((double)(w * (P + kTileCost) + span + kSpanCost) > 0.92 * (double)((w + 1) * (P + kTileCost))) return c;
  c.t0 = (int)(w * sms);
  c.span = (int)span;
  c.spans = (int)((rest * P + span - 1) / span);
  return c;
}

int64_t cut_slots(const CutPlan& p) { return (p.pair ? 4 : 2) * (int64_t)p.spans; }

cudaError_t launch_fused_halfsweep(tu_market* m, int side, int residual, int update, int* nparts_out,
                                   int64_t row0, int64_t nrows) {
  Side& own = side == 0 ? m->X : m->Y;
  Side& partner = side == 0 ? m->Y : m->X;
  const bool whole = nrows < 0;
  if (whole) {
    row0 = 0;
    nrows = own.rows;
  }
  // the caller's split; or, in the default shape, a CTA per span of the cut tiles
  const bool user_split = whole && !m->wide && m->split > 1 && m->split_part != nullptr;
  const bool cuts = !user_split && own.cut.span > 0;
  const bool cut_launch = cuts && whole && m->small_mode == 1 && m->cut_part != nullptr;
  const bool pair = !user_split && whole && own.cut.pair && m->small_mode == 1 && cuts == cut_launch;
  const bool small = !cut_launch && !pair && use_small_tiles(m, nrows);
  FusedParams p = base_params(nrows, row0, 0, partner.rows, m->cmul, small);
  p.g = partner.pvec;
  p.lmax = m->st + kStShift;
  p.ksteps = k_steps(m);
  p.own_off = m->st + kStOwnOff;
  p.grp = whole ? own.grp : nullptr;  // a range of rows does not write the side's groups
  p.b2s = own.b2s;
  p.mass = own.mass;
  p.log_u = own.log_u;
  p.ell = own.ell;
  p.partials = m->partials;
  p.err = m->err_dev;
  p.residual = residual;
  p.update = update;
  p.omega = m->omega_dev;
  p.fs_own = own.fs;
  p.fs_par = partner.fs;
  p.gfold = partner.fold;
  {
    // partner matrices larger than L2: keep a fixed 70 % of L2's worth resident
    const double pbytes = (double)partner.rows * (double)m->kp * (is_fp8(m->dtype) ? 1.0 : 2.0);
    const double keep = 0.7 * (double)m->l2_bytes;
    p.l2_keep = (m->l2_bytes > 0 && pbytes > keep) ? (float)(keep / pbytes) : 0.0f;
  }
  int items = p.num_own_tiles;
  if (user_split) {
    // at most one range per partner tile
    p.split = m->split < p.num_partner_tiles ? m->split : p.num_partner_tiles;
    p.range_major = m->split_blocks ? 1 : 0;
    p.part = m->split_part;
    p.split_cnt = m->split_cnt;
    items *= p.split;
  } else if (cuts) {
    p.cut_t0 = own.cut.t0;
    p.cut_span = own.cut.span;
    p.cut_spans = own.cut.spans;
    p.cut_ptiles = p.num_partner_tiles;
    p.cut_rows = own.cut.pair ? 2 * kFusedOwnRows : kFusedOwnRows;
    if (cut_launch) {
      p.part = m->cut_part;
      p.part_m = m->cut_m;
      p.split_cnt = m->cut_cnt;
      items = p.cut_t0 > 0 ? m->num_sms : (pair ? 2 : 1) * p.cut_spans;
    }
  }
  if (pair && !cut_launch) {
    items = (items + 1) / 2 * 2;
    p.cut_t0 = items / 2;
  }
  const int grid = grid_for_tiles(items, m->num_sms);
  *nparts_out = grid;
  const int fmt = fmt_of(m->dtype);
  const bool split = p.split > 1 || cut_launch;
  if (pair) {
    if (m->wide)
      return launch_wide_pair(k_blocks(m->kp, fmt), fmt, split, &own.tm_own, &partner.tm_half, &partner.tm_fold, &p,
                              grid, m->stream);
    return launch_pair<kModeSweep>(k_blocks(m->kp, fmt), fmt, split, &own.tm_own, &partner.tm_half, &partner.tm_fold, &p,
                              grid, m->stream);
  }
  if (m->wide)
    return launch_wide_sweep(m->kp, fmt, own.tm_own, partner.tm_partner, p, grid, m->stream, small, split);
  return launch_sweep<kModeSweep>(m->kp, fmt, own.tm_own, partner.tm_partner, p, grid, m->stream, small, split);
}

// Ranked lists of own users [row0, row0 + nrows) over all partners (the
// partner vector must have been prepared in log2 mode). hand_v / hand_i:
// nrows x k scratch.
cudaError_t launch_fused_topk(tu_market* m, int side, int k, int64_t row0, int64_t nrows, int32_t* idx,
                              float* logmu, float* hand_v, int32_t* hand_i) {
  Side& own = side == 0 ? m->X : m->Y;
  Side& partner = side == 0 ? m->Y : m->X;
  const bool small = use_small_tiles(m, nrows) || lists_want_small(k, m->kp, fmt_of(m->dtype));
  FusedParams p = base_params(nrows, row0, 0, partner.rows, m->cmul, small);
  p.g = partner.pvec;
  p.lmax = m->st + kStShift;
  p.ell = own.ell;
  p.partials = m->partials;
  p.err = m->err_dev;
  p.k = k;
  p.idx = idx;
  p.logmu = logmu;
  p.hand_v = hand_v;
  p.hand_i = hand_i;
  p.fs_own = own.fs;
  p.fs_par = partner.fs;
  const int grid = grid_for_tiles(p.num_own_tiles, m->num_sms);
  const int fmt = fmt_of(m->dtype);
  return launch_lists(m->kp, fmt, own.tm_own, partner.tm_partner, p, grid, m->stream, small);
}

// Where the partner vector of a mu block from column y0 starts in pvec.
int mu_vector_offset(const tu_market* m, int64_t y0) {
  return m->dtype == TU_DTYPE_FP8E4M3 ? 0 : (int)((4 - (y0 & 3)) & 3);
}

// mu for own X users [x0, x0 + nx) and partners [y0, y0 + ny) (the Y partner
// vector must have been prepared in log2 mode).
cudaError_t launch_fused_mu(tu_market* m, int64_t x0, int64_t nx, int64_t y0, int64_t ny, float* out, int64_t ld) {
  // The bulk copies of g start 16-byte aligned: the vector is prepared with the
  // block's first column there. (Row scales are where they are: the block then
  // starts at the multiple of four before it, and its stores are single floats.)
  const bool scales = m->dtype == TU_DTYPE_FP8E4M3;
  const int64_t c0 = scales ? y0 & ~(int64_t)3 : y0;
  FusedParams p = base_params(nx, x0, c0, y0 + ny - c0, m->cmul);
  // A block is bounded by its stores (128 KB per 256 x 128 tile), so every SM
  // takes part: the partner tiles of an own tile go to several CTAs.
  // (7,150 x 9,336 at d = 50: 795 us on 56 CTAs with each thread storing along
  // its own row, 109 us with the stores turned through shared memory on 140.)
  p.split = best_split(p.num_own_tiles, p.num_partner_tiles, m->num_sms, 64, 1.0);
  p.vec = !scales && (ld & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  p.g = m->Y.pvec + mu_vector_offset(m, y0);
  p.lmax = m->st + kStShift;
  p.ell = m->X.ell;
  p.partials = m->partials;
  p.err = m->err_dev;
  p.out = out;
  p.ld = ld;
  p.y0 = y0;
  p.ny = ny;
  p.fs_own = m->X.fs;
  p.fs_par = m->Y.fs;
  return launch_mu(m->kp, fmt_of(m->dtype), m->X.tm_own, m->Y.tm_partner, p,
                   grid_for_tiles(p.num_own_tiles * p.split, m->num_sms), m->stream);
}

// Same kernel on caller-described buffers (no market object): used by the
// allocation-free entry point. Tensor maps are built on the host stack.
cudaError_t launch_fused_halfsweep_raw(const FusedRaw& r, cudaStream_t stream, int num_sms, int* nparts_out) {
  CUtensorMap own_map, partner_map;
  cudaError_t e;
  if ((e = make_map(&own_map, r.own16, r.rows, r.kp, kFusedOwnRows)) != cudaSuccess) return e;
  if ((e = make_map(&partner_map, r.par16, r.cols, r.kp, kFusedPartnerRows)) != cudaSuccess) return e;
  if ((e = set_kernel_attributes()) != cudaSuccess) return e;
  FusedParams p = base_params(r.rows, 0, 0, r.cols, (float)(1.4426950408889634 / (2.0 * r.sigma)));
  p.ksteps = (int)(r.kp / 16);  // (the caller's rows: whole)
  p.g = r.g;
  p.lmax = r.lmax;
  p.b2s = r.b2s;
  p.mass = r.mass;
  p.log_u = r.log_u;
  p.ell = r.ell;
  p.partials = r.partials;
  p.err = r.err;
  p.residual = r.residual;
  p.update = 1;
  const int grid = grid_for_tiles(p.num_own_tiles, num_sms);
  *nparts_out = grid;
  // (no folded operand here: the instantiation with g from the shared ring)
  if (r.kp == kKBlock) return launch_kernel<1, kModeSweep, false, kFmtBF16, false, false, true>(own_map, partner_map, p,
                                                                                              grid, stream);
  return launch_kernel<2, kModeSweep, false, kFmtBF16, false, false, true>(own_map, partner_map, p, grid, stream);
}

// One half-sweep over the items of many markets (batched launch). The
// per-market tensor maps live in the descriptors, so the kernel's map
// parameters are unused.
cudaError_t launch_fused_batch(const BatchLaunch& b, cudaStream_t stream) {
  static_assert(kEpiWarps / 2 == kBatchSlotWarps, "per-tile partial slots");
  // (the shared-memory opt-in was made when the member markets were prepared)
  FusedParams p{};
  p.ksteps = b.ksteps;
  p.bdesc = b.desc;
  p.items = b.items;
  p.cta_start = b.cta_start;
  p.partials = b.partials;
  p.err = b.err;
  p.residual = b.residual;
  p.update = b.update;
  CUtensorMap unused;
  memset(&unused, 0, sizeof(unused));
  return launch_any<kModeSweep, true>(b.kp, fmt_of(b.dtype), unused, unused, p, b.grid, stream);
}

}  // namespace tu
