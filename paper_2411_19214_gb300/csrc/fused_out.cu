// fused_out.cu -- instantiations of the fused kernel (fused_kernel.cuh) for wide
// half-sweeps, ranked lists and mu blocks.
#include "fused_kernel.cuh"

namespace tu {

cudaError_t set_out_attributes() {
  cudaError_t e = set_attributes_mode<kModeTopK, false>();
  if (e == cudaSuccess) e = set_attributes_mode<kModeMu, false>();
  if (e == cudaSuccess) e = set_attributes_mode<kModeTopKShared, false>();
  if (e == cudaSuccess) e = set_attributes_mode<kModeSweepWide, false>();
  if (e == cudaSuccess) e = set_pair_attributes<kModeSweepWide>();
  return e;
}

cudaError_t launch_wide_sweep(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                              const FusedParams& p, int grid, cudaStream_t stream, bool small, bool split) {
  return launch_sweep<kModeSweepWide>(kp, fmt, own, partner, p, grid, stream, small, split);
}

cudaError_t launch_wide_pair(int kb, int fmt, bool split, const CUtensorMap* own, const CUtensorMap* half,
                             const CUtensorMap* fold, const FusedParams* p, int grid, cudaStream_t stream) {
  return launch_pair<kModeSweepWide>(kb, fmt, split, own, half, fold, p, grid, stream);
}

// Lists longer than kSharedTopK fit in shared memory only with 128-row tiles
// (half of the threads have rows, so each has twice the slots).
bool lists_want_small(int k, int64_t kp, int fmt) {
  return k > kSharedTopK && k <= kSharedTopKSmall && k_blocks(kp, fmt) < 4;
}

cudaError_t launch_lists(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner,
                         const FusedParams& p, int grid, cudaStream_t stream, bool small) {
  if (p.k <= (small ? kSharedTopKSmall : kSharedTopK) && k_blocks(kp, fmt) < 4)
    return launch_any<kModeTopKShared>(kp, fmt, own, partner, p, grid, stream, small);
  return launch_any<kModeTopK>(kp, fmt, own, partner, p, grid, stream, small);
}

cudaError_t launch_mu(int64_t kp, int fmt, const CUtensorMap& own, const CUtensorMap& partner, const FusedParams& p,
                      int grid, cudaStream_t stream) {
  return launch_variant<kModeMu, false, false, true>(kp, fmt, own, partner, p, grid, stream);
}

}  // namespace tu
