// The several-job step kernels whose blocks pull their work items
// (bodex_kernels.cuh).
#include "bodex_kernels.cuh"

// One CTA per resident slot (SMs x CTAs that fit per SM at `bytes` of shared
// memory), at most one per work item, pulling items until none is left.
int launch_multi_pull(bool adapt, bool exact, const MultiArgs& MA, size_t bytes, cudaStream_t st) {
  auto go = [&](auto kernel) -> int {
    if (int r = ensure_smem(kernel, bytes)) return r;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, CTA_LANES, bytes) != cudaSuccess)
      return launch_err("multi_kernel occupancy query");
    kernel<<<std::max(1, std::min(MA.total, sms * std::max(per_sm, 1))), CTA_LANES, bytes, st>>>(MA);
    return launch_err("multi_kernel launch");
  };
  if (exact) return go(multi_kernel<false, true, true>);
  return adapt ? go(multi_kernel<true, false, true>) : go(multi_kernel<false, false, true>);
}
