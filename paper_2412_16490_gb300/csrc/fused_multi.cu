// The several-job step kernels, a block per work item (bodex_kernels.cuh).
#include "bodex_kernels.cuh"

int launch_multi(bool adapt, bool exact, const MultiArgs& MA, size_t bytes, cudaStream_t st) {
  auto go = [&](auto kernel) -> int {
    if (int r = ensure_smem(kernel, bytes)) return r;
    kernel<<<MA.total, CTA_LANES, bytes, st>>>(MA);
    return launch_err("multi_kernel launch");
  };
  if (exact) return go(multi_kernel<false, true>);
  if (few_wrenches(MA)) return adapt ? go(multi_kernel<true>) : go(multi_kernel<false>);
  return adapt ? go(multi_kernel<true, false, false, false>) : go(multi_kernel<false, false, false, false>);
}

int launch_multi_wide(bool soc, const MultiArgs& MA, int threads, size_t bytes, cudaStream_t st) {
  auto go = [&](auto kernel) -> int {
    if (int r = ensure_smem(kernel, bytes)) return r;
    kernel<<<MA.total, threads, bytes, st>>>(MA);
    return launch_err("multi_wide_kernel launch");
  };
  return soc ? go(multi_wide_kernel<CONE_SOC>) : go(multi_wide_kernel<CONE_PYR>);
}
