// Cooperative launches: kernels whose CTAs wait for one another (cg.cu, mlp.cu).
#pragma once

#include <cuda_runtime.h>

namespace pjds {

#ifdef PJDS_CHECKED
// Test of the callers' way out, without a limited context: launches of more CTAs than this are refused (-1: none;
// pjds_checked_cooperative_limit).
extern int g_cooperative_limit;
#endif

// cudaErrorCooperativeLaunchTooLarge: the context does not hold so many CTAs at once; the caller has another way.
// (That error is not kept for the thread's next check.)
inline cudaError_t launch_cooperative(const void *kernel, unsigned grid, unsigned threads, void **args, size_t smem,
                                      cudaStream_t s) {
#ifdef PJDS_CHECKED
  if (g_cooperative_limit >= 0 && grid > (unsigned)g_cooperative_limit) return cudaErrorCooperativeLaunchTooLarge;
#endif
  const cudaError_t e = cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(threads), args, smem, s);
  if (e == cudaErrorCooperativeLaunchTooLarge) cudaGetLastError();
  return e;
}

}  // namespace pjds
