// Programmatic dependent launches of the H application's kernels: a kernel is put in place while its
// predecessor on the stream drains, instead of after it.  Every kernel launched this way begins with
// pdl_wait(), which lets the next one be put in place in turn and then waits until the predecessor has
// completed with all its writes visible, so the kernels' work itself stays in stream order; what
// overlaps is the launch.  An application is 6 to 9 kernels, of 3 to 40 us in the small cells.  Filter
// step of 82 bands of a 12.3 bohr cell 106 -> 88 us, H on 1127 bands of a 10 bohr cell at Gamma 122 -> 107.
// The small FP64 products (gemm_small.cu) are launched plainly: put in place early they held up the FP64
// pipe of the kernels beside them (H on 20 bands: 59 us without, 73 with them, 55 with the others only).
#pragma once

#include <type_traits>

#include "kss_internal.h"

namespace kss {

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;" ::: "memory");
}
#endif

// Lets a kernel be launched with `bytes` of dynamic shared memory (up to 48 KB needs no leave).
template <class K>
void allow_smem(K* kernel, size_t bytes) {
  if (bytes > 48u * 1024u)
    KSS_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// early = false: an ordinary launch (of a kernel that has pdl_wait all the same).
template <class... P>
void launch_pdl_if(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                   std::common_type_t<P>... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  KSS_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
}
template <class... P>
void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                std::common_type_t<P>... args) {
  launch_pdl_if(true, kernel, grid, block, smem, st, args...);
}

}  // namespace kss
