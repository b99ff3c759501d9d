// The sort of dbci.cu (dbci_sort.cu).
#ifndef LCD_DBCI_SORT_H_
#define LCD_DBCI_SORT_H_

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace lcd {

// A launch that may begin while the kernel before it on the stream ends (every kernel here waits for that one first).
template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

bool dbci_sort_takes(int64_t n);
size_t dbci_sort_workspace_bytes(int64_t n);
// weights[n] in ascending order (negative zero and zero are equal and keep their order) to sorted[n], which does not overlap them
cudaError_t launch_dbci_sort(const float* weights, int64_t n, float* sorted, void* workspace, cudaStream_t s);

}  // namespace lcd
#endif
