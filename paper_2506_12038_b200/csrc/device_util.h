// Per-device bookkeeping of the kernel launchers: a kernel's attributes (the opt-in to large dynamic shared memory)
// belong to the device that is current when they are set, and a process may use several devices from several threads.
#ifndef LCD_DEVICE_UTIL_H_
#define LCD_DEVICE_UTIL_H_

#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>

namespace lcd {

// One flag per device (up to 64) for one kernel instance: first() is true until done() was called for the current
// device.  Two threads that race both set the attribute, which is harmless.
struct PerDeviceFlag {
  std::atomic<unsigned long long> mask{0ull};
  bool first(int* dev) const {
    *dev = 0;
    if (cudaGetDevice(dev) != cudaSuccess || *dev < 0 || *dev >= 64) return true;   // unknown device: always set
    return ((mask.load(std::memory_order_acquire) >> *dev) & 1ull) == 0;
  }
  void done(int dev) {
    if (dev >= 0 && dev < 64) mask.fetch_or(1ull << dev, std::memory_order_release);
  }
};

// Multiprocessors of the current device (148 if it cannot be asked).  Asked of the runtime once per device: the query costs
// as much as a tenth of a launch and every call needs the number.
inline int current_sm_count() {
  static std::atomic<int> known[64];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  const bool slot = dev >= 0 && dev < 64;
  if (slot && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 148;
  if (slot) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

#ifdef __CUDACC__
// Loads of what an earlier kernel of the stream writes, behind griddepcontrol.wait.  A kernel launched with programmatic
// stream serialization may be running while that one still writes, and __ldg (ld.global.nc, what loads through const
// __restrict__ pointers become too) is only for data that nobody writes while the reading kernel runs.
__device__ __forceinline__ float ld_global(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ unsigned short ld_global(const unsigned short* p) {
  unsigned short v;
  asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ld_global(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
#endif

// cuTensorMapEncodeTiled, asked of the driver (the library does not link against it); null if there is none.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

}  // namespace lcd
#endif
