// Shared host-side plumbing of the repq library: error reporting and argument checks.
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <string>

#include "../../include/repq.h"

namespace repq {

std::string& last_error_ref();

inline repq_status fail(repq_status code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  last_error_ref() = buf;
  return code;
}

#define REPQ_REQUIRE(cond, code, ...) \
  do {                                \
    if (!(cond)) return ::repq::fail((code), __VA_ARGS__); \
  } while (0)

#define REPQ_CUDA(call)                                                                   \
  do {                                                                                    \
    cudaError_t e__ = (call);                                                             \
    if (e__ != cudaSuccess)                                                               \
      return ::repq::fail(REPQ_CUDA_ERROR, "%s failed: %s", #call, cudaGetErrorString(e__)); \
  } while (0)

#define REPQ_TRY(call)                   \
  do {                                   \
    repq_status s__ = (call);            \
    if (s__ != REPQ_OK) return s__;      \
  } while (0)

// A `bits` value = quantizer width (4, 6, 8) | optional REPQ_BYTE_CODES.
inline int quant_bits(int b) { return b & 0xFF; }
inline bool bits_ok(int b) {
  const int q = quant_bits(b);
  return (b & ~(0xFF | REPQ_BYTE_CODES)) == 0 && (q == 4 || q == 6 || q == 8);
}
inline bool packed4(int b) { return b == 4; }                        // two codes per byte
inline bool packed6(int b) { return b == (6 | REPQ_PACKED6); }       // four codes in three bytes (weights only)
inline bool bits_w_ok(int b) { return bits_ok(b) || packed6(b); }
inline int code_max(int b) { return (1 << quant_bits(b)) - 1; }
inline int64_t code_row_bytes(int64_t n, int bits) { return packed4(bits) ? (n + 1) / 2 : packed6(bits) ? (n * 3 + 3) / 4 : n; }
inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

int sm_count();

// Launch accounting (repq_launch_count).
void note_launch(int n = 1);

// Kernels of one stream that follow each other are launched with programmatic stream serialization: the next
// kernel may be scheduled, and run its prologue (barrier setup, tensor-memory allocation, parameter staging), as
// SMs drain from the one before.  Such a kernel calls grid_dependency_wait() before its first access to global
// memory that an earlier kernel may have written or may still read, and grid_dependency_trigger() once it has
// started (both are no-ops in a kernel launched the plain way).
#ifdef __CUDACC__
// Opt-in of a kernel to more than 48 KB of dynamic shared memory, asked of the runtime once per kernel and device.
template <auto kKernel>
repq_status allow_smem(int bytes) {
  static std::atomic<uint64_t> done{0};                // one bit per device
  int dev = 0;
  REPQ_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
  if (done.load(std::memory_order_relaxed) & bit) return REPQ_OK;
  REPQ_CUDA(cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done.fetch_or(bit, std::memory_order_relaxed);
  return REPQ_OK;
}

// Resident blocks per SM of a kernel, remembered per device for the last dynamic shared-memory size asked for.
struct Residency { std::atomic<uint64_t> last[64]; };   // (bytes << 8) | blocks, 0: nothing yet
template <typename Kernel>
repq_status resident_blocks(Residency& memo, Kernel kern, int block, size_t smem, int* out) {
  int dev = 0;
  REPQ_CUDA(cudaGetDevice(&dev));
  const bool keep = dev >= 0 && dev < 64;
  const uint64_t seen = keep ? memo.last[dev].load(std::memory_order_relaxed) : 0;
  if (seen != 0 && (seen >> 8) == smem) { *out = int(seen & 0xFF); return REPQ_OK; }
  int n = 0;
  REPQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem));
  if (n < 1) n = 1;
  if (keep) memo.last[dev].store((uint64_t(smem) << 8) | uint64_t(n), std::memory_order_relaxed);
  *out = n;
  return REPQ_OK;
}

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// (cluster: CTAs of a thread-block cluster along x)
template <typename... KArgs, typename... Args>
cudaError_t launch_chained_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = unsigned(cluster);
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_chained_cluster(kernel, grid, block, smem, st, 1, static_cast<Args&&>(args)...);
}
#endif

}  // namespace repq
