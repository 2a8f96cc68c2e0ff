// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "ttnn.h"

namespace ttnn {

// --- error reporting ------------------------------------------------------
void set_error(const char* fmt, ...);
const char* last_error();

#define TTNN_TRY_CUDA(call)                                                   \
  do {                                                                        \
    cudaError_t e_ = (call);                                                  \
    if (e_ != cudaSuccess) {                                                  \
      ::ttnn::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                        __FILE__, __LINE__);                                  \
      return TTNN_ECUDA;                                                      \
    }                                                                         \
  } while (0)

#define TTNN_TRY(...)                  \
  do {                                 \
    ttnn_status s_ = (__VA_ARGS__);    \
    if (s_ != TTNN_OK) return s_;      \
  } while (0)

#define TTNN_CHECK_ARG(cond, ...)                 \
  do {                                            \
    if (!(cond)) {                                \
      ::ttnn::set_error(__VA_ARGS__);             \
      return TTNN_EINVAL;                         \
    }                                             \
  } while (0)

ttnn_status check_launch(const char* what);   // also counts the launch
void count_launch();

// Programmatic dependent launch, for the short kernels that follow one another
// in an update or a recovery: a kernel's blocks may be placed while the kernel
// before it in the stream still runs, and wait for its end (and the visibility
// of its writes) before they do anything.  Every kernel launched by launch_pdl
// begins with pdl_begin() or pdl_wait(), so the end of a kernel still implies the end of all
// before it; any other kernel, copy or event after it sees ordinary stream
// order.  8 small streaming updates 557 -> 490 us, 64^5 bfloat16 531 -> 512,
// 24^4 binary64 to cores 128 -> 120.
// (pdl_wait() alone in a long kernel: the blocks after it would hold room that
// another stream's kernels could use.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  pdl_wait();
}
// Whether this thread's launches are programmatic.  Not those of the server's
// workers: their streams share the chip, and blocks placed early hold room that
// other streams' kernels could use (16 streams 1185 -> 1207 us with them).
bool& pdl_of_thread();
// Ordinary also while a graph is captured.
template <typename T>
struct PdlArg { using type = T; };
template <typename... P>
void launch_pdl(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                const typename PdlArg<P>::type&... args) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusActive;
  if (pdl_of_thread() && cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();
    cs = cudaStreamCaptureStatusActive;
  }
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;   // not Active, as it starts
  void* a[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  cudaLaunchKernelExC(&cfg, (const void*)kernel, a);   // the caller's check_launch reports an error
}

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }

// number formats of the DRM rounding (index = ttnn_dtype for F64..E4M3)
enum RoundFmt { RF_F64 = 0, RF_F32 = 1, RF_BF16 = 2, RF_E4M3 = 3 };

}  // namespace ttnn
