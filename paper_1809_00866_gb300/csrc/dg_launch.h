// Kernel launches that overlap their start with the end of the kernel before them in the stream
// (programmatic dependent launch): the grid's CTAs become resident while that kernel's last ones
// run, and wait_previous(), the first statement of every kernel launched this way, holds them until
// all of its work is complete and visible. Nothing a kernel reads or writes comes before that
// statement, so the order of the stream is what it was; a kernel launched in the ordinary way, a
// copy, or an event still waits for the whole kernel ahead of it. At most two kernels are resident at
// a time, since a kernel lets its own successor start only once its wait is over.
//
// Only for grids of at most one CTA per SM, launched into a stream: a Jacobian action at 4^3 P2 22.5 -> 17.7 us,
// an FGMRES stage there 3.66 -> 2.73 ms, a training gradient of 16384 samples 32.8 -> 29.2 us. A grid that
// fills the GPU lands unevenly when its CTAs take the places the kernel before it leaves (a Jacobian action at
// 16^3 P4 206 -> 238 us). Captured into the graphs of a plan such edges cost more than they hide (a stage at
// 12^3 P3 in FP64 22.6 -> 29.0 ms, of 16 small boxes 46.0 -> 49.5 ms). Elsewhere the launch is an ordinary one,
// and the wait returns at once.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace dg {

template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  static const unsigned sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return static_cast<unsigned>(n);
  }();
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool small = grid.x * grid.y * grid.z <= sms && cudaStreamIsCapturing(st, &cap) == cudaSuccess &&
                     cap == cudaStreamCaptureStatusNone;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = small ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);  // errors: cudaGetLastError, as after <<<>>>
}

// True always; kernels begin with `if (!wait_previous()) return;`, a branch that also keeps loads of
// constant memory, which a compiler may move across statements, below the wait.
__device__ __forceinline__ bool wait_previous() {
  unsigned on;
  asm volatile(
      "griddepcontrol.wait;\n\t"
      "griddepcontrol.launch_dependents;\n\t"
      "mov.u32 %0, 1;"
      : "=r"(on)::"memory");
  return on != 0;
}

}  // namespace dg
