// Launches of kernels that follow one another on a stream: programmatic
// dependent launches.  A kernel of such a chain may become resident while its
// predecessor still runs (once every CTA of it has called grid_next()), so its
// launch latency and its set-up (shared memory, barriers, tensor memory)
// overlap the predecessor; grid_wait() then waits until everything before it on
// the stream is complete and visible.  Short kernels call grid_next() first
// thing, the persistent products at their end (waiting CTAs beside a running
// product slowed it).
//
// A product is itself chained only while it is short (kChainChunks k-chunks a
// CTA, about 40 us): chained, the XXZ m = 512 operator in 3xTF32 takes 37.6 us instead of
// 43.0, the Hubbard m = 1024 one in FP64 113 instead of 117 and the FP64 eigensolver 6.38 ms
// instead of 6.48 (an expansion 66 instead of 63), but the cylinder's products slow
// down (environment 991 instead of 917 us), whose launch latency does not count.  Every
// kernel launched this way calls grid_wait() before its first access to global
// memory, whatever the data: the chain stays ordered as plain launches would be.
// Pointers that a predecessor may write through are not declared __restrict__: a
// load from a const __restrict__ pointer counts as invariant for the whole kernel,
// and the compiler may move it before the wait.
#pragma once

#include <cuda_runtime.h>

namespace dmrg3s {

constexpr int kChainChunks = 16;

#ifdef __CUDACC__
__device__ __forceinline__ void grid_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// While one of these exists, the thread's launches are plain (inside a captured
// graph: the replays of chained nodes measured slower than plain ones).
struct PlainLaunches {
  static bool& on() {
    static thread_local bool v = false;
    return v;
  }
  bool before = on();
  explicit PlainLaunches(bool plain = true) { on() = before || plain; }
  ~PlainLaunches() { on() = before; }
  PlainLaunches(const PlainLaunches&) = delete;
  PlainLaunches& operator=(const PlainLaunches&) = delete;
};

template <class... P, class... A>
void launch_chain(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                  A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = PlainLaunches::on() ? 0 : 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

}  // namespace dmrg3s
