// Launches that overlap the end of the previous kernel in the stream
// (programmatic dependent launch).
//
// A chain of short kernels -- an evaluation of T on a tree of 2,047 nodes is
// 24 of them -- pays for each one's launch, its blocks' start and its first
// loads after the one before has ended.  A kernel launched here may start
// while the previous one still runs; it calls pdl_enter() before it touches
// anything that an earlier kernel writes or reads, and until then may only
// read what no kernel of the chain writes (the factors).  pdl_enter() returns
// when the previous grid has completed and its writes are visible -- which had
// waited for the one before it in the same way -- and lets the next one
// start.  After a kernel or a copy launched otherwise the launch is an
// ordinary one.
#pragma once

#include <cuda_runtime.h>

namespace spock {

__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Ordinary launches while one of these lives on the calling thread (event
// records between the kernels, which time them one by one).
struct PlainLaunches {
  static bool& on() {
    static thread_local bool v = false;
    return v;
  }
  bool before;
  explicit PlainLaunches(bool want) : before(on()) { on() = before || want; }
  ~PlainLaunches() { on() = before; }
};

template <typename... K, typename... A>
inline void launch_pdl(void (*kernel)(K...), int grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute a[1];
  a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = a;
  c.numAttrs = PlainLaunches::on() ? 0 : 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<K>(args)...);
}

}  // namespace spock
