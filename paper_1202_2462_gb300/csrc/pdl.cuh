// Programmatic dependent launch for chains of short kernels: a kernel launched so
// starts while its predecessor in the stream still runs, does what does not depend on
// it, and calls pdl_begin() before it reads or writes anything that does.  The wait ends
// when the predecessor has completed, so a chain whose every kernel calls it keeps the
// stream's order; the trigger comes after the wait, so at most one successor is
// early.  Data of the predecessor is read past L1 (__ldcg), which may hold lines from
// before it was written.
#pragma once
#include <cuda_runtime.h>

namespace sapmg {

__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

struct PdlLaunch {
  cudaLaunchAttribute at;
  cudaLaunchConfig_t cfg;
  PdlLaunch(const PdlLaunch&) = delete;
  // early: as above; otherwise an ordinary launch, for which pdl_begin() does nothing
  PdlLaunch(dim3 grid, unsigned threads, size_t smem, cudaStream_t s, bool early) : at{}, cfg{} {
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
  }
};

}  // namespace sapmg
