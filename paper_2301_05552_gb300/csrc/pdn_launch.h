// Kernel launch with programmatic dependent launch: the kernel may be scheduled
// while its predecessor on the stream drains, and waits for it on the device
// (griddepcontrol.wait) before it reads anything.  PDN_PDL=0, read once per
// process, launches plainly, with the same results; every such launch of the
// library goes through here, so that the switch rules out all of that overlap.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>

namespace pdn {

inline bool pdl_on() {
  static const bool on = [] {
    const char *e = std::getenv("PDN_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), int64_t grid, int block, size_t smem, cudaStream_t s, const Args &...args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = pdl_on() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace pdn
