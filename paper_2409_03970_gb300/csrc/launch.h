// Dependent kernel launches, shared by the translation units of libnsort.
#pragma once

#include <cuda_runtime.h>

#include <cstdlib>

namespace nsort {

// Launches a kernel with programmatic stream serialisation: the launch is
// processed while the previous kernel of the stream still runs and its CTAs
// start as soon as that kernel completes, which hides the launch latency
// between the dependent kernels of a sort (about 20% of a 2^20-key sort, 1%
// at 2^28).  Every kernel so launched calls pdl_wait() before it reads or
// writes anything the previous kernels touch.  NSORT_NO_PDL=1 in the
// environment selects plain launches.
inline bool pdl_enabled() {
  static const bool on = [] {
    const char *e = getenv("NSORT_NO_PDL");
    return !(e && e[0] == '1');
  }();
  return on;
}

// CLUSTER: CTAs of a thread-block cluster.
template <int CLUSTER = 1, typename... KArgs, typename... Args>
void launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem,
                cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CLUSTER;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CLUSTER > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace nsort
