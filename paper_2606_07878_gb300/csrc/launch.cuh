// Kernel launches of the library's sequences.
#pragma once
#include <cuda_runtime.h>

namespace still {

// Launches a kernel that executes griddep_wait (ptx.cuh), in clusters of `cluster` CTAs when
// cluster > 1. It begins when the CTAs of the stream's previous kernel have exited, before that
// kernel's completion has passed through the stream: its launch and its set-up (barriers, TMEM,
// tensor map fetches) lie under the previous kernel's end. What bounds a call on a short sequence
// is these gaps, 20 launches of a one-block layer and 34 of two blocks without FFN: 1,024 tokens of
// 2 heads of 64 channels 188 -> 144 us, three windows of 1,024 in the lookahead call 1099 -> 858 us,
// 8,003 tokens with biases 1153 -> 1103 us. Letting
// the next kernel begin earlier still (griddepcontrol.launch_dependents at a kernel's head) puts
// its idle CTAs beside the working ones: 164, 921 and 1202 us, and the 32,768-token layer
// slower than unchained (5389 against 5225 us); behind a kernel's last tile it changes nothing.
// The first kernel of a sequence is launched the ordinary way, so that it waits for everything
// the stream holds, whatever the caller's last kernel did about its own predecessors.
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t stream, int cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace still
