// Seeding and trace kernels of 8-wide trees (trace.cuh).
#include "trace.cuh"

namespace tpmc {

TraceKernel trace_kernel_w8(uint32_t variant, uint32_t block, uint32_t blocks_per_sm) {
  return pick_trace_w<8>(variant, block, blocks_per_sm);
}

cudaError_t launch_seed_w8(const TraceArgs& args, cudaStream_t stream) {
  return launch_seed_w<8>(args, stream);
}

}  // namespace tpmc
