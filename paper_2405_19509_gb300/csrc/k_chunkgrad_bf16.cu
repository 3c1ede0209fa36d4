// Chunk-gradient kernels for bf16 rows, slices on 16-byte boundaries.
#include "k_chunkgrad.cuh"

namespace gc {
namespace cg {
Kernel pick_bf16(int CL, int NT, int NVT) { return pick_cl<__nv_bfloat16, true>(CL, NT, NVT); }
}  // namespace cg
}  // namespace gc
