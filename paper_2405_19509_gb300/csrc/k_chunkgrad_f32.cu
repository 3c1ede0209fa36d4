// Chunk-gradient kernels for fp32 rows, slices on 16-byte boundaries.
#include "k_chunkgrad.cuh"

namespace gc {
namespace cg {
Kernel pick_f32(int CL, int NT, int NVT) { return pick_cl<float, true>(CL, NT, NVT); }
}  // namespace cg
}  // namespace gc
