// Chunk-gradient kernels for fp32 rows, slices at any element.
#include "k_chunkgrad.cuh"

namespace gc {
namespace cg {
Kernel pick_f32_ragged(int CL, int NT, int NVT) { return pick_cl<float, false>(CL, NT, NVT); }
}  // namespace cg
}  // namespace gc
