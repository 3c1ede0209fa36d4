// Chunk-gradient kernels for bf16 rows, slices at any element.
#include "k_chunkgrad.cuh"

namespace gc {
namespace cg {
Kernel pick_bf16_ragged(int CL, int NT, int NVT) { return pick_cl<__nv_bfloat16, false>(CL, NT, NVT); }
}  // namespace cg
}  // namespace gc
