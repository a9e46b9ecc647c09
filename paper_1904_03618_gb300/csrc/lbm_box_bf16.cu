// Box form of the fused step for __nv_bfloat16 population storage (a translation unit of
// its own so that it compiles in parallel with the other kernels).
#include "lbm_fused_box.cuh"

namespace lbm {
template cudaError_t launch_fused_box_storage<__nv_bfloat16>(const void*, void*, const StepArgs&, int,
                                                   cudaStream_t);
}  // namespace lbm
