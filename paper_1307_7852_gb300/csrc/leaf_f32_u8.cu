// FP32 leaf graphs of byte rows (leaf_f32_kernels.cuh).
#include "leaf_f32_kernels.cuh"

namespace knng {
template cudaError_t leaf_f32_full<kDtU8>(const XDesc&, const TreePlan&, const DevPlan&, int, const int32_t*, int, int,
                                            int32_t*, float*, cudaStream_t);
template cudaError_t leaf_f32_cand<kDtU8, false>(const XDesc&, const TreePlan&, const DevPlan&, int,
                                                   const int32_t*, int, uint16_t*, cudaStream_t);
}  // namespace knng
