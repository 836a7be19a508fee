// First-order propagation on half rows (propagate_kernel.cuh).
#include "propagate_kernel.cuh"

namespace knng {
template cudaError_t prop_dispatch<kDtF16>(const XDesc&, int, const int32_t*, const int32_t*, const float*,
                                           const unsigned long long*, int32_t*, float*, unsigned long long*,
                                           const PairOffers&, const uint8_t*, cudaStream_t, unsigned long long*);
}  // namespace knng
