// Neighbourhood propagation (Sec. 3.2 of arXiv:1307.7852), first-order form:
// dispatch to the per-element-type instantiations of the kernel
// (propagate_kernel.cuh).
#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

template <int kDT>
cudaError_t prop_dispatch(const XDesc& x, int k, const int32_t* order, const int32_t* ids_in, const float* d_in,
                          const unsigned long long* fin, int32_t* ids, float* dists, unsigned long long* fout,
                          const PairOffers& po, const uint8_t* tm, cudaStream_t st, unsigned long long* stats);

cudaError_t run_propagate(const XDesc& x, int k, const int32_t* order, const int32_t* ids_in, const float* d_in,
                          const unsigned long long* flags_in, int32_t* ids, float* dists,
                          unsigned long long* flags_out, cudaStream_t st, const PairOffers* offers,
                          const uint8_t* tmask_in, unsigned long long* stats)
{
    const PairOffers po = offers ? *offers : PairOffers{};
    if (x.dtype == kDtF16)
        return prop_dispatch<kDtF16>(x, k, order, ids_in, d_in, flags_in, ids, dists, flags_out, po, tmask_in, st,
                                     stats);
    if (x.dtype == kDtU8)
        return prop_dispatch<kDtU8>(x, k, order, ids_in, d_in, flags_in, ids, dists, flags_out, po, tmask_in, st,
                                    stats);
    return prop_dispatch<kDtF32>(x, k, order, ids_in, d_in, flags_in, ids, dists, flags_out, po, tmask_in, st, stats);
}

}  // namespace knng
