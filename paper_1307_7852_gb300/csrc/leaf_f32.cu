// Leaf graphs, FP32 candidate stage (Sec. 3.1 of arXiv:1307.7852): dispatch
// to the per-element-type instantiations of the kernels (leaf_f32_kernels.cuh).
#include <algorithm>

#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

constexpr int kCandCap = 128;  // candidates per row of the kernel that rescores by itself

template <int kDT>
cudaError_t leaf_f32_full(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm, int k,
                          int kp, int32_t* ids, float* dists, cudaStream_t st);
template <int kDT, bool kAsync>
cudaError_t leaf_f32_cand(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm, int kp,
                          uint16_t* cand, cudaStream_t st);

cudaError_t run_leaf_knn_f32(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T,
                             const int32_t* perm, int k, int kp, int32_t* ids, float* dists, Arena& ar,
                             cudaStream_t st)
{
    if (kp > kCandCap) kp = kCandCap;
    if (!ar.lean && leaf_rescore_staged_ok(kp, P.max_leaf)) {
        // (eight more: the rescoring reads whole groups of eight)
        uint16_t* cand = ar.take<uint16_t>((size_t)T * x.n * kp + 8);
        if (!ar.base) return cudaSuccess;
        cudaError_t e;
        if (x.dtype == kDtF16) e = leaf_f32_cand<kDtF16, false>(x, P, dp, T, perm, kp, cand, st);
        else if (x.dtype == kDtU8) e = leaf_f32_cand<kDtU8, false>(x, P, dp, T, perm, kp, cand, st);
        else if (x.vec && x.ld % 4 == 0) e = leaf_f32_cand<kDtF32, true>(x, P, dp, T, perm, kp, cand, st);
        else e = leaf_f32_cand<kDtF32, false>(x, P, dp, T, perm, kp, cand, st);
        if (e != cudaSuccess) return e;
        return run_leaf_rescore_staged(x, P, dp, T, perm, nullptr, cand, kp, k, ids, dists, st);
    }
    if (!ar.base) return cudaSuccess;
    if (x.dtype == kDtF16) return leaf_f32_full<kDtF16>(x, P, dp, T, perm, k, kp, ids, dists, st);
    if (x.dtype == kDtU8) return leaf_f32_full<kDtU8>(x, P, dp, T, perm, k, kp, ids, dists, st);
    return leaf_f32_full<kDtF32>(x, P, dp, T, perm, k, kp, ids, dists, st);
}

}  // namespace knng
