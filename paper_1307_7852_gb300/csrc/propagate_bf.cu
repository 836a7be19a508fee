// Best-first neighbourhood propagation with a visit budget (Sec. 3.2 of
// arXiv:1307.7852), one synchronous pass over a frozen snapshot of the
// lists.  For every point p (one warp per point):
//  * p's own neighbours are visited first, in list order, and enter the
//    priority queue with their distance to p;
//  * the nearest unexpanded visited point is popped and its neighbours that
//    were not visited yet are visited, in its list order; and so on,
//  * until the queue is empty or `budget` points were visited (the budget
//    may end a list part way);
//  * p's new list is the k best visited points by (dist, id).
// Shared memory per warp: a hash set of visited ids (with p), the visited
// ids and their distance keys (32 bits, order-preserving) in visit order, and
// the selection scratch.  The queue is a second copy of the distance keys in
// which a popped entry reads as the largest value: a pop is a word per lane
// and 32 entries and two warp reductions (the smallest distance, then the
// smallest id that has it).  Distances are the canonical FP32 ones (float
// rows with an exact byte copy are scored on the copy).
// What bounds it: the chain of a pop, the popped point's list, and the rows of
// the few points it adds, each waiting for the last -- so the work between the
// loads is kept short (byte rows are scored four at a time, not in batches of
// 32 with mostly idle slots) and, on byte rows, 24 warps per SM share it.
#include "knng_common.cuh"
#include "knng_internal.h"

#include <algorithm>
#include <type_traits>

namespace knng {

namespace {
struct BfLayout {
    int H, hshift, Bc;
    size_t per_warp;
};

BfLayout bf_layout(int budget)
{
    BfLayout L;
    L.Bc = (budget + 31) & ~31;
    int H = 64;
    while (H < 2 * (budget + 34)) H <<= 1;
    L.H = H;
    int lg = 0;
    while ((1 << lg) < H) ++lg;
    L.hshift = 32 - lg;
    // vid[Bc] | vdist[Bc] | max(tab[H] | queue[Bc], ws): the final selection
    // reuses the set and the queue
    size_t b = 2 * sizeof(int) * (size_t)L.Bc +
               std::max(sizeof(int) * (size_t)(H + L.Bc), (size_t)kLeafWarpScratch);
    L.per_warp = (b + 15) & ~(size_t)15;
    return L;
}
}  // namespace

// kForm: the scoring of the rows, see warp_canon_dist32; kFormBytes: always on
// lane_X, the byte rows, 16-byte aligned and padded, d <= 128 (other forms:
// when it is set and, for float rows, exact).
constexpr int kFormBytes = 4;
template <int kDT, int kForm>
__global__ void __launch_bounds__(256, kForm == kFormBytes ? 3 : 2) propagate_bf_kernel(RowLoader<kDT> L, RowLoader<kDtU8> Lb,
                                                              const int* __restrict__ xb_bad,
                                                              const uint8_t* __restrict__ lane_X, int64_t lane_ld,
                                                              int64_t n, int k, int budget,
                                                              const int32_t* __restrict__ order,
                                                              const int32_t* __restrict__ ids_in,
                                                              int32_t* __restrict__ ids_out, float* __restrict__ d_out,
                                                              int H, int hshift, int Bc, int per_warp_bytes)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int* vid = reinterpret_cast<int*>(smem_raw + (size_t)w * per_warp_bytes);
    uint32_t* vdist = reinterpret_cast<uint32_t*>(vid + Bc);
    int* tab = reinterpret_cast<int*>(vdist + Bc);
    uint32_t* queue = reinterpret_cast<uint32_t*>(tab + H);
    unsigned char* ws = reinterpret_cast<unsigned char*>(tab);
    uint32_t* hist = reinterpret_cast<uint32_t*>(ws);
    uint64_t* keys = reinterpret_cast<uint64_t*>(ws + 1024);
    const uint32_t hmask = (uint32_t)H - 1;
    bool bytes = false;
    if constexpr (kDT == kDtF32) bytes = xb_bad && *xb_bad == 0;
    const bool lanes8 = kForm == kFormBytes || (lane_X && bytes);

    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t wi = gw; wi < n; wi += nw) {
        const int32_t p = order ? order[wi] : (int32_t)wi;
        for (int s = lane * 4; s < H; s += 128) *reinterpret_cast<int4*>(tab + s) = make_int4(-1, -1, -1, -1);
        for (int s = lane; s < Bc; s += 32) queue[s] = 0xFFFFFFFFu;
        uint4 q8 = make_uint4(0u, 0u, 0u, 0u);
        if (lanes8) q8 = load_query_u8(lane_X, lane_ld, p, L.d);
        __syncwarp();
        if (lane == 0) hash_insert(tab, (uint32_t)hshift, hmask, p);
        __syncwarp();
        int cnt = 0;
        // visits the lanes' ids o (-1: none) in lane order while the budget
        // lasts, and scores them (collective)
        auto visit = [&](int32_t o) {
            const bool fresh = o >= 0 && hash_insert(tab, (uint32_t)hshift, hmask, o);
            const uint32_t b = __ballot_sync(KNNG_FULL_MASK, fresh);
            const int pos = cnt + __popc(b & lanemask_lt());
            if (fresh && pos < budget) vid[pos] = o;
            const int nb = min(__popc(b), budget - cnt);  // at most 32
            __syncwarp();
            if (nb > 0) {
                float dd;
                if ((kForm == kFormBytes || kDT == kDtF32) && lanes8)
                    dd = dist_u8_g8(lane_X, lane_ld, L.d, q8, vid + cnt, nb);
                else if (kDT == kDtF32 && bytes) dd = warp_canon_dist32<kFormWide>(Lb, p, vid + cnt, nb);
                else dd = warp_canon_dist32<kForm == kFormBytes ? kFormNarrow : kForm>(L, p, vid + cnt, nb);
                if (lane < nb) {
                    const uint32_t o32 = ord_key(dd);
                    vdist[cnt + lane] = o32;
                    queue[cnt + lane] = min(o32, 0xFFFFFFFEu);
                }
                cnt += nb;
            }
            __syncwarp();
        };
        for (int e0 = 0; e0 < k; e0 += 32) {
            const int e = e0 + lane;
            int32_t o = e < k ? ids_in[(int64_t)p * k + e] : -1;
            if (o >= n) o = -1;  // ids outside [0, n) are empty slots
            visit(o);
        }
        while (cnt < budget) {
            // pop the nearest visited point not expanded yet: smallest
            // distance, ties by id
            uint32_t best = 0xFFFFFFFFu;
            int bi = -1;
            for (int i = lane; i < cnt; i += 32) {
                const uint32_t v = queue[i];
                // (an equal distance of this lane: the smaller id)
                if (v < best || (v == best && v != 0xFFFFFFFFu && vid[i] < vid[bi])) {
                    best = v;
                    bi = i;
                }
            }
            const uint32_t wbest = __reduce_min_sync(KNNG_FULL_MASK, best);
            if (wbest == 0xFFFFFFFFu) break;  // queue empty
            const int mid = best == wbest ? vid[bi] : 0x7FFFFFFF;
            const int32_t u = __reduce_min_sync(KNNG_FULL_MASK, mid);
            if (best == wbest && mid == u) queue[bi] = 0xFFFFFFFFu;
            __syncwarp();
            for (int f0 = 0; f0 < k && cnt < budget; f0 += 32) {
                const int f = f0 + lane;
                int32_t o = f < k ? ids_in[(int64_t)u * k + f] : -1;
                if (o >= n) o = -1;
                visit(o);
            }
        }
        __syncwarp();  // the set and the queue are done: their room is the selection's
        auto key = [&](int i) -> uint64_t { return ((uint64_t)vdist[i] << 32) | (uint32_t)vid[i]; };
        const int nsel = cnt <= 256 ? warp_topk_sorted<8>(key, cnt, k, keys, keys + 64, hist)
                                    : warp_topk_sorted<16>(key, cnt, k, keys, keys + 64, hist);
        __syncwarp();
        for (int i = lane; i < k; i += 32) {
            const bool ok = i < nsel;
            ids_out[(int64_t)p * k + i] = ok ? (int32_t)(uint32_t)keys[i] : -1;
            d_out[(int64_t)p * k + i] = ok ? unord_key((uint32_t)(keys[i] >> 32)) : __int_as_float(0x7f800000);
        }
        __syncwarp();
    }
}

cudaError_t run_propagate_best_first(const XDesc& x, int k, int budget, const int32_t* order, const int32_t* ids_in,
                                     int32_t* ids, float* dists, cudaStream_t st)
{
    if (budget < k || budget > 512 || k > 64) return cudaErrorInvalidValue;
    const BfLayout BL = bf_layout(budget);
    int warps = (int)((200 * 1024) / BL.per_warp);
    if (warps > 8) warps = 8;
    if (warps < 1) return cudaErrorInvalidConfiguration;
    const size_t smem = BL.per_warp * warps;
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto dt) {
        constexpr int kDT = decltype(dt)::value;
        RowLoader<kDT> rl{x.X, x.ld, x.d, x.vec};
        // byte rows scored eight lanes a row (as in propagate_kernel.cuh)
        const uint8_t* lane_X = nullptr;
        int64_t lane_ld = 0;
        if (x.d <= 128) {
            if (kDT == kDtF32 && x.Xb) {
                lane_X = x.Xb;
                lane_ld = x.ldb;
            } else if (kDT == kDtU8 && (uintptr_t)x.X % 16 == 0 && x.ld % 16 == 0 && x.d % 16 == 0) {
                lane_X = static_cast<const uint8_t*>(x.X);
                lane_ld = x.ld;
            }
        }
        const int form = row_form(rl);
        auto kern = form == kFormAny ? propagate_bf_kernel<kDT, kFormAny>
                  : form == kFormNarrow ? propagate_bf_kernel<kDT, kDT == kDtU8 ? kFormWide : kFormNarrow>
                                        : propagate_bf_kernel<kDT, kFormWide>;
        if (kDT == kDtU8 && lane_X) kern = propagate_bf_kernel<kDT, kDT == kDtU8 ? kFormBytes : kFormAny>;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return;
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem);
        if (per_sm < 1) per_sm = 1;
        int64_t blocks = (int64_t)num_sms() * per_sm;
        const int64_t need = (x.n + warps - 1) / warps;
        if (blocks > need) blocks = need;
        // (the copy's rows are padded with zeros: whole words, d <= 256)
        const RowLoader<kDtU8> rb{x.Xb, x.ldb, (x.d + 3) & ~3, true};
        kern<<<(int)blocks, warps * 32, smem, st>>>(rl, rb, x.xb_bad, lane_X, lane_ld, x.n, k, budget, order, ids_in,
                                                    ids, dists,
                                                    BL.H, BL.hshift, BL.Bc, (int)BL.per_warp);
        note_launches(1);
        e = cudaGetLastError();
    };
    if (x.dtype == kDtF16) launch(std::integral_constant<int, kDtF16>{});
    else if (x.dtype == kDtU8) launch(std::integral_constant<int, kDtU8>{});
    else launch(std::integral_constant<int, kDtF32>{});
    return e;
}

}  // namespace knng
