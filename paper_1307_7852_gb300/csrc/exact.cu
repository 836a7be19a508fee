// Exact k-NN lists (Def. 1 of arXiv:1307.7852) of a set of query points
// against all n points, by brute force with the canonical FP32 distance.
// This is the yardstick of the accuracy measure of Sec. 4 (recall on a
// sample of points), not part of the approximate method.
//
// Two forms with the same result:
//
// exact_knn_kernel (small sets, and queries the other form cannot bound):
// one block of QB warps serves QB queries; candidate rows stream through
// shared memory in tiles of 32 rows, so each row is read once per block.
// Every warp keeps a buffer of keys below its current k-th best and shrinks
// it to the k best (warp radix select) whenever it fills.
//
// The filtered form (run_exact_knn_tc) scores the pairs on the tensor cores
// and computes the canonical distance only of those that can be listed:
//   1. x^ = bfloat16(x) of every row, |x^|^2 and the distance |x - x^|; rows
//      far above the others by either are taken out and listed for every
//      query;
//   2. exact_gram_kernel (minima): D^ = |q^|^2 + |x^|^2 - 2 q^.x^ of every
//      pair (tcgen05, FP32 accumulation), reduced to minima over 64 groups of
//      rows per query and CTA;
//   3. exact_bound_kernel: the (k+1)-th smallest minimum is at least the
//      D^ of k rows other than the query.  With e a bound of the error of D^
//      and s = |q - q^| + max |x - x^|, k rows are within
//      U = sqrt(D^ + e) + s of the query, so a row of the answer has
//      D^ <= (U + s)^2 + e (with the relative error of the canonical
//      distance on top);
//   4. exact_gram_kernel (lists): the same products again (cheaper than
//      storing n values per query), rows up to that bound listed per query
//      (a few tens on descriptor data);
//   5. exact_rescore_kernel: canonical distances of the listed rows, the k
//      best by (distance, id).
// Queries whose list overflows or whose own row is a far one, and all of them
// when more rows are not finite than can be taken out or a bounded wait gave
// up, are answered by exact_knn_kernel.  One row 300 times longer than the
// rest (2,000 queries of 200,000 x 128): 52.7 -> 0.6 ms.  What the bounds
// cannot help (more than 1,024 rows nearly as near as the k-th, rows far from
// the origin for their spread) costs the passes beside the direct kernel: 12 %
// at 2,048 rows and 10 queries, 3 % at 16,384 and 1,000, 1 % at 200,000.
// 10,000 queries of 1,000,000 x 128 rows, k = 20: 788 ms with exact_knn_kernel
// alone (seven shuffles per pair and 128 entries), 6.9 ms filtered.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "knng_common.cuh"
#include "knng_internal.h"
#include "tc_ptx.cuh"

namespace knng {

namespace {
constexpr int kQB = 8;  // queries (warps) per block
}

template <int kDT>
__global__ void __launch_bounds__(kQB * 32) exact_knn_kernel(RowLoader<kDT> L, int64_t n,
                                                             const int32_t* __restrict__ queries, int nq,
                                                             int k, int cap, int32_t* __restrict__ out_ids,
                                                             float* __restrict__ out_d,
                                                             const uint8_t* __restrict__ need)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // with need, only the queries marked there are answered
    if (need) {
        const int qn = blockIdx.x * kQB + (int)threadIdx.x;
        if (__syncthreads_or(threadIdx.x < kQB && qn < nq && need[qn] != 0) == 0) return;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int dp = (L.d + 3) & ~3;
    // shared memory: tile[32][dp] | qrow[kQB][dp] | buf[kQB][cap] | hist[kQB][256] | sel[kQB][64]
    float* tile = reinterpret_cast<float*>(smem_raw);
    float* qrow = tile + 32 * dp;
    unsigned long long* buf_all = reinterpret_cast<unsigned long long*>(qrow + kQB * dp);
    uint32_t* hist_all = reinterpret_cast<uint32_t*>(buf_all + (size_t)kQB * cap);
    int* sel_all = reinterpret_cast<int*>(hist_all + 256 * kQB);
    unsigned long long* buf = buf_all + (size_t)w * cap;
    uint32_t* hist = hist_all + 256 * w;
    int* sel = sel_all + 64 * w;

    const int qi = blockIdx.x * kQB + w;
    const int32_t qraw = qi < nq ? queries[qi] : 0;
    const bool valid = qraw >= 0 && qraw < n;  // an out-of-range query gets an empty row
    const bool wanted = qi < nq && (!need || need[qi] != 0);
    const bool active = wanted && valid;
    const int32_t q = valid ? qraw : 0;
    for (int j = 4 * lane; j < dp; j += 128) {
        const float4 v = L.load4(q, j);
        *reinterpret_cast<float4*>(qrow + w * dp + j) = v;
    }
    unsigned long long thr = kKeyMax;
    int nb = 0;
    for (int64_t j0 = 0; j0 < n; j0 += 32) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < 32 * (dp / 4); idx += kQB * 32) {
            const int r = idx / (dp / 4), c = 4 * (idx % (dp / 4));
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j0 + r < n) v = L.load4(j0 + r, c);
            *reinterpret_cast<float4*>(tile + r * dp + c) = v;
        }
        __syncthreads();
        if (!active) continue;
        unsigned long long mine = kKeyMax;
        const int rows = (n - j0) < 32 ? (int)(n - j0) : 32;
        for (int r = 0; r < rows; ++r) {
            // the canonical distance (blocks of 32 entries added in order)
            float tot = 0.f;
            for (int c0 = 0; c0 < L.d; c0 += 128) {
                const int j = c0 + 4 * lane;
                float s = 0.f;
                if (j < dp) {
                    const float4 a = *reinterpret_cast<const float4*>(qrow + w * dp + j);
                    const float4 b = *reinterpret_cast<const float4*>(tile + r * dp + j);
                    float t;
                    t = a.x - b.x; s = fmaf(t, t, s);
                    t = a.y - b.y; s = fmaf(t, t, s);
                    t = a.z - b.z; s = fmaf(t, t, s);
                    t = a.w - b.w; s = fmaf(t, t, s);
                }
                s += __shfl_xor_sync(KNNG_FULL_MASK, s, 4);
                s += __shfl_xor_sync(KNNG_FULL_MASK, s, 2);
                s += __shfl_xor_sync(KNNG_FULL_MASK, s, 1);
                tot = chunk_blocks_add(tot, s);
            }
            if (lane == r && j0 + r != q) mine = pack_key(tot, (uint32_t)(j0 + r));
        }
        const bool take = mine < thr;
        const uint32_t b = __ballot_sync(KNNG_FULL_MASK, take);
        if (take) buf[nb + __popc(b & lanemask_lt())] = mine;
        nb += __popc(b);
        if (nb > cap - 32) {
            __syncwarp();
            auto key = [&](int i) -> uint64_t { return buf[i]; };
            const uint64_t t2 = warp_select_threshold(key, nb, k, hist);
            const int m = warp_compact_le(key, nb, t2, sel);
            __syncwarp();
            unsigned long long keep0 = lane < m ? buf[sel[lane]] : kKeyMax;
            unsigned long long keep1 = lane + 32 < m ? buf[sel[lane + 32]] : kKeyMax;
            __syncwarp();
            if (lane < m) buf[lane] = keep0;
            if (lane + 32 < m) buf[lane + 32] = keep1;
            nb = m;
            thr = t2;
            __syncwarp();
        }
    }
    if (!wanted) return;
    if (!valid) nb = 0;
    __syncwarp();
    auto key = [&](int i) -> uint64_t { return buf[i]; };
    const int want = min(k, nb);
    int m = 0;
    if (want > 0) {
        const uint64_t t2 = warp_select_threshold(key, nb, want, hist);
        m = warp_compact_le(key, nb, t2, sel);
    }
    __syncwarp();
    uint64_t v[2];
    v[0] = 2 * lane < m ? buf[sel[2 * lane]] : kKeyMax;
    v[1] = 2 * lane + 1 < m ? buf[sel[2 * lane + 1]] : kKeyMax;
    warp_bitonic_sort<2>(v);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = 2 * lane + e;
        if (i < k) {
            const bool ok = i < m;
            out_ids[(int64_t)qi * k + i] = ok ? (int32_t)(uint32_t)v[e] : -1;
            out_d[(int64_t)qi * k + i] = ok ? unord_key((uint32_t)(v[e] >> 32)) : __int_as_float(0x7f800000);
        }
    }
}

cudaError_t run_exact_knn(const XDesc& x, const int32_t* queries, int nq, int k, int32_t* ids,
                          float* dists, cudaStream_t st, const uint8_t* need)
{
    const int dp = (x.d + 3) & ~3;
    const int cap = 4 * k + 64;
    const size_t smem = sizeof(float) * (size_t)(32 + kQB) * dp + sizeof(unsigned long long) * (size_t)kQB * cap +
                        sizeof(uint32_t) * 256 * kQB + sizeof(int) * 64 * kQB;
    if (smem > 220 * 1024) return cudaErrorInvalidConfiguration;
    const int grid = (nq + kQB - 1) / kQB;
    auto launch = [&](auto dt) {
        constexpr int kDT = decltype(dt)::value;
        auto kern = exact_knn_kernel<kDT>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        RowLoader<kDT> rl{x.X, x.ld, x.d, x.vec};
        kern<<<grid, kQB * 32, smem, st>>>(rl, x.n, queries, nq, k, cap, ids, dists, need);
        note_launches(1);
    };
    if (x.dtype == kDtF16) launch(std::integral_constant<int, kDtF16>{});
    else if (x.dtype == kDtU8) launch(std::integral_constant<int, kDtU8>{});
    else launch(std::integral_constant<int, kDtF32>{});
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The filtered form
// ---------------------------------------------------------------------------
namespace {
constexpr int kTileM = 128;         // queries per tile
constexpr int kTileN = 256;         // rows per tile
constexpr int kGramStages = 4;
constexpr int kGramThreads = 320;   // copy warp, MMA warp, eight epilogue warps
constexpr int kBatchQ = 16384;      // queries per batch: fewer row tiles than SMs, so that
                                    // every query's rows are split over at least two CTAs
constexpr int kListMax = 1024;      // listed rows per query
constexpr int kRescoreWarps = 4;
constexpr long long kExactWait = 2000000000LL;  // ~1 s at GB300 clocks: the default limit of the
                                                // waits, and the limit of the drains

// The bounds use the largest |x - x^| and |x^|^2 over the rows, so rows far
// above the others (and rows that are not finite) are taken out: at most
// kFarRows by either measure.  They are listed for every query instead.
constexpr int kFarRows = 64;
constexpr int kUnusable = 255;  // histogram bin of rows that no bound holds for

// Over the rows: histograms of the exponents of |x^|^2 and |x - x^|; the rows
// taken out and the largest values of the others (as order-preserving words
// of non-negative floats); bad: more unusable rows than can be taken out.
struct ExactStats {
    uint32_t max_err;
    uint32_t max_nrm;
    uint32_t bad;
    uint32_t nfar;
    uint32_t gave_up;  // a bounded wait of this call's passes
    int32_t far[2 * kFarRows];
    uint32_t nrm_hist[256];
    uint32_t err_hist[256];
};
}  // namespace

// kLanes lanes a row: bfloat16 copy (rows of dq entries, zeros past d), squared
// norm of the copy, distance to it.  Norms of unusable rows and of the padding
// rows are +inf: neither pass finds them.
// kLanes: lanes a row, 16 for rows of one K slice (10 queries of 500,000 x 64
// bytes: 266 -> 234 us).
template <int kDT, int kLanes>
__global__ void __launch_bounds__(256) exact_quant_kernel(RowLoader<kDT> L, int64_t n, int64_t n_pad, int dq,
                                                          __nv_bfloat16* __restrict__ Xq, float* __restrict__ nrm,
                                                          float* __restrict__ err)
{
    const int lane = threadIdx.x & (kLanes - 1);
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kLanes;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) / kLanes;
    // (n_pad and nw are even: a warp's groups go round together)
    for (int64_t r = gw; r < n_pad; r += nw) {
        const int64_t row = r < n ? r : n - 1;  // (padding: the last row once more)
        float s = 0.f, e = 0.f;
        __nv_bfloat16* o = Xq + row * dq;
        for (int j = 4 * lane; j < dq; j += 4 * kLanes) {
            float4 v = j < L.d ? L.load4(row, j) : make_float4(0.f, 0.f, 0.f, 0.f);
            const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
            const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
            s = fmaf(fa.x, fa.x, s); s = fmaf(fa.y, fa.y, s);
            s = fmaf(fb.x, fb.x, s); s = fmaf(fb.y, fb.y, s);
            float t;
            t = v.x - fa.x; e = fmaf(t, t, e);
            t = v.y - fa.y; e = fmaf(t, t, e);
            t = v.z - fb.x; e = fmaf(t, t, e);
            t = v.w - fb.y; e = fmaf(t, t, e);
            uint2 u;
            u.x = *reinterpret_cast<const uint32_t*>(&a);
            u.y = *reinterpret_cast<const uint32_t*>(&b);
            *reinterpret_cast<uint2*>(o + j) = u;
        }
#pragma unroll
        for (int q = kLanes / 2; q >= 1; q >>= 1) {
            s += __shfl_xor_sync(KNNG_FULL_MASK, s, q);
            e += __shfl_xor_sync(KNNG_FULL_MASK, e, q);
        }
        if (r >= n) {
            if (lane == 0) nrm[r] = __int_as_float(0x7f800000);
            continue;
        }
        // (rounded up: the sum's relative error is below (d / 32 + 8) 2^-24,
        // and squares that underflow lose d 2^-149 <= 2^-138 in all)
        e = sqrtf(e) * 1.0001f + 0x1p-69f;
        if (lane == 0) {
            // 1e30 also keeps the bounds' squares finite
            nrm[r] = s <= 1e30f && e <= 1e30f ? s : __int_as_float(0x7f800000);
            err[r] = e;
        }
    }
}

// Histograms of the exponents of the norms and errors.  (A kernel of its own:
// counted by the one above, whose rows are a chain of loads and shuffles at
// 32 registers, 1M x 100 took 179 to 222 us there instead of 160.)
__global__ void __launch_bounds__(256) exact_hist_kernel(int64_t n, const float* __restrict__ nrm,
                                                         const float* __restrict__ err, ExactStats* __restrict__ stats)
{
    __shared__ uint32_t hist[512];
    for (int i = threadIdx.x; i < 512; i += 256) hist[i] = 0u;
    __syncthreads();
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        const float s = nrm[r], e = err[r];
        atomicAdd(&hist[s <= 1e30f ? __float_as_uint(s) >> 23 : kUnusable], 1u);
        if (s <= 1e30f) atomicAdd(&hist[256 + (__float_as_uint(e) >> 23)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 512; i += 256)
        if (hist[i]) atomicAdd(i < 256 ? &stats->nrm_hist[i] : &stats->err_hist[i - 256], hist[i]);
}

// One warp: the exponent above which a histogram's rows are taken out.  Those
// above the smallest exponent with at most kFarRows rows past it, if that
// leaves the usable ones at least 2^(gap - 1) times smaller; else unusable
// rows only.
__device__ __forceinline__ int far_cut(const uint32_t* __restrict__ hist, int gap)
{
    const int lane = threadIdx.x & 31;
    uint32_t c[8], sum = 0;
    int top = -1;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        c[b] = hist[8 * lane + b];
        sum += c[b];
        if (c[b] && 8 * lane + b < kUnusable) top = 8 * lane + b;
    }
    top = __reduce_max_sync(KNNG_FULL_MASK, top);
    uint32_t past = sum;  // rows of this lane's bins and above
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(KNNG_FULL_MASK, past, o);
        if (lane + o < 32) past += v;
    }
    past -= sum;
    int least = 256;
#pragma unroll
    for (int b = 7; b >= 0; --b) {
        if (past <= kFarRows) least = 8 * lane + b;
        past += c[b];
    }
    least = __reduce_min_sync(KNNG_FULL_MASK, least);
    return top - least >= gap ? least : kUnusable - 1;
}

// The batch's query rows, packed (rows of row16 16-byte words; zeros past nq
// and for ids out of range).
__device__ __forceinline__ void gather_queries(const uint4* __restrict__ Xq, int64_t n, int row16,
                                               const int32_t* __restrict__ queries, int nq, int rows,
                                               uint4* __restrict__ Aq)
{
    const int64_t total = (int64_t)rows * row16;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / row16), c = (int)(e - (int64_t)r * row16);
        const int32_t q = r < nq ? queries[r] : -1;
        Aq[e] = q >= 0 && q < n ? Xq[(int64_t)q * row16 + c] : make_uint4(0u, 0u, 0u, 0u);
    }
}
__global__ void __launch_bounds__(256) exact_gather_kernel(const uint4* __restrict__ Xq, int64_t n, int row16,
                                                           const int32_t* __restrict__ queries, int nq, int rows,
                                                           uint4* __restrict__ Aq)
{
    gather_queries(Xq, n, row16, queries, nq, rows, Aq);
}

// Takes the far rows out (norm +inf) and finds the largest norm and error of
// the others.  A factor of 8 in the squared norm or of 2 in the error pays for
// kFarRows more rescored rows a query.  Gathers the first batch's queries as
// well (a launch less).
__global__ void __launch_bounds__(256) exact_far_kernel(int64_t n, float* __restrict__ nrm,
                                                        const float* __restrict__ err, ExactStats* __restrict__ stats,
                                                        const uint4* __restrict__ Xq, int row16,
                                                        const int32_t* __restrict__ queries, int nq, int rows,
                                                        uint4* __restrict__ Aq)
{
    gather_queries(Xq, n, row16, queries, nq, rows, Aq);
    __shared__ int cut[2];
    __shared__ uint32_t most[2][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < 2) {
        const int c = w == 0 ? far_cut(stats->nrm_hist, 4) : far_cut(stats->err_hist, 2);
        if (lane == 0) cut[w] = c;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) stats->bad = stats->nrm_hist[kUnusable] > kFarRows ? 1u : 0u;
    __syncthreads();
    float me = 0.f, mn = 0.f;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        const float s = nrm[r], e = err[r];
        const bool usable = s <= 1e30f;
        if (!usable || (int)(__float_as_uint(s) >> 23) > cut[0] || (int)(__float_as_uint(e) >> 23) > cut[1]) {
            const uint32_t at = atomicAdd(&stats->nfar, 1u);
            if (at < 2 * kFarRows) stats->far[at] = (int32_t)r;
            nrm[r] = __int_as_float(0x7f800000);
        } else {
            me = fmaxf(me, e);
            mn = fmaxf(mn, s);
        }
    }
    for (int o = 16; o >= 1; o >>= 1) {
        me = fmaxf(me, __shfl_xor_sync(KNNG_FULL_MASK, me, o));
        mn = fmaxf(mn, __shfl_xor_sync(KNNG_FULL_MASK, mn, o));
    }
    if (lane == 0) {
        most[0][w] = __float_as_uint(me);
        most[1][w] = __float_as_uint(mn);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        uint32_t m = 0u;
        for (int i = 0; i < 8; ++i) m = max(m, most[threadIdx.x][i]);
        atomicMax(threadIdx.x == 0 ? &stats->max_err : &stats->max_nrm, m);
    }
}

// First tile of CTA c when `total` tiles are dealt evenly to G CTAs.
__host__ __device__ __forceinline__ int64_t tile_begin(int64_t total, int G, int c)
{
    return total * c / G;
}

// Products of the query tiles (tile g: queries 128 (g / CT), rows 256 (g mod
// CT)), tiles dealt to the CTAs in contiguous runs.  Warp 0 copies (TMA,
// 128-byte swizzled K slices of 64 entries; the queries' slices stay in
// shared memory over a run when they fit), warp 1 issues the MMAs into two
// 256-column accumulators, warps 2..9 read them back: a thread has one query
// and 128 of the tile's rows.  A tile of 128 entries a row is 1,024 cycles of
// tensor work and about as much of the eight warps' minima, so the two
// overlap; 10,000 queries of 1M x 128 take 3.2 ms for the minima and 3.4 ms
// for the lists (810 and 755 TFLOP/s).
//  kList == false: minima over 32 groups per thread, written per CTA and
//   query tile (slot c + rt of CTA c) to mins[slot][128][64].
//  kList == true: rows with |x^|^2 - 2 q^.x^ <= thr[query] are appended to
//   the query's list, to the end of the tile that fills it: rows that no bound
//   holds back cost the products, not an atomic per pair.  2,000 queries of
//   200,000 x 128 equal rows, which the direct kernel answers in 52.2 ms: 56.7
//   in all with an atomic per pair, 52.6 so.
// A set with too many unusable rows takes the direct kernel: both passes
// return at once (52.7 -> 52.5 ms).
// kPoll: the waits poll without suspending (limits too short for try_wait).
template <bool kList, bool kPoll>
__global__ void __launch_bounds__(kGramThreads, 1) exact_gram_kernel(
    const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, int nK, int RT, int CT,
    bool a_stays, const float* __restrict__ nrm, ExactStats* __restrict__ stats, float* __restrict__ mins,
    const float* __restrict__ thr, int* __restrict__ counts, int32_t* __restrict__ lists, long long limit, int* err)
{
    if (stats->bad) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr int kA = kTileM * 128, kB = kTileN * 128;  // bytes of a K slice
    const int stage_bytes = a_stays ? kB : kA + kB;
    unsigned char* stages = base + (a_stays ? nK * kA : 0);
    float* norms = reinterpret_cast<float*>(stages + kGramStages * stage_bytes);  // [2][256]
    __shared__ __align__(8) uint64_t full[kGramStages], empty[kGramStages], tfull[2], tempty[2], nfull[2], afull;
    __shared__ uint32_t tslot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < kGramStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&tfull[b], 1);
            tc::mbar_init(&tempty[b], 8);
            tc::mbar_init(&nfull[b], 1);
        }
        tc::mbar_init(&afull, 1);
        tc::fence_mbar_init();
        abort_flag = 0;
    }
    if (w == 1) {
        tc::tmem_alloc(&tslot, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tslot;
    const int64_t total = (int64_t)RT * CT;
    const int64_t g0 = tile_begin(total, gridDim.x, blockIdx.x), g1 = tile_begin(total, gridDim.x, blockIdx.x + 1);
    auto give_up = [&]() {
        abort_flag = 1;
        atomicExch(&stats->gave_up, 1u);
        atomicExch(err, 1);
    };
    // a bounded wait that also ends when another warp gave up
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        if (abort_flag) return false;
        if (kPoll) {
            if (tc::mbar_wait(bar, parity, limit)) return true;
        } else {
            // (the first try without a look at the clock: 144 -> 128 us of
            // the minima of 2,000 queries and 200,000 x 128 rows)
            if (tc::mbar_try_wait(bar, parity)) return true;
            const long long t0 = clock64();
            do {
                if (tc::mbar_try_wait(bar, parity)) return true;
            } while (clock64() - t0 <= limit);
        }
        give_up();
        return false;
    };
    if (w == 0) {
        if (lane == 0 && g0 < g1) {
            int64_t it = 0;  // K slices copied
            int rt_cur = -1;
            uint32_t atimes = 0, ntimes = 0;
            bool ok = true;
            int rt = (int)(g0 / CT), ct = (int)(g0 - (int64_t)rt * CT);
            for (int64_t g = g0; g < g1 && ok; ++g) {
                const int64_t lt = g - g0;
                if (a_stays && rt != rt_cur) {
                    // the MMAs of every earlier tile have read the old slices
                    // once the last copied stage was released
                    if (it > 0) ok = wait(&empty[(it - 1) % kGramStages], (uint32_t)((it - 1) / kGramStages) & 1u);
                    if (!ok) break;
                    tc::mbar_arrive_expect_tx(&afull, (uint32_t)(nK * kA));
                    for (int kc = 0; kc < nK; ++kc)
                        tc::tma_load_2d(base + kc * kA, &amap, &afull, kc * 64, rt * kTileM);
                    ++atimes;
                    rt_cur = rt;
                }
                const int b = (int)(lt & 1);
                if (lt >= 2) ok = wait(&tempty[b], (uint32_t)((lt >> 1) - 1) & 1u);
                if (!ok) break;
                tc::mbar_arrive_expect_tx(&nfull[b], kTileN * 4);
                tc::bulk_load(norms + b * kTileN, nrm + (int64_t)ct * kTileN, kTileN * 4, &nfull[b]);
                ++ntimes;
                for (int kc = 0; kc < nK; ++kc, ++it) {
                    const int s = (int)(it % kGramStages);
                    if (it >= kGramStages) ok = wait(&empty[s], (uint32_t)(it / kGramStages - 1) & 1u);
                    if (!ok) break;
                    unsigned char* dst = stages + (size_t)s * stage_bytes;
                    tc::mbar_arrive_expect_tx(&full[s], (uint32_t)stage_bytes);
                    tc::tma_load_2d(dst, &bmap, &full[s], kc * 64, ct * kTileN);
                    if (!a_stays) tc::tma_load_2d(dst + kB, &amap, &full[s], kc * 64, rt * kTileM);
                }
                if (++ct == CT) {
                    ct = 0;
                    ++rt;
                }
            }
            // every copy has landed before the CTA ends (bounded), also when
            // this warp issued all of its own and another one gave up on them
            for (int64_t q = it > kGramStages ? it - kGramStages : 0; q < it; ++q)
                tc::mbar_wait(&full[q % kGramStages], (uint32_t)(q / kGramStages) & 1u, kExactWait);
            for (uint32_t q = ntimes > 2 ? ntimes - 2 : 0; q < ntimes; ++q)
                tc::mbar_wait(&nfull[q & 1u], (q >> 1) & 1u, kExactWait);
            if (atimes) tc::mbar_wait(&afull, (atimes - 1) & 1u, kExactWait);
        }
        __syncwarp();
    } else if (w == 1) {
        if (lane == 0) {
            const uint32_t idesc = tc::make_idesc(1u, kTileM, kTileN);
            int64_t it = 0, done = 0;  // K slices, whole tiles
            int rt_cur = -1;
            uint32_t atimes = 0;
            bool ok = true;
            int rt = (int)(g0 / CT), ct = (int)(g0 - (int64_t)rt * CT);
            for (int64_t g = g0; g < g1 && ok; ++g) {
                const int64_t lt = g - g0;
                if (a_stays && rt != rt_cur) {
                    ok = wait(&afull, atimes & 1u);
                    ++atimes;
                    rt_cur = rt;
                }
                const int b = (int)(lt & 1);
                if (ok && lt >= 2) ok = wait(&tempty[b], (uint32_t)((lt >> 1) - 1) & 1u);
                for (int kc = 0; kc < nK && ok; ++kc, ++it) {
                    const int s = (int)(it % kGramStages);
                    ok = wait(&full[s], (uint32_t)(it / kGramStages) & 1u);
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint32_t sb = tc::smem_u32(stages + (size_t)s * stage_bytes);
                    const uint32_t sa = a_stays ? tc::smem_u32(base + kc * kA) : sb + kB;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc::mma_f16(tbase + (uint32_t)b * kTileN, tc::sw128_desc(sa + kk * 32),
                                    tc::sw128_desc(sb + kk * 32), idesc, (kc | kk) ? 1u : 0u);
                    tc::mma_commit(&empty[s]);
                }
                if (ok) {
                    tc::mma_commit(&tfull[b]);
                    ++done;
                }
                if (++ct == CT) {
                    ct = 0;
                    ++rt;
                }
            }
            // the MMAs have ended (and signalled) before the accumulators are
            // freed and the CTA ends, also when all were issued and a warp
            // that reads them gave up
            if (it > 0)
                tc::mbar_wait(&empty[(it - 1) % kGramStages], (uint32_t)((it - 1) / kGramStages) & 1u, kExactWait);
            if (done > 0) tc::mbar_wait(&tfull[(done - 1) & 1], (uint32_t)((done - 1) >> 1) & 1u, kExactWait);
        }
        __syncwarp();
    } else {
        const int quad = w & 3, half = (w - 2) >> 2;
        const int lr = 32 * quad + lane;
        const float kInf = __int_as_float(0x7f800000);
        const uint32_t trow = tbase + ((uint32_t)(32 * quad) << 16) + (uint32_t)(128 * half);
        float gm[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) gm[e] = kInf;
        float lim = kInf;
        bool full = false;  // the query's list is: it is handed back, no need to count on
        int rt_cur = -1;
        int rt = (int)(g0 / CT), ct = (int)(g0 - (int64_t)rt * CT);
        for (int64_t g = g0; g < g1; ++g) {
            const int64_t lt = g - g0;
            const int b = (int)(lt & 1);
            if (kList && rt != rt_cur) {
                lim = thr[rt * kTileM + lr];
                full = false;
            }
            rt_cur = rt;
            bool ok = wait(&tfull[b], (uint32_t)(lt >> 1) & 1u);
            ok = ok && wait(&nfull[b], (uint32_t)(lt >> 1) & 1u);
            if (!__all_sync(KNNG_FULL_MASK, ok)) break;
            tc::fence_after_sync();
            if (kList && full) lim = -kInf;  // (not within a tile: each test would wait for the counter)
            const float* nv = norms + b * kTileN + 128 * half;
            const uint32_t tcol = trow + (uint32_t)b * kTileN;
            // |x^|^2 - 2 q^.x^ of chunk c (32 rows), packed pairs
            auto body = [&](const uint32_t (&r)[32], int c) {
                float v[32];
                const float2 two = make_float2(-2.f, -2.f);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 q = *reinterpret_cast<const float4*>(nv + 32 * c + 4 * i);
                    const float2 lo = __ffma2_rn(
                        two, make_float2(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1])),
                        make_float2(q.x, q.y));
                    const float2 hi = __ffma2_rn(
                        two, make_float2(__uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])),
                        make_float2(q.z, q.w));
                    v[4 * i] = lo.x;
                    v[4 * i + 1] = lo.y;
                    v[4 * i + 2] = hi.x;
                    v[4 * i + 3] = hi.y;
                }
                if (!kList) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) gm[e] = fminf(gm[e], v[e]);
                } else {
                    float mn[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) mn[e] = fminf(fminf(v[e], v[e + 8]), fminf(v[e + 16], v[e + 24]));
#pragma unroll
                    for (int o = 4; o >= 1; o >>= 1)
#pragma unroll
                        for (int e = 0; e < o; ++e) mn[e] = fminf(mn[e], mn[e + o]);
                    if (mn[0] <= lim) {
                        // one counter update for the chunk's rows (one per
                        // row: lists of hundreds, 474 us instead of 187)
                        uint32_t hit = 0;
#pragma unroll
                        for (int e = 0; e < 32; ++e) hit |= v[e] <= lim ? 1u << e : 0u;
                        const int qi = rt * kTileM + lr;
                        int at = atomicAdd(&counts[qi], __popc(hit));
                        int32_t* o = lists + (int64_t)qi * kListMax;
                        const int row0 = ct * kTileN + 128 * half + 32 * c;
                        for (; hit && at < kListMax; hit &= hit - 1u, ++at) o[at] = row0 + __ffs((int)hit) - 1;
                        full |= hit != 0u;
                    }
                }
            };
            uint32_t ra[32], rb[32];
            tc::tmem_ld32(tcol, ra);
            tc::tmem_ld_wait(ra);
            tc::tmem_ld32(tcol + 32u, rb);
            body(ra, 0);
            tc::tmem_ld_wait(rb);
            tc::tmem_ld32(tcol + 64u, ra);
            body(rb, 1);
            tc::tmem_ld_wait(ra);
            tc::tmem_ld32(tcol + 96u, rb);
            body(ra, 2);
            tc::tmem_ld_wait(rb);
            body(rb, 3);
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[b]);
            if (!kList && (ct == CT - 1 || g + 1 == g1)) {
                float* o = mins + (((int64_t)blockIdx.x + rt) * kTileM + lr) * 64 + 32 * half;
#pragma unroll
                for (int e = 0; e < 32; e += 4)
                    *reinterpret_cast<float4*>(o + e) = make_float4(gm[e], gm[e + 1], gm[e + 2], gm[e + 3]);
#pragma unroll
                for (int e = 0; e < 32; ++e) gm[e] = kInf;
            }
            if (++ct == CT) {
                ct = 0;
                ++rt;
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (w == 1) tc::tmem_dealloc(tbase, 512);
}

// One warp per query: the bound of step 3 as a limit of |x^|^2 - 2 q^.x^ (in
// thr; -inf: nothing is listed), the list with the far rows, and the mark of
// queries left to exact_knn_kernel.
__global__ void __launch_bounds__(256) exact_bound_kernel(int64_t n, int d, int k, const int32_t* __restrict__ queries,
                                                          int nq, int rows, int G, int CT, int64_t total,
                                                          const float* __restrict__ mins,
                                                          const float* __restrict__ nrm, const float* __restrict__ err,
                                                          const ExactStats* __restrict__ stats,
                                                          float* __restrict__ thr, int* __restrict__ counts,
                                                          int32_t* __restrict__ lists, uint8_t* __restrict__ need)
{
    __shared__ uint32_t hist_all[8][256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int qi = blockIdx.x * 8 + w;
    if (qi >= rows) return;
    const float kInf = __int_as_float(0x7f800000);
    const int32_t q = qi < nq ? queries[qi] : -1;
    const bool valid = q >= 0 && q < n;
    float lim = -kInf;
    bool left = false;
    if (valid && (stats->bad || !(nrm[q] <= 1e30f))) left = true;  // (its own row is a far one)
    if (valid && !left) {
        // the CTAs with tiles of this query's row tile
        const int rt = qi / kTileM, lr = qi % kTileM;
        const int64_t first = (int64_t)rt * CT, last = first + CT - 1;
        int c0 = (int)(first * G / total), c1 = (int)(last * G / total);
        while (c0 + 1 < G && tile_begin(total, G, c0 + 1) <= first) ++c0;
        while (c0 > 0 && tile_begin(total, G, c0) > first) --c0;
        while (c1 + 1 < G && tile_begin(total, G, c1 + 1) <= last) ++c1;
        while (c1 > 0 && tile_begin(total, G, c1) > last) --c1;
        // (G <= total: every CTA has tiles)
        const int cnt = (c1 - c0 + 1) * 64;
        const float* mrow = mins + (((int64_t)c0 + rt) * kTileM + lr) * 64;
        auto key = [&](int i) -> uint64_t {
            return pack_key(mrow[(int64_t)(i >> 6) * (kTileM * 64) + (i & 63)], (uint32_t)i);
        };
        float vk = kInf;
        if (k + 1 <= cnt) {
            // largest of the k + 1 smallest (unique) keys
            const uint64_t t = warp_select_threshold(key, cnt, k + 1, hist_all[w]);
            float mx = -kInf;
            for (int i = lane; i < cnt; i += 32) {
                const uint64_t kv = key(i);
                if (kv <= t) mx = fmaxf(mx, unord_key((uint32_t)(kv >> 32)));
            }
            for (int o = 16; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(KNNG_FULL_MASK, mx, o));
            vk = mx;
        }
        if (vk < 1e30f) {
            const float ni = nrm[q];
            const float ymax = __uint_as_float(stats->max_nrm);
            // error of D^: each of the d additions of a product errs by at
            // most 2^-22 of |q^| |x^| <= (|q^|^2 + |x^|^2) / 2; the norms and
            // the combination add less.  Twice that, for the roundings of
            // this bound itself.  Below the normal range the errors are
            // absolute: 2^-126 for a product or a partial sum flushed to zero
            // (twice, for the factor 2), 2^-149 for a rounding of the norms or
            // of the canonical distances; 2^-122 an entry covers them twice.
            const float e = (float)(d + 16) * (0x1p-20f * (ni + ymax) + 0x1p-122f);
            const float s = (err[q] + __uint_as_float(stats->max_err)) * 1.0001f;
            const float u = sqrtf(fmaxf(ni + vk, 0.f) + e) * 1.0001f + 2.f * s;
            lim = (u * u * 1.0001f + e) - ni;
            // (rounding of the difference)
            lim += 0x1p-22f * (fabsf(lim) + ni);
        } else {
            left = true;
        }
    }
    // the far rows are listed at once
    const int nfar = valid && !left ? (int)stats->nfar : 0;
    for (int i = lane; i < nfar; i += 32) lists[(int64_t)qi * kListMax + i] = stats->far[i];
    if (lane == 0) {
        thr[qi] = lim;
        counts[qi] = nfar;
        if (qi < nq) need[qi] = left ? 1 : 0;
    }
}

// One warp per query: canonical distances of its listed rows, the k best by
// (distance, id).  Marks queries whose list overflowed, and all of them once a
// bounded wait gave up, for exact_knn_kernel.
template <int kDT>
__global__ void __launch_bounds__(kRescoreWarps * 32) exact_rescore_kernel(
    RowLoader<kDT> L, int64_t n, const int32_t* __restrict__ queries, int nq, int k, const int* __restrict__ counts,
    const int32_t* __restrict__ lists, uint8_t* __restrict__ need,
    const ExactStats* __restrict__ stats, int32_t* __restrict__ out_ids, float* __restrict__ out_d)
{
    __shared__ uint64_t buf_all[kRescoreWarps][kListMax];
    __shared__ uint32_t hist_all[kRescoreWarps][256];
    __shared__ int sel_all[kRescoreWarps][64];
    __shared__ int cid_all[kRescoreWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int qi = blockIdx.x * kRescoreWarps + w;
    if (qi >= nq) return;
    if (need[qi]) return;
    const int cnt = counts[qi];
    // (a wait that gave up leaves rows unlisted: the direct kernel answers)
    if (cnt > kListMax || stats->gave_up) {
        if (lane == 0) need[qi] = 1;
        return;
    }
    const int32_t q = queries[qi];  // (an id out of range listed nothing)
    uint64_t* buf = buf_all[w];
    uint32_t* hist = hist_all[w];
    int* sel = sel_all[w];
    int* cid = cid_all[w];
    int nb = 0;
    for (int c0 = 0; c0 < cnt; c0 += 32) {
        const int i = c0 + lane;
        const int32_t id = i < cnt ? lists[(int64_t)qi * kListMax + i] : -1;
        const bool take = id >= 0 && id != q;
        const uint32_t b = __ballot_sync(KNNG_FULL_MASK, take);
        __syncwarp();
        if (take) cid[__popc(b & lanemask_lt())] = id;
        __syncwarp();
        const int m = __popc(b);
        const float dd = warp_canon_dist32(L, q, cid, m);
        if (lane < m) buf[nb + lane] = pack_key(dd, (uint32_t)cid[lane]);
        nb += m;
    }
    __syncwarp();
    auto key = [&](int i) -> uint64_t { return buf[i]; };
    const int want = min(k, nb);
    int m = 0;
    if (want > 0) {
        const uint64_t t2 = warp_select_threshold(key, nb, want, hist);
        m = warp_compact_le(key, nb, t2, sel);
    }
    __syncwarp();
    uint64_t v[2];
    v[0] = 2 * lane < m ? buf[sel[2 * lane]] : kKeyMax;
    v[1] = 2 * lane + 1 < m ? buf[sel[2 * lane + 1]] : kKeyMax;
    warp_bitonic_sort<2>(v);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = 2 * lane + e;
        if (i < k) {
            const bool ok = i < m;
            out_ids[(int64_t)qi * k + i] = ok ? (int32_t)(uint32_t)v[e] : -1;
            out_d[(int64_t)qi * k + i] = ok ? unord_key((uint32_t)(v[e] >> 32)) : __int_as_float(0x7f800000);
        }
    }
}

static bool exact_rows_map(CUtensorMap* map, void* base, int dq, int64_t rows, int box_rows)
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    if (!fn) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)dq, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)dq * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int kDT>
std::integral_constant<int, kDT> dtype_of(const RowLoader<kDT>&);

// The filtered form from 2,048 rows on: exact_knn_kernel streams all rows per
// block, 0.50 ms at 2,048 x 128 for 10 or 1,000 queries and 3.8 ms at 16,384
// for 1,000, the filtered form 0.08 and 0.13 ms; smaller sets keep the form
// that needs no scratch.  n below 2^31 - 256: row numbers of a tile stay
// in an int.
bool exact_tc_ok(const XDesc& x, int nq)
{
    return x.n >= 2048 && x.n < ((int64_t)1 << 31) - kTileN && nq > 0;
}

// Scratch from ar (measured with ar.base == nullptr).  wait_cycles: limit of
// the tensor-core passes' waits (0: about one second); *err: word set when one
// gave up (the direct kernel then answers the queries).
cudaError_t run_exact_knn_tc(const XDesc& x, const int32_t* queries, int nq, int k, int32_t* ids, float* dists,
                             int* err, Arena& ar, cudaStream_t st, long long wait_cycles)
{
    const long long limit = wait_cycles > 0 ? wait_cycles : kExactWait;
    const int dq = (x.d + 63) / 64 * 64, nK = dq / 64;
    const int CT = (int)((x.n + kTileN - 1) / kTileN);
    const int64_t n_pad = (int64_t)CT * kTileN;
    const int G = num_sms();
    const int bq = std::min(nq, kBatchQ);
    const int brows = (bq + kTileM - 1) / kTileM * kTileM;
    __nv_bfloat16* Xq = ar.take<__nv_bfloat16>((size_t)x.n * dq);
    float* nrm = ar.take<float>((size_t)n_pad);
    float* xerr = ar.take<float>((size_t)x.n);
    ExactStats* stats = ar.take<ExactStats>(1);
    __nv_bfloat16* Aq = ar.take<__nv_bfloat16>((size_t)brows * dq);
    float* mins = ar.take<float>((size_t)(G + brows / kTileM) * kTileM * 64);
    float* thr = ar.take<float>((size_t)brows);
    int* counts = ar.take<int>((size_t)brows);
    uint8_t* need = ar.take<uint8_t>((size_t)brows);
    int32_t* lists = ar.take<int32_t>((size_t)brows * kListMax);
    if (!ar.base) return cudaSuccess;

    CUtensorMap bmap, amap;
    if (!exact_rows_map(&bmap, Xq, dq, x.n, kTileN) || !exact_rows_map(&amap, Aq, dq, brows, kTileM))
        return run_exact_knn(x, queries, nq, k, ids, dists, st);
    const bool a_stays = nK <= 4;
    const size_t smem = 1024 + (a_stays ? (size_t)nK * kTileM * 128 : 0) +
                        kGramStages * (size_t)((a_stays ? 0 : kTileM * 128) + kTileN * 128) + 2 * kTileN * sizeof(float);
    const bool poll = limit < tc::kPollBelow;
    auto minima = poll ? exact_gram_kernel<false, true> : exact_gram_kernel<false, false>;
    auto listing = poll ? exact_gram_kernel<true, true> : exact_gram_kernel<true, false>;
    cudaError_t e = cudaFuncSetAttribute(minima, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(listing, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaMemsetAsync(stats, 0, sizeof(ExactStats), st);
    if (e != cudaSuccess) return e;
    auto typed = [&](auto&& f) {
        if (x.dtype == kDtF16) f(RowLoader<kDtF16>{x.X, x.ld, x.d, x.vec});
        else if (x.dtype == kDtU8) f(RowLoader<kDtU8>{x.X, x.ld, x.d, x.vec});
        else f(RowLoader<kDtF32>{x.X, x.ld, x.d, x.vec});
    };
    typed([&](auto rl) {
        constexpr int kDT = decltype(dtype_of(rl))::value;
        const int grid = (int)std::min<int64_t>((n_pad + 7) / 8, (int64_t)G * 8);
        auto quant = dq == 64 ? exact_quant_kernel<kDT, 16> : exact_quant_kernel<kDT, 32>;
        quant<<<grid, 256, 0, st>>>(rl, x.n, n_pad, dq, Xq, nrm, xerr);
    });
    exact_hist_kernel<<<(int)std::min<int64_t>((x.n + 255) / 256, (int64_t)G * 2), 256, 0, st>>>(x.n, nrm, xerr, stats);
    exact_far_kernel<<<G * 2, 256, 0, st>>>(x.n, nrm, xerr, stats, reinterpret_cast<const uint4*>(Xq), dq / 8, queries,
                                           bq, brows, reinterpret_cast<uint4*>(Aq));
    note_launches(3);
    for (int q0 = 0; q0 < nq; q0 += kBatchQ) {
        const int cq = std::min(nq - q0, kBatchQ);
        const int RT = (cq + kTileM - 1) / kTileM, rows = RT * kTileM;
        const int64_t total = (int64_t)RT * CT;
        const int Gb = (int)std::min<int64_t>(G, total);  // no CTA without a tile
        const int32_t* qs = queries + q0;
        int32_t* oi = ids + (int64_t)q0 * k;
        float* od = dists + (int64_t)q0 * k;
        if (q0 > 0) {
            const int grid = (int)std::min<int64_t>(((int64_t)rows * (dq / 8) + 255) / 256, (int64_t)G * 8);
            exact_gather_kernel<<<grid, 256, 0, st>>>(reinterpret_cast<const uint4*>(Xq), x.n, dq / 8, qs, cq, rows,
                                                      reinterpret_cast<uint4*>(Aq));
            note_launches(1);
        }
        minima<<<Gb, kGramThreads, smem, st>>>(amap, bmap, nK, RT, CT, a_stays, nrm, stats, mins, nullptr,
                                                                nullptr, nullptr, limit, err);
        exact_bound_kernel<<<(rows + 7) / 8, 256, 0, st>>>(x.n, x.d, k, qs, cq, rows, Gb, CT, total, mins, nrm, xerr,
                                                           stats, thr, counts, lists, need);
        listing<<<Gb, kGramThreads, smem, st>>>(amap, bmap, nK, RT, CT, a_stays, nrm, stats, nullptr, thr,
                                                               counts, lists, limit, err);
        note_launches(3);
        typed([&](auto rl) {
            exact_rescore_kernel<<<(cq + kRescoreWarps - 1) / kRescoreWarps, kRescoreWarps * 32, 0, st>>>(
                rl, x.n, qs, cq, k, counts, lists, need, stats, oi, od);
            note_launches(1);
        });
        e = run_exact_knn(x, qs, cq, k, oi, od, st, need);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace knng
