// FP32 rescoring of the reduced-precision leaf candidates (the leaf graphs of
// Sec. 3.1 of arXiv:1307.7852 with a BF16 / FP8 candidate stage), one CTA per
// (tree, leaf).
//
// The tensor-core leaf kernel leaves, for every row of a leaf that is not
// exact in reduced precision, its k' candidates (local indices in the leaf).
// Rescoring them with the canonical FP32 distance reads k' rows of d floats
// per point; fetched one pair at a time from L2 that is k' * d * 4 bytes per
// point (0.6 TB over the eight trees of a 1M x 960 build).  Here the leaf's
// rows stream through shared memory instead, in 32-entry slices (one block
// of the canonical distance), double-buffered, so each row of the leaf
// crosses L2 once per tree:
//   * one thread per row holds its own slice in registers and one running
//     sum per candidate; per slice it forms the eight 4-entry partials of
//     every candidate pair, closes the block by the butterfly and adds it to
//     the pair's sum -- exactly the canonical distance, block by block;
//   * thread r reads the slice's eight 16-byte columns in the order
//     u ^ (r mod 8), so the eight threads of a quarter warp touch eight
//     different bank groups whatever rows they read;
//   * at the end every row sorts its candidates by (distance, id) and keeps
//     the k best.
// What bounds it: shared-memory bandwidth, 128 bytes a pair and slice (four
// wavefronts per 16-byte load of a warp), so a pair listed by both of its
// rows is scored by one of them only, and each thread's own pairs come first
// in its list: a warp's loop ends at its longest list of own pairs.
// 16-byte aligned FP32 rows are copied by cp.async; other rows (FP16, bytes,
// unaligned) are loaded a slice ahead into registers and widened on the way
// to shared memory.
// Leaves that are exact in reduced precision (their lists are final) are
// skipped by a flag the leaf kernel writes.
#include <algorithm>
#include <type_traits>

#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

namespace {
constexpr int kSlice = 32;       // floats per row and slice (one block of the distance)
constexpr int kMaxCand = 40;     // candidates per row handled here
}  // namespace

// Canonical block value of a pair: own slice a (columns in the order
// u ^ x, u = 0..7, already in registers), candidate slice b in shared
// memory.  s[u] is the partial of column u ^ x; since the block's butterfly
// pairs columns by xor (q with q ^ 4, then q ^ 2, then q ^ 1), relabelling
// them by xor with x only swaps the operands of some additions, so the tree
// below over s[] gives the block value bit for bit -- and, t = a - b and
// b - a squaring alike, the same value whichever row is the own one.
// (Scalar FP32: packed pairs need their operands in adjacent registers,
// which these columns are not, and measured slower.)
__device__ __forceinline__ float slice_block(const float4 (&a)[8], const float4* __restrict__ b, int x)
{
    float s[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 v = b[u ^ x];
        float acc = 0.f, t;
        t = a[u].x - v.x; acc = fmaf(t, t, acc);
        t = a[u].y - v.y; acc = fmaf(t, t, acc);
        t = a[u].z - v.z; acc = fmaf(t, t, acc);
        t = a[u].w - v.w; acc = fmaf(t, t, acc);
        s[u] = acc;
    }
    return ((s[0] + s[4]) + (s[2] + s[6])) + ((s[1] + s[5]) + (s[3] + s[7]));
}

// grid (nleaves, T); blockDim >= the largest leaf (multiple of 32, <= 512).
// cand: [T * n][kp] local indices (u16) of every row's candidates, the first
// want = min(kp, m - 1) valid, kp <= KC.  kAsync: FP32 rows, 16-byte aligned,
// ld % 4 == 0.  nbuf: slices in shared memory, 2 or (kAsync) 3 -- with three
// a slice needs one barrier instead of two.
//
// A pair listed by both of its rows (r in c's list and c in r's) is scored
// once: the canonical distance is symmetric bit for bit, so the other row
// takes the value from a table in shared memory.  The smaller row scores it
// when r + c is odd, the larger one when it is even, so that rows anywhere
// in the leaf score about the same number.  Membership is a bitmap per row,
// and a candidate's slot in the table is its rank in its row's bitmap: the
// scoring row finds the slot by a prefix count, without a search.  (Dealing
// the pairs out evenly, both rows then read from shared memory, measured
// slower: the row-per-thread form keeps the own slice in registers.)
constexpr int kBitRow = 21;      // words of a row's bitmap (16) and prefix counts (4); odd: no bank conflicts
constexpr int kNoSlot = 63;

template <int KC, int kDT, bool kAsync>
__global__ void __launch_bounds__(512, 1) leaf_rescore_staged_kernel(
    RowLoader<kDT> L, int64_t n, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ leaf_off, int nleaves, const uint8_t* __restrict__ leaf_exact,
    const uint16_t* __restrict__ cand, int kp, uint32_t kp_magic, int nbuf, int k, int32_t* __restrict__ out_ids,
    float* __restrict__ out_d)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int t = blockIdx.y, leaf = blockIdx.x;
    if (leaf_exact && leaf_exact[(int64_t)t * nleaves + leaf]) return;
    const int off = leaf_off[leaf];
    const int m = leaf_off[leaf + 1] - off;
    const int mp = (m + 7) & ~7;
    const int d = L.d;
    // [nbuf][mp][8] float4 slices | lid[mp] | list[kp][mp] u16
    float4* buf = reinterpret_cast<float4*>(smem_raw);
    int32_t* lid = reinterpret_cast<int32_t*>(buf + (size_t)nbuf * mp * 8);
    uint16_t* list = reinterpret_cast<uint16_t*>(lid + mp);
    // over the slices: bits[mp][kBitRow] before them, res[kp][mp] after
    uint32_t* bits = reinterpret_cast<uint32_t*>(buf);
    float* res = reinterpret_cast<float*>(buf);
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t rowbase = (int64_t)t * n + off;
    for (int j = tid; j < m; j += blockDim.x) lid[j] = perm[rowbase + j];

    const bool active = tid < m;
    const int want = min(kp, m - 1);
    for (int e = tid; e < mp * kBitRow; e += blockDim.x) bits[e] = 0u;
    __syncthreads();
    // the leaf's candidates are contiguous; entry e is candidate e mod kp of
    // row e / kp (kp_magic = 2^32 / kp rounded up: exact below 2^16)
    const uint16_t* cleaf = cand + rowbase * kp;
    for (int e = tid; e < m * kp; e += blockDim.x) {
        const int r = kp == 1 ? e : (int)__umulhi((uint32_t)e, kp_magic);
        if (e - r * kp < want) {
            const int c = cleaf[e];
            atomicOr(&bits[r * kBitRow + (c >> 5)], 1u << (c & 31));
        }
    }
    __syncthreads();
    // prefix counts of the row's bitmap, a byte per word
    if (active) {
        uint32_t run = 0, pk = 0;
        for (int z = 0; z < 16; ++z) {
            pk |= run << (8 * (z & 3));
            run += __popc(bits[tid * kBitRow + z]);
            if ((z & 3) == 3) {
                bits[tid * kBitRow + 16 + (z >> 2)] = pk;
                pk = 0;
            }
        }
    }
    __syncthreads();
    // the row's list, an entry being candidate | slot << 9: the pairs it
    // scores from the front, with the slot in the candidate's table row
    // (kNoSlot: the candidate does not list this row), the others from the
    // end, with the slot in the own table row
    int nown = 0;
    if (active) {
        int back = want, rank = 0;
        const int myw = tid >> 5;
        for (int z = 0; z < 16 && rank < want; ++z) {
            uint32_t word = bits[tid * kBitRow + z];
            while (word) {
                const int c = 32 * z + __ffs((int)word) - 1;
                word &= word - 1u;
                const uint32_t cw = bits[c * kBitRow + myw];
                const bool listed = (cw >> lane) & 1u;
                if (!listed || ((c > tid) == (((c + tid) & 1) != 0))) {
                    const uint32_t pre = (bits[c * kBitRow + 16 + (myw >> 2)] >> (8 * (myw & 3))) & 0xFFu;
                    const int slot = listed ? (int)pre + __popc(cw & lanemask_lt()) : kNoSlot;
                    list[nown * mp + tid] = (uint16_t)(c | (slot << 9));
                    ++nown;
                } else {
                    --back;
                    list[back * mp + tid] = (uint16_t)(c | (rank << 9));
                }
                ++rank;
            }
        }
    }
    const int wmax = __reduce_max_sync(KNNG_FULL_MASK, nown);
    __syncthreads();  // the bitmaps are read before the slices replace them

    const int nslices = (d + kSlice - 1) / kSlice;
    // slice sl into buffer b: cp.async, or loads a slice ahead (fetch) that
    // put() widens into the buffer; thread u copies columns u, u + blockDim, ...
    auto stage = [&](int sl, int b) {
        float4* dst = buf + (size_t)b * mp * 8;
        for (int u = tid; u < m * 8; u += blockDim.x) {
            const int r = u >> 3, col = u & 7;
            const int j = sl * kSlice + 4 * col;
            const int avail = d - j;
            const float* src = static_cast<const float*>(L.X) + L.row_off(lid[r]);
            const int bytes = avail >= 4 ? 16 : (avail > 0 ? 4 * avail : 0);
            cp_async16(dst + (size_t)r * 8 + col, bytes > 0 ? src + j : src, bytes);
        }
        cp_async_commit();
    };
    float4 pf[kAsync ? 1 : 8];
    auto fetch = [&](int sl) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int u = tid + i * blockDim.x;
            const int j = sl * kSlice + 4 * (u & 7);
            pf[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (u < m * 8 && j < d) pf[i] = L.load4(lid[u >> 3], j);
        }
    };
    auto put = [&](int b) {
        float4* dst = buf + (size_t)b * mp * 8;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int u = tid + i * blockDim.x;
            if (u < m * 8) dst[u] = pf[i];
        }
    };
    const int x8 = tid & 7;  // columns read in the order u ^ x8: a quarter warp hits eight bank groups

    float tot[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) tot[i] = 0.f;
    if constexpr (kAsync) {
        stage(0, 0);
        if (nbuf == 3 && nslices > 1) stage(1, 1);
    } else {
        fetch(0);
        put(0);
    }
    int bsl = 0;  // buffer of slice sl
    for (int sl = 0; sl < nslices; ++sl) {
        if constexpr (kAsync) {
            if (nbuf == 2 && sl + 1 < nslices) stage(sl + 1, bsl ^ 1);
            if (sl + 1 < nslices) cp_async_wait<1>();
            else cp_async_wait<0>();
        } else {
            if (sl + 1 < nslices) fetch(sl + 1);
        }
        __syncthreads();
        // (three buffers: the one of slice sl - 1, whose readers passed the
        // barrier)
        if (kAsync && nbuf == 3 && sl + 2 < nslices) stage(sl + 2, bsl == 0 ? 2 : bsl - 1);
        if (wmax > 0) {
            const float4* B = buf + (size_t)bsl * mp * 8;
            float4 a[8];
            const int self = active ? tid : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] = B[(size_t)self * 8 + (u ^ x8)];
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                if (i >= wmax) break;  // uniform over the warp
                const int c = i < nown ? list[i * mp + tid] & 511 : self;
                tot[i] = tot[i] + slice_block(a, B + (size_t)c * 8, x8);
            }
        }
        if constexpr (!kAsync) {
            if (sl + 1 < nslices) put(bsl ^ 1);  // its last readers passed the barrier above
        } else if (nbuf == 2) {
            __syncthreads();  // the buffer of this slice is staged again two slices on
        }
        bsl = bsl + 1 == nbuf ? 0 : bsl + 1;
    }
    __syncthreads();
    // exchange: the pairs another row is to take go to its slot
    if (active) {
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < nown) {
                const int e = list[i * mp + tid];
                if ((e >> 9) != kNoSlot) res[(e >> 9) * mp + (e & 511)] = tot[i];
            }
    }
    __syncthreads();
    if (!active) return;
    uint64_t key[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) {
        key[i] = kKeyMax;
        if (i < want) {
            const int e = list[i * mp + tid];
            const float dist = i < nown ? tot[i] : res[(e >> 9) * mp + tid];
            key[i] = pack_key(dist, (uint32_t)lid[e & 511]);
        }
    }
    // the k best of the row's candidates by (distance, point id)
    reg_oddeven_sort(key);
    const int gi = lid[tid];
    int32_t* oi = out_ids + ((int64_t)t * n + gi) * k;
    float* od = out_d + ((int64_t)t * n + gi) * k;
    const float kInf = __int_as_float(0x7f800000);
    // entries four or two at a time where rows of k start aligned for it
    const uintptr_t al = (uintptr_t)out_ids | (uintptr_t)out_d;
    auto id_of = [&](int i) { return i < want ? (int32_t)(uint32_t)key[i] : -1; };
    auto d_of = [&](int i) { return i < want ? unord_key((uint32_t)(key[i] >> 32)) : kInf; };
    if ((k & 3) == 0 && (al & 15) == 0) {
#pragma unroll
        for (int i = 0; i < KC; i += 4)
            if (i < k) {
                *reinterpret_cast<int4*>(oi + i) = make_int4(id_of(i), id_of(i + 1), id_of(i + 2), id_of(i + 3));
                *reinterpret_cast<float4*>(od + i) = make_float4(d_of(i), d_of(i + 1), d_of(i + 2), d_of(i + 3));
            }
    } else if ((k & 1) == 0 && (al & 7) == 0) {
#pragma unroll
        for (int i = 0; i < KC; i += 2)
            if (i < k) {
                *reinterpret_cast<int2*>(oi + i) = make_int2(id_of(i), id_of(i + 1));
                *reinterpret_cast<float2*>(od + i) = make_float2(d_of(i), d_of(i + 1));
            }
    } else {
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < k) {
                oi[i] = id_of(i);
                od[i] = d_of(i);
            }
    }
}

static size_t staged_smem(int max_leaf, int kp, int nbuf)
{
    const size_t mp = (size_t)((max_leaf + 7) & ~7);
    return std::max(nbuf * mp * 8 * sizeof(float4), mp * kBitRow * sizeof(uint32_t)) + mp * sizeof(int32_t) +
           mp * kp * sizeof(uint16_t);
}

bool leaf_rescore_staged_ok(int kp, int max_leaf)
{
    return kp <= kMaxCand && max_leaf <= 512 && staged_smem(max_leaf, kp, 2) <= 220 * 1024;
}

template <int KC, int kDT, bool kAsync>
static cudaError_t launch_staged(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm,
                                 const uint8_t* leaf_exact, const uint16_t* cand, int kp, int k, int32_t* ids,
                                 float* dists, cudaStream_t st)
{
    const int nleaves = (int)P.leaf_off.size() - 1;
    const int threads = std::max(32, (P.max_leaf + 31) & ~31);
    // a third slice where it costs no resident CTA: more than 256 threads
    // leave registers for one CTA per SM anyway
    const int nbuf = kAsync && threads > 256 && staged_smem(P.max_leaf, kp, 3) <= 220 * 1024 ? 3 : 2;
    const size_t smem = staged_smem(P.max_leaf, kp, nbuf);
    const uint32_t kp_magic = (uint32_t)((((uint64_t)1 << 32) + kp - 1) / kp);
    auto kern = leaf_rescore_staged_kernel<KC, kDT, kAsync>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    RowLoader<kDT> rl{x.X, x.ld, x.d, x.vec};
    kern<<<dim3(nleaves, T), threads, smem, st>>>(rl, x.n, perm, dp.leaf_off, nleaves, leaf_exact, cand, kp,
                                                  kp_magic, nbuf, k, ids, dists);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t run_leaf_rescore_staged(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T,
                                    const int32_t* perm, const uint8_t* leaf_exact, const uint16_t* cand, int kp,
                                    int k, int32_t* ids, float* dists, cudaStream_t st)
{
    // candidate capacity per row: the smaller of 24, 40 holding k'
    auto go = [&](auto dt, auto async) {
        constexpr int kDT = decltype(dt)::value;
        constexpr bool kAsync = decltype(async)::value;
        return kp <= 24 ? launch_staged<24, kDT, kAsync>(x, P, dp, T, perm, leaf_exact, cand, kp, k, ids, dists, st)
                        : launch_staged<40, kDT, kAsync>(x, P, dp, T, perm, leaf_exact, cand, kp, k, ids, dists, st);
    };
    if (x.dtype == kDtF16) return go(std::integral_constant<int, kDtF16>{}, std::false_type{});
    if (x.dtype == kDtU8) return go(std::integral_constant<int, kDtU8>{}, std::false_type{});
    if (x.vec && x.ld % 4 == 0) return go(std::integral_constant<int, kDtF32>{}, std::true_type{});
    return go(std::integral_constant<int, kDtF32>{}, std::false_type{});
}

}  // namespace knng
