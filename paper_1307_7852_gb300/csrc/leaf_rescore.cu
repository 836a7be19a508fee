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
//   * one thread per row holds its own slice in registers; per slice it
//     forms the eight 4-entry partials of every candidate pair, closes the
//     block by the butterfly and adds it to the pair's running sum in shared
//     memory -- exactly the canonical distance, block by block;
//   * thread r reads the slice's eight 16-byte columns in the order
//     u ^ (r mod 8), so the eight threads of a quarter warp touch eight
//     different bank groups whatever rows they read;
//   * at the end every row sorts its candidates by (distance, id) and keeps
//     the k best.
// What bounds it: shared-memory bandwidth, 128 bytes a pair and slice (four
// wavefronts per 16-byte load of a warp; the running sum adds two).  So a
// pair listed by both of its rows is scored by one of them only, the threads
// take the rows in order of their number of pairs (a warp's loop ends at its
// longest list), and the next pair's slice is loaded while one is summed.
// 16-byte aligned FP32 rows are copied by cp.async a slice ahead; other rows
// (FP16, bytes, unaligned) are loaded, widened and stored.
// Leaves that are exact in reduced precision (their lists are final) are
// skipped by a flag the leaf kernel writes.
// 1M x 960, 8 trees, k' = 20: 24.7 -> 19.8 ms with the rows in order of their
// pairs, slots instead of searches, candidates read as 16-byte groups and a
// third slice; 300k x 384, 6 trees, k' = 40: 9.9 -> 6.2 ms.  (Rolled, sums in
// shared memory, at k' = 20: 28.4 ms.)
#include <algorithm>
#include <type_traits>

#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

namespace {
constexpr int kSlice = 32;       // floats per row and slice (one block of the distance)
constexpr int kMaxCand = 40;     // candidates per row handled here
}  // namespace

// Canonical block value of a pair: own slice a and candidate slice b, columns
// in the order u ^ x, u = 0..7.  s[u] is the partial of column u ^ x; since the block's butterfly
// pairs columns by xor (q with q ^ 4, then q ^ 2, then q ^ 1), relabelling
// them by xor with x only swaps the operands of some additions, so the tree
// below over s[] gives the block value bit for bit -- and, t = a - b and
// b - a squaring alike, the same value whichever row is the own one.
// (Scalar FP32: packed pairs need their operands in adjacent registers,
// which these columns are not, and measured slower.)
__device__ __forceinline__ float slice_block(const float4 (&a)[8], const float4 (&b)[8])
{
    float s[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 v = b[u];
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
// ld % 4 == 0.  nbuf: slices in shared memory; with 2 the next one is loaded
// while one is scored, with 1 between two of them, with 3 (kAsync) a slice
// needs one barrier instead of two.
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

// Bytes of the slices (and, over them, the bitmaps and the table).
__host__ __device__ constexpr size_t slice_bytes(int mp, int kp, int nbuf)
{
    const size_t sl = (size_t)nbuf * 8 * sizeof(float4), tb = (size_t)kp * sizeof(float);
    return (size_t)mp * (sl > tb ? sl : tb);
}

// Up to 24 pairs a row keep their running sums in registers (the pair loop
// unrolled); more keep them in shared memory (rolled).
__host__ __device__ constexpr bool regs_hold(int kc) { return kc <= 24; }

template <int KC, int kDT, bool kAsync>
__global__ void __launch_bounds__(512, 1) leaf_rescore_staged_kernel(
    RowLoader<kDT> L, int64_t n, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ leaf_off, int nleaves, const uint8_t* __restrict__ leaf_exact,
    const uint16_t* __restrict__ cand, int kp, uint32_t kp_magic, int nbuf, int k, int32_t* __restrict__ out_ids,
    float* __restrict__ out_d)
{
    constexpr bool kRegs = regs_hold(KC);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int hist[64];
    const int t = blockIdx.y, leaf = blockIdx.x;
    if (leaf_exact && leaf_exact[(int64_t)t * nleaves + leaf]) return;
    const int off = leaf_off[leaf];
    const int m = leaf_off[leaf + 1] - off;
    const int mp = (m + 7) & ~7;
    const int d = L.d;
    // [nbuf][mp][8] float4 slices | lid[mp] | tot[kp][mp] f32 (!kRegs) | list[kp][mp] u16 | order[mp] u16
    float4* buf = reinterpret_cast<float4*>(smem_raw);
    int32_t* lid = reinterpret_cast<int32_t*>(smem_raw + slice_bytes(mp, kp, nbuf));
    float* tot = reinterpret_cast<float*>(lid + mp);
    uint16_t* list = reinterpret_cast<uint16_t*>(tot + (kRegs ? 0 : (size_t)kp * mp));
    uint16_t* order = list + (size_t)kp * mp;
    // over the slices: bits[mp][kBitRow] before them, res[kp][mp] after
    uint32_t* bits = reinterpret_cast<uint32_t*>(buf);
    float* res = reinterpret_cast<float*>(buf);
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t rowbase = (int64_t)t * n + off;
    for (int j = tid; j < m; j += blockDim.x) lid[j] = perm[rowbase + j];

    const bool active = tid < m;
    const int want = min(kp, m - 1);
    for (int e = tid; e < mp * kBitRow; e += blockDim.x) bits[e] = 0u;
    for (int e = tid; e < 64; e += blockDim.x) hist[e] = 0;  // (a block may have 32 threads)
    __syncthreads();
    // the leaf's candidates are contiguous, read as aligned groups of eight;
    // entry e is candidate e mod kp of row e / kp (kp_magic = 2^32 / kp
    // rounded up: exact below 2^16)
    {
        const int64_t first = rowbase * kp;
        const int lead = (int)(first & 7);
        const uint4* src = reinterpret_cast<const uint4*>(cand + (first - lead));
        const int groups = (m * kp + lead + 7) >> 3;
        for (int g0 = tid; g0 < groups; g0 += 4 * blockDim.x) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int g = g0 + q * blockDim.x;
                v[q] = g < groups ? src[g] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t wv[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int e = 8 * (g0 + q * (int)blockDim.x) + j - lead;
                    if (e < 0 || e >= m * kp) continue;
                    const int r = kp == 1 ? e : (int)__umulhi((uint32_t)e, kp_magic);
                    if (e - r * kp < want) {
                        const uint32_t c = (wv[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
                        if (c < (uint32_t)m) atomicOr(&bits[r * kBitRow + (c >> 5)], 1u << (c & 31u));
                    }
                }
            }
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
    // row tid's list, an entry being candidate | slot << 9: the pairs it
    // scores from the front, with the slot in the candidate's table row
    // (kNoSlot: the candidate does not list this row), the others from the
    // end, with the slot in the own table row
    int mine = 0;
    if (active) {
        int back = want, z = 0;
        const int myw = tid >> 5;
        uint32_t word = bits[tid * kBitRow];
        for (int rank = 0; rank < want; ++rank) {
            while (word == 0u && z < 15) word = bits[tid * kBitRow + ++z];
            if (word == 0u) break;
            const int c = 32 * z + __ffs((int)word) - 1;
            word &= word - 1u;
            const uint32_t cw = bits[c * kBitRow + myw];
            const bool listed = (cw >> lane) & 1u;
            if (!listed || ((c > tid) == (((c + tid) & 1) != 0))) {
                const uint32_t pre = (bits[c * kBitRow + 16 + (myw >> 2)] >> (8 * (myw & 3))) & 0xFFu;
                const int slot = listed ? (int)pre + __popc(cw & lanemask_lt()) : kNoSlot;
                list[mine * mp + tid] = (uint16_t)(c | (slot << 9));
                ++mine;
            } else {
                --back;
                list[back * mp + tid] = (uint16_t)(c | (rank << 9));
            }
        }
        // (a leaf whose candidate kernel gave up lists fewer)
        for (int i = mine; i < back; ++i) list[i * mp + tid] = (uint16_t)tid;
        atomicAdd(&hist[mine], 1);
    }
    __syncthreads();  // the bitmaps are read before the slices replace them

    const int nslices = (d + kSlice - 1) / kSlice;
    // slice sl into buffer b
    auto stage = [&](int sl, int b) {
        float4* dst = buf + (size_t)b * mp * 8;
        if constexpr (kAsync) {
            // (blockDim is a multiple of 8: a thread copies one column)
            const int j = sl * kSlice + 4 * (tid & 7);
            const int bytes = min(max(4 * (d - j), 0), 16);
            const float* base = static_cast<const float*>(L.X) + (bytes > 0 ? j : 0);
            for (int u = tid; u < m * 8; u += blockDim.x)
                cp_async16(dst + u, base + L.row_off(lid[u >> 3]), bytes);
            cp_async_commit();
        } else {
            // eight columns a thread at most (blockDim >= m), four loads in flight
#pragma unroll
            for (int i0 = 0; i0 < 8; i0 += 4) {
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int u = tid + (i0 + i) * blockDim.x;
                    const int j = sl * kSlice + 4 * (u & 7);
                    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (u < m * 8 && j < d) v[i] = L.load4(lid[u >> 3], j);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int u = tid + (i0 + i) * blockDim.x;
                    if (u < m * 8) dst[u] = v[i];
                }
            }
        }
    };
    stage(0, 0);
    // the rows in order of their number of pairs (a counting sort, longest
    // first; the order of equal ones does not matter)
    if (tid < 32) {
        const int a = hist[63 - 2 * tid], b2 = hist[62 - 2 * tid];
        int incl = a + b2;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(KNNG_FULL_MASK, incl, o);
            if (lane >= o) incl += v;
        }
        __syncwarp();
        hist[63 - 2 * tid] = incl - a - b2;
        hist[62 - 2 * tid] = incl - b2;
    }
    __syncthreads();
    if (active) order[atomicAdd(&hist[mine], 1)] = (uint16_t)(tid | (mine << 9));
    __syncthreads();
    const int row = active ? order[tid] & 511 : 0;
    const int nown = active ? order[tid] >> 9 : 0;
    const int wmax = __reduce_max_sync(KNNG_FULL_MASK, nown);
    const int x8 = tid & 7;  // columns read in the order u ^ x8: a quarter warp hits eight bank groups
    auto load_slice = [&](float4 (&v)[8], const float4* __restrict__ b) {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = b[u ^ x8];
    };
    // pair i's candidate (past the own pairs: the row itself, whose sum is
    // not kept)
    auto cand_of = [&](int i) { return i < nown ? list[i * mp + row] & 511 : row; };
    float sum[kRegs ? KC : 1];
    if constexpr (kRegs) {
#pragma unroll
        for (int i = 0; i < KC; ++i) sum[i] = 0.f;
    } else {
        for (int i = 0; i < wmax; ++i) tot[i * mp + (active ? tid : 0)] = 0.f;
    }
    if (nbuf == 3 && nslices > 1) stage(1, 1);
    int bsl = 0;  // buffer of slice sl
    for (int sl = 0; sl < nslices; ++sl) {
        const bool ahead = nbuf >= 2 && sl + 1 < nslices;
        if (nbuf == 2 && ahead) stage(sl + 1, bsl ^ 1);
        if constexpr (kAsync) {
            if (ahead) cp_async_wait<1>();
            else cp_async_wait<0>();
        }
        __syncthreads();
        // (three buffers: the one of slice sl - 1, whose readers passed the
        // barrier)
        if (nbuf == 3 && sl + 2 < nslices) stage(sl + 2, bsl == 0 ? 2 : bsl - 1);
        if (wmax > 0) {
            const float4* B = buf + (size_t)bsl * mp * 8;
            float4 a[8];
            load_slice(a, B + (size_t)row * 8);
            if constexpr (kRegs) {
#pragma unroll
                for (int i = 0; i < KC; ++i) {
                    if (i >= wmax) break;  // uniform over the warp
                    float4 v[8];
                    load_slice(v, B + (size_t)cand_of(i) * 8);
                    sum[i] = sum[i] + slice_block(a, v);
                }
            } else {
                float4 v0[8], v1[8];
                load_slice(v0, B + (size_t)cand_of(0) * 8);
                int c1 = cand_of(1);
                float* tp = tot + (active ? tid : 0);
                for (int i = 0; i < wmax; i += 2) {
                    load_slice(v1, B + (size_t)c1 * 8);
                    const int c2 = cand_of(i + 2), c3 = cand_of(i + 3);
                    const float s0 = tp[i * mp] + slice_block(a, v0);
                    if (i < nown) tp[i * mp] = s0;
                    load_slice(v0, B + (size_t)c2 * 8);
                    if (i + 1 < nown) tp[(i + 1) * mp] = tp[(i + 1) * mp] + slice_block(a, v1);
                    c1 = c3;
                }
            }
        }
        if (nbuf < 3) __syncthreads();  // the buffer of this slice is staged again
        if (nbuf == 1 && sl + 1 < nslices) stage(sl + 1, 0);
        bsl = bsl + 1 == nbuf ? 0 : bsl + 1;
    }
    __syncthreads();
    // exchange: the pairs another row is to take go to its slot
    if constexpr (kRegs) {
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < nown) {
                const int e = list[i * mp + row];
                if ((e >> 9) != kNoSlot) res[(e >> 9) * mp + (e & 511)] = sum[i];
            }
    } else {
        for (int i = 0; i < nown; ++i) {
            const int e = list[i * mp + row];
            if ((e >> 9) != kNoSlot) res[(e >> 9) * mp + (e & 511)] = tot[i * mp + tid];
        }
    }
    __syncthreads();
    if (!active) return;
    uint64_t key[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) {
        key[i] = kKeyMax;
        if (i < want) {
            const int e = list[i * mp + row];
            float dist = kRegs ? sum[kRegs ? i : 0] : 0.f;
            if (i >= nown) dist = res[(e >> 9) * mp + row];
            else if (!kRegs) dist = tot[i * mp + tid];
            key[i] = pack_key(dist, (uint32_t)lid[e & 511]);
        }
    }
    // the k best of the row's candidates by (distance, point id)
    reg_oddeven_sort(key);
    const int gi = lid[row];
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

static size_t staged_smem(int max_leaf, int kp, int nbuf, bool regs)
{
    const size_t mp = (size_t)((max_leaf + 7) & ~7);
    static_assert(8 * sizeof(float4) >= kBitRow * sizeof(uint32_t), "the bitmaps fit one slice");
    return slice_bytes((int)mp, kp, nbuf) + mp * (sizeof(int32_t) + sizeof(uint16_t)) +
           mp * kp * ((regs ? 0 : sizeof(float)) + sizeof(uint16_t));
}

bool leaf_rescore_staged_ok(int kp, int max_leaf)
{
    return kp <= kMaxCand && max_leaf <= 512 && staged_smem(max_leaf, kp, 1, false) <= 226 * 1024;
}

template <int KC, int kDT, bool kAsync>
static cudaError_t launch_staged(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm,
                                 const uint8_t* leaf_exact, const uint16_t* cand, int kp, int k, int32_t* ids,
                                 float* dists, cudaStream_t st)
{
    const int nleaves = (int)P.leaf_off.size() - 1;
    const int threads = std::max(32, (P.max_leaf + 31) & ~31);
    // as many slices as there is room for, with at most 256 threads beside
    // the second CTA that the registers allow
    constexpr bool regs = regs_hold(KC);
    const size_t room = (threads <= 256 ? 112 : 226) * (size_t)1024;
    int nbuf = kAsync ? 3 : 2;
    while (nbuf > 1 && staged_smem(P.max_leaf, kp, nbuf, regs) > room) --nbuf;
    const size_t smem = staged_smem(P.max_leaf, kp, nbuf, regs);
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
