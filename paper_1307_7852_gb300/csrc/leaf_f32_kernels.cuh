// Leaf graphs, FP32 candidate stage (Sec. 3.1 of arXiv:1307.7852: a brute-
// force k-NN graph inside every leaf subset).
//
// Up to k' = 40 candidates per row (leaf_cand_f32_kernel): one block per
// (leaf, tree, block of up to 64 rows), a warp per eight rows and all columns
// of the leaf.  The leaf's rows stream through shared memory in slices of 32
// entries; a lane holds the FP32 sums of its columns (lane + 32 c) for the
// warp's rows, so a row's distances D~ = |x|^2 + |y|^2 - 2 S end up in the
// registers of one warp, which picks the k' smallest (D~, column) without
// storing them.  The staged rescoring (leaf_rescore.cu) finishes the rows.
// Bound by FP32 issue in the products (8 rows x 8 columns a lane: 256 FMAs
// per 16 shared loads) and by the selection.  400k x 128 rows, 4 trees,
// leaves of 195, k' = 40: 10.1 ms with the kernel below (which re-stages the
// leaf per 32 rows and rescores row by row from L2), 5.2 + 2.2 ms so.
//
// More candidates (leaf_knn_f32_kernel): one block per (leaf, tree).  For
// every block of 32 rows of the leaf:
//   1. Gram S = X_rows X_leaf^T in FP32 SIMT (register-tiled, K in slices of
//      32 staged transposed in shared memory), D~ = |x|^2 + |y|^2 - 2 S;
//   2. one warp per row picks the k' smallest (D~, id) by radix select;
//   3. the k' candidates are rescored by the canonical FP32 direct-difference
//      distance and sorted; the k best are written.
// Leaf members are in ascending id order, so a local index ranks like the id.
#pragma once
// Kernels and launchers; one instantiation per element type in
// leaf_f32_f32.cu / leaf_f32_f16.cu / leaf_f32_u8.cu, the dispatch in leaf_f32.cu.
#include <algorithm>

#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

namespace {
constexpr int kRB = 32;   // rows per block pass
constexpr int kKC = 32;   // K slice
constexpr int kNT = 256;  // threads

struct LeafSmem {
    int32_t* lid;
    float* nrm;
    float* Bt;
    float* D;
    unsigned char* ws;  // kLeafWarpScratch per warp
};

__host__ __device__ inline size_t leaf_smem_bytes(int m_pad)
{
    return sizeof(int32_t) * m_pad + sizeof(float) * m_pad + sizeof(float) * kKC * (m_pad + 1) +
           sizeof(float) * kRB * m_pad + 16 + (kNT / 32) * kLeafWarpScratch;
}
}  // namespace

template <int CT, int kDT>
__global__ void __launch_bounds__(kNT) leaf_knn_f32_kernel(RowLoader<kDT> L, int64_t n,
                                                           const int32_t* __restrict__ perm,
                                                           const int32_t* __restrict__ leaf_off, int k,
                                                           int kp, int32_t* __restrict__ out_ids,
                                                           float* __restrict__ out_d)
{
    constexpr int m_pad = 32 * CT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LeafSmem sm;
    {
        unsigned char* p = smem_raw;
        sm.lid = reinterpret_cast<int32_t*>(p); p += sizeof(int32_t) * m_pad;
        sm.nrm = reinterpret_cast<float*>(p); p += sizeof(float) * m_pad;
        sm.Bt = reinterpret_cast<float*>(p); p += sizeof(float) * kKC * (m_pad + 1);
        sm.D = reinterpret_cast<float*>(p); p += sizeof(float) * kRB * m_pad;
        sm.ws = reinterpret_cast<unsigned char*>(((uintptr_t)p + 15) & ~(uintptr_t)15);
    }
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int tx = tid & 31, ty = tid >> 5;
    const int t = blockIdx.y;
    const int b = leaf_off[blockIdx.x];
    const int m = leaf_off[blockIdx.x + 1] - b;
    const int32_t* prow = perm + (int64_t)t * n + b;
    for (int j = tid; j < m_pad; j += kNT) {
        sm.lid[j] = j < m ? prow[j] : -1;
        sm.nrm[j] = 0.f;
    }
    __syncthreads();
    // squared norms (any order: they only feed the candidate distances)
    for (int r = w; r < m; r += kNT / 32) {
        float s = 0.f;
        for (int j = 4 * lane; j < L.d; j += 128) {
            const float4 x = L.load4(sm.lid[r], j);
            s = fmaf(x.x, x.x, s); s = fmaf(x.y, x.y, s); s = fmaf(x.z, x.z, s); s = fmaf(x.w, x.w, s);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(KNNG_FULL_MASK, s, o);
        if (lane == 0) sm.nrm[r] = s;
    }
    unsigned char* ws = sm.ws + (size_t)kLeafWarpScratch * w;
    constexpr int mp1 = m_pad + 1;

    for (int rb = 0; rb < m; rb += kRB) {
        float acc[4][CT];
#pragma unroll
        for (int rr = 0; rr < 4; ++rr)
#pragma unroll
            for (int c = 0; c < CT; ++c) acc[rr][c] = 0.f;
        for (int k0 = 0; k0 < L.d; k0 += kKC) {
            __syncthreads();
            // four entries a load (zero past d), stored transposed
            for (int idx = tid; idx < m_pad * (kKC / 4); idx += kNT) {
                const int row = idx / (kKC / 4), kk = 4 * (idx % (kKC / 4));
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row < m && k0 + kk < L.d) v = L.load4(sm.lid[row], k0 + kk);
                sm.Bt[(kk + 0) * mp1 + row] = v.x;
                sm.Bt[(kk + 1) * mp1 + row] = v.y;
                sm.Bt[(kk + 2) * mp1 + row] = v.z;
                sm.Bt[(kk + 3) * mp1 + row] = v.w;
            }
            __syncthreads();
#pragma unroll 4
            for (int kk = 0; kk < kKC; ++kk) {
                float a[4], bb[CT];
#pragma unroll
                for (int rr = 0; rr < 4; ++rr) a[rr] = sm.Bt[kk * mp1 + rb + ty * 4 + rr];
#pragma unroll
                for (int c = 0; c < CT; ++c) bb[c] = sm.Bt[kk * mp1 + tx + 32 * c];
#pragma unroll
                for (int rr = 0; rr < 4; ++rr)
#pragma unroll
                    for (int c = 0; c < CT; ++c) acc[rr][c] = fmaf(a[rr], bb[c], acc[rr][c]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            const int r = ty * 4 + rr;
            const float ni = sm.nrm[min(rb + r, m_pad - 1)];
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                const int col = tx + 32 * c;
                sm.D[r * m_pad + col] = ni + sm.nrm[col] - 2.f * acc[rr][c];
            }
        }
        __syncthreads();
        for (int r = w; r < kRB; r += kNT / 32) {
            const int row = rb + r;
            if (row >= m) break;
            const float* Drow = sm.D + r * m_pad;
            const int gi = sm.lid[row];
            leaf_row_finish<CT, kDT>(L, [&](int j) { return Drow[j]; }, m, row, sm.lid, k, kp, ws,
                                  out_ids + ((int64_t)t * n + gi) * k, out_d + ((int64_t)t * n + gi) * k);
        }
    }
}

// ---------------------------------------------------------------------------
// Candidates of up to kMaxStaged per row, for the staged rescoring
// ---------------------------------------------------------------------------
namespace {
constexpr int kSliceF = 32;      // entries of a slice
constexpr int kRowF = 36;        // floats of a row in shared memory: eight lanes' 16-byte
                                 // loads of consecutive rows fall in distinct bank groups
constexpr int kScratchF = 128;   // words of selection scratch per warp

__host__ __device__ constexpr int rows_per_warp(int ct) { return ct > 8 ? 4 : 8; }

__host__ __device__ constexpr size_t cand_smem_bytes(int ct)
{
    return sizeof(float) * (2 * (size_t)32 * ct * kRowF + 32 * ct) + sizeof(int32_t) * 32 * ct +
           sizeof(uint32_t) * kScratchF * (kNT / 32);
}
}  // namespace

// The want smallest of a row's distances by (key, column), lane's column e
// being lane + 32 e (key 0xFFFFFFFF: no column), as columns to out[0..want)
// in any order.  scr: kScratchF words of the warp.
template <int CT>
__device__ __forceinline__ void warp_pick_columns(const uint32_t (&h)[CT], int want, uint32_t* scr, uint16_t* out)
{
    const int lane = threadIdx.x & 31;
    // bound: the want-th smallest of the lanes' one or two smallest keys
    uint32_t a = 0xFFFFFFFFu, b = 0xFFFFFFFFu;
#pragma unroll
    for (int e = 0; e < CT; ++e) {
        const uint32_t mx = max(a, h[e]);
        a = min(a, h[e]);
        b = min(b, mx);
    }
    uint32_t tau;
    if (want <= 32) {
        uint32_t s1[1] = {a};
        warp_bitonic_sort32<1>(s1);
        tau = __shfl_sync(KNNG_FULL_MASK, s1[0], want - 1);
    } else {
        uint32_t s2[2] = {a, b};
        warp_bitonic_sort32<2>(s2);
        tau = __shfl_sync(KNNG_FULL_MASK, ((want - 1) & 1) ? s2[1] : s2[0], (want - 1) >> 1);
    }
    int c = 0;
#pragma unroll
    for (int e = 0; e < CT; ++e) {
        const uint32_t bl = __ballot_sync(KNNG_FULL_MASK, h[e] <= tau);
        if (h[e] <= tau) {
            const int at = c + __popc(bl & lanemask_lt());
            if (at < kScratchF) scr[at] = h[e];
        }
        c += __popc(bl);
    }
    if (c > want) {
        // the want-th smallest of the listed keys
        __syncwarp();
        if (c <= 64) {
            uint32_t v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) v[e] = 32 * e + lane < c ? scr[32 * e + lane] : 0xFFFFFFFFu;
            warp_bitonic_sort32<2>(v);
            tau = __shfl_sync(KNNG_FULL_MASK, ((want - 1) & 1) ? v[1] : v[0], (want - 1) >> 1);
        } else if (c <= kScratchF) {
            uint32_t v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = 32 * e + lane < c ? scr[32 * e + lane] : 0xFFFFFFFFu;
            warp_bitonic_sort32<4>(v);
            uint32_t x = v[0];
#pragma unroll
            for (int e = 1; e < 4; ++e) x = ((want - 1) & 3) == e ? v[e] : x;
            tau = __shfl_sync(KNNG_FULL_MASK, x, (want - 1) >> 2);
        } else {
            // bit by bit: the largest value with fewer than want keys below it
            uint32_t t = 0;
            for (int bit = 31; bit >= 0; --bit) {
                const uint32_t cand = t | (1u << bit);
                int below = 0;
#pragma unroll
                for (int e = 0; e < CT; ++e) below += h[e] < cand ? 1 : 0;
                if ((int)__reduce_add_sync(KNNG_FULL_MASK, below) < want) t = cand;
            }
            tau = t;
        }
        __syncwarp();
    }
    int below = 0;
#pragma unroll
    for (int e = 0; e < CT; ++e) below += h[e] < tau ? 1 : 0;
    int equal = want - (int)__reduce_add_sync(KNNG_FULL_MASK, below);  // keys equal to tau to take, smallest columns first
    int base = 0;
#pragma unroll
    for (int e = 0; e < CT; ++e) {
        const uint32_t be = __ballot_sync(KNNG_FULL_MASK, h[e] == tau);
        const bool take = h[e] < tau || (h[e] == tau && __popc(be & lanemask_lt()) < equal);
        const uint32_t bt = __ballot_sync(KNNG_FULL_MASK, take);
        if (take) out[base + __popc(bt & lanemask_lt())] = (uint16_t)(lane + 32 * e);
        base += __popc(bt);
        equal -= min(equal, __popc(be));
    }
}

// Block (leaf, row block, tree).  kAsync: 16-byte aligned FP32 rows, ld % 4 == 0.
template <int CT, int kDT, bool kAsync>
__global__ void __launch_bounds__(kNT, CT > 8 ? 1 : 2) leaf_cand_f32_kernel(RowLoader<kDT> L, int64_t n,
                                                                          const int32_t* __restrict__ perm,
                                                                          const int32_t* __restrict__ leaf_off, int kp,
                                                                          uint16_t* __restrict__ cand)
{
    constexpr int M = 32 * CT, R = rows_per_warp(CT), W = kNT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* buf = reinterpret_cast<float*>(smem_raw);  // [2][M][kRowF]
    float* nrm = buf + 2 * M * kRowF;
    int32_t* lid = reinterpret_cast<int32_t*>(nrm + M);
    uint32_t* scr = reinterpret_cast<uint32_t*>(lid + M) + kScratchF * (threadIdx.x >> 5);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int t = blockIdx.z;
    const int off = leaf_off[blockIdx.x];
    const int m = leaf_off[blockIdx.x + 1] - off;
    // rows dealt evenly to the leaf's blocks, whole warps' shares
    const int blocks = (m + R * W - 1) / (R * W);
    if ((int)blockIdx.y >= blocks) return;
    const int share = ((m + blocks - 1) / blocks + R - 1) / R * R;
    const int rb = blockIdx.y * share + R * w;  // the warp's first row
    const bool busy = R * w < share && rb < m;
    const int64_t rowbase = (int64_t)t * n + off;
    for (int j = tid; j < M; j += kNT) lid[j] = j < m ? perm[rowbase + j] : -1;
    // rows past the leaf stay zero in both buffers
    for (int e = tid; e < 2 * (M - m) * (kRowF / 4); e += kNT) {
        const int per = (M - m) * (kRowF / 4);
        const int b = e >= per ? 1 : 0, q = e - b * per;
        reinterpret_cast<float4*>(buf + (b * M + m) * kRowF)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const int nslices = (L.d + kSliceF - 1) / kSliceF;
    auto stage = [&](int sl, int b) {
        float* dst = buf + b * M * kRowF;
        const int q = tid & 7, j = sl * kSliceF + 4 * q;  // (kNT is a multiple of 8: one column per thread)
        if constexpr (kAsync) {
            const int bytes = min(max(4 * (L.d - j), 0), 16);
            const float* src = static_cast<const float*>(L.X) + (bytes > 0 ? j : 0);
            for (int r = tid >> 3; r < m; r += kNT / 8)
                cp_async16(dst + r * kRowF + 4 * q, src + L.row_off(lid[r]), bytes);
            cp_async_commit();
        } else {
            for (int r0 = tid >> 3; r0 < m; r0 += 4 * (kNT / 8)) {
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r0 + i * (kNT / 8);
                    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r < m && j < L.d) v[i] = L.load4(lid[r], j);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r0 + i * (kNT / 8);
                    if (r < m) *reinterpret_cast<float4*>(dst + r * kRowF + 4 * q) = v[i];
                }
            }
        }
    };
    float acc[R][CT];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < CT; ++c) acc[r][c] = 0.f;
    // squared norms of rows tid, tid + kNT: sums and what their rounding lost
    // (one chain of d additions errs by 1.7e-7 of the norm at 128 entries and
    // 9e-7 at 4,096, a sum by 32 lanes by 4e-8 and 5e-8, this one by 3e-8)
    float nr[(M + kNT - 1) / kNT] = {}, lost[(M + kNT - 1) / kNT] = {};
    stage(0, 0);
    for (int sl = 0; sl < nslices; ++sl) {
        const bool ahead = sl + 1 < nslices;
        if (ahead) stage(sl + 1, (sl + 1) & 1);
        if constexpr (kAsync) {
            if (ahead) cp_async_wait<1>();
            else cp_async_wait<0>();
        }
        __syncthreads();
        const float* B = buf + (sl & 1) * M * kRowF;
#pragma unroll
        for (int i = 0; i < (M + kNT - 1) / kNT; ++i) {
            const int row = tid + i * kNT;
            if (row < m) {
#pragma unroll
                for (int q = 0; q < kSliceF; q += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(B + row * kRowF + q);
                    const float p = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, v.x * v.x)));
                    const float t = nr[i] + p, b = t - nr[i];
                    lost[i] += (nr[i] - (t - b)) + (p - b);
                    nr[i] = t;
                }
            }
        }
        if (busy) {
#pragma unroll 1
            for (int q = 0; q < kSliceF; q += 4) {
                float4 a[R];
#pragma unroll
                for (int r = 0; r < R; ++r) a[r] = *reinterpret_cast<const float4*>(B + (rb + r) * kRowF + q);
#pragma unroll
                for (int c = 0; c < CT; ++c) {
                    const float4 b = *reinterpret_cast<const float4*>(B + (lane + 32 * c) * kRowF + q);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        acc[r][c] = fmaf(a[r].x, b.x, acc[r][c]);
                        acc[r][c] = fmaf(a[r].y, b.y, acc[r][c]);
                        acc[r][c] = fmaf(a[r].z, b.z, acc[r][c]);
                        acc[r][c] = fmaf(a[r].w, b.w, acc[r][c]);
                    }
                }
            }
        }
        __syncthreads();  // the buffer is staged again
    }
#pragma unroll
    for (int i = 0; i < (M + kNT - 1) / kNT; ++i)
        // (a sum past the range has lost nothing that counts)
        if (tid + i * kNT < M) nrm[tid + i * kNT] = nr[i] < __int_as_float(0x7f800000) ? nr[i] + lost[i] : nr[i];
    __syncthreads();
    const int want = min(kp, m - 1);
    if (!busy || want < 1) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int row = rb + r;
        if (row >= m || (row - (int)blockIdx.y * share) >= share) break;
        const float ni = nrm[row];
        uint32_t h[CT];
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            const int col = lane + 32 * c;
            const float dist = ni + nrm[col] - 2.f * acc[r][c];
            // (a distance that is not a number comes after all others, whatever
            // its sign bit: as a key it came before them)
            const uint32_t o = dist == dist ? ord_key(dist) : 0xFFFFFFFEu;
            h[c] = (col < m && col != row) ? min(o, 0xFFFFFFFEu) : 0xFFFFFFFFu;
        }
        warp_pick_columns<CT>(h, want, scr, cand + (rowbase + row) * kp);
        __syncwarp();
    }
}

template <int CT, int kDT, bool kAsync>
static cudaError_t launch_cand_f32(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm,
                                   int kp, uint16_t* cand, cudaStream_t st)
{
    const size_t smem = cand_smem_bytes(CT);
    auto kern = leaf_cand_f32_kernel<CT, kDT, kAsync>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    RowLoader<kDT> rl{x.X, x.ld, x.d, x.vec};
    const int nleaves = (int)P.leaf_off.size() - 1;
    const int per = rows_per_warp(CT) * (kNT / 32);
    kern<<<dim3(nleaves, (P.max_leaf + per - 1) / per, T), kNT, smem, st>>>(rl, x.n, perm, dp.leaf_off, kp, cand);
    note_launches(1);
    return cudaGetLastError();
}

template <int kDT, bool kAsync>
cudaError_t leaf_f32_cand(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T, const int32_t* perm,
                                 int kp, uint16_t* cand, cudaStream_t st)
{
    // columns per lane: the smallest of 1, 2, 4, 6, 8, 12, 16 that hold the
    // widest leaf (lanes past the leaf's end multiply zeros)
    const int m = P.max_leaf;
    if (m <= 32) return launch_cand_f32<1, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    if (m <= 64) return launch_cand_f32<2, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    if (m <= 128) return launch_cand_f32<4, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    if (m <= 192) return launch_cand_f32<6, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    if (m <= 256) return launch_cand_f32<8, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    if (m <= 384) return launch_cand_f32<12, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
    return launch_cand_f32<16, kDT, kAsync>(x, P, dp, T, perm, kp, cand, st);
}

template <int CT, int kDT>
static cudaError_t launch_leaf_f32(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T,
                                   const int32_t* perm, int k, int kp, int32_t* ids, float* dists,
                                   cudaStream_t st)
{
    const size_t smem = leaf_smem_bytes(32 * CT);
    auto kern = leaf_knn_f32_kernel<CT, kDT>;
    static bool attr_done = false;
    if (!attr_done) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)leaf_smem_bytes(32 * CT));
        if (e != cudaSuccess) return e;
        attr_done = true;
    }
    RowLoader<kDT> rl{x.X, x.ld, x.d, x.vec};
    const int nleaves = (int)P.leaf_off.size() - 1;
    kern<<<dim3(nleaves, T), kNT, smem, st>>>(rl, x.n, perm, dp.leaf_off, k, kp, ids, dists);
    note_launches(1);
    return cudaGetLastError();
}

template <int kDT>
cudaError_t leaf_f32_full(const XDesc& x, const TreePlan& P, const DevPlan& dp, int T,
                               const int32_t* perm, int k, int kp, int32_t* ids, float* dists,
                               cudaStream_t st)
{
    const int m = P.max_leaf;
    if (m <= 32) return launch_leaf_f32<1, kDT>(x, P, dp, T, perm, k, kp, ids, dists, st);
    if (m <= 64) return launch_leaf_f32<2, kDT>(x, P, dp, T, perm, k, kp, ids, dists, st);
    if (m <= 128) return launch_leaf_f32<4, kDT>(x, P, dp, T, perm, k, kp, ids, dists, st);
    if (m <= 256) return launch_leaf_f32<8, kDT>(x, P, dp, T, perm, k, kp, ids, dists, st);
    return launch_leaf_f32<16, kDT>(x, P, dp, T, perm, k, kp, ids, dists, st);
}

}  // namespace knng
