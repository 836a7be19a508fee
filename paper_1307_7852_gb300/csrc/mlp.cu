// Learned partitioner: training of the split-feature network.
//
// The paper splits along random principal directions (Sec. 3.4) or random
// projections (appendix after Lemma 1); this library can also split along
// learned features: a network x -> z in (-1, 1)^C (d -> H -> C, GELU, output
// tanh), where level
// l of tree t splits every node at the median of feature pi_t(l).  The
// network is trained on edges (i, j) of k-NN graphs built by the method
// itself, to keep neighbours on the same side of those medians:
//
//   L = sum_c mean_b (z_c(i_b) - z_c(j_b))^2 / (V_c + eps)
//       + lam * sum_{c != c'} corr(z_c, z_c')^2 + mu * sum_c (1 - V_c)^2
// (batch statistics; the last term stops an output from collapsing to a
// constant, which would zero the first two)
//
// All training arithmetic is FP32 in the kernels below: batch sampling
// (Philox), forward and backward GEMMs (tiled SIMT), the loss and its
// gradient through the batch statistics, and Adam.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "../../include/knng.h"
#include "knng_common.cuh"
#include "knng_internal.h"

namespace knng {

// ---------------------------------------------------------------------------
// Tiled FP32 GEMM: C[M][N] = sum_k A(m, k) B(k, n) with A(m, k) = TA ?
// A[k*lda + m] : A[m*lda + k] and B(k, n) = TB ? B[n*ldb + k] : B[k*ldb + n].
// Epilogue: EPI 1 = + bias[n], store pre-activation to aux and GELU to C, 3 =
// tanh(. + bias[n]), 4 = times GELU'(aux) (the backward pass through the
// activation), 5 = one K slice of a reduction: slice z of K (kper entries)
// goes to C + z * (M*N + M), followed by the slice's row sums of A(m, .) (the
// bias gradient), for grad_reduce_kernel.
//
// A thread block holds a TM x TN tile, 256 threads of (TM/16) x (TN/16)
// entries each; the next K step of 32 is loaded into registers while the
// current one is multiplied from shared memory.  TM = 16 / TN = 16 serve the
// network's 16 or 32 outputs, where a 64-wide tile would be mostly padding.
// The weight gradients contract over the batch (K = 8192 rows of a
// 4,096-edge batch against 256 x 96 outputs): without the K slices 8 blocks
// did each whole contraction, most of the call's 3.4 ms; 20 + 9 us with slices
// over about two blocks per SM, and 5 us to add them up.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float gelu_f(float a)
{
    return 0.5f * a * (1.0f + erff(a * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad_f(float a)
{
    return 0.5f * (1.0f + erff(a * 0.70710678118654752f)) + a * 0.39894228040143268f * __expf(-0.5f * a * a);
}

constexpr int kGemmTK = 32;

template <bool TA, bool TB, int EPI, int TM, int TN>
__global__ void __launch_bounds__(256) gemm_kernel(int M, int N, int K, int kper, const float* __restrict__ A, int lda,
                                                   const float* __restrict__ B, int ldb, float* __restrict__ C,
                                                   int ldc, const float* __restrict__ bias, float* __restrict__ aux)
{
    constexpr int TK = kGemmTK, RM = TM / 16, RN = TN / 16;
    constexpr int LA = TM * TK / 256, LB = TN * TK / 256;
    __shared__ float As[TK][TM + 4];
    __shared__ float Bs[TK][TN + 4];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    const int kbeg = blockIdx.z * kper, kend = min(K, kbeg + kper);
    float acc[RM][RN] = {};
    float rsum[RM] = {};
    float ra[LA], rb[LB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int e = tid + 256 * i;
            const int mm = TA ? e % TM : e / TK, kk = TA ? e / TM : e % TK;
            const int m = m0 + mm, k = k0 + kk;
            ra[i] = (m < M && k < kend) ? (TA ? A[(int64_t)k * lda + m] : A[(int64_t)m * lda + k]) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int e = tid + 256 * i;
            const int nn = TB ? e / TK : e % TN, kk = TB ? e % TK : e / TN;
            const int n = n0 + nn, k = k0 + kk;
            rb[i] = (n < N && k < kend) ? (TB ? B[(int64_t)n * ldb + k] : B[(int64_t)k * ldb + n]) : 0.f;
        }
    };
    fetch(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += TK) {
        if (k0 > kbeg) __syncthreads();
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int e = tid + 256 * i;
            As[TA ? e / TM : e % TK][TA ? e % TM : e / TK] = ra[i];
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int e = tid + 256 * i;
            Bs[TB ? e % TK : e / TN][TB ? e / TK : e % TN] = rb[i];
        }
        __syncthreads();
        if (k0 + TK < kend) fetch(k0 + TK);
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float a[RM], b[RN];
#pragma unroll
            for (int i = 0; i < RM; ++i) a[i] = As[kk][ty * RM + i];
#pragma unroll
            for (int j = 0; j < RN; ++j) b[j] = Bs[kk][tx * RN + j];
#pragma unroll
            for (int i = 0; i < RM; ++i) {
#pragma unroll
                for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
                if (EPI == 5) rsum[i] += a[i];
            }
        }
    }
    if (EPI == 5) C += (int64_t)blockIdx.z * ((int64_t)M * N + M);
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int m = m0 + ty * RM + i;
#pragma unroll
        for (int j = 0; j < RN; ++j) {
            const int n = n0 + tx * RN + j;
            if (m >= M || n >= N) continue;
            float v = acc[i][j];
            if (EPI == 1) {
                v += bias[n];
                aux[(int64_t)m * ldc + n] = v;
                v = gelu_f(v);
            } else if (EPI == 3) {
                v = tanhf(v + bias[n]);
            } else if (EPI == 4) {
                v *= gelu_grad_f(aux[(int64_t)m * ldc + n]);
            }
            C[(int64_t)m * ldc + n] = v;
        }
        if (EPI == 5 && blockIdx.x == 0 && tx == 0 && m < M) C[(int64_t)M * N + m] = rsum[i];
    }
}

template <bool TA, bool TB, int EPI, int TM, int TN>
static void gemm(int M, int N, int K, int kper, const float* A, int lda, const float* B, int ldb, float* C, int ldc,
                 const float* bias, float* aux, cudaStream_t st)
{
    dim3 grid((N + TN - 1) / TN, (M + TM - 1) / TM, (K + kper - 1) / kper);
    gemm_kernel<TA, TB, EPI, TM, TN><<<grid, 256, 0, st>>>(M, N, K, kper, A, lda, B, ldb, C, ldc, bias, aux);
    note_launches(1);
}

// K entries per slice of a weight-gradient contraction: about two blocks per
// SM over the output tiles and slices, whole K steps, at least four of them.
static int slice_len(int tiles, int K)
{
    const int slices = std::max(1, 2 * num_sms() / std::max(1, tiles));
    const int len = (K + slices - 1) / slices;
    return std::max(4 * kGemmTK, (len + kGemmTK - 1) / kGemmTK * kGemmTK);
}

// Packed gradient from the slices: entry e of the first c1 (W1 | b1) sums its
// s1 slices, the rest (W2 | b2, c2 entries) its s2.
__global__ void grad_reduce_kernel(int c1, int s1, const float* __restrict__ p1, int c2, int s2,
                                   const float* __restrict__ p2, float* __restrict__ g)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= c1 + c2) return;
    const bool first = e < c1;
    const float* p = first ? p1 + e : p2 + (e - c1);
    const int c = first ? c1 : c2, s = first ? s1 : s2;
    // four running sums keep four loads in flight
    float a[4] = {0.f, 0.f, 0.f, 0.f};
    int z = 0;
    for (; z + 4 <= s; z += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] += p[(int64_t)(z + q) * c];
    for (; z < s; ++z) a[0] += p[(int64_t)z * c];
    g[e] = (a[0] + a[1]) + (a[2] + a[3]);
}

// ---------------------------------------------------------------------------
// Batch sampling: edge b takes a Philox-random point i and a random valid
// slot of its list; row b of Xb is x_i, row B + b is x_j (FP32).
// ---------------------------------------------------------------------------
template <int kDT>
__global__ void sample_batch_kernel(RowLoader<kDT> L, int64_t n, const int32_t* __restrict__ ids, int k, int B,
                                    uint64_t seed, uint32_t step, float* __restrict__ Xb)
{
    const int lane = threadIdx.x & 31;
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= B) return;
    const uint4 w = philox4x32_10(make_uint4((uint32_t)b, step, 0x4C4E4E42u, 0u),
                                  make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const int64_t i = (int64_t)(((uint64_t)w.x << 32 | w.y) % (uint64_t)n);
    int32_t j = -1;
    for (int t = 0; t < k && j < 0; ++t) {
        const int slot = (int)((w.z + (uint32_t)t) % (uint32_t)k);
        j = ids[i * k + slot];
    }
    if (j < 0 || j >= n) j = (int32_t)i;
    for (int c = 4 * lane; c < L.d; c += 128) {
        const float4 a = L.load4(i, c), v = L.load4(j, c);
        const float av[4] = {a.x, a.y, a.z, a.w}, vv[4] = {v.x, v.y, v.z, v.w};
        for (int e = 0; e < 4 && c + e < L.d; ++e) {
            Xb[(int64_t)b * L.d + c + e] = av[e];
            Xb[(int64_t)(B + b) * L.d + c + e] = vv[e];
        }
    }
}

// ---------------------------------------------------------------------------
// Loss and dL/dZ through the batch statistics.  Z: N x C rows, N = 2B.
// Four passes over blocks of kLossRows rows (one block did it all before:
// 0.70 ms of an 8192 x 16 batch, now 49 us in all): column sums; centred second
// moments and the pairs' differences; the statistics and the loss (one
// block, sums of the row blocks in FP64); the gradient.
//   K = corr, S = (z - mean) / sqrt(var + eps), dS = (2/N) S G with
//   G = 2 lam offdiag(K).  S has zero column means, so mean(dS) = 0 and
//   mean(dS_c S_c) = (2/N) sum_{a != c} 2 lam K_ac^2: no pass over the rows
//   is needed for them.
// ---------------------------------------------------------------------------
constexpr int kLossRows = 128;
constexpr int kLossTile = 32;  // rows summed in FP32 before the FP64 sum

// sums[block][C]
__global__ void __launch_bounds__(256) loss_sum_kernel(const float* __restrict__ Z, int N, int C,
                                                       double* __restrict__ sums)
{
    __shared__ double red[256];
    const int tid = threadIdx.x, c = tid % C, per = 256 / C;
    const int rend = min(N, ((int)blockIdx.x + 1) * kLossRows);
    double s = 0.0;
    for (int r = blockIdx.x * kLossRows + tid / C; r < rend; r += per) s += (double)Z[(int64_t)r * C + c];
    red[tid] = s;
    __syncthreads();
    if (tid < C) {
        for (int q = 1; q < per; ++q) s += red[q * C + tid];
        sums[(int64_t)blockIdx.x * C + tid] = s;
    }
}

__device__ __forceinline__ void loss_means(const double* __restrict__ sums, int nblk, int N, int C, float* mu)
{
    const int lane = threadIdx.x & 31;
    for (int c = threadIdx.x >> 5; c < C; c += blockDim.x >> 5) {
        double s = 0.0;
        for (int b = lane; b < nblk; b += 32) s += sums[(int64_t)b * C + c];
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(KNNG_FULL_MASK, s, o);
        if (lane == 0) mu[c] = (float)(s / N);
    }
}

// mom[block][C*C + C]: sums of z_a z_b (centred) and of the squared
// differences of the block's edges.
__global__ void __launch_bounds__(256) loss_moment_kernel(const float* __restrict__ Z, int N, int C,
                                                          const double* __restrict__ sums, double* __restrict__ mom)
{
    __shared__ float mu[32];
    __shared__ float zt[kLossTile][33];
    __shared__ float dt[kLossTile][33];
    const int tid = threadIdx.x, B = N / 2;
    loss_means(sums, gridDim.x, N, C, mu);
    __syncthreads();
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    double accp = 0.0;
    const int rbeg = blockIdx.x * kLossRows, rend = min(N, rbeg + kLossRows);
    const int pairs = C * C;  // 256 or 1024: one or four per thread
    for (int t0 = rbeg; t0 < rend; t0 += kLossTile) {
        __syncthreads();
        for (int e = tid; e < kLossTile * C; e += 256) {
            const int r = t0 + e / C, c = e % C;
            const float z = r < rend ? Z[(int64_t)r * C + c] : mu[c];
            const float dd = (r < rend && r < B) ? z - Z[(int64_t)(r + B) * C + c] : 0.f;
            zt[e / C][c] = z - mu[c];
            dt[e / C][c] = dd;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int pr = tid + 256 * q;
            if (pr < pairs) {
                const int a = pr / C, b = pr % C;
                float s = 0.f;
#pragma unroll 8
                for (int r = 0; r < kLossTile; ++r) s = fmaf(zt[r][a], zt[r][b], s);
                acc[q] += (double)s;
            }
        }
        if (tid < C) {
            float s = 0.f;
#pragma unroll 8
            for (int r = 0; r < kLossTile; ++r) s = fmaf(dt[r][tid], dt[r][tid], s);
            accp += (double)s;
        }
    }
    double* o = mom + (int64_t)blockIdx.x * (pairs + C);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (tid + 256 * q < pairs) o[tid + 256 * q] = acc[q];
    if (tid < C) o[pairs + tid] = accp;
}

// stats: mean[C] | var[C] | P[C] | K[C*C] (floats), and the loss.
__global__ void __launch_bounds__(1024) loss_stats_kernel(int N, int C, int nblk, float lam, float eps, float mus,
                                                          const double* __restrict__ sums,
                                                          const double* __restrict__ mom, float* __restrict__ stats,
                                                          float* __restrict__ loss)
{
    __shared__ double var[32], P[32], part[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int pairs = C * C, tot = pairs + C;
    float* Kc = stats + 3 * C;
    loss_means(sums, nblk, N, C, stats);
    // the diagonal and the differences first: a warp per column
    for (int c = w; c < C; c += 32) {
        double sv = 0.0, sp = 0.0;
        for (int b = lane; b < nblk; b += 32) {
            sv += mom[(int64_t)b * tot + c * C + c];
            sp += mom[(int64_t)b * tot + pairs + c];
        }
        for (int o = 16; o >= 1; o >>= 1) {
            sv += __shfl_xor_sync(KNNG_FULL_MASK, sv, o);
            sp += __shfl_xor_sync(KNNG_FULL_MASK, sp, o);
        }
        if (lane == 0) {
            var[c] = sv / N;
            P[c] = sp / (N / 2);
            stats[C + c] = (float)var[c];
            stats[2 * C + c] = (float)P[c];
        }
    }
    __syncthreads();
    // correlations: 1024 / pairs threads per pair, neighbours in the block
    // sums' order so that a warp's loads are contiguous
    double off = 0.0;
    __shared__ double seg[1024];
    const int grp = 1024 / pairs, pr = tid % pairs, g0 = tid / pairs;
    double s = 0.0;
    for (int b = g0; b < nblk; b += grp) s += mom[(int64_t)b * tot + pr];
    seg[tid] = s;
    __syncthreads();
    if (tid < pairs) {
        for (int q = 1; q < grp; ++q) s += seg[q * pairs + tid];
        const int a = tid / C, b = tid % C;
        const double k = s / N / sqrt((var[a] + eps) * (var[b] + eps));
        Kc[tid] = (float)k;
        if (a != b) off = k * k;
    }
    for (int o = 16; o >= 1; o >>= 1) off += __shfl_xor_sync(KNNG_FULL_MASK, off, o);
    if (lane == 0) part[w] = off;
    __syncthreads();
    if (tid == 0) {
        double L = 0.0, Ld = 0.0, Ls = 0.0;
        for (int a = 0; a < C; ++a) {
            L += P[a] / (var[a] + eps);
            Ls += (1.0 - var[a]) * (1.0 - var[a]);
        }
        for (int q = 0; q < 32; ++q) Ld += part[q];
        *loss = (float)(L + lam * Ld + mus * Ls);
    }
}

// dL/dZ of every entry, taken through the output tanh: dZpre = dZ (1 - Z^2).
__global__ void __launch_bounds__(256) loss_grad_kernel(const float* __restrict__ Z, int N, int C, float lam, float eps,
                                                        float mus, const float* __restrict__ stats,
                                                        float* __restrict__ dZ)
{
    __shared__ float mu[32], isig[32], P[32], var[32], m2[32];
    __shared__ float Kc[32 * 33];
    __shared__ float st[256];
    const int tid = threadIdx.x, B = N / 2;
    for (int e = tid; e < C * C; e += 256) Kc[(e / C) * 33 + e % C] = stats[3 * C + e];
    if (tid < C) {
        mu[tid] = stats[tid];
        var[tid] = stats[C + tid];
        P[tid] = stats[2 * C + tid];
        isig[tid] = 1.f / sqrtf(var[tid] + eps);
    }
    __syncthreads();
    if (tid < C) {
        float s = 0.f;
        for (int a = 0; a < C; ++a)
            if (a != tid) s = fmaf(Kc[a * 33 + tid], Kc[a * 33 + tid], s);
        m2[tid] = 2.f * lam * s * (2.f / N);
    }
    const int c = tid % C, rl = tid / C, per = 256 / C;
    const int r = blockIdx.x * per + rl;
    const float z = r < N ? Z[(int64_t)r * C + c] : mu[c];
    const float zc = z - mu[c];
    st[tid] = zc * isig[c];  // S of the block's rows
    __syncthreads();
    if (r >= N) return;
    const float ve = var[c] + eps;
    float g = (-P[c] / (ve * ve) - 2.f * mus * (1.f - var[c])) * (2.f / N) * zc;
    const float other = Z[(int64_t)(r < B ? r + B : r - B) * C + c];
    g += (1.f / ve) * (2.f / B) * (z - other);
    float ds = 0.f;
    for (int a = 0; a < C; ++a)
        if (a != c) ds = fmaf(st[rl * C + a], 2.f * lam * Kc[a * 33 + c], ds);
    ds *= 2.f / N;
    g += (ds - st[tid] * m2[c]) * isig[c];
    dZ[(int64_t)r * C + c] = g * (1.f - z * z);
}

// Adam step on the packed parameters.
__global__ void adam_kernel(int count, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= count) return;
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.f - b1) * gg;
    const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    w[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// ---------------------------------------------------------------------------
// Model object
// ---------------------------------------------------------------------------
constexpr float kLam = 0.05f, kEps = 1e-4f, kSpread = 1.0f;

// Sizes of one batch's scratch: row blocks of the loss, length and number of
// the K slices of the two weight gradients, entries per slice.
struct GradScratch {
    int nblk, k1, s1, c1, k2, s2, c2;
    size_t bytes;
};
static GradScratch grad_scratch(const MlpModel* M, int N)
{
    GradScratch g;
    const int d = M->d, H = M->H, C = M->C;
    g.nblk = (N + kLossRows - 1) / kLossRows;
    g.k1 = slice_len(((H + 63) / 64) * ((d + 63) / 64), N);
    g.s1 = (N + g.k1 - 1) / g.k1;
    g.c1 = H * d + H;
    g.k2 = slice_len(((C + 15) / 16) * ((H + 63) / 64), N);
    g.s2 = (N + g.k2 - 1) / g.k2;
    g.c2 = C * H + C;
    g.bytes = sizeof(double) * (size_t)g.nblk * (C * C + 2 * C) +
              sizeof(float) * (3 * (size_t)C + (size_t)C * C + (size_t)g.s1 * g.c1 + (size_t)g.s2 * g.c2);
    return g;
}

static int ensure_rows(MlpModel* M, int rows)
{
    // (fewer rows can need a little more: their slices are shorter)
    const size_t need = grad_scratch(M, rows).bytes;
    if (need > M->part_bytes) {
        cudaFree(M->part);
        M->part = nullptr;
        M->part_bytes = 0;
        if (cudaMalloc(&M->part, need) != cudaSuccess) {
            cudaGetLastError();
            return KNNG_ERR_OOM;
        }
        M->part_bytes = need;
    }
    if (rows <= M->cap_rows) return KNNG_OK;
    cudaFree(M->Xb);
    cudaFree(M->A);
    cudaFree(M->Hh);
    cudaFree(M->Z);
    cudaFree(M->dZ);
    M->Xb = M->A = M->Hh = M->Z = M->dZ = nullptr;
    M->cap_rows = 0;
    if (cudaMalloc(&M->Xb, sizeof(float) * (size_t)rows * M->d) != cudaSuccess ||
        cudaMalloc(&M->A, sizeof(float) * (size_t)rows * M->H) != cudaSuccess ||
        cudaMalloc(&M->Hh, sizeof(float) * (size_t)rows * M->H) != cudaSuccess ||
        cudaMalloc(&M->Z, sizeof(float) * (size_t)rows * M->C) != cudaSuccess ||
        cudaMalloc(&M->dZ, sizeof(float) * (size_t)rows * M->C) != cudaSuccess) {
        cudaGetLastError();
        return KNNG_ERR_OOM;
    }
    M->cap_rows = rows;
    return KNNG_OK;
}

// Loss and packed gradient of the batch Xb (rows = 2B) into M->g.
static cudaError_t loss_grad(MlpModel* M, const float* Xb, int B, cudaStream_t st)
{
    const int N = 2 * B, d = M->d, H = M->H, C = M->C;
    gemm<false, true, 1, 64, 64>(N, H, d, d, Xb, d, M->W1(), d, M->Hh, H, M->b1(), M->A, st);
    gemm<false, true, 3, 64, 16>(N, C, H, H, M->Hh, H, M->W2(), H, M->Z, C, M->b2(), nullptr, st);
    // scratch of this batch: FP64 sums of the row blocks | statistics |
    // slices of the two weight gradients (sizes: grad_scratch)
    const GradScratch gs = grad_scratch(M, N);
    char* base = reinterpret_cast<char*>(M->part);
    double* sums = reinterpret_cast<double*>(base);
    double* mom = sums + (size_t)gs.nblk * C;
    float* stats = reinterpret_cast<float*>(mom + (size_t)gs.nblk * (C * C + C));
    float* p1 = stats + 3 * C + C * C;
    float* p2 = p1 + (size_t)gs.s1 * gs.c1;
    loss_sum_kernel<<<gs.nblk, 256, 0, st>>>(M->Z, N, C, sums);
    loss_moment_kernel<<<gs.nblk, 256, 0, st>>>(M->Z, N, C, sums, mom);
    loss_stats_kernel<<<1, 1024, 0, st>>>(N, C, gs.nblk, kLam, kEps, kSpread, sums, mom, stats, M->loss);
    loss_grad_kernel<<<(N + 256 / C - 1) / (256 / C), 256, 0, st>>>(M->Z, N, C, kLam, kEps, kSpread, stats, M->dZ);
    note_launches(4);
    // dW2 = dZ^T Hh and db2, in slices of the batch
    gemm<true, false, 5, 16, 64>(C, H, N, gs.k2, M->dZ, C, M->Hh, H, p2, H, nullptr, nullptr, st);
    // dA = (dZ W2) GELU'(A) (into Hh)
    gemm<false, false, 4, 64, 64>(N, H, C, C, M->dZ, C, M->W2(), H, M->Hh, H, nullptr, M->A, st);
    // dW1 = dA^T X and db1
    gemm<true, false, 5, 64, 64>(H, d, N, gs.k1, M->Hh, H, Xb, d, p1, d, nullptr, nullptr, st);
    grad_reduce_kernel<<<(gs.c1 + gs.c2 + 255) / 256, 256, 0, st>>>(gs.c1, gs.s1, p1, gs.c2, gs.s2, p2, M->g);
    note_launches(1);
    return cudaGetLastError();
}

int mlp_dims(const MlpModel* M, int* d, int* H, int* C)
{
    *d = M->d;
    *H = M->H;
    *C = M->C;
    return KNNG_OK;
}

}  // namespace knng

using namespace knng;

struct knng_mlp {
    MlpModel m;
};

extern "C" {

int knng_mlp_create(int32_t device, int32_t d_in, int32_t hidden, int32_t d_out, uint64_t seed, knng_mlp** out)
{
    if (!out) return KNNG_ERR_INVALID_ARG;
    *out = nullptr;
    if (d_in < 1 || d_in > 1024 || hidden < 16 || hidden > 256 || hidden % 16 || (d_out != 16 && d_out != 32))
        return KNNG_ERR_INVALID_ARG;
    int cnt = 0;
    if (cudaGetDeviceCount(&cnt) != cudaSuccess || device < 0 || device >= cnt) {
        cudaGetLastError();
        return KNNG_ERR_INVALID_ARG;
    }
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(device);
    knng_mlp* o = new knng_mlp();
    MlpModel& M = o->m;
    M.device = device;
    M.d = d_in;
    M.H = hidden;
    M.C = d_out;
    M.count = (int64_t)hidden * d_in + hidden + (int64_t)d_out * hidden + d_out;
    std::vector<float> host(M.count, 0.f);
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    for (int64_t e = 0; e < (int64_t)hidden * d_in; ++e) host[e] = (float)(nd(rng) / std::sqrt((double)d_in));
    float* w2 = host.data() + (int64_t)hidden * d_in + hidden;
    for (int64_t e = 0; e < (int64_t)d_out * hidden; ++e) w2[e] = (float)(nd(rng) / std::sqrt((double)hidden));
    int rc = KNNG_OK;
    if (cudaMalloc(&M.w, sizeof(float) * M.count) != cudaSuccess ||
        cudaMalloc(&M.g, sizeof(float) * M.count) != cudaSuccess ||
        cudaMalloc(&M.am, sizeof(float) * M.count) != cudaSuccess ||
        cudaMalloc(&M.av, sizeof(float) * M.count) != cudaSuccess || cudaMalloc(&M.loss, sizeof(float)) != cudaSuccess)
        rc = KNNG_ERR_OOM;
    if (rc == KNNG_OK) {
        cudaMemcpy(M.w, host.data(), sizeof(float) * M.count, cudaMemcpyHostToDevice);
        cudaMemset(M.am, 0, sizeof(float) * M.count);
        cudaMemset(M.av, 0, sizeof(float) * M.count);
    }
    cudaSetDevice(prev);
    if (rc != KNNG_OK) {
        cudaGetLastError();
        knng_mlp_destroy(o);
        return rc;
    }
    *out = o;
    return KNNG_OK;
}

int knng_mlp_destroy(knng_mlp* o)
{
    if (!o) return KNNG_ERR_INVALID_ARG;
    MlpModel& M = o->m;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(M.device);
    cudaDeviceSynchronize();
    for (float* p : {M.w, M.g, M.am, M.av, M.Xb, M.A, M.Hh, M.Z, M.dZ, M.part, M.loss}) cudaFree(p);
    cudaFree(M.img);
    cudaSetDevice(prev);
    delete o;
    return KNNG_OK;
}

int knng_mlp_param_count(const knng_mlp* o, int64_t* count)
{
    if (!o || !count) return KNNG_ERR_INVALID_ARG;
    *count = o->m.count;
    return KNNG_OK;
}

int knng_mlp_get_params(const knng_mlp* o, float* host)
{
    if (!o || !host) return KNNG_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(o->m.device);
    const cudaError_t e = cudaMemcpy(host, o->m.w, sizeof(float) * o->m.count, cudaMemcpyDeviceToHost);
    cudaSetDevice(prev);
    return e == cudaSuccess ? KNNG_OK : KNNG_ERR_CUDA;
}

int knng_mlp_set_params(knng_mlp* o, const float* host)
{
    if (!o || !host) return KNNG_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(o->m.device);
    const cudaError_t e = cudaMemcpy(o->m.w, host, sizeof(float) * o->m.count, cudaMemcpyHostToDevice);
    o->m.img_stale = true;
    cudaSetDevice(prev);
    return e == cudaSuccess ? KNNG_OK : KNNG_ERR_CUDA;
}

int knng_mlp_get_adam_state(const knng_mlp* o, float* m1_host, float* m2_host, int64_t* t)
{
    if (!o || !m1_host || !m2_host || !t) return KNNG_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(o->m.device);
    cudaError_t e = cudaMemcpy(m1_host, o->m.am, sizeof(float) * o->m.count, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(m2_host, o->m.av, sizeof(float) * o->m.count, cudaMemcpyDeviceToHost);
    *t = o->m.adam_t;
    cudaSetDevice(prev);
    return e == cudaSuccess ? KNNG_OK : KNNG_ERR_CUDA;
}

int knng_mlp_set_adam_state(knng_mlp* o, const float* m1_host, const float* m2_host, int64_t t)
{
    if (!o || !m1_host || !m2_host || t < 0) return KNNG_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(o->m.device);
    cudaError_t e = cudaMemcpy(o->m.am, m1_host, sizeof(float) * o->m.count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(o->m.av, m2_host, sizeof(float) * o->m.count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) o->m.adam_t = t;
    cudaSetDevice(prev);
    return e == cudaSuccess ? KNNG_OK : KNNG_ERR_CUDA;
}

int knng_mlp_loss_grad(knng_mlp* o, const float* Xpairs, int32_t B, float* loss, float* grad, void* stream)
{
    if (!o || !Xpairs || B < 2 || !loss || !grad) return KNNG_ERR_INVALID_ARG;
    MlpModel& M = o->m;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(M.device);
    int rc = ensure_rows(&M, 2 * B);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (rc == KNNG_OK) {
        cudaError_t e = loss_grad(&M, Xpairs, B, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(grad, M.g, sizeof(float) * M.count, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(loss, M.loss, sizeof(float), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = KNNG_ERR_CUDA;
    }
    cudaSetDevice(prev);
    return rc;
}

int knng_mlp_train(knng_mlp* o, const void* X, int32_t dtype, int64_t n, int32_t d, int64_t ld, const int32_t* ids,
                   int32_t k, int32_t steps, int32_t batch_edges, float lr, uint64_t seed, float* last_loss,
                   void* stream)
{
    if (!o || !X || !ids || n < 2 || k < 1 || steps < 0 || batch_edges < 2 || lr <= 0.f) return KNNG_ERR_INVALID_ARG;
    if (dtype != KNNG_DTYPE_F32 && dtype != KNNG_DTYPE_F16 && dtype != KNNG_DTYPE_U8) return KNNG_ERR_INVALID_ARG;
    MlpModel& M = o->m;
    if (d != M.d || ld < d || ld >= (int64_t)1 << 31 || n >= (int64_t)1 << 31) return KNNG_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(M.device);
    int rc = ensure_rows(&M, 2 * batch_edges);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t es = dtype == KNNG_DTYPE_F16 ? 2 : dtype == KNNG_DTYPE_U8 ? 1 : 4;
    const size_t align = dtype == KNNG_DTYPE_F16 ? 8 : dtype == KNNG_DTYPE_U8 ? 4 : 16;
    const bool vec = ((uintptr_t)X % align == 0) && ((size_t)ld * es % align == 0);
    for (int s = 0; s < steps && rc == KNNG_OK; ++s) {
        const int blocks = (batch_edges * 32 + 255) / 256;
        if (dtype == KNNG_DTYPE_F16) {
            RowLoader<kDtF16> L{X, ld, d, vec};
            sample_batch_kernel<kDtF16><<<blocks, 256, 0, st>>>(L, n, ids, k, batch_edges, seed, (uint32_t)s, M.Xb);
        } else if (dtype == KNNG_DTYPE_U8) {
            RowLoader<kDtU8> L{X, ld, d, vec};
            sample_batch_kernel<kDtU8><<<blocks, 256, 0, st>>>(L, n, ids, k, batch_edges, seed, (uint32_t)s, M.Xb);
        } else {
            RowLoader<kDtF32> L{X, ld, d, vec};
            sample_batch_kernel<kDtF32><<<blocks, 256, 0, st>>>(L, n, ids, k, batch_edges, seed, (uint32_t)s, M.Xb);
        }
        note_launches(1);
        cudaError_t e = loss_grad(&M, M.Xb, batch_edges, st);
        ++M.adam_t;
        const float c1 = 1.f - powf(0.9f, (float)M.adam_t), c2 = 1.f - powf(0.999f, (float)M.adam_t);
        adam_kernel<<<(int)((M.count + 255) / 256), 256, 0, st>>>((int)M.count, M.w, M.g, M.am, M.av, lr, 0.9f,
                                                                 0.999f, 1e-8f, c1, c2);
        note_launches(1);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) rc = KNNG_ERR_CUDA;
    }
    M.img_stale = true;
    if (rc == KNNG_OK && last_loss) {
        if (cudaMemcpyAsync(last_loss, M.loss, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            rc = KNNG_ERR_CUDA;
    }
    cudaSetDevice(prev);
    return rc;
}

int knng_mlp_save(const knng_mlp* o, const char* path)
{
    if (!o || !path) return KNNG_ERR_INVALID_ARG;
    std::vector<float> host(o->m.count);
    if (knng_mlp_get_params(o, host.data()) != KNNG_OK) return KNNG_ERR_CUDA;
    FILE* f = fopen(path, "wb");
    if (!f) return KNNG_ERR_INVALID_ARG;
    const int32_t hdr[4] = {0x4B4E4D31 /* "KNM1" */, o->m.d, o->m.H, o->m.C};
    const bool ok = fwrite(hdr, sizeof hdr, 1, f) == 1 && fwrite(host.data(), sizeof(float), host.size(), f) == host.size();
    fclose(f);
    return ok ? KNNG_OK : KNNG_ERR_INVALID_ARG;
}

int knng_mlp_load(knng_mlp* o, const char* path)
{
    if (!o || !path) return KNNG_ERR_INVALID_ARG;
    FILE* f = fopen(path, "rb");
    if (!f) return KNNG_ERR_INVALID_ARG;
    int32_t hdr[4];
    std::vector<float> host(o->m.count);
    bool ok = fread(hdr, sizeof hdr, 1, f) == 1 && hdr[0] == 0x4B4E4D31 && hdr[1] == o->m.d && hdr[2] == o->m.H &&
              hdr[3] == o->m.C && fread(host.data(), sizeof(float), host.size(), f) == host.size();
    fclose(f);
    if (!ok) return KNNG_ERR_INVALID_ARG;
    return knng_mlp_set_params(o, host.data());
}

}  // extern "C"

namespace knng {
MlpModel* mlp_model(knng_mlp* o) { return o ? &o->m : nullptr; }
}  // namespace knng
