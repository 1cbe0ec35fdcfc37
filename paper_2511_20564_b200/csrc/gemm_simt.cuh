// fp32-FMA tiled GEMM for the true-fp32 path (rel 1e-5 against float64 rules out TF32) and as
// the reference path for shapes the tensor-core kernels do not take.
//   C(m, n) = sum_k A(m, k) * B(n, k)
// A_KM: A is stored k-major (element (m,k) at A[k*lda + m]) instead of m-major (A[m*lda + k]).
// B_KN: B is stored k-major (element (n,k) at B[k*ldb + n]) instead of n-major (B[n*ldb + k]).
// M and/or K may live on the device (m_dev / k_dev); the grid is sized for the caps.
// gridDim.z splits K; the epilogue receives the split index.
#pragma once

#include <cooperative_groups.h>
#include <string.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"

namespace e2egrec {

// gemm_simt_kernel, for bf16 operands and large fp32 products (the others: gemm_async_kernel below).  At the sizes of a batch the
// time is the K loop's chain of loads, not its arithmetic: the next 64 x 32 tiles are loaded into registers (four values at a
// time where rows are aligned) while the current ones are multiplied out of shared memory, two buffers, one barrier per step.
// Loading, storing and multiplying in turn with steps of 16 took 1.7 us a step.
constexpr int kGemmBM = 64, kGemmBN = 64, kGemmBK = 32, kGemmThreads = 256;

// four values from p on, `n` of them there
template <typename T> __device__ __forceinline__ float4 gemm_load4(const T *p, int n, bool vec)
{
    if (vec && n >= 4) {
        if constexpr (sizeof(T) == 4) {
            return *reinterpret_cast<const float4 *>(p);
        } else {
            const uint2 r = *reinterpret_cast<const uint2 *>(p);
            return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16),
                               __uint_as_float(r.y & 0xFFFF0000u));
        }
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) v.x = to_float<T>(p[0]);
    if (n > 1) v.y = to_float<T>(p[1]);
    if (n > 2) v.z = to_float<T>(p[2]);
    if (n > 3) v.w = to_float<T>(p[3]);
    return v;
}

// One operand's 64 x kGemmBK tile: two groups of four values per thread, along k (rows of the matrix are rows of the tile)
// or along the tile's rows (KM: rows of the matrix are lines of k).
template <typename T, bool KM>
struct GemmTile {
    static constexpr int kLd = 64 + 4;
    const T *p;
    int64_t ld, rows, r0;
    bool vec;
    __device__ GemmTile(const T *p_, int64_t ld_, int64_t rows_, int64_t r0_) : p(p_), ld(ld_), rows(rows_), r0(r0_)
    {
        vec = (ld * (int64_t)sizeof(T)) % (4 * sizeof(T)) == 0 && reinterpret_cast<uintptr_t>(p) % (4 * sizeof(T)) == 0;
    }
    __device__ __forceinline__ void load(float4 (&v)[2], int64_t k0, int64_t ke) const
    {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int id = threadIdx.x + t * kGemmThreads;
            v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (KM) {
                const int64_t k = k0 + (id >> 4), r = r0 + (id & 15) * 4;
                if (k < ke && r < rows) v[t] = gemm_load4(p + k * ld + r, (int)min((int64_t)4, rows - r), vec);
            } else {
                const int64_t r = r0 + (id >> 3), k = k0 + (id & 7) * 4;
                if (r < rows && k < ke) v[t] = gemm_load4(p + r * ld + k, (int)min((int64_t)4, ke - k), vec);
            }
        }
    }
    __device__ __forceinline__ void store(const float4 (&v)[2], float (*s)[kLd]) const
    {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int id = threadIdx.x + t * kGemmThreads;
            if (KM) {
                *reinterpret_cast<float4 *>(&s[id >> 4][(id & 15) * 4]) = v[t];
            } else {
                const int r = id >> 3, k = (id & 7) * 4;
                s[k][r] = v[t].x; s[k + 1][r] = v[t].y; s[k + 2][r] = v[t].z; s[k + 3][r] = v[t].w;
            }
        }
    }
};

template <typename T, bool A_KM, bool B_KN, class Epi>
__global__ void __launch_bounds__(kGemmThreads)
gemm_simt_kernel(const T *A, int64_t lda, const T *B, int64_t ldb, int64_t M_host, int N, int64_t K_host, const int32_t *m_dev,
                 const int32_t *k_dev, Epi epi)
{
    __shared__ __align__(16) float As[2][kGemmBK][kGemmBM + 4];
    __shared__ __align__(16) float Bs[2][kGemmBK][kGemmBN + 4];
    pdl_wait();
    const int64_t M = m_dev ? min((int64_t)__ldcg(m_dev), M_host) : M_host;
    const int64_t K = k_dev ? min((int64_t)__ldcg(k_dev), K_host) : K_host;
    const int64_t m0 = (int64_t)blockIdx.x * kGemmBM;
    const int n0 = blockIdx.y * kGemmBN;
    if (m0 >= M) return;
    // K range of this split, a multiple of the k tile
    const int64_t k_per = ceil_div(ceil_div(K, (int64_t)gridDim.z), kGemmBK) * kGemmBK;
    const int64_t kb = (int64_t)blockIdx.z * k_per;
    const int64_t ke = min(K, kb + k_per);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    // kFold (products that contract over the rows of a batch, thousands of terms): every K step is summed by itself and added
    // to `total`, so that a chain of additions is 32 + K / 32 long and not K
    constexpr bool kFold = A_KM && B_KN;
    float acc[4][4], total[kFold ? 4 : 1][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc[i][j] = 0.f;
            if (kFold) total[i][j] = 0.f;
        }

    const GemmTile<T, A_KM> ta(A, lda, M, m0);
    const GemmTile<T, B_KN> tb(B, ldb, N, n0);
    float4 va[2], vb[2];
    if (kb < ke) {
        ta.load(va, kb, ke);
        tb.load(vb, kb, ke);
        ta.store(va, As[0]);
        tb.store(vb, Bs[0]);
    }
    __syncthreads();
    int cur = 0;
    for (int64_t k0 = kb; k0 < ke; k0 += kGemmBK, cur ^= 1) {
        const bool more = k0 + kGemmBK < ke;
        if (more) {
            ta.load(va, k0 + kGemmBK, ke);
            tb.load(vb, k0 + kGemmBK, ke);
        }
#pragma unroll 8
        for (int kk = 0; kk < kGemmBK; ++kk) {
            const float4 a4 = *reinterpret_cast<const float4 *>(&As[cur][kk][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4 *>(&Bs[cur][kk][tx * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (more) {
            ta.store(va, As[cur ^ 1]);
            tb.store(vb, Bs[cur ^ 1]);
        }
        __syncthreads();
        if (kFold) {                           // behind the barrier: before it, the stores waited (35.3 and 36.9 us, 1000 x 320 x 320 gate)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    total[i][j] += acc[i][j];
                    acc[i][j] = 0.f;
                }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t m = m0 + ty * 4 + i;
            const int n = n0 + tx * 4 + j;
            if (m < M && n < N) epi(m, n, kFold ? total[kFold ? i : 0][j] : acc[i][j], blockIdx.z);
        }
}

// The same product of fp32 operands, for batches whose few tiles leave most of an SM idle: the tiles are copied to shared memory
// asynchronously, as they lie in memory (rows of k, or lines of k), kGemmStages - 1 K steps ahead, and two groups of 256
// threads take half of every K step each; their sums are added at the end.  What bounds it is latency at 16 warps per SM (products
// of the forward pass, 86 registers) or 32 (the others, 64 registers).
// B200, fp32 step of 777 seeds at fanouts 25, 15, 100 and 72 values, its six products together (us) and the step: loads through
// registers one step ahead, one group 88, 163; copies, one group 74, 154; two groups 144; four groups (64 registers, spills) 166;
// 128 threads of 8 x 4 values instead of 256 of 4 x 4 164.  No chain of additions is longer than in gemm_simt_kernel.
constexpr int kGemmStages = 4, kGemmGroups = 2, kAsyncThreads = kGemmThreads * kGemmGroups;
template <bool KM> struct AsyncTile {
    static constexpr int kLd = KM ? 64 + 4 : kGemmBK + 4;        // floats per line: 64 values of a k, or kGemmBK of a row
    static constexpr int kFloats = (KM ? kGemmBK : 64) * kLd;
    // requests the tile of rows r0 .. r0 + 63 and k0 .. k0 + kGemmBK - 1; values beyond `rows` and `ke` read zero
    static __device__ __forceinline__ void request(float *s, const float *__restrict__ p, int64_t ld, int64_t rows, int64_t r0, int64_t k0,
                                                   int64_t ke, bool vec)
    {
#pragma unroll
        for (int t = 0; t < (512 + kAsyncThreads - 1) / kAsyncThreads; ++t) {
            const int id = threadIdx.x + t * kAsyncThreads;
            if (512 % kAsyncThreads && id >= 512) break;
            const int line = KM ? id >> 4 : id >> 3, col = (KM ? id & 15 : id & 7) * 4;
            const int64_t l = (KM ? k0 : r0) + line, c = (KM ? r0 : k0) + col, l_end = KM ? ke : rows, c_end = KM ? rows : ke;
            const int n = l < l_end ? (int)max((int64_t)0, min((int64_t)4, c_end - c)) : 0;
            const float *src = n > 0 ? p + l * ld + c : p;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s + line * kLd + col);
            if (vec) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n * 4) : "memory");
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * e), "l"(e < n ? src + e : p), "r"(e < n ? 4 : 0)
                                 : "memory");
            }
        }
    }
};
template <bool A_KM, bool B_KN> constexpr size_t gemm_async_smem() { return (size_t)kGemmStages * (AsyncTile<A_KM>::kFloats + AsyncTile<B_KN>::kFloats) * 4; }

template <bool A_KM, bool B_KN, class Epi>
__global__ void __launch_bounds__(kAsyncThreads)
gemm_async_kernel(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t M_host, int N, int64_t K_host, const int32_t *m_dev,
                  const int32_t *k_dev, Epi epi)
{
    using TA = AsyncTile<A_KM>;
    using TB = AsyncTile<B_KN>;
    extern __shared__ __align__(16) float gemm_sm[];
    pdl_wait();
    const int64_t M = m_dev ? min((int64_t)__ldcg(m_dev), M_host) : M_host;
    const int64_t K = k_dev ? min((int64_t)__ldcg(k_dev), K_host) : K_host;
    const int64_t m0 = (int64_t)blockIdx.x * kGemmBM;
    const int n0 = blockIdx.y * kGemmBN;
    if (m0 >= M) return;
    const int64_t k_per = ceil_div(ceil_div(K, (int64_t)gridDim.z), kGemmBK) * kGemmBK;
    const int64_t kb = (int64_t)blockIdx.z * k_per;
    const int64_t ke = min(K, kb + k_per);
    const int steps = kb < ke ? (int)ceil_div(ke - kb, kGemmBK) : 0;
    const int tx = threadIdx.x & 15, ty = (threadIdx.x & (kGemmThreads - 1)) >> 4, g = threadIdx.x / kGemmThreads;
    constexpr bool kFold = A_KM && B_KN;                         // as in gemm_simt_kernel
    float acc[4][4], total[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            acc[i][j] = 0.f;
            if (kFold) total[i][j] = 0.f;
        }
    const bool vec_a = lda % 4 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0, vec_b = ldb % 4 == 0 && reinterpret_cast<uintptr_t>(B) % 16 == 0;
    auto request = [&](int step) {
        if (step < steps) {
            float *s = gemm_sm + (step % kGemmStages) * (TA::kFloats + TB::kFloats);
            TA::request(s, A, lda, M, m0, kb + (int64_t)step * kGemmBK, ke, vec_a);
            TB::request(s + TA::kFloats, B, ldb, N, n0, kb + (int64_t)step * kGemmBK, ke, vec_b);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kGemmStages - 1; ++i) request(i);
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGemmStages - 2) : "memory");
        __syncthreads();                                         // step's tiles are there, and everybody has left the buffer that is filled next
        request(step + kGemmStages - 1);
        const float *sa = gemm_sm + (step % kGemmStages) * (TA::kFloats + TB::kFloats), *sb = sa + TA::kFloats;
#pragma unroll
        for (int q0 = 0; q0 < kGemmBK / 4 / kGemmGroups; ++q0) {
            const int q = g * (kGemmBK / 4 / kGemmGroups) + q0;
            // rows ty * 4 + i; columns tx + 16 j (rows of k: 16 lines side by side, no bank twice) or tx * 4 + j (lines of k)
            float a[4][4], b[4][4];                              // [k][row], [k][column]
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(A_KM ? sa + (4 * q + i) * TA::kLd + ty * 4 : sa + (ty * 4 + i) * TA::kLd + 4 * q);
                const float x[4] = {v.x, v.y, v.z, v.w};
                const float4 w = *reinterpret_cast<const float4 *>(B_KN ? sb + (4 * q + i) * TB::kLd + tx * 4 : sb + (tx + 16 * i) * TB::kLd + 4 * q);
                const float y[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    a[A_KM ? i : e][A_KM ? e : i] = x[e];
                    b[B_KN ? i : e][B_KN ? e : i] = y[e];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[k][i], b[k][j], acc[i][j]);
        }
        if (kFold) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    total[i][j] += acc[i][j];
                    acc[i][j] = 0.f;
                }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // the groups' sums in the order of the groups
    float (*sum)[4] = kFold ? total : acc;
    __syncthreads();
    if (g > 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(gemm_sm + (((g - 1) * 4 + i) * kGemmThreads + (threadIdx.x & (kGemmThreads - 1))) * 4) =
                make_float4(sum[i][0], sum[i][1], sum[i][2], sum[i][3]);
    }
    __syncthreads();
    if (g > 0) return;
#pragma unroll
    for (int o = 0; o < kGemmGroups - 1; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(gemm_sm + ((o * 4 + i) * kGemmThreads + threadIdx.x) * 4);
            sum[i][0] += v.x; sum[i][1] += v.y; sum[i][2] += v.z; sum[i][3] += v.w;
        }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t m = m0 + ty * 4 + i;
            const int n = n0 + (B_KN ? tx * 4 + j : tx + 16 * j);
            if (m < M && n < N) epi(m, n, sum[i][j], blockIdx.z);
        }
}

// Which of the two takes an fp32 product.  The asynchronous one needs tiles that wait for their loads: up to 65536 rows of capacity
// (as M or as K) and, in products over rows, 4096 tiles.  Beyond, tiles hide each other's loads, and most of them hold no live row
// at all: one or two blocks of 512 threads per SM, four of the other kernel's 256, have to come and go for those.  B200, us by
// the asynchronous / the other kernel: forward of 2048 and 8192 seeds of 256 values at fanouts 15, 10 (32768 and 131072 rows) 155 / 173
// and 393 / 369, training step of 2048 and 8192 seeds of 128 values 169 / 188 and 377 / 348, of 4096 seeds of 64 at 25, 15 185 / 167.
constexpr int64_t kAsyncRows = 65536, kAsyncTiles = 4096;
template <typename T, bool A_KM, bool B_KN, class Epi>
inline void launch_gemm_simt(bool chain, dim3 grid, cudaStream_t st, const T *A, int64_t lda, const T *B, int64_t ldb, int64_t M, int N,
                             int64_t K, const int32_t *m_dev, const int32_t *k_dev, const Epi &epi)
{
    note_launch();
    if constexpr (sizeof(T) == 4) {
        if (A_KM ? K <= kAsyncRows : M <= kAsyncRows && (int64_t)grid.x * grid.y <= kAsyncTiles) {
            constexpr size_t smem = gemm_async_smem<A_KM, B_KN>();
            static std::atomic<bool> set[64] = {};               // per device; two threads may both raise the limit
            int dev = 0;
            cudaGetDevice(&dev);
            if (dev < 0 || dev >= 64 || !set[dev].load(std::memory_order_relaxed)) {
                cudaFuncSetAttribute(gemm_async_kernel<A_KM, B_KN, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (dev >= 0 && dev < 64) set[dev].store(true, std::memory_order_relaxed);
            }
            launch_pdl(chain, gemm_async_kernel<A_KM, B_KN, Epi>, grid, dim3(kAsyncThreads), smem, st, A, lda, B, ldb, M, N, K, m_dev, k_dev, epi);
            return;
        }
    }
    launch_pdl(chain, gemm_simt_kernel<T, A_KM, B_KN, Epi>, grid, dim3(kGemmThreads), 0, st, A, lda, B, ldb, M, N, K, m_dev, k_dev, epi);
}

// Splits over `rows` (a capacity) of an m x n weight gradient on this kernel, at most `most` (148): two blocks per SM over all
// output tiles and at least 64 rows each.  With 148 splits whatever the shape, a 320 x 320 result was 3700 blocks of at
// most 16 rows and 60 MB of partial sums (24 + 12 us; the gated joint step 331 -> 273 us with this and the narrower products).
// Wide results get more, up to five, at 4096 rows each: a sum's rounding error goes with the square root of its longest chain
// of additions, K / 32 / splits + 32 + splits here and K / 148 + 148 before, and K / 160 is below K / 148 for every K.
// Relative error of 256 x 512 weights over 12 k, 50 k and 200 k rows: 2.8e-7, 4.2e-7 and 7.1e-7 with 148 splits, 1.6e-7, 2.8e-7
// and 4.7e-7 now (6.5e-7, 1.3e-6 and 2.8e-6 with ten splits and no folding).
inline int simt_splits(int64_t rows, int m, int n, int most)
{
    const int64_t tiles = ceil_div(m, kGemmBM) * ceil_div(n, kGemmBN);
    const int64_t wanted = std::max<int64_t>(ceil_div(2 * 148, tiles), std::min<int64_t>(5, ceil_div(rows, 4096)));
    return (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)most, wanted, ceil_div(rows, 64)}));
}

// h' = act(z + b), stored in the feature dtype
template <typename T>
struct EpiUpdate {
    T *out; int64_t ldo; const float *bias; int relu;
    __device__ void operator()(int64_t m, int n, float z, int) const {
        if (bias) z += bias[n];
        if (relu && z < 0.f) z = 0.f;
        out[m * ldo + n] = from_float<T>(z);
    }
};

// dCat = [dSelf | dAgg * (1/|S|)], stored in the feature dtype
template <typename T>
struct EpiDCat {
    T *out; int64_t ldo; int d_in; const float *inv_cnt;
    __device__ void operator()(int64_t m, int n, float v, int) const {
        if (n >= d_in) v *= inv_cnt[m];
        out[m * ldo + n] = from_float<T>(v);
    }
};

// split-K partial sums, fp32
struct EpiPartial {
    float *out; int64_t ldo; int64_t split_stride;
    __device__ void operator()(int64_t m, int n, float v, int z) const { out[z * split_stride + m * ldo + n] = v; }
};

// out = (accumulate ? out : 0) + sum_z partial[z], z ascending.  With rows_dev the partials come from the
// tensor-core weight-gradient kernel, which only fills the first ceil(total / per) splits
// (total = ceil(rows / 64) k-blocks, per = max(8, ceil(total / splits))); without it all splits are added.
static __global__ void splitk_reduce_kernel(const float *__restrict__ partial, int64_t n, int splits, int accumulate,
                                            float *__restrict__ out, const int32_t *rows_dev, int n_rhs = 1)
{
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int active = splits;
    if (rows_dev) {
        const int64_t total = (((int64_t)__ldcg(rows_dev) + 63) / 64) * n_rhs;
        const int64_t per = max((int64_t)8, (total + splits - 1) / splits);
        active = (int)max((int64_t)1, (total + per - 1) / per);
    }
    float s = accumulate ? out[i] : 0.f;
    // eight loads in flight, added in order
#pragma unroll 8
    for (int z = 0; z < active; ++z) s += __ldcg(partial + (int64_t)z * n + i);
    out[i] = s;
}

// dZ = dH where the stored output is positive (or everywhere for the identity activation);
// rows in [n, rows_alloc) are set to zero.  gridDim.y = 2: a second gradient dH1 goes to the block of rows_alloc
// rows behind the first in dZ (two right-hand sides sent through the backward pass together).  zero: zero16 times 16 bytes that
// the launches behind this one want cleared (a memset of its own ended the chain of dependent launches).
// d is a multiple of a 16-byte chunk, H and dZ have rows of d values on 16-byte boundaries; dH may lie anywhere.
// 16 bytes per thread: one value per thread took 6, 9 and 16 us for 4096 x 128, twice that and 8192 x 256 bf16 values (B200).
template <typename T>
__global__ void __launch_bounds__(256)
relu_mask_kernel(const T *__restrict__ dH, int64_t ld_dh, const T *__restrict__ H, const int32_t *n_dev, int64_t rows_alloc, int d, int relu,
                 T *__restrict__ dZ, const T *__restrict__ dH1, int64_t ld_dh1, uint4 *__restrict__ zero, int64_t zero16)
{
    constexpr int E = Chunk<T>::kElems;
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.y == 0)
        for (int64_t k = i; k < zero16; k += (int64_t)gridDim.x * blockDim.x) zero[k] = make_uint4(0, 0, 0, 0);
    if (blockIdx.y == 1) {
        dH = dH1;
        ld_dh = ld_dh1;
        dZ += rows_alloc * d;
    }
    const int chunks = d / E;
    const int64_t r = i / chunks;
    const int k = (int)(i - r * chunks) * E;
    if (r >= rows_alloc) return;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (r < __ldcg(n_dev)) {
        const T *src = dH + r * ld_dh + k;
        T x[E];
        if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
            v = __ldcg(reinterpret_cast<const uint4 *>(src));
            memcpy(x, &v, 16);
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = __ldcg(src + e);
        }
        if (relu) {
            const uint4 hv = __ldcg(reinterpret_cast<const uint4 *>(H + r * d + k));
            T h[E];
            memcpy(h, &hv, 16);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (!(to_float<T>(h[e]) > 0.f)) x[e] = from_float<T>(0.f);
        }
        memcpy(&v, x, 16);
    }
    *reinterpret_cast<uint4 *>(dZ + r * d + k) = v;
}

// out[k] = (accumulate ? out[k] : 0) + sum over rows r of (wgt ? wgt[r] : 1) * a[r, k], rows in a fixed order.
//
// A cluster of kColCtas blocks owns 4 chunks of 16 bytes (64 bytes of every row); each of its kColCtas * 64 row lanes takes
// every (kColCtas * 64)-th row, eight loads in flight.  Lanes are added by shuffles, warps through shared memory, blocks
// through the cluster's shared memory, each in a fixed order.  Latency-bound at the sizes of a batch: one block per 32
// columns with eight row lanes walked 4096 rows in 512 dependent steps (B200, 4096 x 256 bf16 with weights 51 us,
// 4096 x 512 bf16 30 us, 10 k x 72 fp32 24 us; now 5 to 6 us each).
constexpr int kColCtas = 8;
template <typename T>
__global__ void __cluster_dims__(kColCtas, 1, 1) __launch_bounds__(256)
colsum_kernel(const T *__restrict__ a, int64_t ld, const float *__restrict__ wgt, const int32_t *n_dev, int64_t n_host, int d,
              int accumulate, float *__restrict__ out)
{
    constexpr int E = Chunk<T>::kElems;
    constexpr int U = 8;
    __shared__ float red[8][4 * E];
    __shared__ float part[4 * E];
    const auto cluster = cooperative_groups::this_cluster();
    const int cta = (int)cluster.block_rank();
    const int cl = threadIdx.x & 3;                              // chunk within the block's four
    const int col0 = ((int)(blockIdx.x / kColCtas) * 4 + cl) * E;
    const int64_t n = n_dev ? (int64_t)*n_dev : n_host;
    const int64_t step = kColCtas * 64;
    const bool vec = (ld * (int64_t)sizeof(T)) % 16 == 0 && reinterpret_cast<uintptr_t>(a) % 16 == 0 && col0 + E <= d;
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    if (col0 < d)
        for (int64_t r0 = cta * 64 + (threadIdx.x >> 2); r0 < n; r0 += U * step) {
            uint4 v[U];
            float w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = r0 + u * step;
                v[u] = make_uint4(0, 0, 0, 0);
                w[u] = r < n ? (wgt ? wgt[r] : 1.f) : 0.f;
                if (r < n) {
                    if (vec) {
                        v[u] = Chunk<T>::load_raw(a + r * ld + col0);
                    } else {                                     // rows that are no multiple of 16 bytes, the last columns
                        T x[E];
#pragma unroll
                        for (int e = 0; e < E; ++e) x[e] = col0 + e < d ? a[r * ld + col0 + e] : from_float<T>(0.f);
                        memcpy(&v[u], x, 16);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float x[E];
                Chunk<T>::unpack(v[u], x);
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = wgt ? fmaf(w[u], x[e], acc[e]) : acc[e] + x[e];
            }
        }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if ((threadIdx.x & 31) < 4) {
#pragma unroll
        for (int e = 0; e < E; ++e) red[threadIdx.x >> 5][cl * E + e] = acc[e];
    }
    __syncthreads();
    if (threadIdx.x < 4 * E) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
        part[threadIdx.x] = s;
    }
    cluster.sync();
    const int col = (int)(blockIdx.x / kColCtas) * 4 * E + threadIdx.x;
    if (cta == 0 && threadIdx.x < 4 * E && col < d) {
        float s = accumulate ? out[col] : 0.f;
#pragma unroll
        for (int c = 0; c < kColCtas; ++c) s += cluster.map_shared_rank(part, c)[threadIdx.x];
        out[col] = s;
    }
    cluster.sync();                                              // the other blocks' sums stay until they have been read
}

template <typename T>
inline void launch_colsum(const T *a, int64_t ld, const float *wgt, const int32_t *n_dev, int64_t n_host, int d, int accumulate,
                          float *out, cudaStream_t st)
{
    note_launch();
    colsum_kernel<T><<<(unsigned)(ceil_div(d, 4 * Chunk<T>::kElems) * kColCtas), 256, 0, st>>>(a, ld, wgt, n_dev, n_host, d, accumulate, out);
}

// Wt[j][o] = W[o][j]: the dCat product reads the layer weight with d_out as the contraction index.
template <typename T>
__global__ void transpose_kernel(const T *__restrict__ W, int rows, int cols, T *__restrict__ Wt)
{
    __shared__ T tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y)
        if (r0 + i < rows && c0 + threadIdx.x < cols) tile[i][threadIdx.x] = W[(int64_t)(r0 + i) * cols + c0 + threadIdx.x];
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y)
        if (c0 + i < cols && r0 + threadIdx.x < rows) Wt[(int64_t)(c0 + i) * rows + r0 + threadIdx.x] = tile[threadIdx.x][i];
}

// masked copy of the gradient of a dense layer input: out = acc where mask > 0 (no mask: plain store)
template <typename T>
struct EpiMasked {
    T *out; int64_t ldo; const T *mask; int64_t ld_mask;
    __device__ void operator()(int64_t m, int n, float v, int) const {
        if (mask && !(to_float<T>(mask[m * ld_mask + n]) > 0.f)) v = 0.f;
        out[m * ldo + n] = from_float<T>(v);
    }
};

}  // namespace e2egrec
