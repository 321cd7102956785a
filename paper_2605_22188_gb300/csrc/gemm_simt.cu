// CUDA-core GEMMs of the FP64 and FP32 paths: S = X B and G = X^T R of §4.2
// Eq. (gradient_matrix_form) in the node-major layout, with the loss/link of
// §4.2 fused into the epilogue of S (R = dl(S, y) is written, S is not).
//
// C[r][c] = sum_k A[r][k] B[c][k]: both operands are K-contiguous (node rows
// of V or R against rows of X or X^T).  Each CTA computes a BM x BN tile (in FP64
// with TM x TN contiguous outputs per thread); the next K slice is prefetched into
// registers while the current one is multiplied from shared memory.
//
// Split-K: when the output has too few tiles to fill the GPU (X^T R is only
// m x p while K = n), the K range is cut into `splits` chunks (grid z).  Each
// CTA stores its partial tile in a scratch buffer, fences, and increments the
// tile's arrival counter; the CTA that arrives last sums the partials in the
// fixed order s = 0..splits-1 (so the result does not depend on arrival
// order), applies the epilogue and sets the counter back to 0.  No CTA waits
// for another.
#include <algorithm>

#include "common.cuh"
#include "engine.h"

namespace kglm {
namespace {

template <typename T>
struct EpiStore {
    T* out;
    int ldo;
    __device__ __forceinline__ void operator()(int r, int c, T v) const { out[(size_t)r * ldo + c] = v; }
};

template <typename T>
struct EpiLink {
    T* out;
    int ldo;
    const T* y;
    int kind;
    __device__ __forceinline__ void operator()(int r, int c, T v) const {
        out[(size_t)r * ldo + c] = dloss(v, y[c], kind);
    }
};

template <typename T> struct Vec4;
template <> struct Vec4<double> { using type = double2; };   // 16-byte vector

template <typename T, int BM, int BN, int BK, int TM, int TN, bool VEC, typename Epi>
__global__ __launch_bounds__((BM / TM) * (BN / TN)) void k_gemm_nt(int R, int C, int K, const T* __restrict__ A,
                                                                   int lda, const T* __restrict__ B, int ldb,
                                                                   Epi epi, int kchunk, T* __restrict__ part,
                                                                   int* __restrict__ counters) {
    constexpr int NTX = BN / TN, NTY = BM / TM, NT = NTX * NTY;
    constexpr int VW = 16 / sizeof(T);                 // elements per 16-byte vector
    constexpr int PAD = VW;
    constexpr int AV = BM * BK / VW, BV = BN * BK / VW; // vectors per tile
    constexpr int AL = (AV + NT - 1) / NT, BL = (BV + NT - 1) / NT;
    static_assert(BK % VW == 0, "BK must be a multiple of the vector width");
    __shared__ __align__(16) T As[BK][BM + PAD];
    __shared__ __align__(16) T Bs[BK][BN + PAD];
    __shared__ int s_last;

    const int tid = threadIdx.x, tx = tid % NTX, ty = tid / NTX;
    const int r0 = blockIdx.y * BM, c0 = blockIdx.x * BN;
    const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);

    T ra[AL][VW], rb[BL][VW];
    auto load = [&](int k0) {
#pragma unroll
        for (int l = 0; l < AL; ++l) {
            const int v = tid + l * NT;
            const int row = v / (BK / VW), kk = (v % (BK / VW)) * VW;
            const int gr = r0 + row, gk = k0 + kk;
            if (v < AV) {
                if (VEC && gr < R && gk + VW <= kend) {
                    const auto x = *reinterpret_cast<const typename Vec4<T>::type*>(A + (size_t)gr * lda + gk);
                    const T* px = reinterpret_cast<const T*>(&x);
#pragma unroll
                    for (int q = 0; q < VW; ++q) ra[l][q] = px[q];
                } else {
#pragma unroll
                    for (int q = 0; q < VW; ++q)
                        ra[l][q] = (gr < R && gk + q < kend) ? A[(size_t)gr * lda + gk + q] : T(0);
                }
            }
        }
#pragma unroll
        for (int l = 0; l < BL; ++l) {
            const int v = tid + l * NT;
            const int col = v / (BK / VW), kk = (v % (BK / VW)) * VW;
            const int gc = c0 + col, gk = k0 + kk;
            if (v < BV) {
                if (VEC && gc < C && gk + VW <= kend) {
                    const auto x = *reinterpret_cast<const typename Vec4<T>::type*>(B + (size_t)gc * ldb + gk);
                    const T* px = reinterpret_cast<const T*>(&x);
#pragma unroll
                    for (int q = 0; q < VW; ++q) rb[l][q] = px[q];
                } else {
#pragma unroll
                    for (int q = 0; q < VW; ++q)
                        rb[l][q] = (gc < C && gk + q < kend) ? B[(size_t)gc * ldb + gk + q] : T(0);
                }
            }
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int l = 0; l < AL; ++l) {
            const int v = tid + l * NT;
            if (v < AV) {
                const int row = v / (BK / VW), kk = (v % (BK / VW)) * VW;
#pragma unroll
                for (int q = 0; q < VW; ++q) As[kk + q][row] = ra[l][q];
            }
        }
#pragma unroll
        for (int l = 0; l < BL; ++l) {
            const int v = tid + l * NT;
            if (v < BV) {
                const int col = v / (BK / VW), kk = (v % (BK / VW)) * VW;
#pragma unroll
                for (int q = 0; q < VW; ++q) Bs[kk + q][col] = rb[l][q];
            }
        }
    };

    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);

    if (kbeg < kend) load(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
        store();
        __syncthreads();
        if (k0 + BK < kend) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; i += VW) {
                const auto x = *reinterpret_cast<const typename Vec4<T>::type*>(&As[kk][ty * TM + i]);
                const T* px = reinterpret_cast<const T*>(&x);
#pragma unroll
                for (int q = 0; q < VW; ++q) a[i + q] = px[q];
            }
#pragma unroll
            for (int j = 0; j < TN; j += VW) {
                const auto x = *reinterpret_cast<const typename Vec4<T>::type*>(&Bs[kk][tx * TN + j]);
                const T* px = reinterpret_cast<const T*>(&x);
#pragma unroll
                for (int q = 0; q < VW; ++q) b[j + q] = px[q];
            }
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }

    if (gridDim.z == 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const int r = r0 + ty * TM + i, c = c0 + tx * TN + j;
                if (r < R && c < C) epi(r, c, acc[i][j]);
            }
        return;
    }
    // split-K: publish the partial tile, the last arriving CTA reduces it
    const int tile = blockIdx.y * gridDim.x + blockIdx.x;
    const int ntile = gridDim.x * gridDim.y;
    T* my = part + ((size_t)blockIdx.z * ntile + tile) * (BM * BN);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) my[(ty * TM + i) * BN + tx * TN + j] = acc[i][j];
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&counters[tile], 1) == (int)gridDim.z - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    for (int s = 0; s < (int)gridDim.z; ++s) {
        const T* ps = part + ((size_t)s * ntile + tile) * (BM * BN);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] += __ldcg(ps + (ty * TM + i) * BN + tx * TN + j);
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int r = r0 + ty * TM + i, c = c0 + tx * TN + j;
            if (r < R && c < C) epi(r, c, acc[i][j]);
        }
    if (tid == 0) counters[tile] = 0;
}

// The FP32 product: 128 x 128 tiles of 16 of K, double-buffered in shared memory as
// [K][row], the next slice prefetched into registers.  What bounds it: sm_103a takes a
// scalar FMA at half the rate of the packed one (fma.rn.f32x2; 36 against some 72
// TFLOP/s over the chip), and the scalar kernel ran at its 36.  So a thread's 8 x 8
// outputs are 8 rows x 4 pairs of columns, each half of a pair the same IEEE operation
// in the same order of K as before.  The four 16-byte quarters of a slice's rows are
// stored at columns rotated by 8 (an exclusive or), so that neither the transposing
// stores nor the 16-byte reads conflict.  2048 x 10000 by 1000 columns: 1139 us (36
// TFLOP/s) with scalar FMAs, now 914 (45); 512 x 5000 by 1000: 181, now 131.  (A's entries
// stored twice, in place of the eight packing moves per step: 1059 and 150.)
constexpr int kF32K = 16;
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t& c, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

template <bool VEC, typename Epi>
__global__ __launch_bounds__(256, 2) void k_gemm_f32(int R, int C, int K, const float* __restrict__ A, int lda,
                                                     const float* __restrict__ B, int ldb, Epi epi, int kchunk,
                                                     float* __restrict__ part, int* __restrict__ counters) {
    __shared__ __align__(16) float As[2][kF32K][128];
    __shared__ __align__(16) float Bs[2][kF32K][128];
    __shared__ int s_last;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int r0 = blockIdx.y * 128, c0 = blockIdx.x * 128;
    const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
    // a warp loads 8 rows x 64 bytes; quarter kv of row `lr` (and lr + 64)
    const int lr = tid >> 2, kv = tid & 3;
    float4 ra[2], rb[2];
    auto fetch = [&](const float* P, int ld, int row, int rows, int k) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < rows) {
            const float* q = P + (size_t)row * ld + k;
            if (VEC && k + 4 <= kend) {
                v = __ldg(reinterpret_cast<const float4*>(q));
            } else {
                if (k < kend) v.x = __ldg(q);
                if (k + 1 < kend) v.y = __ldg(q + 1);
                if (k + 2 < kend) v.z = __ldg(q + 2);
                if (k + 3 < kend) v.w = __ldg(q + 3);
            }
        }
        return v;
    };
    auto load = [&](int k0) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            ra[l] = fetch(A, lda, r0 + lr + 64 * l, R, k0 + 4 * kv);
            rb[l] = fetch(B, ldb, c0 + lr + 64 * l, C, k0 + 4 * kv);
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int at = (lr + 64 * l) ^ (8 * kv);
            As[s][4 * kv][at] = ra[l].x; As[s][4 * kv + 1][at] = ra[l].y;
            As[s][4 * kv + 2][at] = ra[l].z; As[s][4 * kv + 3][at] = ra[l].w;
            Bs[s][4 * kv][at] = rb[l].x; Bs[s][4 * kv + 1][at] = rb[l].y;
            Bs[s][4 * kv + 2][at] = rb[l].z; Bs[s][4 * kv + 3][at] = rb[l].w;
        }
    };
    // rows 4 ty + i and 64 + 4 ty + i, columns 4 tx + .. and 64 + 4 tx + ..
    uint64_t acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    const int nt = kbeg < kend ? (kend - kbeg + kF32K - 1) / kF32K : 0;
    if (nt > 0) {
        load(kbeg);
        store(0);
    }
    __syncthreads();
    for (int it = 0; it < nt; ++it) {
        if (it + 1 < nt) load(kbeg + (it + 1) * kF32K);
        const int s = it & 1;
#pragma unroll
        for (int k = 0; k < kF32K; ++k) {
            const int x = 8 * (k >> 2);
            const float4 a0 = *reinterpret_cast<const float4*>(&As[s][k][(4 * ty) ^ x]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[s][k][64 + ((4 * ty) ^ x)]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[s][k][(4 * tx) ^ x]);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[s][k][64 + ((4 * tx) ^ x)]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint64_t aa = pack2(a[i], a[i]);
                fma2(acc[i][0], aa, b0.x);
                fma2(acc[i][1], aa, b0.y);
                fma2(acc[i][2], aa, b1.x);
                fma2(acc[i][3], aa, b1.y);
            }
        }
        if (it + 1 < nt) store(s ^ 1);
        __syncthreads();
    }
    auto out = [&] {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 v = unpack2(acc[i][j]);
                const int r = r0 + 4 * ty + (i & 3) + 64 * (i >> 2), c = c0 + 4 * tx + 2 * (j & 1) + 64 * (j >> 1);
                if (r < R && c < C) epi(r, c, v.x);
                if (r < R && c + 1 < C) epi(r, c + 1, v.y);
            }
    };
    if (gridDim.z == 1) {
        out();
        return;
    }
    // split-K: publish the partial tile, the last arriving CTA reduces it (k_gemm_nt)
    const int tile = blockIdx.y * gridDim.x + blockIdx.x, ntile = gridDim.x * gridDim.y;
    uint64_t* my = reinterpret_cast<uint64_t*>(part + ((size_t)blockIdx.z * ntile + tile) * (128 * 128)) + tid;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) my[(i * 4 + j) * 256] = acc[i][j];
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&counters[tile], 1) == (int)gridDim.z - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    float2 sum[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[i][j] = make_float2(0.f, 0.f);
    for (int z = 0; z < (int)gridDim.z; ++z) {
        const float2* ps = reinterpret_cast<const float2*>(part + ((size_t)z * ntile + tile) * (128 * 128)) + tid;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 v = __ldcg(ps + (i * 4 + j) * 256);
                sum[i][j].x += v.x;
                sum[i][j].y += v.y;
            }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = pack2(sum[i][j].x, sum[i][j].y);
    out();
    if (tid == 0) counters[tile] = 0;
}

constexpr int kSMs = 152;

// The FP64 product for outputs that would leave most of a 64 x 64 tile empty
// (the few nodes of a search's first batches, few features): a CTA computes
// RT rows x 32 columns, a column per lane, its eight warps taking eight of
// every 64 of K each, their partial sums added in warp order at the end.
// What bounds it: GB300 retires about two FP64 FMAs per SM and cycle, so one
// warp instruction holds the pipe for 16 cycles and the shared-memory loads
// hide behind it whatever the tile; time is the FP64 work of the busiest SM,
// padding included.  A 64 x 64 tile multiplies 262k FMAs per 64 of K for
// output of any size: 207 us per launch of X^T R at n = 200, p = 30, m <= 8,
// 8 us here (both between events of their own; S = X V 39 us before, 7 us here).
template <int RT, typename Epi>
__global__ __launch_bounds__(256) void k_gemm_f64_small(int R, int C, int K, const double* __restrict__ A, int lda,
                                                        const double* __restrict__ B, int ldb, Epi epi, int kchunk,
                                                        double* __restrict__ part, int* __restrict__ counters) {
    constexpr int KT = 64, NW = 8;
    __shared__ double Bs[32][KT + 1];                  // odd row stride: a column per lane without bank conflicts
    __shared__ double As[RT][KT];
    __shared__ double red[NW][RT][32];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = blockIdx.y * RT, c0 = blockIdx.x * 32;
    const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
    constexpr int BL = 32 * KT / 256;
    double rb[BL], ra = 0.0, rc = 0.0;
    auto load = [&](int k0) {
#pragma unroll
        for (int l = 0; l < BL; ++l) {
            const int v = tid + l * 256, col = v / KT, k = k0 + v % KT;
            rb[l] = (c0 + col < C && k < kend) ? __ldg(B + (size_t)(c0 + col) * ldb + k) : 0.0;
        }
        // RT x 64 entries of A: at most two per thread
        const int row = tid / KT, k = k0 + tid % KT;
        ra = (row < RT && r0 + row < R && k < kend) ? __ldg(A + (size_t)(r0 + row) * lda + k) : 0.0;
        if (RT > 4) rc = (r0 + row + 4 < R && k < kend) ? __ldg(A + (size_t)(r0 + row + 4) * lda + k) : 0.0;
    };
    double acc[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[r] = 0.0;
    if (kbeg < kend) load(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += KT) {
#pragma unroll
        for (int l = 0; l < BL; ++l) {
            const int v = tid + l * 256;
            Bs[v / KT][v % KT] = rb[l];
        }
        if (tid / KT < RT) As[tid / KT][tid % KT] = ra;
        if (RT > 4) As[(tid / KT + 4) % RT][tid % KT] = rc;
        __syncthreads();
        if (k0 + KT < kend) load(k0 + KT);
        if (k0 + warp * (KT / NW) < kend) {            // the tail of K: no FP64 work on the zeros past it
#pragma unroll
            for (int kk = 0; kk < KT / NW; ++kk) {
                const double b = Bs[lane][warp * (KT / NW) + kk];
#pragma unroll
                for (int r = 0; r < RT; ++r) acc[r] = fma(As[r][warp * (KT / NW) + kk], b, acc[r]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) red[warp][r][lane] = acc[r];
    __syncthreads();
    const int row = tid / 32;                          // RT <= 8 rows, a warp each
    const bool mine = row < RT && r0 + row < R && c0 + lane < C;
    double v = 0.0;
    if (mine) {
#pragma unroll
        for (int w = 0; w < NW; ++w) v += red[w][row][lane];
    }
    if (gridDim.z > 1) {
        // split-K as in k_gemm_nt: the last CTA of a tile sums the partials in order
        const int tile = blockIdx.y * gridDim.x + blockIdx.x, ntile = gridDim.x * gridDim.y;
        if (row < RT) part[((size_t)blockIdx.z * ntile + tile) * (RT * 32) + row * 32 + lane] = v;
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = (atomicAdd(&counters[tile], 1) == (int)gridDim.z - 1);
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        v = 0.0;
        if (mine)
            for (int s = 0; s < (int)gridDim.z; ++s)
                v += __ldcg(part + ((size_t)s * ntile + tile) * (RT * 32) + row * 32 + lane);
        if (tid == 0) counters[tile] = 0;
    }
    if (mine) epi(r0 + row, c0 + lane, v);
}

// out[r] = A[r] . v, a CTA per row (X^T y of an instance: a 32-column tile for its one column
// took 310 us at n = 5000, p = 1000).
__global__ __launch_bounds__(256) void k_gemv_f64(int K, const double* __restrict__ A, const double* __restrict__ v,
                                                  double* __restrict__ out) {
    __shared__ double red[8];
    const double* a = A + (size_t)blockIdx.x * K;
    double q[1] = {0.0};
    for (int k = threadIdx.x; k < K; k += 256) q[0] = fma(__ldg(a + k), __ldg(v + k), q[0]);
    block_sum<256, 1, double>(q, red);
    if (threadIdx.x == 0) out[blockIdx.x] = q[0];
}

// One step of the power iteration on the symmetric Gram matrix: w = G v / ||v||,
// a warp per row; every CTA forms ||v|| itself (the same sum in the same order),
// CTA 0 records it.  A step reads G once (p x p from L2 where it fits).
__global__ __launch_bounds__(256) void k_power_step(int p, const double* __restrict__ G, const double* __restrict__ v,
                                                    double* __restrict__ w, double* __restrict__ norm) {
    __shared__ double red[8];
    double q[1] = {0.0};
    for (int j = threadIdx.x; j < p; j += 256) q[0] = fma(v[j], v[j], q[0]);
    block_sum<256, 1, double>(q, red);
    const double nv = sqrt(q[0]);
    if (blockIdx.x == 0 && threadIdx.x == 0) *norm = nv;
    const int lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= p) return;
    const double* g = G + (size_t)r * p;
    double s0 = 0.0, s1 = 0.0;
    int j = lane;
    for (; j + 32 < p; j += 64) {
        s0 = fma(__ldg(g + j), v[j], s0);
        s1 = fma(__ldg(g + j + 32), v[j + 32], s1);
    }
    if (j < p) s0 = fma(__ldg(g + j), v[j], s0);
    const double s = warp_sum(s0 + s1);
    if (lane == 0) w[r] = nv > 0.0 ? s / nv : 0.0;
}

template <typename T>
struct Tile;
template <> struct Tile<float> { static constexpr int BM = 128, BN = 128, BK = 8; };   // BK: what a chunk of K is a multiple of
template <> struct Tile<double> { static constexpr int BM = 64, BN = 64, BK = 8, TM = 4, TN = 4; };

// Resident CTAs per SM of the tile configuration (2 for the FP32 tile, 128
// registers x 256 threads; queried once from the runtime, with that default).
template <typename T>
int ctas_per_sm();

// Split-K factor: the one whose CTA count best fills whole waves of
// (SMs x resident CTAs), with a small penalty per split for the partial-tile
// traffic; each CTA keeps at least 64 of the K range and the grid stays
// within about two waves (so splits x tiles < 3 x SMs x resident CTAs).
inline int choose_splits(int tiles, int K, int BK, int per_sm) {
    const int slots = kSMs * per_sm;
    if (tiles >= slots) return 1;
    // at least 64 of K per CTA, and at most about two waves of CTAs
    const int max_split = max(1, min(min(64, K / 64), (2 * slots + tiles - 1) / tiles));
    int best = 1;
    double best_score = -1.0;
    for (int s = 1; s <= max_split; ++s) {
        const long ctas = (long)tiles * s;
        const long waves = (ctas + slots - 1) / slots;
        const double eff = (double)ctas / (double)(waves * slots);
        const double score = eff - 0.01 * s;
        if (score > best_score + 1e-12) { best_score = score; best = s; }
    }
    return best;
}

template <typename T>
GemmPlan plan_for(int R, int C, int K) {
    using TL = Tile<T>;
    GemmPlan g{};
    g.gx = (C + TL::BN - 1) / TL::BN;
    g.gy = (R + TL::BM - 1) / TL::BM;
    const int tiles = g.gx * g.gy;
    int splits = choose_splits(tiles, K, TL::BK, ctas_per_sm<T>());
    int kchunk = (K + splits - 1) / splits;
    kchunk = (kchunk + TL::BK - 1) / TL::BK * TL::BK;                 // keep vector alignment per chunk
    splits = (K + kchunk - 1) / kchunk;
    g.splits = max(1, splits);
    g.kchunk = kchunk;
    g.part_elems = g.splits > 1 ? (size_t)g.splits * tiles * TL::BM * TL::BN : 0;
    g.tiles = tiles;
    return g;
}

// FP64: the small-tile kernel where the FP64 work of its busiest SM (tiles of
// RT x 32, padding included) is below that of the 64 x 64 tiles; true if it ran.
// The work is counted in FMAs per SM, since the FP64 pipe is what both wait for:
// at p = 30, m = 2 the small tiles do 1/80 of the 64 x 64 tile's, at m = 64,
// n = 2000 the same, and the larger tile reads less.
template <typename Epi>
bool launch_small(cudaStream_t s, int R, int C, int K, const double* A, int lda, const double* B, int ldb, Epi epi,
                  const GemmScratch* scr, const GemmPlan& big) {
    if (K <= 0) return false;
    const long bw = ((long)big.tiles * big.splits + kSMs - 1) / kSMs;
    const double big_work = (double)bw * Tile<double>::BM * Tile<double>::BN * big.kchunk;
    const int ct = (C + 31) / 32;
    int best_rt = 0, best_split = 1, best_kc = K;
    double best = big_work;
    for (int rt = 1; rt <= 8; rt *= 2) {
        const long tiles = (long)ct * ((R + rt - 1) / rt);
        const bool can = scr != nullptr && scr->part != nullptr && scr->counters != nullptr && tiles <= scr->n_counters;
        for (int sp = 1; sp <= 16; ++sp) {
            int kc = (K + sp - 1) / sp;
            kc = (kc + 63) / 64 * 64;
            const int used = (K + kc - 1) / kc;
            if (used != sp) continue;
            if (sp > 1 && (!can || tiles * sp > 2 * kSMs ||
                           (size_t)tiles * sp * rt * 32 * sizeof(double) > scr->part_bytes))
                break;
            const long waves = (tiles * sp + kSMs - 1) / kSMs;
            // a split costs a pass over the partials: about 64 of K per split
            const double work = (double)waves * rt * 32 * ((double)std::min(kc, K) + (sp > 1 ? 16.0 * sp : 0.0));
            if (work < 0.9 * best) {
                best = work;
                best_rt = rt;
                best_split = sp;
                best_kc = kc;
            }
        }
    }
    if (best_rt == 0) return false;
    const long rows = (R + best_rt - 1) / best_rt;
    if (rows > 65535) return false;
    const dim3 grid(ct, (unsigned)rows, best_split);
    double* part = best_split > 1 ? static_cast<double*>(scr->part) : nullptr;
    int* cnt = best_split > 1 ? scr->counters : nullptr;
#define KGLM_SMALL(RT_) \
    k_gemm_f64_small<RT_, Epi><<<grid, 256, 0, s>>>(R, C, K, A, lda, B, ldb, epi, best_kc, part, cnt)
    if (best_rt == 1) KGLM_SMALL(1);
    else if (best_rt == 2) KGLM_SMALL(2);
    else if (best_rt == 4) KGLM_SMALL(4);
    else KGLM_SMALL(8);
#undef KGLM_SMALL
    return true;
}

// The tiles of a plan: k_gemm_f32, or k_gemm_nt in FP64.
template <typename T, typename Epi>
void launch_tiles(cudaStream_t s, int R, int C, int K, const T* A, int lda, const T* B, int ldb, Epi epi,
                  const GemmPlan& g, T* part, int* cnt) {
    using TL = Tile<T>;
    constexpr int VW = 16 / sizeof(T);
    const bool vec = (lda % VW == 0) && (ldb % VW == 0) && ((uintptr_t)A % 16 == 0) && ((uintptr_t)B % 16 == 0);
    const dim3 grid(g.gx, g.gy, g.splits);
    if constexpr (sizeof(T) == 4) {
        if (vec) k_gemm_f32<true, Epi><<<grid, 256, 0, s>>>(R, C, K, A, lda, B, ldb, epi, g.kchunk, part, cnt);
        else k_gemm_f32<false, Epi><<<grid, 256, 0, s>>>(R, C, K, A, lda, B, ldb, epi, g.kchunk, part, cnt);
    } else {
        constexpr int NT = (TL::BM / TL::TM) * (TL::BN / TL::TN);
        if (vec)
            k_gemm_nt<T, TL::BM, TL::BN, TL::BK, TL::TM, TL::TN, true, Epi><<<grid, NT, 0, s>>>(
                R, C, K, A, lda, B, ldb, epi, g.kchunk, part, cnt);
        else
            k_gemm_nt<T, TL::BM, TL::BN, TL::BK, TL::TM, TL::TN, false, Epi><<<grid, NT, 0, s>>>(
                R, C, K, A, lda, B, ldb, epi, g.kchunk, part, cnt);
    }
}

template <typename T, typename Epi>
void launch(cudaStream_t s, int R, int C, int K, const T* A, int lda, const T* B, int ldb, Epi epi,
            const GemmScratch* scr) {
    if (R <= 0 || C <= 0) return;
    using TL = Tile<T>;
    GemmPlan g = plan_for<T>(R, C, K);
    if constexpr (sizeof(T) == 8) {
        if (launch_small(s, R, C, K, A, lda, B, ldb, epi, scr, g)) return;
    }
    T* part = nullptr;
    int* cnt = nullptr;
    if (g.splits > 1) {
        if (scr == nullptr || scr->part == nullptr || scr->part_bytes < g.part_elems * sizeof(T) ||
            scr->counters == nullptr || scr->n_counters < g.tiles) {
            g.splits = 1;                                               // no scratch: one pass over K
            g.kchunk = K;
        } else {
            part = static_cast<T*>(scr->part);
            cnt = scr->counters;
        }
    }
    if (K <= 0) g.kchunk = 1;
    launch_tiles<T>(s, R, C, K, A, lda, B, ldb, epi, g, part, cnt);
}

// Like launch(), but when the scratch cannot hold the planned partials the
// split factor is lowered to what it holds instead of dropping to one pass.
template <typename T, typename Epi>
void launch_clamped(cudaStream_t s, int R, int C, int K, const T* A, int lda, const T* B, int ldb, Epi epi,
                    const GemmScratch& scr) {
    if (R <= 0 || C <= 0) return;
    using TL = Tile<T>;
    GemmPlan g = plan_for<T>(R, C, K);
    const size_t tile_bytes = (size_t)TL::BM * TL::BN * sizeof(T);
    if (g.splits > 1) {
        const size_t fit = (g.tiles > scr.n_counters || scr.part == nullptr) ? 1
                         : scr.part_bytes / ((size_t)g.tiles * tile_bytes);
        if ((size_t)g.splits > fit) {
            const int splits = (int)(fit < 1 ? 1 : fit);
            int kchunk = (K + splits - 1) / splits;
            kchunk = (kchunk + TL::BK - 1) / TL::BK * TL::BK;
            g.kchunk = kchunk;
            g.splits = (K + kchunk - 1) / kchunk;
        }
    }
    if (g.splits <= 1) {
        g.splits = 1;
        g.kchunk = K > 0 ? K : 1;
    }
    T* part = g.splits > 1 ? static_cast<T*>(scr.part) : nullptr;
    int* cnt = g.splits > 1 ? scr.counters : nullptr;
    launch_tiles<T>(s, R, C, K, A, lda, B, ldb, epi, g, part, cnt);
}

template <typename T>
int ctas_per_sm() {
    // computed once per process (a function-local static initialiser is
    // thread-safe; calls may come from several host threads at once)
    static const int cached = [] {
        using TL = Tile<T>;
        int n = 0;
        cudaError_t e;
        if constexpr (sizeof(T) == 4) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gemm_f32<true, EpiStore<T>>, 256, 0);
        } else {
            constexpr int NT = (TL::BM / TL::TM) * (TL::BN / TL::TN);
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &n, k_gemm_nt<T, TL::BM, TL::BN, TL::BK, TL::TM, TL::TN, true, EpiStore<T>>, NT, 0);
        }
        if (e != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 2;
        }
        return n;
    }();
    return cached;
}

}  // namespace

size_t gemm_scratch_bytes(int is_f64) {
    // splits x tiles < 3 x (SMs x resident CTAs), each partial tile BM x BN
    if (is_f64) return (size_t)3 * kSMs * ctas_per_sm<double>() * Tile<double>::BM * Tile<double>::BN * sizeof(double);
    return (size_t)3 * kSMs * ctas_per_sm<float>() * Tile<float>::BM * Tile<float>::BN * sizeof(float);
}
int gemm_scratch_counters(int is_f64) { return 3 * kSMs * (is_f64 ? ctas_per_sm<double>() : ctas_per_sm<float>()); }

GemmPlan gemm_plan(int R, int C, int K, int is_f64) {
    return is_f64 ? plan_for<double>(R, C, K) : plan_for<float>(R, C, K);
}

void gemm_nt_f64(cudaStream_t s, int R, int C, int K, const double* A, int lda, const double* B, int ldb,
                 double* out, int ldo, const GemmScratch* scr) {
    launch<double>(s, R, C, K, A, lda, B, ldb, EpiStore<double>{out, ldo}, scr);
}
void gemm_nt_f32(cudaStream_t s, int R, int C, int K, const float* A, int lda, const float* B, int ldb,
                 float* out, int ldo, const GemmScratch* scr) {
    launch<float>(s, R, C, K, A, lda, B, ldb, EpiStore<float>{out, ldo}, scr);
}
void gemm_nt_f32_clamped(cudaStream_t s, int R, int C, int K, const float* A, int lda, const float* B, int ldb,
                         float* out, int ldo, const GemmScratch& scr) {
    launch_clamped<float>(s, R, C, K, A, lda, B, ldb, EpiStore<float>{out, ldo}, scr);
}
int gemm_tile_rows_f32() { return Tile<float>::BM; }
int gemm_tile_cols_f32() { return Tile<float>::BN; }
void gemm_link_f64(cudaStream_t s, int m, int n, int p, const double* V, const double* X, const double* y,
                   int kind, double* out, const GemmScratch* scr) {
    launch<double>(s, m, n, p, V, p, X, p, EpiLink<double>{out, n, y, kind}, scr);
}
void gemm_link_f32(cudaStream_t s, int m, int n, int p, const float* V, const float* X, const float* y,
                   int kind, float* out, const GemmScratch* scr) {
    launch<float>(s, m, n, p, V, p, X, p, EpiLink<float>{out, n, y, kind}, scr);
}

void gemv_f64(cudaStream_t s, int rows, int K, const double* A, const double* v, double* out) {
    if (rows > 0) k_gemv_f64<<<rows, 256, 0, s>>>(K, A, v, out);
}

void gram_power_step(cudaStream_t s, int p, const double* G, const double* v, double* w, double* norm) {
    k_power_step<<<(p + 7) / 8, 256, 0, s>>>(p, G, v, w, norm);
}

}  // namespace kglm
