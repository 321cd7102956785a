// FP64 products on the BF16 tensor cores, by the error-free splitting of
// cert_exact.cu (Ozaki et al. 2012) carried to the end of an FP64 significand.
//
// GB300 retires two FP64 FMAs per SM and cycle (about 1.1 TFLOP/s over the
// chip), 1/1700 of its BF16 tensor rate, so an FP64 product is the whole cost
// of an FP64 iteration, and 36 exact BF16 products in its place are some 40
// times cheaper.  X^T R of 256 nodes at n = 5000, p = 1000: 2.17 ms on the FP64
// pipe, 69 us as digits; a whole FISTA iteration 4.55 -> 0.29 ms.
//
// Row r of an operand (K-contiguous) is scaled by 2^e > 2 max_k |v_rk| and
// rounded to the 64-bit integer V = rint(v 2^(64 - e)), |V| < 2^63, which is cut
// exactly into eight signed bytes from the bottom, v = 2^e sum_a d_a 2^(-8a),
// |d_a| <= 128: exact in BF16.  The digit pairs (a, c) of one level l = a + c
// share the weight 2^(-8l) and are concatenated along K (the second operand's
// digits are stored in reverse order, so that level l is a prefix of one row
// against a window of the other).  Sums of digit products over 16 slices of 64 are
// integers of at most 16 * 64 * 2^14 = 2^24, exact in the tensor core's FP32
// accumulator; the product's epilogue adds such chunks up in 32-bit integers
// (gemm_tc.cu, INT; the pieces of a level that are taken by several SMs are added in
// global memory), and the kernels here add the levels 2 .. 9 in 64-bit integers:
//   H = sum_{l <= 5} 2^(8 (5 - l)) I_l,  L = sum_{l >= 6} 2^(8 (9 - l)) I_l,
//   C = 2^(ea + eb) (2^-40 H + 2^-72 L),
// |H| < 2^38 K (1 + 2^-6), |L| < 2^41 K (1 + 2^-6): no overflow for K < 2^21.
// Left out are the levels 10 .. 16, at most 7 K 2^14 2^-80 (1 + 2^-7) of the
// scales' product, and the rounding of the operands, 2^-65 of each scale; the last
// FMA rounds once.  So the error is a few K 2^-64 of (2 max |a_r|)(2 max |b_c|)
// plus half an ulp of the result.  An FP64 FMA chain has K 2^-53 of
// sum_k |a_rk b_ck| as its bound and rounds at every one of the K partial sums:
// against exact sums (tests/test_gpu_fp64_split.py) its root-mean-square error is
// 4.3e-16 to 8e-16 of the results' size over n = 640 .. 20011, p = 111 .. 2000,
// this one's 5e-20 to 4e-17.
// The two bounds part where the entries of a row span many binades: the error here is
// normwise, an entry more than 2^11 below its row's largest keeps fewer bits than its
// double.  The engine takes this path only for instances whose rows are not spread so
// (the flag of k_split_digits over X, y and the R of kglm_xtr; the iterates and residuals
// of an evaluation are not looked at), with the columns of X scaled to comparable size
// (powers of two moved from X to the other operand, exactly).
#include <algorithm>

#include "common.cuh"
#include "engine.h"
#include "fixed.cuh"

namespace kglm {
namespace {

// Rows of V (rows x n, stride ldv; entry j times 2^ce[j], or 2^-ce[j] with inv) into
// digit rows of D (8 npad entries each, zero past n; NULL: none) and their scales'
// exponents (kBadRow for a row with a non-finite entry).  GS threads per row.  No
// FP64 operation: the scale is an exponent, the rounding a shift (with FP64 maxima and
// conversions 256 rows of 1000 took 16 us, now 9).  flag: set for a row whose
// largest magnitude is above 2^10 times the mean of its nonzero ones, whose scale is
// outside 2^(-+400), or with a non-finite entry.
template <int GS>
__global__ __launch_bounds__(256) void k_split_digits(const double* __restrict__ V, int rows, int n, size_t ldv,
                                                      int npad, const int* __restrict__ ce, int inv, int reversed,
                                                      __nv_bfloat16* __restrict__ D, int* __restrict__ scale,
                                                      int* flag) {
    __shared__ int redi[8];
    __shared__ float redf[3 * 8];
    const int g = threadIdx.x / GS, t = threadIdx.x % GS;
    const int r = blockIdx.x * (256 / GS) + g;
    if (GS == 32 && r >= rows) return;                       // whole warps; one CTA per row otherwise
    const double* v = V + (size_t)r * ldv;
    auto shift = [&](int i) { return ce == nullptr ? 0 : inv ? -ce[i] : ce[i]; };
    int key = -(1 << 27);
    for (int i = t; i < n; i += GS) {
        const int k = exp_key(v[i]);
        if (k) key = max(key, k + shift(i));
    }
    key = __reduce_max_sync(0xffffffffu, key);
    if (GS != 32) key = block_max<256, int>(key, redi);
    const bool none = key == -(1 << 27);
    // with a column shift the key may be below 1: no clamp, only "none" is a zero row
    const int e = key >= kBadRow / 2 ? kBadRow : none ? 0 : key - 1021;
    if (t == 0 && scale) scale[r] = e;
    if (flag) {
        float q[3] = {0.f, 0.f, 0.f};
        if (e != kBadRow)
            for (int i = t; i < n; i += GS) {
                const double x = v[i];
                if (x == 0.0) continue;
                const long long z = fixed64(x, e - shift(i));
                const float m = (float)((z < 0 ? -z : z) >> 32);
                q[0] = fmaxf(q[0], m);
                q[1] += m;
                q[2] += 1.f;
            }
        if (GS == 32) {
            q[0] = warp_max(q[0]);
            q[1] = warp_sum(q[1]);
            q[2] = warp_sum(q[2]);
        } else {
            const float mx = block_max<256, float>(q[0], redf);
            __syncthreads();
            block_sum<256, 3, float>(q, redf);
            q[0] = mx;
        }
        if (t == 0 && (e == kBadRow || e < -400 || e > 400 || q[0] * q[2] > 1024.f * q[1])) atomicOr(flag, 1);
    }
    if (!D) return;
    __nv_bfloat16* d = D + (size_t)r * 8 * npad;
    for (int i = 4 * t; i < npad; i += 4 * GS) {
        long long z[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = (i + q < n && e != kBadRow) ? fixed64(v[i + q], e - shift(i + q)) : 0ll;
        store_digits<8>(z, d, (size_t)npad, i, reversed);
    }
}

// One entry of the product from its levels' integers, times 2^x (x: the sum of the scales'
// exponents; kBadRow makes it a NaN).
__device__ __forceinline__ double combine(const int* __restrict__ I, size_t stride, size_t idx, int parts, int x) {
    long long H, L;
    level_sums<8>(I, stride, idx, parts, H, L);
    if (x >= kBadRow / 2) return bits_f64(0x7ff8000000000000ull);
    return combine_f64(H, L, x - 72);
}

// out[b][j] of a rows x cols product of digits (scales 2^er[b], 2^ec[j]).
__global__ __launch_bounds__(256) void k_split_combine(int cols, const int* __restrict__ I, size_t stride, int parts,
                                                       const int* __restrict__ er, const int* __restrict__ ec,
                                                       double* __restrict__ out) {
    const int b = blockIdx.y;
    const int s = er[b];
    const size_t base = (size_t)b * cols;
    for (int j = blockIdx.x * 256 + threadIdx.x; j < cols; j += gridDim.x * 256)
        out[base + j] = combine(I, stride, base + j, parts, s + ec[j]);
}

// S = X V of a node, its loss derivative R and R's digits: a cluster of CTAs per node,
// each with a part of the samples in shared memory between the two, so that neither
// S nor R is written in FP64; they exchange the largest exponent.  The parts of a
// row keep 304 CTAs in flight where the batch is small (a CTA per node left most SMs
// idle at 8 nodes).  Integer arithmetic but for the least-squares residual (two FP64
// operations): with FP64 sums, exp and division 1024 nodes of 2000 samples (logistic)
// took about 220 us, now 57 (38 million warp instructions, issue slots 60 % busy; its 69 MB would
// take 10).
constexpr int kLinkNT = 256;
__global__ __launch_bounds__(kLinkNT) void k_split_link(int n, int npad, int parts, int seg, const int* __restrict__ I,
                                                        size_t stride, int parts_k, const int* __restrict__ ev, const int* __restrict__ ex,
                                                        const double* __restrict__ y, int kind,
                                                        __nv_bfloat16* __restrict__ D, int* __restrict__ er) {
    extern __shared__ __align__(16) double row[];
    __shared__ unsigned long long tab[64];
    __shared__ int redi[kLinkNT / 32];
    __shared__ int s_key;
    const int t = threadIdx.x;
    const int b = blockIdx.x / parts, part = blockIdx.x - b * parts;
    const int i0 = part * seg, i1 = min(n, i0 + seg);
    if (t < 64) tab[t] = kExp2Dev[t];
    __syncthreads();
    const size_t base = (size_t)b * n;
    const int s = ev[b];
    int key = 0;
    for (int i = i0 + t; i < i1; i += kLinkNT) {
        const double r = dloss_fixed(combine(I, stride, base + i, parts_k, s + ex[i]), y[i], kind, tab);
        row[i - i0] = r;
        key = max(key, exp_key(r));
    }
    key = __reduce_max_sync(0xffffffffu, key);
    key = block_max<kLinkNT, int>(key, redi);                // its barriers also publish the row
    if (parts > 1) {
        if (t == 0) s_key = key;
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(&s_key);
        for (int q = 0; q < parts; ++q) {
            uint32_t peer, v;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(at), "r"(q));
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer) : "memory");
            key = max(key, (int)v);
        }
        // no CTA leaves (or reuses s_key) before its peers have read it
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    const int e = row_exp(key);
    if (t == 0 && part == 0) er[b] = e;
    __nv_bfloat16* d = D + (size_t)b * 8 * npad;
    const int iend = part == parts - 1 ? npad : min(npad, i0 + seg);
    for (int i = i0 + 4 * t; i < iend; i += 4 * kLinkNT) {
        long long z[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = (i + q < i1 && e != kBadRow) ? fixed64(row[i + q - i0], e) : 0ll;
        store_digits<8>(z, d, (size_t)npad, i, 1);
    }
}

constexpr size_t kLinkSmem = 96 * 1024;    // a part of at most 12288 samples

}  // namespace

bool split_plan(int M, int N, int K, int nd, int bn, bool pair, SplitPlan* out) {
    const int kbs = (K + 63) / 64, chunk = kSplitChunk;
    const int mt = (M + 127) / 128, nt = (N + bn - 1) / bn;
    pair = pair && mt >= 2 && bn >= kPairMinCols;
    const long tiles = (long)(pair ? (mt + 1) / 2 : mt) * nt;
    const int workers = pair ? 76 : 152;
    const double total = 0.5 * nd * (nd + 1) * kbs * (double)tiles;
    // microseconds of one K slice of a tile (operands at ~68 bytes per cycle and SM, as
    // the link product measures), of a unit's start and end, and of a slice of integers:
    // written and read, or with levels in pieces zeroed, added to piece by piece and read
    const double us_kb = (128.0 + (pair ? bn / 2 : bn)) * 128.0 / 68.0 / 1900.0;
    const double us_unit = 2.0, mn = (double)M * N * 4.0;
    double best = 1e300;
    for (int w : {0, 1, 2, 3, 4, 6, 8}) {
        // pieces of at most J slices (whole chunks); w = 0: as few as possible
        long J = w == 0 ? kSplitPart : (long)(total / ((double)workers * w)) + 1;
        J = std::min<long>(kSplitPart, std::max<long>(chunk, (J + chunk - 1) / chunk * chunk));
        SplitPlan p{};
        p.nd = nd;
        p.kbs = kbs;
        p.parts = split_parts(K, nd);
        bool fits = true;
        for (int l = nd + 1; l >= 2 && fits; --l)
            for (int q0 = 0; q0 < (l - 1) * kbs && fits; q0 += kSplitPart) {   // a part, in even pieces
                const int kb = std::min(kSplitPart, (l - 1) * kbs - q0), cnt = (int)((kb + J - 1) / J);
                const int per = ((kb + cnt - 1) / cnt + chunk - 1) / chunk * chunk;
                for (int u0 = 0; u0 < kb; u0 += per) {
                    if (p.njobs >= kTcMaxJobs) { fits = false; break; }
                    p.jobs[p.njobs++] = {(nd + 1 - l) * kbs + q0 + u0, q0 + u0, std::min(per, kb - u0),
                                         q0 / kSplitPart * nd + l - 2};
                }
            }
        if (!fits) continue;
        std::stable_sort(p.jobs, p.jobs + p.njobs, [](const TcJob& a, const TcJob& b) { return a.nkb > b.nkb; });
        // the busiest worker: units dealt forwards and backwards in turn (gemm_tc.cu)
        double worst;
        const long units = tiles * p.njobs;
        if (units > 64L * workers) {
            worst = (total * us_kb + units * us_unit) / workers;
        } else {
            double load[152] = {};
            for (long u = 0; u < units; ++u) {
                const long pass = u / workers, a = u - pass * workers;
                const long width = std::min<long>(workers, units - pass * workers);
                load[(pass & 1) ? width - 1 - a : a] += p.jobs[u / tiles].nkb * us_kb + us_unit;
            }
            worst = *std::max_element(load, load + workers);
        }
        const double cost = worst + (p.njobs > nd ? 2.0 + (p.njobs / 2.5e6 + 2.0 * nd / 6.0e6) * mn : 2.0 * nd / 6.0e6 * mn);
        if (cost < best) {
            best = cost;
            *out = p;
        }
    }
    return best < 1e300;
}

void split_digits(cudaStream_t s, const double* V, int rows, int n, size_t ldv, int npad, const int* ce, int inv,
                  int reversed, __nv_bfloat16* D, int* scale, int* flag) {
    if (rows <= 0) return;
    if (n <= 512) k_split_digits<32><<<(rows + 7) / 8, 256, 0, s>>>(V, rows, n, ldv, npad, ce, inv, reversed, D, scale, flag);
    else k_split_digits<256><<<rows, 256, 0, s>>>(V, rows, n, ldv, npad, ce, inv, reversed, D, scale, flag);
}

void split_combine(cudaStream_t s, int rows, int cols, const int* I, size_t stride, int parts, const int* er,
                   const int* ec, double* out) {
    // rows on the grid's y axis, in runs of at most 65535
    for (int b0 = 0; b0 < rows; b0 += 65535) {
        const int rr = std::min(65535, rows - b0);
        const dim3 grid(std::max(1, std::min(8, (cols + 255) / 256)), rr);
        k_split_combine<<<grid, 256, 0, s>>>(cols, I + (size_t)b0 * cols, stride, parts, er + b0, ec, out + (size_t)b0 * cols);
    }
}

int split_prepare() {
    static const int rc = cudaFuncSetAttribute(k_split_link, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kLinkSmem) == cudaSuccess ? 0 : -1;
    return rc;
}

int split_link(cudaStream_t s, int m, int n, int npad, const int* I, size_t stride, int parts_k, const int* ev,
               const int* ex, const double* y, int kind, __nv_bfloat16* D, int* er) {
    if (m <= 0) return 0;
    int parts = 1;
    while (parts < 8 && ((long)m * parts < 2 * 152 || (size_t)n * 8 > kLinkSmem * parts) &&
           (n / parts >= 1024 || (size_t)n * 8 > kLinkSmem * parts))
        parts *= 2;
    const int seg = ((n + parts - 1) / parts + 3) / 4 * 4;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)m * parts);
    cfg.blockDim = dim3(kLinkNT);
    cfg.dynamicSmemBytes = (size_t)seg * sizeof(double);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = parts > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_split_link, n, npad, parts, seg, I, stride, parts_k, ev, ex, y, kind, D,
                              er) ==
                   cudaSuccess ? 0 : -1;
}

}  // namespace kglm
