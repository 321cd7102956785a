// The certificate product X^T zeta (§4.4 Eq. (batched_dual_candidate_matrix_form))
// of the reduced-precision modes, on the BF16 tensor cores by error-free
// splitting (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 59, 2012; on tensor cores: Mukunoki,
// Ozaki, Ogita and Imamura, ICCS 2020).
//
// Column j of X is scaled by sigma_j = 2^e > 2 max_i |X_ij| and the dual point
// of node b by tau_b = 2^f > 2 max_i |zeta_ib| (exact).  A scaled value v in
// (-1/2, 1/2) is rounded to the integer V = rint(v 2^48) (error at most 2^-49 of the
// scale) and cut exactly into s = 6 signed bytes, v = sum_a d_a 2^(-8a) + r, |d_a| <=
// 128, |r| <= 2^-49: the digits are exact in BF16, their products in FP32.
// The digit pairs (a, c) of one level l = a + c share the weight 2^(-8l), so each
// level is one product with its pairs concatenated along K:
//   I_l[b][j] = sum_{a + c = l} sum_i dz_c(i, b) dx_a(i, j).
// X's digits are stored a = 1 .. s along K and zeta's in reverse, so level l
// reads a prefix of X's row and a window of zeta's.  Sums over 16 slices of 64 are
// integers of at most 2^24, exact in the FP32 accumulator whatever the order; the
// product's epilogue adds them up as 32-bit integers (gemm_tc.cu).  Levels 2 .. s + 1
// are formed, put together in 64-bit integers and rounded to FP64 once:
//   Q~_bj = sigma_j tau_b sum_l 2^(-8l) I_l[b][j],
// |Q~_bj - (X^T zeta)_jb| <= sigma_j tau_b n E' with
//   E' = 2 2^-49 + 2^-98 + sum_{l = s+2}^{2s} (2s - l + 1) 2^14 2^(-8l) + 2^-53 / 4
//      < 2^-47 + 2^-49 (levels left out: 5 2^-50 and less; the rounding of |Q~| <= n / 4).
// The bound that is used, n E per unit of scale with E = 2^-42.7, is the one of seven
// 6-bit digits under scales of half the size (28 level products, 30 FP32 slices at
// n = 10000 against 21 and 6 to 8 integer ones): some 20 times above E', and kept so
// that bounds stay comparable with those stored in checkpoints.  The certificate
// uses |Q~| + sigma tau n E, an entrywise upper bound of |X^T zeta|; H_M and the
// TopSum are increasing in |q|, so the bound remains a valid lower bound.
#include <math.h>

#include "common.cuh"
#include "engine.h"
#include "exact.cuh"

namespace kglm {
namespace {

constexpr int NT = 256;

// One CTA per row r of V (rows x n, row stride ldv): scale[r] = 2^e > 2 max |V_r| (0 for a
// zero row, NaN with a non-finite entry), digits of V_r / 2^e into D row r (segments of
// npad BF16 values, zero past n), in order or reversed.
__global__ __launch_bounds__(NT) void k_digits(const double* V, int n, size_t ldv, int npad, int reversed,
                                               __nv_bfloat16* D, double* scale) {
    __shared__ int red[NT / 32];
    const int r = blockIdx.x;
    const double* v = V + (size_t)r * ldv;
    int key = 0;
    for (int i = threadIdx.x; i < n; i += NT) key = max(key, exp_key(v[i]));
    key = block_max<NT, int>(key, red);
    const int e = row_exp(key);
    if (threadIdx.x == 0) scale[r] = e == kBadRow ? bits_f64(0x7ff8000000000000ull) : key > 0 ? ldexp(1.0, e) : 0.0;
    __nv_bfloat16* d = D + (size_t)r * kCertDigits * npad;
    for (int i = 4 * threadIdx.x; i < npad; i += 4 * NT) {
        long long z[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = i + q < n && e != kBadRow ? fixed64<8 * kCertDigits>(v[i + q], e) : 0ll;
        store_digits<kCertDigits>(z, d, (size_t)npad, i, reversed);
    }
}

// Q[b][j] and its bound from the jobs' integers (kglm_xtz).
__global__ void k_exact_combine(int m, int p, const int* Qi, size_t stride, int parts,
                                const double* sigma, const double* tau, double ebound, double* Q, double* E) {
    const size_t total = (size_t)m * p;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(idx / p), j = (int)(idx % p);
        double err;
        Q[idx] = exact_q(Qi, stride, idx, parts, sigma[j] * tau[b], ebound, &err);
        if (E) E[idx] = err;
    }
}

}  // namespace

void exact_digits(cudaStream_t s, const double* V, int rows, int n, size_t ldv, int npad, int reversed,
                  __nv_bfloat16* D, double* scale) {
    if (rows <= 0) return;
    k_digits<<<rows, NT, 0, s>>>(V, n, ldv, npad, reversed, D, scale);
}

void exact_combine(cudaStream_t s, int m, int p, const int* Qi, size_t stride, int parts, const double* sigma,
                   const double* tau, double ebound, double* Q, double* E) {
    if (m <= 0) return;
    k_exact_combine<<<2 * 152, 256, 0, s>>>(m, p, Qi, stride, parts, sigma, tau, ebound, Q, E);
}

bool exact_plan(int n, ExactPlan* pl) {
    // The slices the footprint counts: the pieces of at most 2^24 that 28 level products of
    // 6-bit digits (the first of 7 bits) take, 17 at n = 5000, 30 at n = 10000, none past 64.
    // The product needs kCertDigits of them; every batch that was chosen for a budget
    // rests on the count, so it stays.
    const int nd = 7, kbs = (n + 63) / 64;
    pl->npad = 64 * kbs;
    pl->njobs = 0;
    for (int l = 2; l <= nd + 1; ++l) {
        const int nkb = (l - 1) * kbs;
        double acc = 0.0;
        for (int u = 0; u <= nkb; ++u) {
            const int a = u / kbs + 1, c = l - a;
            const double add = u < nkb ? 64.0 * (a == 1 ? 64.0 : 32.0) * (c == 1 ? 64.0 : 32.0) : 0.0;
            if (u == nkb || acc + add > 16777216.0) {
                if (pl->njobs >= kTcMaxJobs) return false;
                ++pl->njobs;
                acc = 0.0;
            }
            acc += add;
        }
    }
    // n E: seven 6-bit digits under scales of half the size
    const double r = ldexp(1.0, -43) + ldexp(1.0, -63);
    double E = 2.0 * r + r * r + ldexp(1.0, -44);
    for (int l = nd + 2; l <= 2 * nd; ++l) E += (2 * nd - l + 1) * ldexp(1.0, 10 - 6 * l);
    pl->ebound = 0.25 * (double)n * E * (1.0 + 1e-12);
    return true;
}

}  // namespace kglm
