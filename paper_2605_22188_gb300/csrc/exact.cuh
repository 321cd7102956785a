// Shared by the certificate kernels: one entry of X^T zeta from the exact-splitting
// product's integers, with its error bound.
#pragma once

#include "engine.h"
#include "fixed.cuh"

namespace kglm {

// Entry (b, j) of X^T zeta from the levels' integers (slice t at Qi + t * stride, entry
// idx = b p + j): tau_b sigma_j (2^-40 H + 2^-72 L), correctly rounded.  scale: sigma_j tau_b, a
// power of two (0 for a zero row, whose product is exactly 0).  err: scale n E, a bound on
// the distance to the exact product.
__device__ __forceinline__ double exact_q(const int* Qi, size_t stride, size_t idx, int parts, double scale,
                                          double ebound, double* err) {
    long long H, L;
    level_sums<kCertDigits>(Qi, stride, idx, parts, H, L);
    *err = scale * ebound;
    const int ex = (int)((f64_bits(scale) >> 52) & 0x7ff);
    if (ex == 0 || ex == 2047) return scale == 0.0 ? 0.0 : combine_f64(H, L, -72) * scale;
    return combine_f64(H, L, ex - 1023 - 72);
}

}  // namespace kglm
