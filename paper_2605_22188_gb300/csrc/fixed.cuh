// FP64 values by integer arithmetic.  GB300's FP64 pipe takes one warp instruction
// per SM in 16 cycles, its integer pipes two per cycle, so that a 64 x 64-bit
// high product (some eight instructions) costs a quarter of an FP64 FMA and a
// conversion or a rounding done with shifts a tenth of one done in FP64.  The
// functions compile for the host too, where tests/test_fixed_host.py checks them against
// decimal arithmetic; tests/test_gpu_fp64_digits.py takes the device's sigmoid_neg.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"

namespace kglm {

__host__ __device__ __forceinline__ uint64_t f64_bits(double v) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    union { double d; uint64_t u; } x;
    x.d = v;
    return x.u;
#endif
}
__host__ __device__ __forceinline__ double bits_f64(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    union { double d; uint64_t u; } x;
    x.u = u;
    return x.d;
#endif
}
__host__ __device__ __forceinline__ int64_t mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ uint64_t mulhi_u(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int clz64(uint64_t a) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}

// +-top 2^x (rest != 0: a fraction above top, for the rounding) to the nearest double, ties to even;
// top has its highest bit set.
__host__ __device__ __forceinline__ double round_f64(bool neg, uint64_t top, bool rest, int x) {
    uint64_t m = top >> 11;
    const uint32_t rem = (uint32_t)top & 0x7ffu;
    m += (rem > 0x400u || (rem == 0x400u && (rest || (m & 1u)))) ? 1u : 0u;
    const int be = x + 11 + 52 + 1023;                  // biased exponent: m in [2^52, 2^53]
    const uint64_t sign = (uint64_t)neg << 63;
    if (be >= 1 && be <= 2046) return bits_f64(sign + ((uint64_t)(be - 1) << 52) + m);
    if (be > 2046) return bits_f64(sign | 0x7ff0000000000000ull);
    // a subnormal result: rounded once, at its own last place
    const int sh = 12 - be;
    if (sh > 64) return bits_f64(sign);
    const uint64_t half = 1ull << (sh - 1), low = sh < 64 ? top & ((1ull << (sh & 63)) - 1) : top;
    uint64_t d = sh < 64 ? top >> (sh & 63) : 0ull;
    d += (low > half || (low == half && (rest || (d & 1u)))) ? 1u : 0u;
    return bits_f64(sign | d);
}

// The row exponent's marker of a row with a non-finite entry: its products are NaN.
constexpr int kBadRow = 1 << 28;

// Biased exponent of v (1 for subnormals), 0 for zero, kBadRow for a non-finite value.
__host__ __device__ __forceinline__ int exp_key(double v) {
    const uint64_t u = f64_bits(v) & 0x7fffffffffffffffull;
    const int ex = (int)(u >> 52);
    if (ex == 2047) return kBadRow;
    return ex ? ex : (u ? 1 : 0);
}
// 2^e > 2 |v| for the largest key (plus column shift) of a row; a zero row takes e = 0.
__host__ __device__ __forceinline__ int row_exp(int key) { return key >= kBadRow / 2 ? kBadRow : key > 0 ? key - 1021 : 0; }

// rint(v 2^(BITS - e)) for |v| < 2^(e - 1) (halves away from zero).
template <int BITS = 64>
__host__ __device__ __forceinline__ int64_t fixed64(double v, int e) {
    const uint64_t u = f64_bits(v);
    const int ex = (int)(u >> 52) & 0x7ff;
    const uint64_t m = (u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
    const int sh = (ex ? ex : 1) - 1075 + BITS - e;     // at most BITS - 54
    uint64_t z;
    if (sh >= 0) z = m << (sh & 63);
    else if (sh > -54) z = (m + (1ull << ((-sh - 1) & 63))) >> (-sh & 63);
    else z = 0;
    return (int64_t)u < 0 ? -(int64_t)z : (int64_t)z;
}

// The same for an FP32 value (0 for a non-finite one), |v| < 2^(e - 1).
template <int BITS>
__device__ __forceinline__ int64_t fixed64f(float v, int e) {
    const uint32_t u = __float_as_uint(v);
    const int ex = (int)(u >> 23) & 0xff;
    const uint64_t m = (u & 0x7fffffu) | (ex ? 0x800000u : 0u);
    const int sh = (ex ? ex : 1) - 150 + BITS - e;
    uint64_t z = 0;
    if (ex != 255) {
        if (sh >= 0) z = m << (sh & 63);
        else if (sh > -26) z = (m + (1ull << ((-sh - 1) & 63))) >> (-sh & 63);
    }
    return (int32_t)u < 0 ? -(int64_t)z : (int64_t)z;
}

// The ND signed bytes of z, the last the lowest (|z| < 2^(8 ND - 1)), as BF16: exact.
template <int ND>
__device__ __forceinline__ void cut_digits(long long z, __nv_bfloat16 (&d)[ND]) {
#pragma unroll
    for (int a = ND - 1; a >= 1; --a) {
        const int v = (int)(signed char)z;
        z = (z - v) >> 8;
        d[a] = __int2bfloat16_rn(v);
    }
    d[0] = __int2bfloat16_rn((int)z);
}

// Digits of four consecutive entries i .. i + 3 (a multiple of 4) of a row into its ND
// segments of npad, in order or reversed.
template <int ND>
__device__ __forceinline__ void store_digits(const long long (&z)[4], __nv_bfloat16* row, size_t npad, int i, int reversed) {
    __nv_bfloat16 d[4][ND];
#pragma unroll
    for (int t = 0; t < 4; ++t) cut_digits<ND>(z[t], d[t]);
#pragma unroll
    for (int a = 0; a < ND; ++a) {
        __nv_bfloat162 lo, hi;
        lo.x = d[0][a]; lo.y = d[1][a];
        hi.x = d[2][a]; hi.y = d[3][a];
        uint2 w;
        w.x = *reinterpret_cast<const uint32_t*>(&lo);
        w.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(row + (size_t)(reversed ? ND - 1 - a : a) * npad + i) = w;
    }
}

// H and L of one entry of a product of ND digits from its levels' integers (level l of
// part q in slice q ND + l - 2): 2^-40 H + 2^-72 L, levels 2 .. 5 in H.
template <int ND>
__device__ __forceinline__ void level_sums(const int* __restrict__ I, size_t stride, size_t idx, int parts,
                                           long long& H, long long& L) {
    H = L = 0;
    for (int q = 0; q < parts; ++q) {
        int v[ND];
#pragma unroll
        for (int t = 0; t < ND; ++t) v[t] = __ldg(I + (size_t)(q * ND + t) * stride + idx);
#pragma unroll
        for (int t = 0; t < ND; ++t) {
            if (t < 4) H += (long long)v[t] << (8 * (3 - t));
            else L += (long long)v[t] << (8 * (7 - t));
        }
    }
}

// (2^32 H + L) 2^x, correctly rounded.
__host__ __device__ __forceinline__ double combine_f64(int64_t H, int64_t L, int x) {
    uint64_t lo = (uint64_t)H << 32;
    int64_t hi = H >> 32;
    const uint64_t l0 = lo;
    lo += (uint64_t)L;
    hi += (L >> 63) + (lo < l0 ? 1 : 0);
    const bool neg = hi < 0;
    if (neg) {
        lo = ~lo + 1;
        hi = ~hi + (lo == 0 ? 1 : 0);
    }
    uint64_t h = (uint64_t)hi;
    if ((h | lo) == 0) return 0.0;
    if (h == 0) {
        h = lo;
        lo = 0;
        x -= 64;
    }
    const int lz = clz64(h);
    if (lz) {
        h = (h << lz) | (lo >> (64 - lz));
        lo <<= lz;
    }
    return round_f64(neg, h, lo != 0, x + 64 - lz);
}

// 2^(j / 64) in units of 2^-62, rounded (j = 0 .. 63)
#define KGLM_EXP2_TABLE \
    0x4000000000000000ull, 0x40b268f9de0183baull, 0x4166c34c5615d0ecull, 0x421d1461d66f2023ull, \
    0x42d561b3e6243d8aull, 0x438fb0cb4f468808ull, 0x444c0740496d4294ull, 0x450a6abaa4b77ecdull, \
    0x45cae0f1f545eb73ull, 0x468d6fadbf2dd4f3ull, 0x47521cc5a2e6a9e0ull, 0x4818ee218a3358eeull, \
    0x48e1e9b9d588e19bull, 0x49ad159789f37496ull, 0x4a7a77d47f7b84b1ull, 0x4b4a169b900c2d00ull, \
    0x4c1bf828c6dc54b8ull, 0x4cf022c9905bfd32ull, 0x4dc69cdceaa72a9cull, 0x4e9f6cd3967fdba8ull, \
    0x4f7a993048d088d7ull, 0x50582887dcb8a7e1ull, 0x513821818624b40cull, 0x521a8ad704f3404full, \
    0x52ff6b54d8a89c75ull, 0x53e6c9da74b29ab5ull, 0x54d0ad5a753e077cull, 0x55bd1cdad49f699cull, \
    0x56ac1f752150a563ull, 0x579dbc56b48521baull, 0x5891fac0e95612c8ull, 0x5988e20954889245ull, \
    0x5a827999fcef3242ull, 0x5b7ec8f19468bbc9ull, 0x5c7dd7a3b17dcf75ull, 0x5d7fad59099f22feull, \
    0x5e8451cfac061b5full, 0x5f8bccdb3d398841ull, 0x6096266533384a2bull, 0x61a3666d124bb204ull, \
    0x62b39508aa836d6full, 0x63c6ba6455dcd8aeull, 0x64dcdec3371793d1ull, 0x65f60a7f79393e2eull, \
    0x6712460a8fc24072ull, 0x683199ed779592caull, 0x69540ec8f895722dull, 0x6a79ad55e7f6fd10ull, \
    0x6ba27e656b4eb57aull, 0x6cce8ae13c57ebdbull, 0x6dfddbcbed791babull, 0x6f307a412f074892ull, \
    0x70666f76154a7089ull, 0x719fc4b95f452d29ull, 0x72dc8373be41a454ull, 0x741cb5281e25ee34ull, \
    0x75606373ee921c97ull, 0x76a7980f6cca15c2ull, 0x77f25ccdee6d7ae6ull, 0x7940bb9e2cffd89dull, \
    0x7a92be8a92436616ull, 0x7be86fb985689ddcull, 0x7d41d96db915019dull, 0x7e9f06067a4360baull

#ifdef __CUDACC__
static __device__ const unsigned long long kExp2Dev[64] = {KGLM_EXP2_TABLE};
#endif

// 1 / (1 + e^t) for |t| <= 708, in fixed point: t = N ln 2 / 64 + r with |r| < 0.0056 in
// units of 2^-70 (differences modulo 2^64), e^r by its Taylor series to r^6 (r^7 / 5040 <
// 2^-64), times the table's 2^(j / 64); the reciprocal from an FP32 seed by one step
// of third order, y (1 + e + e^2).  Table lookup and series as in Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic", ACM
// TOMS 1989.  Errors before the final rounding are below 2^-58 relative: below 0.54 ulp in
// all, 0.502 at worst over the arguments of its test (exp, an addition and a division in
// FP64: 1.9 over the same).  With et, *et = e^t too (the same bound).
__host__ __device__ __forceinline__ double sigmoid_neg(double t, const unsigned long long* tab, double* et = nullptr) {
    const uint64_t u = f64_bits(t);
    const bool neg = (int64_t)u < 0;
    const int ex = (int)(u >> 52) & 0x7ff;
    const uint64_t m = (u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
    // t in units of 2^-70, modulo 2^64
    const int s = ex - 1005;                             // 2^(ex - 1075 + 70); at most 27
    uint64_t q = s >= 0 ? m << (s & 63) : s > -54 ? (m + (1ull << ((-s - 1) & 63))) >> (-s & 63) : 0ull;
    if (neg) q = ~q + 1;
    // N = rint(t 64 / ln 2) from t in FP32 (a unit of error in its last place moves r by 2^-17)
    const uint32_t fx = ex >= 1003 ? ((uint32_t)(ex - 1023 + 127) << 23) | (uint32_t)((u >> 29) & 0x7fffffu) : 0u;
#ifdef __CUDA_ARCH__
    float tf = __uint_as_float(fx);
#else
    union { uint32_t u; float f; } cv;
    cv.u = fx;
    float tf = cv.f;
#endif
    if (neg) tf = -tf;
    const int N = (int)rintf(tf * 92.33248261893609f);
    // ln 2 / 64 in units of 2^-70 and 2^-102
    const uint64_t c70 = 0xb17217f7d1cf79abull;
    const int64_t clo = 3387143064ll;
    const int64_t r = (int64_t)(q - (uint64_t)(int64_t)N * c70) - ((N * clo) >> 32);
    // e^r - 1 = r (1 + r (1/2 + r (1/6 + r g))), g = 1/24 + r (1/120 + r / 720)
    const int32_t r38 = (int32_t)(r >> 32);              // units of 2^-38
    // g in units of 2^-34 (r38 in 2^-38: the product's high word is 2^-40 of a 2^-34 factor)
    const int32_t g5 = 143165577 + (int32_t)(((int64_t)r38 * 23860929) >> 38);
    const int32_t g4 = 715827883 + (int32_t)(((int64_t)r38 * g5) >> 38);
    const int64_t h3 = 0x0aaaaaaaaaaaaaabll + (mulhi_s(r, (int64_t)g4 << 28) >> 6);   // units of 2^-62
    const int64_t h2 = 0x2000000000000000ll + (mulhi_s(r, h3) >> 6);
    const int64_t h1 = 0x4000000000000000ll + (mulhi_s(r, h2) >> 6);
    const int64_t w = mulhi_s(r, h1) >> 4;               // e^r - 1 in units of 2^-64
    const int j = N & 63, k0 = N >> 6;
    const int64_t T = (int64_t)tab[j];
    const uint64_t E = (uint64_t)(T + mulhi_s(T, w));    // 2^(j/64) e^r in units of 2^-62
    if (et) {
        const int le = clz64(E);
        *et = round_f64(false, E << le, false, k0 - 62 - le);
    }
    // 1 + e^t = 2^k d in units of 2^-62
    uint64_t d;
    int k = 0;
    if (k0 >= 0) {
        d = E + (k0 <= 62 ? 0x4000000000000000ull >> k0 : 0ull);
        k = k0;
    } else {
        d = 0x4000000000000000ull + (k0 > -64 ? E >> (-k0) : 0ull);
    }
    const int lz = clz64(d);
    d <<= lz;                                            // [2^63, 2^64)
    // 1 / d: seed y of 32 bits (units of 2^-32 of 1 / (d 2^-63))
    const uint32_t dt = (uint32_t)(d >> 32);
#ifdef __CUDA_ARCH__
    const float yf = __fdividef(9.2233720368547758e18f, __uint2float_rn(dt));
    const uint64_t y = min(__float2uint_rz(yf), 0xffffff00u);
#else
    const float yf = 9.2233720368547758e18f / (float)dt;
    const uint64_t y = yf >= 4294967040.f ? 0xffffff00u : (uint32_t)yf;
#endif
    const int64_t e = (int64_t)(0x8000000000000000ull - mulhi_u(d, y << 32));   // 1 - d y in units of 2^-63
    const int64_t es = e >> 11;                          // units of 2^-52; below 2^31
    const int64_t c = e + ((es * es) >> 41);
    uint64_t R = y << 32;                                // 1 / d in units of 2^-64
    R += (uint64_t)(mulhi_s((int64_t)(y << 31), c << 19) >> 17);
    if (!(R >> 63)) R = (R >> 62) ? 0x8000000000000000ull : 0xffffffffffffffffull;   // just below 1/2, or wrapped at 1
    return round_f64(false, R, false, lz - 65 - k);
}

// dl/ds of dloss: the least-squares form as it is there (its doubling is exact), the
// logistic one through sigmoid_neg where that covers it.
__device__ __forceinline__ double dloss_fixed(double s, double y, int kind, const unsigned long long* tab) {
    if (kind == kLSQ) return dloss(s, y, kind);
    const double t = y < 0.0 ? -s : s;                   // y s, y = -1 or 1
    if (!(fabs(t) <= 708.0)) return dloss(s, y, kind);
    const double q = sigmoid_neg(t, tab);
    return y < 0.0 ? q : -q;
}

}  // namespace kglm
