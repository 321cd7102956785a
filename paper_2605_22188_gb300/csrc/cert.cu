// The safe lower bound of §3 "Safe Lower Bound and Pruning", batched as in §4.4:
//   zeta_b = -dl(X beta_b, y)                       (Eq. (dual_candidate_vector_form))
//   q_b    = X^T zeta_b / (2 lambda2)               (Eq. (batched_dual_candidate_matrix_form))
//   LB_b   = -sum_i l*(-zeta_ib, y_i) - 2 lambda2 [ sum_{J1} H_M(q_j) + TopSum_kbar {H_M(q_j)}_{Jf} ]
//                                                   (Eq. (batched_dual_value_component))
// for every node whatever precision the iterations used: by weak duality it
// is a valid bound for any zeta.  X^T zeta, the Huber/TopSum terms and all
// sums are FP64; in the reduced-precision modes the conjugate terms are FP32
// evaluations with explicit rounding margins (k_dual_point_f32), so the
// returned value is a rigorous lower estimate of Psi(zeta).  The same per-node pass
// evaluates Phi_b = sum l + 2 lambda2 g(beta_b) with g from Theorem 4.1, the
// rounded support J1 cup top-kbar |beta| and the branching index
// argmax_{Jf} |beta_j| of §4.3 (ties to the smaller index).
#include <float.h>

#include <algorithm>

#include "common.cuh"
#include "engine.h"
#include "exact.cuh"

namespace kglm {
namespace {

constexpr double kFeasRtol = 1e-12;

// Reduced-precision modes: the dual point is built in FP32 and the conjugate
// sum is an upper bound with an explicit rounding margin, so that the bound
// stays below Psi(zeta) for the zeta actually used (the FP32 value, exact in
// FP64).  Least squares: zeta = -2 r with r = fl(s - fl(y)) (any zeta is
// admissible), l*(-zeta) = w y + w^2/4 with w = 2 r and the data y:
//   w y + w^2/4 = 2 r y + r^2 = 2 r y32 + 2 r ylo + r^2,   y32 + ylo = y to ~2^-48,
// where 2 r y32 and r^2 are formed exactly as FP32 pairs (product and its
// FMA residual) and 2 r ylo (below 2^-24 of 2 r y) in FP32.  Logistic:
// a = sigma(-y s) in FP32, zeta = y a (exact), and
//   l*(-zeta) = a ln a + (1-a) ln(1-a)
// with logf / log1pf, whose maximum errors in the CUDA C Programming Guide's
// accuracy table are 1 and 2 ulp (taken as 2^-23 and 2^-22 relative).  With
// one rounding per product and 1-a exact for a >= 1/2 (one rounding below):
//   |t1 - a ln a| <= (2^-23 + 2^-24)|a ln a|             <= 2^-22 |t1|,
//   |t2 - (1-a) ln(1-a)| <= (2^-22 + 2 * 2^-24)|...|     <= 2^-21 |t2|,
// so each term carries the margin 2^-22|t1| + 2^-21|t2| + 2^-125 (the last
// for denormal products); a term plus its margin is formed in FP32 rounded
// upward (never below the exact sum of the same parts).
// The running sums of a thread are FP32 pairs (hi, lo) updated by the exact
// two-sum of Knuth (hi + a = s + err exactly in round-to-nearest), about 2^-44
// relative per term, far below the logistic margins and of the order of the
// FP64 rounding of the least-squares terms; they reach FP64 once per thread,
// so that the GPU's slow FP64 pipe carries only the FP64 copy of zeta.
// (The _rn intrinsics keep the compiler from contracting a product into the
// two-sum's first addition, which would break its exactness.)
struct FPair {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float s = __fadd_rn(hi, v);
        const float bb = __fsub_rn(s, hi);
        lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(v, bb));
        hi = s;
    }
    // the exact product a b as its rounded value plus the FMA residual
    __device__ __forceinline__ void add_prod(float a, float b) {
        const float pr = __fmul_rn(a, b);
        add(pr);
        lo += fmaf(a, b, -pr);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// zeta of one sample in the reduced-precision modes (the value the certificate uses).
__device__ __forceinline__ float dual_z(float s, float yi, int kind) {
    if (kind == kLSQ) return -2.0f * (s - yi);
    const float t = yi * s;
    const float e = __expf(-fabsf(t));
    return yi * (t >= 0.f ? e / (1.0f + e) : 1.0f / (1.0f + e));   // y sigma(-t)
}

// A cluster of `parts` CTAs per node where the batch is small (one CTA per node took 28 us
// at one node of 5000 samples), each with `seg` of its samples: they exchange the
// largest |zeta| and their sums, which the first adds in order.
template <int NT>
__global__ __launch_bounds__(NT) void k_dual_point_f32(const __grid_constant__ CertArgs a, int parts, int seg) {
    __shared__ double red[2 * (NT / 32)];
    __shared__ float redf[NT / 32];
    __shared__ struct { double acc[2]; float zmax; } mine;
    const int b = blockIdx.x / parts, part = blockIdx.x - b * parts;
    const size_t base = (size_t)b * a.n;
    const int i0 = part * seg, i1 = min(a.n, i0 + seg);
    const bool digits = a.DZ != nullptr;               // zeta is kept as the FP32 value it is
    float* zf = reinterpret_cast<float*>(a.zeta);
    FPair sl, sc;
    float zmax = 0.f;
    const float* S = static_cast<const float*>(a.S);
    for (int i = i0 + threadIdx.x; i < i1; i += NT) {
        const float s = S[base + i];
        const float yi = a.y32[i];
        const float z = dual_z(s, yi, a.kind);
        zmax = fmaxf(zmax, fabsf(z));
        if (digits) zf[base + i] = z;
        else a.zeta[base + i] = (double)z;
        if (a.kind == kLSQ) {
            const float r = s - yi;
            sl.add(__fmul_rn(r, r));                         // the loss term as the iterations form it
            const float r2 = 2.0f * r;                        // w = -zeta, exact
            sc.add_prod(r2, yi);                              // 2 r y32, exact as a pair
            sc.add_prod(r, r);                                // r^2 = w^2 / 4, exact as a pair
            sc.lo += r2 * a.ylo[i];                           // 2 r ylo
        } else {
            const float t = yi * s;
            const float e = __expf(-fabsf(t));
            const float sg = t >= 0.f ? e / (1.0f + e) : 1.0f / (1.0f + e);     // sigma(-t)
            sl.add(fmaxf(-t, 0.f) + log1pf(e));
            float t1 = 0.f, t2 = 0.f;
            if (sg > 0.f) t1 = sg * logf(sg);
            if (sg < 1.f) t2 = (1.0f - sg) * log1pf(-sg);
            // margin and term in FP32 rounded upward (an upper bound of the exact term)
            const float mg = __fadd_ru(__fadd_ru(fabsf(t1) * 0x1p-22f, fabsf(t2) * 0x1p-21f), 0x1p-125f);
            sc.add(__fadd_ru(__fadd_ru(t1, t2), mg));
        }
    }
    double acc[2] = {sl.value(), sc.value()};
    block_sum<NT, 2, double>(acc, red);
    float mx = digits ? block_max<NT, float>(zmax, redf) : 0.f;
    if (parts > 1) {
        if (threadIdx.x == 0) {
            mine.acc[0] = acc[0];
            mine.acc[1] = acc[1];
            mine.zmax = mx;
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(&mine);
        acc[0] = acc[1] = 0.0;
        for (int q = 0; q < parts; ++q) {
            uint32_t peer;
            double v0, v1;
            float z;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(at), "r"(q));
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v0) : "r"(peer) : "memory");
            asm volatile("ld.shared::cluster.f64 %0, [%1 + 8];" : "=d"(v1) : "r"(peer) : "memory");
            asm volatile("ld.shared::cluster.f32 %0, [%1 + 16];" : "=f"(z) : "r"(peer) : "memory");
            acc[0] += v0;
            acc[1] += v1;
            mx = fmaxf(mx, z);
        }
        // no CTA leaves before its peers have read its values
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0 && part == 0) {
        a.sum_loss[b] = acc[0];
        a.sum_conj[b] = acc[1];
    }
    if (!digits) return;
    // the digits of zeta for the exact-splitting X^T zeta: the row's scale from the
    // first pass, then zeta again (written by this CTA) and its bytes from its FP32 bits
    const bool scaled = mx > 0.f && mx <= FLT_MAX;                 // (an infinite zeta has an infinite sum_conj)
    const int e = scaled ? ilogbf(mx) + 2 : 0;                     // 2^e > 2 mx
    if (threadIdx.x == 0 && part == 0) a.ztau[b] = scaled ? ldexp(1.0, e) : 0.0;   // a zero row is exact
    __nv_bfloat16* d = a.DZ + (size_t)b * kCertDigits * a.dz_npad;
    const int iend = part == parts - 1 ? a.dz_npad : min(a.dz_npad, i0 + seg);
    for (int i = i0 + 4 * threadIdx.x; i < iend; i += 4 * NT) {
        long long z[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = i + q < i1 ? fixed64f<8 * kCertDigits>(zf[base + i + q], e) : 0ll;
        store_digits<kCertDigits>(z, d, (size_t)a.dz_npad, i, 1);
    }
}

template <int NT>
__global__ __launch_bounds__(NT) void k_dual_point(CertArgs a) {
    __shared__ double red[2 * (NT / 32)];
    const int b = blockIdx.x;
    const size_t base = (size_t)b * a.n;
    double acc[2] = {0.0, 0.0};
    for (int i = threadIdx.x; i < a.n; i += NT) {
        const double s = a.s_is_f64 ? static_cast<const double*>(a.S)[base + i]
                                    : (double)static_cast<const float*>(a.S)[base + i];
        const double yi = a.y[i];
        const double d = dloss(s, yi, a.kind);       // zeta = -d
        a.zeta[base + i] = -d;
        acc[0] += loss64(s, yi, a.kind);
        acc[1] += loss_conj64(d, yi, a.kind);        // l*(-zeta) = l*(d)
    }
    block_sum<NT, 2, double>(acc, red);
    if (threadIdx.x == 0) {
        a.sum_loss[b] = acc[0];
        a.sum_conj[b] = acc[1];
    }
}

struct CertShared {
    SelectShared sel;
    double red[6 * 32];
    int ired[32];
    int cnt;
    double topv[kMaxK];
    int topi[kMaxK];
    double sv[kMaxK];
    int si[kMaxK];
    int sup[kMaxK];
    int sups[kMaxK];
    double gfree;
};

template <int NT, int E>
__global__ __launch_bounds__(NT) void k_cert_bound(const __grid_constant__ CertArgs a) {
    using K = unsigned long long;
    __shared__ CertShared sh;
    const int b = blockIdx.x, p = a.p;
    const size_t base = (size_t)b * p;
    const double M = a.M, inv2l = 1.0 / (2.0 * a.lam2);
    const uint32_t* im = a.in_mask + (size_t)b * a.W;
    const uint32_t* om = a.out_mask + (size_t)b * a.W;
    double q[E], be[E];
    uint32_t valid = 0, fin = 0, fout = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = threadIdx.x + e * NT;
        q[e] = be[e] = 0.0;
        if (j < p) {
            valid |= 1u << e;
            q[e] = a.Q[base + j] * inv2l;
            be[e] = a.b_is_f64 ? static_cast<const double*>(a.B)[base + j]
                               : (double)static_cast<const float*>(a.B)[base + j];
            if ((im[j >> 5] >> (j & 31)) & 1u) fin |= 1u << e;
            else if ((om[j >> 5] >> (j & 31)) & 1u) fout |= 1u << e;
        }
    }
    const uint32_t ffree = valid & ~fin & ~fout;
    const int kb = a.kbar[b], pf = a.pf[b];

    // ---- TopSum_kbar of H_M(q) over Jf (H_M is increasing in |q|)
    double hthr = 0.0;
    int need = 0;
    K thr = 0;
    const bool topsum_sel = (kb > 0 && pf > kb);
    if (topsum_sel) {
        K key[E];
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] = mag_key(fabs(q[e]));
        block_kth_largest<NT, E, K>(key, ffree, kb, sh.sel, thr, need);
        hthr = huber64(__longlong_as_double((long long)thr), M);
    }
    // sums: [J1 Huber, J1 beta^2, free |beta|, free nnz, free beta^2, infeasible, topsum part]
    double acc[6] = {0, 0, 0, 0, 0, 0};
    double ts[1] = {0.0};
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (!((valid >> e) & 1u)) continue;
        const double ab = fabs(be[e]);
        if ((fin >> e) & 1u) {
            acc[0] += huber64(q[e], M);
            acc[1] += be[e] * be[e];
            if (ab > M * (1.0 + kFeasRtol)) acc[5] += 1.0;
        } else if ((fout >> e) & 1u) {
            if (be[e] != 0.0) acc[5] += 1.0;
        } else {
            acc[2] += ab;
            acc[3] += ab > 0.0 ? 1.0 : 0.0;
            acc[4] += ab * ab;
            if (ab > M * (1.0 + kFeasRtol)) acc[5] += 1.0;
            if (kb > 0) {
                if (!topsum_sel) ts[0] += huber64(q[e], M);
                else if (mag_key(fabs(q[e])) > thr) ts[0] += huber64(q[e], M);
            }
        }
    }
    block_sum<NT, 6, double>(acc, sh.red);
    block_sum<NT, 1, double>(ts, sh.red);
    const double topsum = ts[0] + (topsum_sel ? need * hthr : 0.0);
    const double gconj = acc[0] + topsum;
    const double lb = -a.sum_conj[b] - 2.0 * a.lam2 * gconj;

    // ---- top-kbar |beta| over Jf (ties to the smaller index): rounding, j*, Theorem 4.1
    if (threadIdx.x == 0) sh.cnt = 0;
    __syncthreads();
    const bool leaf = (kb == 0 || pf <= kb);
    uint32_t sel = 0;
    if (!leaf) {
        K key[E];
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] = mag_key(fabs(be[e]));
        sel = block_topk_select<NT, E, K>(key, ffree, kb, sh.sel, sh.ired);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((sel >> e) & 1u) {
                const int s = atomicAdd(&sh.cnt, 1);
                sh.topv[s] = fabs(be[e]);
                sh.topi[s] = threadIdx.x + e * NT;
            }
        __syncthreads();
        warp_rank_sort_desc<double>(sh.topv, sh.topi, kb, sh.sv, sh.si);
    } else if (kb > 0) {
        sel = ffree;                                   // every free coordinate fits the budget
    }
    __syncthreads();
    // support = J1 cup selected free, ascending
    if (threadIdx.x == 0) sh.cnt = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e)
        if ((((fin | sel) >> e) & 1u)) {
            const int c = atomicAdd(&sh.cnt, 1);
            if (kglm_check(c < kMaxK, a.chk, kChkCert)) sh.sup[c] = threadIdx.x + e * NT;
        }
    __syncthreads();
    const int ns = sh.cnt;
    if (threadIdx.x < 32) {
        for (int i = threadIdx.x; i < ns; i += 32) {
            const int v = sh.sup[i];
            int r = 0;
            for (int j = 0; j < ns; ++j) r += sh.sup[j] < v;
            sh.sups[r] = v;
        }
    }
    // Theorem 4.1 on the free part (thread 0)
    if (threadIdx.x == 0) {
        const double total = acc[2], nnz = acc[3], sumsq = acc[4];
        double gf;
        if (acc[5] > 0.0) gf = INFINITY;
        else if (kb == 0) gf = total > 0.0 ? INFINITY : 0.0;
        else if (total / M > kb * (1.0 + kFeasRtol)) gf = INFINITY;
        else if (nnz <= kb) gf = 0.5 * sumsq;
        else {
            // s = the smallest index with tau_s >= |beta|_(s+1); then |beta|_(s) > tau_s
            // too, as Theorem 4.1 requires.  s = kbar - 1 qualifies in exact
            // arithmetic; it is also taken if rounding in total - pre says otherwise.
            double pre = 0.0, presq = 0.0;
            int s = 0;
            for (; s < kb - 1; ++s) {
                if ((total - pre) / (kb - s) >= sh.sv[s]) break;
                pre += sh.sv[s];
                presq += sh.sv[s] * sh.sv[s];
            }
            const double tail = total - pre;
            gf = 0.5 * (presq + tail / (kb - s) * tail);
        }
        sh.gfree = gf;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.lb[b] = lb;
        const double g = 0.5 * acc[1] + sh.gfree;
        a.primal[b] = isinf(g) ? INFINITY : a.sum_loss[b] + 2.0 * a.lam2 * g;
        a.jstar[b] = leaf ? -1 : sh.si[0];
    }
    for (int i = threadIdx.x; i < a.k; i += NT) a.support[(size_t)b * a.k + i] = i < ns ? sh.sups[i] : -1;
}

// ---- the same bound, primal, support and branching index for FP32 beta with X^T zeta as
// the exact-splitting product's integers (the reduced-precision modes): a CTA per
// node.  FP64 operations are what GB300 has least of (one warp instruction per SM in 16
// cycles), so an entry takes three of them, v_j = (|q~_j| + err_j) / (2 lambda2) from the
// correctly rounded integer combine; the selections work on the bits of v and |beta|,
// the beta sums of Theorem 4.1 are FP64 up to 512 coordinates and FP32 pairs per thread
// beyond (a pair's squares keep some 48 bits and FP32's range: few entries per thread, added
// up in FP64), and only the at most 64 selected values reach FP64 sums, in the order of
// their ranks.  8192 nodes of p = 2000: 0.61 ms (1.25 with a warp per node over 30 FP32
// slices); one node of p = 1000: 32 us between its events (76).  What bounds it: the chain of
// selections at 33 % of the warps an SM holds, issue slots 29 % busy, 235 MB in 312 us.
struct CertNodeShared {
    SelectShared sel;
    double red[2 * 32];
    float redf[4 * 32];
    int ired[32];
    int ncand, nj1;
    double topv[kMaxK];      // selected v (then |beta|), unordered
    int topi[kMaxK];
    double sv[kMaxK];        // sorted, descending
    int si[kMaxK];
    double vj1[kMaxK];       // v of the J1 coordinates
    int j1[kMaxK];
    int sup[2 * kMaxK];
};

// compensated FP32 accumulation (Knuth's two-sum; the product error by an FMA)
__device__ __forceinline__ void acc2(float& hi, float& lo, float x) {
    const float s = __fadd_rn(hi, x), bp = __fsub_rn(s, hi);
    lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
}
__device__ __forceinline__ void acc2_sq(float& hi, float& lo, float x) {
    const float pr = __fmul_rn(x, x);
    acc2(hi, lo, pr);
    lo += fmaf(x, x, -pr);
}
template <int NT, int E>
__global__ __launch_bounds__(NT) void k_cert_node(const __grid_constant__ CertArgs a) {
    using K = unsigned long long;
    constexpr int NW = NT / 32;
    __shared__ CertNodeShared sh;
    const int row = blockIdx.x, b = a.rowmap ? a.rowmap[row] : row;
    if (b < 0) return;
    const int p = a.p, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t base = (size_t)b * p, qbase = (size_t)row * p;
    const double M = a.M, inv2l = 1.0 / (2.0 * a.lam2), ztau = a.ztau[row];
    const double mth = M * (1.0 + kFeasRtol);
    const float mth_f = __double2float_rd(mth);                // |b| > mth  <=>  |b| > mth_f for FP32 b
    const uint32_t* im = a.in_mask + (size_t)b * a.W;
    const uint32_t* om = a.out_mask + (size_t)b * a.W;
    const int kb = a.kbar[b], pf = a.pf[b];
    const bool leaf = kb == 0 || pf <= kb;
    if (threadIdx.x == 0) sh.ncand = sh.nj1 = 0;
    __syncthreads();
    K key[E];                                                  // bits of v (non-negative)
    uint32_t bkey[E];                                          // bits of |beta|
    uint32_t ffree = 0;
    constexpr bool F64 = NT * E <= 512;
    float s1h = 0.f, s1l = 0.f, s2h = 0.f, s2l = 0.f;          // free sum |beta|, sum beta^2
    double s1 = 0.0, s2 = 0.0;
    int nnz = 0, infeas = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = threadIdx.x + e * NT;
        key[e] = 0;
        bkey[e] = 0;
        if (j >= p) continue;
        const bool in = (im[j >> 5] >> (j & 31)) & 1u, out = !in && ((om[j >> 5] >> (j & 31)) & 1u);
        const float ab = fabsf(static_cast<const float*>(a.B)[base + j]);
        if (out) {
            infeas += ab != 0.f;
            continue;
        }
        double err;
        const double qv = exact_q(a.Qi, a.qi_stride, qbase + j, a.qi_parts, a.xsig[j] * ztau, a.ebound, &err);
        // |X^T zeta| bounded from above: |Q~| + its distance bound (H_M, TopSum increase in |q|)
        const double v = (fabs(qv) + err) * inv2l;
        if (in) {
            const int c = atomicAdd(&sh.nj1, 1);
            if (kglm_check(c < kMaxK, a.chk, kChkCert) && c < kMaxK) {
                sh.j1[c] = j;
                sh.vj1[c] = v;
            }
            infeas += ab > mth_f;
            continue;
        }
        ffree |= 1u << e;
        key[e] = (K)__double_as_longlong(v);
        bkey[e] = __float_as_uint(ab);
        if constexpr (F64) {
            const double d = (double)ab;
            s1 += d;
            s2 = fma(d, d, s2);
        } else {
            acc2(s1h, s1l, ab);
            acc2_sq(s2h, s2l, ab);
        }
        nnz += ab > 0.f;
        infeas += ab > mth_f;
    }
    if constexpr (!F64) {
        s1 = (double)s1h + (double)s1l;
        s2 = (double)s2h + (double)s2l;
    }
    // both sums in one butterfly, half of the lanes each: five FP64 additions for ten
    const bool up = lane >= 16;
    double both = (up ? s2 : s1) + __shfl_xor_sync(0xffffffffu, up ? s1 : s2, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) both += __shfl_xor_sync(0xffffffffu, both, o);
    nnz = __reduce_add_sync(0xffffffffu, nnz);
    infeas = __reduce_add_sync(0xffffffffu, infeas);
    if ((lane & 15) == 0) sh.red[2 * warp + (lane >> 4)] = both;
    if (lane == 0) {
        sh.redf[2 * warp] = __int_as_float(nnz);
        sh.redf[2 * warp + 1] = __int_as_float(infeas);
    }
    // ---- TopSum_kbar {H_M(v_j)}_{j in Jf}: the selected values in shared memory
    int ntop = 0;
    if (!leaf) {
        K thr;
        int need;
        block_kth_largest<NT, E, K>(key, ffree, kb, sh.sel, thr, need);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (((ffree >> e) & 1u) && key[e] > thr) {
                const int c = atomicAdd(&sh.ncand, 1);
                sh.topv[c] = __longlong_as_double((long long)key[e]);
                sh.topi[c] = threadIdx.x + e * NT;
            }
        __syncthreads();
        const int gt = sh.ncand;
        // the remaining kbar - gt equal the threshold
        for (int c = gt + threadIdx.x; c < kb; c += NT) {
            sh.topv[c] = __longlong_as_double((long long)thr);
            sh.topi[c] = p + c;
        }
        ntop = kb;
    } else if (kb > 0) {
        // every free coordinate fits the budget (pf <= kbar <= kMaxK)
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((ffree >> e) & 1u) {
                const int c = atomicAdd(&sh.ncand, 1);
                if (kglm_check(c < kMaxK, a.chk, kChkCert) && c < kMaxK) {
                    sh.topv[c] = __longlong_as_double((long long)key[e]);
                    sh.topi[c] = threadIdx.x + e * NT;
                }
            }
        __syncthreads();
        ntop = min(sh.ncand, kMaxK);
    }
    __syncthreads();
    const int n1 = min(sh.nj1, kMaxK);
    if (warp == 0) {
        // sums in the order of the ranks (v descending) and of the J1 indices
        warp_rank_sort_desc<double>(sh.topv, sh.topi, ntop, sh.sv, sh.si);
        __syncwarp();
        double part = 0.0, hj1 = 0.0, bj1 = 0.0;
        for (int i = lane; i < ntop; i += 32) part += huber64(sh.sv[i], M);
        for (int i = lane; i < n1; i += 32) {
            int r = 0;
            for (int q = 0; q < n1; ++q) r += sh.j1[q] < sh.j1[i];
            sh.sup[r] = i;
        }
        __syncwarp();
        for (int i = lane; i < n1; i += 32) {
            const int at = sh.sup[i];
            hj1 += huber64(sh.vj1[at], M);
            const double bv = (double)static_cast<const float*>(a.B)[base + sh.j1[at]];
            bj1 += bv * bv;
        }
        part = warp_sum(part);
        hj1 = warp_sum(hj1);
        bj1 = warp_sum(bj1);
        if (lane == 0) {
            a.lb[b] = -a.sum_conj[row] - 2.0 * a.lam2 * (hj1 + part);
            sh.vj1[0] = bj1;                                   // (the J1 values are spent)
        }
        __syncwarp();
        if (lane == 0) sh.ncand = 0;
    }
    __syncthreads();
    // ---- top-kbar |beta| over Jf (ties to the smaller index): rounding, j*, Theorem 4.1
    if (!leaf) {
        const uint32_t sel = block_topk_select<NT, E, uint32_t>(bkey, ffree, kb, sh.sel, sh.ired);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((sel >> e) & 1u) {
                const int c = atomicAdd(&sh.ncand, 1);
                sh.topv[c] = (double)__uint_as_float(bkey[e]);
                sh.topi[c] = threadIdx.x + e * NT;
            }
        __syncthreads();
    }
    if (warp != 0) return;
    // ---- the first warp: sorted |beta|, the support ascending, Theorem 4.1 and the outputs
    if (!leaf) {
        warp_rank_sort_desc<double>(sh.topv, sh.topi, kb, sh.sv, sh.si);
        __syncwarp();
    }
    const int nf = leaf ? ntop : kb, ns = min(n1 + nf, kMaxK);
    for (int i = lane; i < ns; i += 32) {
        const int v = i < n1 ? sh.j1[i] : sh.topi[i - n1];
        int r = 0;
        for (int q = 0; q < ns; ++q) r += (q < n1 ? sh.j1[q] : sh.topi[q - n1]) < v;
        sh.sup[r] = v;
    }
    __syncwarp();
    for (int i = lane; i < a.k; i += 32) a.support[(size_t)b * a.k + i] = i < ns ? sh.sup[i] : -1;
    if (lane == 0) {
        double total = 0.0, sumsq = 0.0;
        int nz = 0, bad = 0;
        for (int w = 0; w < NW; ++w) {
            total += sh.red[2 * w];
            sumsq += sh.red[2 * w + 1];
            nz += __float_as_int(sh.redf[2 * w]);
            bad += __float_as_int(sh.redf[2 * w + 1]);
        }
        double gf;
        if (bad > 0) gf = INFINITY;
        else if (kb == 0) gf = total > 0.0 ? INFINITY : 0.0;
        else if (total / M > kb * (1.0 + kFeasRtol)) gf = INFINITY;
        else if (nz <= kb) gf = 0.5 * sumsq;
        else {
            // s = the smallest index with tau_s >= |beta|_(s+1) (Theorem 4.1), s = kbar - 1
            // taken also if rounding in total - pre says otherwise
            double pre = 0.0, presq = 0.0;
            int s = 0;
            for (; s < kb - 1; ++s) {
                if ((total - pre) / (kb - s) >= sh.sv[s]) break;
                pre += sh.sv[s];
                presq += sh.sv[s] * sh.sv[s];
            }
            const double tail = total - pre;
            gf = 0.5 * (presq + tail / (kb - s) * tail);
        }
        const double g = 0.5 * sh.vj1[0] + gf;
        a.primal[b] = isinf(g) ? INFINITY : a.sum_loss[row] + 2.0 * a.lam2 * g;
        a.jstar[b] = leaf ? -1 : sh.si[0];
    }
}

}  // namespace

void cert_dual_point(cudaStream_t s, const CertArgs& a) {
    if (a.m <= 0) return;
    if (a.s_is_f64) k_dual_point<256><<<a.m, 256, 0, s>>>(a);
    else {
        int parts = 1;
        while (parts < 8 && (long)a.m_batch * parts < 2 * 152 && a.n / parts >= 1024) parts *= 2;
        const int seg = ((a.n + parts - 1) / parts + 3) / 4 * 4;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)a.m * parts);
        cfg.blockDim = dim3(256);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = parts;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = parts > 1 ? 1 : 0;
        cudaLaunchKernelEx(&cfg, k_dual_point_f32<256>, a, parts, seg);   // errors surface at the caller's check
    }
}

int cert_bound(cudaStream_t s, const CertArgs& a) {
    const int p = a.p, m = a.m;
    if (m <= 0) return 0;
    if (a.Qi) {
#define KGLM_CERT(NT_, E_) k_cert_node<NT_, E_><<<m, NT_, 0, s>>>(a)
        if (p <= 128) KGLM_CERT(64, 2);
        else if (p <= 512) KGLM_CERT(128, 4);
        else if (p <= 1024) KGLM_CERT(256, 4);
        else if (p <= 2048) KGLM_CERT(256, 8);
        else if (p <= 4096) KGLM_CERT(512, 8);
        else if (p <= 8192) KGLM_CERT(512, 16);
        else return -1;
#undef KGLM_CERT
        return 0;
    }
#define KGLM_CERT(NT_, E_) k_cert_bound<NT_, E_><<<m, NT_, 0, s>>>(a)
    if (p <= 64) KGLM_CERT(32, 2);
    else if (p <= 128) KGLM_CERT(64, 2);
    else if (p <= 256) KGLM_CERT(64, 4);
    else if (p <= 512) KGLM_CERT(128, 4);
    else if (p <= 1024) KGLM_CERT(128, 8);
    else if (p <= 2048) KGLM_CERT(256, 8);
    else if (p <= 4096) KGLM_CERT(512, 8);
    else if (p <= 8192) KGLM_CERT(512, 16);
    else return -1;
#undef KGLM_CERT
    return 0;
}

}  // namespace kglm
