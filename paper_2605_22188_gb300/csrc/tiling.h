// The rule that picks the tiles of the tensor-core products where nobody set them (host
// arithmetic only).
#pragma once

#include <algorithm>

namespace kglm {

// Column tile, CTA pairs and split-K slices (0: the launcher's own count) of a product.
struct Tiling {
    int bn;
    bool pair;
    int splits;
};

// A product to be tiled: M rows (of a batch of Mb, which sets the split-K), N columns, nkb K
// slices of 128 bytes, na and nb parts of its operands.
struct TileShape {
    int M, Mb, N, nkb, na, nb;
    int def, max_bn;        // the default column tile, and the widest to look at
    int grad_splits;        // G = X^T R: the cap of its split-K slices; 0: a product that sums its own
    bool can_pair;          // whether the launcher takes CTA pairs for it
    int pair;               // 1 on, 0 off, -1 by the rule
};

// Microseconds of an M x N product over nkb K slices of 128 bytes at column tile bn: the
// busiest worker's units, each bound by its products (2 cycles per column, slice and
// part product) or by its operands' way from L2.  Measured on S = X V of 2048 nodes, n =
// 10000, p = 2000: single CTAs take 0.50 us a slice whether the tile has 128 columns or
// 224 (up to 87 KB/us), pairs 0.39 to 0.41 us at 192 to 256 columns (78 KB/us per CTA).
// Plus the last unit's epilogue and a pair's cluster launch.
inline double tiling_cost(int M, int N, int nkb, int na, int nb, int bn, bool pair, int splits) {
    const int mt = (M + 127) / 128, nt = (N + bn - 1) / bn;
    const long units = (long)(pair ? (mt + 1) / 2 : mt) * nt * splits;
    const int workers = pair ? 76 : 152;
    const double per = (nkb + splits - 1) / splits;
    const double mma = 2.0 * bn * (na + nb - 1) / 1900.0;
    const double load = pair ? std::max((128.0 + bn / 2) * 0.128 / 78.0, 0.38)
                             : std::max((128.0 * na + (double)bn * nb) * 0.128 / 87.0, 0.48);
    const double unit = per * std::max(mma, load) + 0.5;
    return (double)((units + workers - 1) / workers) * unit + 2.5 * bn / 256.0 + (pair ? 1.5 : 0.0);
}

// The column tile and CTA pairs of a product of M nodes.  The
// default widths leave SMs idle in the last wave (2048 nodes, p = 2000: 128 units on
// 152 SMs) and take in twice the operand bytes a pair does.  The number of split-K
// slices stays the default width's, and a product's sums run over K in the same order at
// any width and in pairs, so that no bit of a result depends on the choice.  2048
// nodes, n = 10000, p = 2000: S 147 -> 70 us per launch, G 81 -> 65,
// X beta 420 -> 365; 64 nodes,
// n = 1373, p = 611: G 16.3 -> 11.3 us.
inline Tiling choose_tiling(const TileShape& q) {
    const bool grad = q.grad_splits > 0;
    const int tiles = ((q.Mb + 127) / 128) * ((q.N + q.def - 1) / q.def);
    // the default's split-K (tc_gemm)
    const int splits = grad ? std::max(1, std::min(q.grad_splits, std::min((q.nkb + 3) / 4, std::max(1, 152 / tiles))))
                            : (tiles < 152 ? std::min((q.nkb + 3) / 4, std::max(1, 152 / tiles)) : 1);
    Tiling best{q.def, q.pair == 1 && q.can_pair, splits};
    if (grad || splits == 1) {
        double cost = tiling_cost(q.M, q.N, q.nkb, q.na, q.nb, q.def, best.pair, splits);
        for (int bn = 64; bn <= q.max_bn; bn += 16)
            for (int pr = 0; pr <= (q.can_pair ? 1 : 0); ++pr) {
                if (q.pair >= 0 && (pr != 0) != (q.pair == 1 && q.can_pair)) continue;   // as the caller set them
                const double t = tiling_cost(q.M, q.N, q.nkb, q.na, q.nb, bn, pr != 0, splits);
                if (t < 0.97 * cost) {
                    cost = t;
                    best = {bn, pr != 0, splits};
                }
            }
    }
    return best;
}

}  // namespace kglm
