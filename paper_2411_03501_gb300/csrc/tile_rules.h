// tile_rules.h -- default tiles chosen by an estimate of a stage's time: host
// arithmetic alone.
#pragma once
#include <algorithm>
#include <cmath>

namespace lsp {

struct RuleTile {
    int tb, ta, ch;  // ch = 0: no tile
};

// The 16 x 16 tile of the paired shared-face WENO5 kernel (stage_pair.cuh) in
// chunks for about three waves of 3 CTAs per SM, of even length (its planes
// are paired).  d = 3 or 4 axes.
inline RuleTile pair_square_tile(int d, const int* n, long long sms)
{
    const long long nplane = (long long)((n[d - 1] + 15) / 16) * ((n[d - 2] + 15) / 16) * (d == 4 ? n[0] : 1);
    const int nS = n[d - 3];
    const long long nch = std::max(1LL, std::min((9 * sms + nplane - 1) / nplane, (long long)nS / 4));
    const int ch = (int)((nS + nch - 1) / nch);
    return {16, 16, ch + (ch & 1)};
}

// Estimated time in us of a stage of that kernel on a 3-D grid, back to back
// with others of its kind.
//  - A pair of planes takes f(k) = (1.88^2.4 + (0.128 k u)^2.4)^(1/2.4) us with k
//    CTAs on the SM that started together and u = warps (1 + 0.19 frame / tile):
//    the latency of one chain, or the issue slots of all.  A chunk takes its
//    pairs and 0.32 more for its start.
//  - 24 warps of 80 registers fit on an SM: R = 24 / warps CTAs.
//  - A launch of one wave: its CTAs start beside the previous stage's, so above
//    half a wave some SMs fill up to R while others wait (16 x 16 tiles of 6
//    planes: 9.5 us up to one CTA per SM, 11.8 up to 1.5, 15.5 up to 3).
//  - More: R CTAs out of step take 0.74 of f(R) a pair (0.73 pairs for a start),
//    and the tail of the last is 0.42 of a chunk.
// Fitted to 42,800 timings on 870 random grids (root mean square error 5 %).
struct PairCost {
    int nS, R;
    double unit, columns, sms, full_pair;
    PairCost(const int* n, int tb, int ta, long long sms_)
    {
        const int nA = n[1], nB = n[2], G = 3, warps = (tb * ta + 31) / 32;
        nS = n[0];
        R = 24 / warps;
        unit = 0.128 * warps * (1.0 + 0.19 * 2 * G * (tb + ta) / (tb * ta));
        columns = (double)((nB + tb - 1) / tb) * ((nA + ta - 1) / ta);
        sms = (double)sms_;
        full_pair = pair_us(R);
    }
    double pair_us(double k) const
    {
        return std::pow(4.5498 + std::pow(k * unit, 2.4), 1.0 / 2.4);  // 1.88^2.4
    }
    double operator()(int ch) const
    {
        const double chunks = (nS + ch - 1) / ch, per_sm = columns * chunks / sms;
        const double chunk = 0.5 * std::min(ch, nS) + 0.32, full = chunk * full_pair;
        if (per_sm <= 0.5 * R) return 2.9 + chunk * pair_us(std::ceil(per_sm));
        if (per_sm <= R) return 2.9 + full;
        return 2.9 + std::max(full, 0.74 * columns * (0.5 * nS + 0.73 * chunks) / sms * full_pair / R + 0.42 * full);
    }
};

// Tile of that kernel on a 3-D grid: the lowest estimate over tiles of 64 to
// 256 threads that split both axes evenly and a few even chunk lengths, where
// it is 5 % below the square tile's, else none (the square tile is used).
// On 360 other grids (7 to 3000 nodes an axis) the geometric mean is 0.757 of
// the square tile's time; four are slower by more than 3 % (1.13 on 9 x 262 x
// 206, else 1.04).  us per stage, square tile and this rule: 41^3 9.7, 5.4; 97 x
// 113 x 85 25.4, 22.5; 429 x 286 x 8 40.8, 25.6; 3000 x 148 x 19 228, 146; 201^3
// (square) 123.6.
inline RuleTile pair_rule(const int* n, long long sms)
{
    const int nS = n[0], nA = n[1], nB = n[2], G = 3;
    RuleTile best{0, 0, 0};
    double best_cost = 0.0;
    const auto even = [](int axis, int t) {  // t splits the axis evenly
        const int k = (axis + t - 1) / t;
        return (axis + k - 1) / k == t;
    };
    for (int tb = std::min(64, nB); tb >= 8; --tb) {
        if (!even(nB, tb)) continue;
        for (int ta = std::min(256 / tb, nA); ta >= 4 && tb * ta >= 64; --ta) {
            if (!even(nA, ta) || (nA + ta - 1) / ta > 65535) continue;
            // the haloed tile in 3 values per thread
            if ((ta + 2 * G) * (tb + 2 * G) > 3 * ta * tb) continue;
            const PairCost cost(n, tb, ta, sms);
            for (const int ch : {2, 4, 6, 8, 10, 12, 16, 20, 26, 34, 50, 66, 102}) {
                if (ch > nS + 1) break;
                if ((nS + ch - 1) / ch > 65535) continue;
                const double c = cost(ch);
                if (best.ch == 0 || c < best_cost) {
                    best = {tb, ta, ch};
                    best_cost = c;
                }
            }
        }
    }
    const RuleTile square = pair_square_tile(3, n, sms);
    if (best.ch && PairCost(n, square.tb, square.ta, sms)(square.ch) <= 1.05 * best_cost) best.ch = 0;
    return best;
}

// Would the marching kernel's tile (stage_march.cuh) compute more than two
// nodes per node of a 4-D grid, in more than one wave of CTAs?  Its tiles are
// moved back from an axis' end, nodes under two of them computed twice, and a
// chunk starts at the cost of two planes.  ENO3 with 7 rows (the shortest axis;
// its frame allows tiles of 6 there) is then slower than the scalar kernel: 69
// x 14 x 7 x 800 (2.01) 120 us per stage against 104, 7 x 7 x 7 x 3000 (2.5)
// 40 against 34; 25 x 39 x 7 x 263 (2.24) 49.2, 49.6; 47 x 72 x 7 x 169 (1.996)
// 89, 97.  A single wave is bound by latency, and the march is faster (7 x 53 x
// 7 x 497, 2.4: 36 against 42).
inline bool march_wasteful(const int* n, const RuleTile& t, int threads, long long sms)
{
    const auto up = [](int a, int b) { return (a + b - 1) / b; };
    const int ch = std::min(t.ch, n[1]);
    const double computed = (double)up(n[3], t.tb) * t.tb * up(n[2], t.ta) * t.ta * up(n[0], 2) * 2 * (ch + 2) / ch;
    const double ctas = (double)up(n[3], t.tb) * up(n[2], t.ta) * up(n[0], 2) * up(n[1], t.ch);
    return computed > 2.0 * n[3] * n[2] * n[0] && ctas * threads > 512.0 * sms;
}

}  // namespace lsp
