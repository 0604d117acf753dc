// Launch shape of the direct pair sum's row kernel (sg_direct.cu): host arithmetic
// alone, so that a test can compile it and see which instances its sizes reach.
#pragma once

#include <algorithm>
#include <cmath>

namespace sg {

constexpr int kDirectLagTile = 128;    // lags per tile
constexpr int kDirectMaxThreads = 256; // threads per CTA, at most

// Targets per thread, warps per CTA and CTAs per cluster (source-row split):
// the shape with the least warp instructions on the fullest SM (152 of them).  Per row
// pair and lag tile a warp spends about 72 on barriers and limits, 45 per staged
// source and 160 per lag of its threads' share, and per lag 2 and 25.5 a
// target (FP32); CTAs of few warps wait at the barriers (an eighth longer with one), and
// fewer than 25 resident warps leave the pipes idle.  Fitted to 50 shapes on 8 discs of 24 x 48 to
// 256 x 512, where the choice is within 8 % of the best: 53 x 603 gas 1.34 ms with (2, 2, 8)
// against 1.96 with (4, 5, 8), 128 x 256 gas + dust 4.59 with (2, 4, 8) against 4.24 with (2, 2, 8).
// FP64: its instructions count alone, 36 a pair and 60 a lag (within 11 % on 4
// discs).  KT: 1, 2, 4 (FP32), 1, 2 (FP64: registers).
struct DirectTile { int KT, W, S, nchunk; };
inline DirectTile direct_tile(int nr, int nphi, bool f64)
{
    DirectTile best{1, 1, 1, 0};
    double best_t = 1e300;
    const int DLT = kDirectLagTile;
    const double tiles = (nphi + DLT - 1) / DLT;
    for (int KT = 1; KT <= (f64 ? 2 : 4); KT *= 2)
        for (int W = 1; W <= kDirectMaxThreads / 32; ++W) {
            const int TJ = 32 * W * KT;
            if (W > 1 && 32 * (W - 1) * KT >= nphi) break;
            const long long nchunk = (nphi + TJ - 1) / TJ;
            for (int S = 1; S <= 8 && S <= nr; S *= 2) {
                const double ctas = std::ceil((double)nr * nchunk * S / 152.0);   // per SM
                const double rows = std::ceil((double)nr / S);
                double t;
                if (f64) {
                    const double work = rows * nphi * (TJ * 36.0 + 60.0 + 2.0 * KT * W * 32 / DLT * 30);
                    t = ctas * work * std::max(1.0, 12.0 / (std::min(ctas * W, 32.0) * std::min(KT, 2)));
                } else {
                    const double share = (double)nphi / (32.0 * W);               // lags of a thread, over all tiles
                    const double work = rows * W * (tiles * 72 + 45 * (KT * tiles + share) + 160 * share + nphi * (KT * 25.5 + 2));
                    t = ctas * work * (1 + 0.12 / W) * std::max(1.0, 25.0 / (ctas * W));
                }
                if (t < best_t * 0.999) {
                    best_t = t;
                    best = {KT, W, S, (int)nchunk};
                }
            }
        }
    return best;
}

}  // namespace sg
