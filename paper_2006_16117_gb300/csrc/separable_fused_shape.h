// The launch shape of the fused separable apply (separable_fused.cu).
#pragma once

#include <stddef.h>

#include <algorithm>
#include <cmath>

namespace sim {

constexpr int SF_T = 256;     // threads of a CTA
constexpr int SF_STAGES = 3;  // of rows of Q in shared memory

constexpr int sf_pad4(int n) { return (n + 3) / 4 * 4; }
// rows of Q per stage: three stages within 48 KB
constexpr int sf_stage_rows(int ldq) { return ldq <= 256 ? 16 : (ldq <= 512 ? 8 : 4); }
constexpr size_t sf_stage_floats(int N) { return (size_t)sf_stage_rows(sf_pad4(N)) * sf_pad4(N); }

// (rows, columns) a thread forms at a time, from few to many
constexpr int kSepTiles[3][2] = {{1, 4}, {2, 4}, {4, 4}};

struct FusedShape {
    int C = 0, Rc = 0, Cc = 0, tile = 2;
    size_t smem = 0;
    double cost = 1e300;
};

// Cluster size and tile by an estimate of the clocks of an apply.  A product takes,
// per two reduction steps and round of 256 threads, 1.5 times its loads' way into
// the registers (a 16-byte load of a warp takes 4 clocks), at least 200 clocks, and
// a round's results 100 clocks a value (measured on 30 to 250 points a side: 40,000
// clocks at 60 points with four CTAs and 1 x 4, 185,000 at 250 with 16 and 4 x 4,
// where 2 x 4 takes 260,000 and 4 x 8, on half the threads, 220,000).
// Clusters of at most `most` CTAs, on `sms` multiprocessors.
inline FusedShape fused_shape(int N0, int N1, int na, int sms, int most) {
    FusedShape best;
    for (int C = 1; C <= most; ++C) {
        FusedShape f;
        f.Rc = (N1 + C - 1) / C;
        f.Cc = (N0 + C - 1) / C;
        if (C > 1 && ((C - 1) * f.Rc >= N1 || (C - 1) * f.Cc >= N0)) continue;  // a CTA without lines
        f.C = C;
        f.smem = 16 * (size_t)std::max(f.Rc * sf_pad4(N0), f.Cc * sf_pad4(N1)) +
                 SF_STAGES * sizeof(float) * std::max(sf_stage_floats(N0), sf_stage_floats(N1));
        if (f.smem > 220 * 1024) continue;
        const double per_sm = std::ceil((double)na * C / sms);  // CTAs that share an SM, in turn or at once
        for (int t = 0; t < 3; ++t) {
            const int RT = kSepTiles[t][0], KT = kSepTiles[t][1];
            auto product = [&](int rows, int N) {
                const int items = (N + KT - 1) / KT * ((rows + RT - 1) / RT);
                const double rounds = std::ceil((double)items / SF_T);
                const double warps = std::min<double>(SF_T / 32, std::ceil(items / 32.0));
                const double lsu = warps * (RT + KT / 2.0) * 4.0;
                return rounds * (N / 2.0 * std::max(200.0, 1.5 * lsu) + 100.0 * warps * RT * KT / 2.0);
            };
            const double cost = per_sm * (2.0 * product(f.Rc, N0) + 2.0 * product(f.Cc, N1)) + (C > 1 ? 9000.0 : 4000.0);
            if (cost < best.cost) {
                best = f;
                best.tile = t;
                best.cost = cost;
            }
        }
    }
    return best;
}

// The best shape that the device places, as fits(shape) says; C = 0 if there is none.
template <class Fits> FusedShape fused_shape_that_fits(int N0, int N1, int na, int sms, Fits fits) {
    FusedShape f = fused_shape(N0, N1, na, sms, 16);
    while (f.C > 0 && !fits(f)) f = fused_shape(N0, N1, na, sms, f.C - 1);
    return f;
}

}  // namespace sim
