// Shapes of the line sweep (host only, no CUDA): CTAs per team and right-hand sides per cluster.
#pragma once
#include <algorithm>

namespace helm {

// CTAs of a team of cs that own rows when each takes ceil(nz / cs): the number a team is launched with.
// The exchange has two buffers and no release: a CTA runs at most a step ahead because it waits for
// the rows of every other CTA of its team, so a CTA without rows would bound nobody, and bytes of two
// steps could meet in one phase of its barrier (n_z = 49 on eight CTAs: seven rows each, the eighth none).
inline int sweep_filled_ctas(int nz, int cs) {
    const int rpc = (nz + cs - 1) / cs;
    return (nz + rpc - 1) / rpc;
}

struct SweepShape {
    int cs, R;   // CTAs per team, right-hand sides per cluster (0: the caller's rule)
};
// FP64: the products, not the exchange, are the length of a step (2 lanes a cycle per SM: 8 us of
// a 10 us step at 64 rows x 8 right-hand sides on 4 CTAs).  CTAs per team (from cs on) and right-hand
// sides per cluster are taken for the least time of (waves of clusters) x (products of a step + about
// 3500 cycles of exchange), the line product's 2 multiply-adds of 2 lanes per entry.  64^2 with 8
// right-hand sides: 649 -> 278 us.  Shorter lines are bound by the exchange (40 x 37 ran 210 us as it
// was, 249 spread out).  active(c, R): clusters of teams * c CTAs that run at once.
template <typename Active> SweepShape sweep_shape_fp64(int nz, int teams, int n_sys, int nrhs, int cs, Active active) {
    SweepShape s{cs, 0};
    if (nz < 48) return s;
    double best = 0.0;
    for (int c = cs; c <= 16 / teams; c = c < 8 && 2 * c > 8 ? 8 : 2 * c) {
        const int rp = (nz + c - 1) / c, cf = sweep_filled_ctas(nz, c);
        for (int r = 1; r <= std::min(16, nrhs); ++r) {
            if (rp * r > 128) break;   // (128 outputs per CTA measured best)
            const int act = std::max(1, active(cf, r));
            const long waves = ((long)n_sys * ((nrhs + r - 1) / r) + act - 1) / act;
            const double t = (double)waves * (2.0 * rp * r * nz + 3500.0);
            if (s.R == 0 || t < best) { best = t; s = SweepShape{cf, r}; }
        }
    }
    return s;
}

}  // namespace helm
