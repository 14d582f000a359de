// Shapes of the line sweep (host only, no CUDA): CTAs per team and right-hand sides per cluster.
#pragma once
#include <algorithm>
#include <cstddef>

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
    int cs, R;   // CTAs per team, right-hand sides per cluster
};
struct SweepFit {   // a shape as it is launched (R right-hand sides; 0: it does not fit the shared memory)
    int R;
    bool slab;      // G's rows of the next line prefetched (else streamed)
    int tpo;        // threads per output
    size_t smem;
};
constexpr int kSweepMaxPerSm = 3;   // CTAs of the FP64 sweep on an SM (its registers)
// clusters of a size that run at once with up to 1, 2 and 3 CTAs on an SM (0: cannot be scheduled)
struct SweepActive {
    int n[kSweepMaxPerSm];
};

// Time of an FP64 sweep, in cycles of a step.  A step of a cluster is the exchange, about 6100 cycles, and
// the products of a CTA's rows, 2 cycles an entry of whole warps (the FP64 pipe takes 2 lanes a cycle
// per SM, idle ones too), plus the reads of G, a quarter of a right-hand side (0.65 where it is
// streamed).  So k CTAs on an SM take k times the products, and share the exchange but for 0.3 of it
// each.  Clusters beyond those that run at once follow as others end.
inline double sweep_time_fp64(int nz, int cs, long clusters, const SweepActive &active, const SweepFit &f) {
    constexpr double kExchange = 6100.0;
    const int rpc = (nz + cs - 1) / cs;
    const int kmax = std::max(1, std::min<int>(kSweepMaxPerSm, (int)(228 * 1024 / (f.smem + 1224))));
    const double outputs = 32.0 * ((rpc * f.R * f.tpo + 31) / 32) / f.tpo;
    const double w = 2.0 * nz * (outputs + rpc * (f.slab ? 0.25 : 0.65));
    auto wave = [&](int k) { return kExchange * (1.0 + 0.3 * (k - 1)) + k * w; };
    const long all = active.n[kmax - 1];
    if (clusters <= all) {
        int k = 1;
        while (clusters > active.n[k - 1]) ++k;
        return wave(k);
    }
    const long rest = clusters % all;
    return (double)(clusters / all) * wave(kmax) + (rest ? wave(kmax) * (double)rest / (double)all + 0.63 * wave(1) : 0.0);
}

// FP64: the shape of the least time, where that is 8 % below that of the given one (`s`: nz / 16 CTAs and 128 outputs
// a CTA, the rule where a step is all exchange), from 48 nodes a line on (shorter ones: 40 x 37 ran 210 us as it
// was, 249 spread out).  active(c): of clusters of teams * c CTAs; fit(c, R): the launch.
// Measured on 60 lines of 48 to 160 nodes, 1 to 8 systems of 1 to 64 right-hand sides, every shape (25000
// points, which the model meets to 8 %): 1.43 times as fast as the given shape on average and 2 % above
// the best, 5 % slower than the given one in 3 of 498 calls.  64^2 with 8 right-hand sides: a call 770 -> 324 us.  Counting
// CTAs that share an SM as free took 60 to 72 nodes with 24 to 64 right-hand sides twice as long.
template <typename Active, typename Fit>
SweepShape sweep_shape_fp64(int nz, int teams, int n_sys, int nrhs, SweepShape s, Active active, Fit fit) {
    if (nz < 48) return s;
    auto time = [&](int c, int R, const SweepActive &a) -> double {   // < 0: not possible
        const SweepFit f = a.n[0] > 0 ? fit(c, R) : SweepFit{0, false, 1, 0};
        return f.R > 0 ? sweep_time_fp64(nz, c, (long)n_sys * ((nrhs + f.R - 1) / f.R), a, f) : -1.0;
    };
    const double t0 = time(s.cs, s.R, active(s.cs));
    double best = t0 < 0 ? -1.0 : t0 / 1.08;
    constexpr int kR[] = {1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 16};
    int last = 0;
    for (int c = (nz + 63) / 64; c <= 16 / teams; ++c) {
        const int cf = sweep_filled_ctas(nz, c);
        if (cf == last) continue;
        last = cf;
        const SweepActive a = active(cf);
        for (int R : kR) {
            if (R > 1 && (R > nrhs || (nz + cf - 1) / cf * R > 256)) break;
            const double t = time(cf, R, a);
            if (t >= 0 && (best < 0 || t < best)) { best = t; s = SweepShape{cf, R}; }
        }
    }
    return s;
}

}  // namespace helm
