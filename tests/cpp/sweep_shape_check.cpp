// Shapes of the line sweep (sweep_shape.h): every CTA of a team owns rows, the rows are covered, clusters
// stay within sixteen CTAs, and the FP64 rule leaves the given shape only for one that its model has faster.
#include <cstdio>
#include "sweep_shape.h"

using namespace helm;

int main() {
    for (int nz = 4; nz <= 700; ++nz)
        for (int cs = 1; cs <= 16; ++cs) {
            const int f = sweep_filled_ctas(nz, cs), rp = (nz + f - 1) / f;
            if (f < 1 || f > cs || (f - 1) * rp >= nz || f * rp < nz || rp != (nz + cs - 1) / cs) {
                printf("nz %d cs %d: %d CTAs of %d rows\n", nz, cs, f, rp);
                return 1;
            }
        }
    // SMs in groups of 19, a cluster within one
    for (int few = 0; few < 2; ++few)   // few: clusters of more than eight CTAs cannot be scheduled
        for (int teams = 1; teams <= 2; ++teams)
            for (int nz = 4; nz <= 700; ++nz)
                for (int nrhs : {1, 3, 8, 17, 64})
                    for (int ns : {1, 3, 8}) {
                        int cs0 = nz / 16, R0 = 1;
                        cs0 = cs0 < 1 ? 1 : (cs0 > 16 / teams ? 16 / teams : cs0);
                        while (R0 * 2 <= 16 && (nz + cs0 - 1) / cs0 * R0 * 2 <= 128) R0 *= 2;
                        auto active = [&](int c) {
                            SweepActive a;
                            for (int k = 0; k < kSweepMaxPerSm; ++k) a.n[k] = few && teams * c > 8 ? 0 : 8 * (19 * (k + 1) / (teams * c));
                            return a;
                        };
                        auto fit = [&](int c, int R) {
                            const size_t rp = (nz + c - 1) / c;
                            R = R < nrhs ? R : nrhs;
                            while (R > 1 && 80 * (size_t)R * nz + 32 * rp * nz > 200 * 1024) R = (R + 1) / 2;
                            const bool slab = 80 * (size_t)R * nz + 32 * rp * nz <= 200 * 1024;
                            return SweepFit{R, slab, 1, slab ? 80 * (size_t)R * nz + 32 * rp * nz : 80 * (size_t)R * nz + 1024 * rp};
                        };
                        const SweepShape s = sweep_shape_fp64(nz, teams, ns, nrhs, SweepShape{cs0, R0}, active, fit);
                        const int rp = (nz + s.cs - 1) / s.cs;
                        const bool kept = s.cs == cs0 && s.R == R0;
                        bool ok = s.cs >= 1 && s.cs * teams <= 16 && (s.cs - 1) * rp < nz && s.R >= 1 && s.R <= 16 &&
                                  (kept || (nz >= 48 && active(s.cs).n[0] > 0 && (s.R == 1 || s.R <= nrhs)));
                        if (ok && !kept && active(cs0).n[0] > 0) {
                            const SweepFit a = fit(cs0, R0), b = fit(s.cs, s.R);
                            ok = sweep_time_fp64(nz, s.cs, (long)ns * ((nrhs + b.R - 1) / b.R), active(s.cs), b) * 1.079 <
                                 sweep_time_fp64(nz, cs0, (long)ns * ((nrhs + a.R - 1) / a.R), active(cs0), a);
                        }
                        if (!ok) {
                            printf("teams %d nz %d nrhs %d systems %d: %d CTAs of %d rows, R %d\n", teams, nz, nrhs, ns, s.cs, rp, s.R);
                            return 1;
                        }
                    }
    printf("ok\n");
    return 0;
}
