// Shapes of the line sweep (sweep_shape.h): every CTA of a team owns rows, the rows are covered, and
// clusters stay within sixteen CTAs.
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
    const int rhs[] = {1, 3, 8, 17, 64}, sys[] = {1, 3, 8};
    for (int teams = 1; teams <= 2; ++teams)
        for (int nz = 4; nz <= 700; ++nz)
            for (int nrhs : rhs)
                for (int ns : sys) {
                    int cs0 = nz / 16;
                    cs0 = cs0 < 1 ? 1 : (cs0 > 16 / teams ? 16 / teams : cs0);
                    const SweepShape s = sweep_shape_fp64(nz, teams, ns, nrhs, cs0, [&](int c, int) { return 140 / (teams * c); });
                    const int rp = (nz + s.cs - 1) / s.cs;
                    if (s.cs < 1 || s.cs * teams > 16 || (s.cs - 1) * rp >= nz || s.R < 0 || s.R > 16 || s.R > nrhs) {
                        printf("teams %d nz %d nrhs %d systems %d: %d CTAs of %d rows, R %d\n", teams, nz, nrhs, ns, s.cs, rp, s.R);
                        return 1;
                    }
                }
    printf("ok\n");
    return 0;
}
