// The memory rule of the automatic factor choice (factor_choice.h).
#include <cstdio>
#include "factor_choice.h"

using namespace helm;

int main() {
    const size_t G = (size_t)1 << 30;
    const struct { size_t bytes, avail; bool want, asked; } t[] = {
        {G, 0, true, false},           {G + 1, 8 * G, false, true},  {2 * G, 16 * G, true, true},
        {2 * G, 16 * G - 8, false, true}, {16 * G, 128 * G, true, true}, {16 * G + 1, 1000 * G, false, false}};
    for (auto &c : t) {
        bool asked = false;
        const bool got = short_bcr_fits(c.bytes, [&]() { asked = true; return c.avail; });
        if (got != c.want || asked != c.asked) {
            printf("%zu of %zu: %d (asked %d)\n", c.bytes, c.avail, got, asked);
            return 1;
        }
    }
    if (short_bcr_bytes(3, 128, 128) != (size_t)48 * 3 * 128 * 128 * 128) { printf("bytes\n"); return 1; }
    printf("ok\n");
    return 0;
}
