// Host check that pairs too close for the fixed-point formats are recognised:
// random pairs from distance zero, over the units of the two words, to the near
// radius.  argv: pairs, seed.  Prints how many pairs well inside the radius
// were not taken for near, and how many well outside were.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "pair_fx.cuh"

using namespace hsma;

int main(int argc, char **argv)
{
    const int count = atoi(argv[1]);
    std::mt19937_64 g(atoi(argv[2]));
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    const int src_lim = (3 << 29) - 1, tgt_lim = 1 << 29;
    int missed = 0, wrong = 0;
    for (int it = 0; it < count; ++it) {
        double t[3], s[3], r2 = 0;
        const double size = std::ldexp(1.0, it % 65 - 62);  // 2^-62 .. 4
        for (int c = 0; c < 3; ++c) {
            t[c] = 0.5 * u(g);
            if (it % 3 == 0) t[c] = (std::floor(t[c] * 0x1p30) + 0.5) * 0x1p-30;  // between two values of the high word
            s[c] = t[c] + (it % 5 == c ? 0.0 : size * u(g));
            if (std::fabs(s[c]) > 1.5) s[c] = t[c];
            r2 += (s[c] - t[c]) * (s[c] - t[c]);
        }
        int dh[3], dl[3];
        for (int c = 0; c < 3; ++c) {
            int hs, ls, ht, lt;
            float f;
            fx_split(fx_fixed(s[c], 60), src_lim, hs, ls, f);
            fx_split(fx_fixed(t[c], 60), tgt_lim, ht, lt, f);
            dh[c] = hs - ht, dl[c] = ls - lt;
        }
        const bool near = fx_near(fx_distance2(dh, dl));
        if (std::sqrt(r2) < kFxNearR * 0.999 && !near) ++missed;
        if (std::sqrt(r2) > kFxNearR * 1.001 && near) ++wrong;
    }
    printf("%d %d\n", missed, wrong);
    return 0;
}
