// Host check of the fixed-point pair arithmetic (csrc/pair_fx.cuh) against
// long double.  argv: mode, count, seed.  Prints the largest potential error
// relative to 1/r, the largest field error relative to 1/r^2 and the largest
// |e|; the sources and targets are scaled coordinates of a sphere of radius
// 1.5 and a box of half-width 0.5.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "pair_fx.cuh"

using namespace hsma;
typedef long double ld;

int main(int argc, char **argv)
{
    const int mode = atoi(argv[1]), count = atoi(argv[2]);
    std::mt19937_64 g(atoi(argv[3]));
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    const int src_lim = (3 << 29) - 1, tgt_lim = 1 << 29;
    ld wp = 0, wf = 0, we = 0;
    for (int it = 0; it < count; ++it) {
        double t[3], s[3], q = u(g);
        for (int c = 0; c < 3; ++c) t[c] = 0.5 * u(g), s[c] = 0.86 * u(g);
        int reps = 1;
        if (mode == 1) {  // just outside the near radius, in every direction
            double n = 0.0, d[3];
            for (int c = 0; c < 3; ++c) d[c] = u(g), n += d[c] * d[c];
            for (int c = 0; c < 3; ++c) s[c] = t[c] + d[c] / std::sqrt(n) * kFxNearR * (1.0 + 0.2 * std::fabs(u(g)));
        }
        if (mode == 2) {  // a full tile of the strongest pairs, the largest charge
            double n = 0.0, d[3];
            for (int c = 0; c < 3; ++c) d[c] = u(g), n += d[c] * d[c];
            for (int c = 0; c < 3; ++c) s[c] = t[c] + d[c] / std::sqrt(n) * kFxNearR * (1.0 + 1e-9);
            q = it % 2 ? 1.0 - 0x1p-53 : -(1.0 - 0x1p-53);
            reps = 256;
        }
        if (mode == 3) {  // the largest differences
            const int c = it % 3;
            for (int k = 0; k < 3; ++k) t[k] = it & (1 << k) ? 0.5 : -0.5, s[k] = 0.0;
            s[c] = (t[c] > 0 ? -1.5 : 1.5) * (1.0 - 0x1p-53);
            if (it % 5 == 0) t[(c + 1) % 3] = u(g) * 0x1p-40;  // and tiny coordinates
        }
        FxSource f;
        bool in = fx_split(fx_fixed(s[0], 60), src_lim, f.hx, f.lx, f.fx);
        in = fx_split(fx_fixed(s[1], 60), src_lim, f.hy, f.ly, f.fy) && in;
        in = fx_split(fx_fixed(s[2], 60), src_lim, f.hz, f.lz, f.fz) && in;
        fx_split_charge(fx_fixed(q, 63), f.qh, f.ql, f.fq);
        FxTarget tg;
        for (int c = 0; c < 3; ++c) {
            in = fx_split(fx_fixed(t[c], 60), tgt_lim, tg.h[c], tg.l[c], tg.f[c]) && in;
            int h, l;  // the form with an origin gives the same words
            float fl;
            in = fx_split_from(t[c] * 0x1p30 + 0x1p40, 0x1p40, tgt_lim, h, l, fl) && in;
            if (std::abs(t[c]) > 0x1p-10 && std::abs(h - tg.h[c]) > 1) in = false;
        }
        if (!in || fx_fits(4.0, 60) ||
            !fx_fits(3.9, 60) || fx_fits(NAN, 60)) {
            printf("range\n");
            return 1;
        }
        const int dh[3] = {f.hx - tg.h[0], f.hy - tg.h[1], f.hz - tg.h[2]};
        const int dl[3] = {f.lx - tg.l[0], f.ly - tg.l[1], f.lz - tg.l[2]};
        const float df[3] = {f.fx - tg.f[0], f.fy - tg.f[1], f.fz - tg.f[2]};
        const uint64_t A = fx_distance2(dh, dl);
        if (A < kFxNearA) continue;
        const FxPair r = fx_inverse(A, false, f.qh, f.ql);
        FxSums sum;
        fx_clear(sum);
        double gf[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < reps; ++k) {
            fx_add_potential(sum, r, f.fq);
            fx_add_field(sum, r, dh, df, f.qh >> 31, f.fq);
            for (int c = 0; c < 3; ++c) gf[c] += sum.gf[c], sum.gf[c] = 0.f;
        }
        ld d[3], r2 = 0;
        for (int c = 0; c < 3; ++c) d[c] = (ld)s[c] - (ld)t[c], r2 += d[c] * d[c];
        const ld ri = 1 / sqrtl(r2);
        we = std::max(we, fabsl(1 - r2 * (ld)r.y * (ld)r.y));
        wp = std::max(wp, fabsl((ld)fx_potential(sum) / reps - q * ri) / ri);
        for (int c = 0; c < 3; ++c)
            wf = std::max(wf, fabsl((ld)fx_field(sum, c, gf[c]) / reps - q * ri * ri * ri * d[c]) * r2);
        // a pair left to the caller adds nothing, whatever the sign of q
        const FxPair z = fx_inverse(A, true, f.qh, f.ql);
        fx_clear(sum);
        fx_add_potential(sum, z, f.fq);
        fx_add_field(sum, z, dh, df, f.qh >> 31, f.fq);
        if (fx_potential(sum) != 0.0 || fx_field(sum, 0, sum.gf[0]) != 0.0) wp = 1;
    }
    printf("%.3Le %.3Le %.3Le\n", wp, wf, we);
    return 0;
}
