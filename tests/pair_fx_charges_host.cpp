// Host check of the fixed-point pair arithmetic (csrc/pair_fx.cuh) where the
// charges of a tile differ: the sums of a target that skips the tile's largest
// charge, against long double and against the FP64 loop.
// argv: distribution, sources, parameter, tiles, seed.  Prints over the tiles
// that fx_charges_fit accepts: their number, the rms error of the potential and
// field over the FP64 loop's, and the largest error relative to the sums of
// |q|/r and |q|/r^2 of the sources that are not skipped.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "pair_fx.cuh"

using namespace hsma;
typedef long double ld;

int main(int argc, char **argv)
{
    const char *dist = argv[1];
    const int n = atoi(argv[2]), tiles = atoi(argv[4]);
    const double par = atof(argv[3]);
    std::mt19937_64 g(atoi(argv[5]));
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    std::normal_distribution<double> normal;
    const int src_lim = (3 << 29) - 1, tgt_lim = 1 << 29;
    auto sign = [&] { return g() & 1 ? 1.0 : -1.0; };
    int accepted = 0;
    ld fx_p = 0, nat_p = 0, fx_f = 0, nat_f = 0, worst_p = 0, worst_f = 0;
    for (int it = 0; it < tiles; ++it) {
        std::vector<double> q(n);
        for (int i = 0; i < n; ++i) {
            if (!strcmp(dist, "normal")) q[i] = par * normal(g);
            if (!strcmp(dist, "ions")) q[i] = i % 2 ? par : -par;
            if (!strcmp(dist, "heavy")) q[i] = i == 0 ? 1.0 : sign() * par;  // one charge 1, the others +-par
            if (!strcmp(dist, "lognormal")) q[i] = sign() * std::exp(par * normal(g));
            if (!strcmp(dist, "uniform")) q[i] = par * u(g);
            if (!strcmp(dist, "zeros")) q[i] = i % 4 ? 0.0 : sign() * (1.0 + par * u(g));
        }
        const int big = (int)(std::max_element(q.begin(), q.end(), [](double a, double b) {
                                  return std::fabs(a) < std::fabs(b);
                              }) - q.begin());
        int eq = 0;
        std::frexp(q[big], &eq);  // the charges in units of 2^eq
        FxTarget tg;
        double t[3];
        for (int c = 0; c < 3; ++c) t[c] = 0.5 * u(g), fx_split(fx_fixed(t[c], 60), tgt_lim, tg.h[c], tg.l[c], tg.f[c]);
        FxSums sum;
        fx_clear(sum);
        uint32_t tally = 0;
        double gf[3] = {0, 0, 0}, np = 0, nf[3] = {0, 0, 0};
        ld p = 0, f[3] = {0, 0, 0}, ap = 0, af = 0;
        for (int i = 0; i < n; ++i) {
            FxSource s;
            double x[3];
            int dh[3], dl[3];
            uint64_t A;
            do {
                for (double &v : x) v = 0.86 * u(g);
                fx_split(fx_fixed(x[0], 60), src_lim, s.hx, s.lx, s.fx);
                fx_split(fx_fixed(x[1], 60), src_lim, s.hy, s.ly, s.fy);
                fx_split(fx_fixed(x[2], 60), src_lim, s.hz, s.lz, s.fz);
                dh[0] = s.hx - tg.h[0], dh[1] = s.hy - tg.h[1], dh[2] = s.hz - tg.h[2];
                dl[0] = s.lx - tg.l[0], dl[1] = s.ly - tg.l[1], dl[2] = s.lz - tg.l[2];
                A = fx_distance2(dh, dl);
            } while (A < kFxNearA);
            fx_split_charge(fx_fixed(q[i], 63 - eq), s.qh, s.ql, s.fq);
            tally += fx_charge_tally(s.fq, q[i] != 0.0);
            if (i == big) continue;
            const float df[3] = {s.fx - tg.f[0], s.fy - tg.f[1], s.fz - tg.f[2]};
            const FxPair r = fx_inverse(A, false, s.qh, s.ql);
            fx_add_potential(sum, r, s.fq);
            fx_add_field(sum, r, dh, df, s.qh >> 31, s.fq);
            for (int c = 0; c < 3; ++c) gf[c] += sum.gf[c], sum.gf[c] = 0.f;
            const double d[3] = {x[0] - t[0], x[1] - t[1], x[2] - t[2]};
            const double ri = 1.0 / std::sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]), q3 = q[i] * ri * ri * ri;
            np += q[i] * ri;
            for (int c = 0; c < 3; ++c) nf[c] += q3 * d[c];
            ld e[3], r2 = 0;
            for (int c = 0; c < 3; ++c) e[c] = (ld)x[c] - (ld)t[c], r2 += e[c] * e[c];
            const ld Ri = 1 / sqrtl(r2);
            p += q[i] * Ri, ap += std::fabs(q[i]) * Ri, af += std::fabs(q[i]) * Ri * Ri;
            for (int c = 0; c < 3; ++c) f[c] += q[i] * Ri * Ri * Ri * e[c];
        }
        if (!fx_charges_fit(tally, (uint32_t)(std::ldexp(std::fabs(q[big]), -eq) * 16384.0))) continue;
        ++accepted;
        const ld scale = std::ldexp(1.0, eq), ep = fx_potential(sum) * scale - p;
        fx_p += ep * ep, nat_p += (np - p) * (np - p), worst_p = std::max(worst_p, fabsl(ep) / ap);
        for (int c = 0; c < 3; ++c) {
            const ld ef = fx_field(sum, c, gf[c]) * scale - f[c];
            fx_f += ef * ef, nat_f += (nf[c] - f[c]) * (nf[c] - f[c]), worst_f = std::max(worst_f, fabsl(ef) / af);
        }
    }
    printf("%d %.3Lf %.3Lf %.3Le %.3Le\n", accepted, accepted ? sqrtl(fx_p / nat_p) : 0, accepted ? sqrtl(fx_f / nat_f) : 0,
           worst_p, worst_f);
    return 0;
}
