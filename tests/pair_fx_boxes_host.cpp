// Host check of the scale of a direct sum (csrc/pair_fx.cuh) for sources and
// targets in boxes of their own: sides and offset along each axis in argv, then
// the number of targets and a seed; 256 charges +-1 per target.  Prints the
// halvings, the share of near pairs and, over the others, the rms error of
// potential and field over the FP64 loop's.
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
    double side[3], tside[3], off[3];
    for (int c = 0; c < 3; ++c) side[c] = atof(argv[1 + c]), tside[c] = atof(argv[4 + c]), off[c] = atof(argv[7 + c]);
    const int count = atoi(argv[10]), n = 256, lim = 1 << 30;
    std::mt19937_64 g(atoi(argv[11]));
    std::uniform_real_distribution<double> u(0.0, 1.0);
    float slo[3], shi[3], tlo[3], thi[3], half = 0.f;
    double mid[3];
    for (int c = 0; c < 3; ++c) {
        slo[c] = 0.f, shi[c] = (float)side[c], tlo[c] = (float)off[c], thi[c] = (float)(off[c] + tside[c]);
        const float lo = std::min(slo[c], tlo[c]), hi = std::max(shi[c], thi[c]);
        mid[c] = 0.5 * ((double)lo + (double)hi);
        half = std::max(half, 0.5f * (hi - lo) * 1.0000002f);
    }
    int e = 0;
    std::frexp(half * 1.000001f, &e);  // half < 2^e
    const int k = fx_halvings(slo, shi, tlo, thi, (float)std::ldexp(kFxNearR, e));
    const double scale = std::ldexp(1.0, -e - k);
    auto split = [&](const double *v, int *h, int *l, float *f) {
        bool in = true;
        for (int c = 0; c < 3; ++c)
            in = fx_split_from(v[c] * scale * 0x1p30, std::rint(mid[c] * scale * 0x1p30), lim - 1, h[c], l[c], f[c]) && in;
        return in;
    };
    ld fp = 0, np = 0, ff = 0, nf = 0;
    long long near = 0;
    for (int it = 0; it < count; ++it) {
        double t[3], phi = 0, fld[3] = {0, 0, 0}, gf[3] = {0, 0, 0};
        int th[3], tl[3];
        float tf[3];
        for (int c = 0; c < 3; ++c) t[c] = off[c] + tside[c] * u(g);
        if (!split(t, th, tl, tf)) return 1;
        FxSums sum;
        fx_clear(sum);
        ld P = 0, F[3] = {0, 0, 0};
        for (int i = 0; i < n; ++i) {
            double s[3];
            int sh[3], sl[3];
            float sf[3];
            for (int c = 0; c < 3; ++c) s[c] = side[c] * u(g);
            if (!split(s, sh, sl, sf)) return 1;
            const double q = i % 2 ? 1.0 : -1.0;
            const int dh[3] = {sh[0] - th[0], sh[1] - th[1], sh[2] - th[2]};
            const int dl[3] = {sl[0] - tl[0], sl[1] - tl[1], sl[2] - tl[2]};
            const float df[3] = {sf[0] - tf[0], sf[1] - tf[1], sf[2] - tf[2]};
            const uint64_t A = fx_distance2(dh, dl);
            if (fx_near(A)) {
                ++near;
                continue;
            }
            int qh;
            uint32_t ql;
            float fq;
            fx_split_charge(fx_fixed(q, 62), qh, ql, fq);
            const FxPair r = fx_inverse(A, false, qh, ql);
            fx_add_potential(sum, r, fq);
            fx_add_field(sum, r, dh, df, qh >> 31, fq);
            for (int c = 0; c < 3; ++c) gf[c] += sum.gf[c], sum.gf[c] = 0.f;
            const double d[3] = {s[0] - t[0], s[1] - t[1], s[2] - t[2]};
            const double ri = 1.0 / std::sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]), q3 = q * ri * ri * ri;
            phi += q * ri;
            ld D[3], r2 = 0;
            for (int c = 0; c < 3; ++c) fld[c] += q3 * d[c], D[c] = (ld)s[c] - (ld)t[c], r2 += D[c] * D[c];
            const ld Ri = 1 / sqrtl(r2);
            P += q * Ri;
            for (int c = 0; c < 3; ++c) F[c] += q * Ri * Ri * Ri * D[c];
        }
        const ld ep = (ld)fx_potential(sum) * 2 * scale - P;
        fp += ep * ep, np += (phi - P) * (phi - P);
        for (int c = 0; c < 3; ++c) {
            const ld ef = (ld)fx_field(sum, c, gf[c]) * 2 * scale * scale - F[c];
            ff += ef * ef, nf += (fld[c] - F[c]) * (fld[c] - F[c]);
        }
    }
    printf("%d %.5f %.3Lf %.3Lf\n", k, (double)near / ((double)n * count), sqrtl(fp / np), sqrtl(ff / nf));
    return 0;
}
