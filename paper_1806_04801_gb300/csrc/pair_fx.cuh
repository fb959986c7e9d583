// Fixed-point pair arithmetic of the FP64 near-field sums: one Coulomb pair
// to FP64 accuracy on the integer and FP32 pipes.
//
// Why: this part issues two FP64 lanes per SM and cycle, against 128 FP32 and
// 64 integer-multiply lanes, and a pair takes about 20 FP64 instructions --
// ten cycles per pair and SM, whatever the tiling.  Here a pair takes about
// 150 issue slots of the wide pipes.
//
// Number formats (coordinates scaled by a power of two, the charges of a tile
// by one so that |q| < 1; both scalings are exact):
//   position   x = h 2^-30 + l 2^-60, two integers (|l| <= 2^29); for sources
//              and targets |h| is limited so that no difference overflows
//   charge     q = qh 2^-31 + ql 2^-63, qh signed, ql unsigned
//   distance^2 A 2^-60: sum dh^2 + 2 sum dh dl 2^-30, exact but for the last
//              unit
//   y          the SFU's 1/r after one FP32 Newton step, as the integer
//              Y = y 2^28 (exact: 24 bits)
//   e          1 - r^2 y^2, |e| <= 2^-22, in units 2^-52 from the 128-bit
//              product A Y^2
//   q / r      q y (1 + e/2 + 3 e^2/8)
//   q / r^3    V 2^-51 = q y^3 (1 + 3 e/2 + 15 e^2/8), a 64-bit integer
// and the sums of q y and of V dh run in 96-bit integers, exactly, with FP32
// sums for the terms below 2^-44 of these.  Pairs closer than kFxNearR (in
// scaled units) exceed the formats; the caller sums them in native FP64,
// which also covers a target's own slot.
//
// The units are fixed by the tile's largest charge, so the rounding of a sum is
// the same whatever the charges in it: up to 2^-50 of the charge 1 per pair.  A
// tile is summed this way only where its other charges make up for that
// (fx_charges_fit); the caller sums the rest in native FP64.
//
// Plain C++ so that the arithmetic can be checked on the host.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define HSMA_HD __host__ __device__ __forceinline__
#else
#define HSMA_HD inline
#endif

namespace hsma {

// y < 7.9 keeps Y below 2^31, and 256 terms |q| / r^2 <= 62.5 below 2^63 in
// the units of FxSums::g1.
constexpr double kFxNearR = 1.0 / 7.9;
constexpr uint64_t kFxNearA = (uint64_t)(kFxNearR * kFxNearR * 1152921504606846976.0) >> 32 << 32;

struct FxSource {
    int hx, hy, hz, qh;
    int lx, ly, lz;
    uint32_t ql;
    float fx, fy, fz;  // l 2^-30 in FP32
    float fq;          // q in FP32
};

struct FxTarget {
    int h[3], l[3];
    float f[3];
};

// Sums over one tile (at most 256 sources) for one target.
struct FxSums {
    uint32_t p0, p1;     // sum q y in units 2^-59, 96 bits
    int p2;
    int64_t px;          // correction of q y for 1/r^3 (to first order 3x that of 1/r), units 2^-59
    float pf;            // second-order terms of q / r, units 2^-59
    uint32_t g0[3];      // sum V (dh + 2^31): low 32 of 96 bits, units 2^-81
    int64_t g1[3];
    uint64_t vl;         // sum of V's low words (the 2^31 above)
    float gf[3];         // sum V dl, units 2^-30: the caller folds it every few sources
};

HSMA_HD void fx_clear(FxSums &s)
{
    s.p0 = s.p1 = 0u;
    s.p2 = 0;
    s.px = 0;
    s.pf = 0.f;
    s.vl = 0;
    for (int c = 0; c < 3; ++c) {
        s.g0[c] = 0u;
        s.g1[c] = 0;
        s.gf[c] = 0.f;
    }
}

// a b / 2^32 to within 2^17: where only its upper half matters, half the cost
// of the full product on the pipe that bounds the loop.
HSMA_HD uint32_t fx_mulhi16(uint32_t a, uint32_t b) { return (a >> 16) * (b >> 16); }

HSMA_HD float fx_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return (float)(1.0 / sqrt((double)x));
#endif
}

HSMA_HD int fx_f2i(float x)  // to nearest
{
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int)lrintf(x);
#endif
}

HSMA_HD uint64_t fx_bits(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    memcpy(&b, &v, sizeof b);
    return b;
#endif
}

// v 2^k rounded to an integer, by integer operations (a conversion through
// the FP64 pipe costs as much as 64 of these); |v 2^k| < 2^63.
HSMA_HD int64_t fx_fixed(double v, int k)
{
    const uint64_t b = fx_bits(v);
    const int e = (int)(b >> 52) & 0x7ff, sh = (e > 0 ? e : 1) - 1075 + k;
    const uint64_t m = (b & 0xfffffffffffffull) | (e > 0 ? 0x10000000000000ull : 0ull);
    const uint64_t r = sh >= 0 ? m << sh : (sh > -64 ? ((m >> (-sh - 1)) + 1) >> 1 : 0ull);
    return (int64_t)b < 0 ? -(int64_t)r : (int64_t)r;
}

// Whether |v 2^k| < 2^62 (no for a NaN).
HSMA_HD bool fx_fits(double v, int k) { return ((int)(fx_bits(v) >> 52) & 0x7ff) <= 1084 - k; }

// Coordinate X in units of 2^-60: h within +-lim; whether it lies there.
HSMA_HD bool fx_split(int64_t X, int lim, int &h, int &l, float &f)
{
    const int64_t n = (X + 0x20000000LL) >> 30;
    h = (int)(n < -lim ? -lim : (n > lim ? lim : n));
    const int64_t d = X - ((int64_t)h << 30);
    l = (int)d;
    f = (float)l * 0x1p-30f;
    return d <= 0x40000000LL && d >= -0x40000000LL;
}

// The same from an origin o (an integer in units 2^-30) that may be far off,
// v in units of 2^-30, |v| < 2^51: exact, with FP64 operations.
HSMA_HD bool fx_split_from(double v, double o, int lim, int &h, int &l, float &f)
{
#ifdef __CUDA_ARCH__
    const double magic = 6755399441055744.0;  // 1.5 2^52: a sum's low word is the nearest integer
    const double n = (v + magic) - magic, w = n - o, t = fmin(fmax(w, -(double)lim), (double)lim),
                 d = (v - n) + (w - t);
    h = __double2loint(t + magic);
    l = __double2loint(fma(d, 0x1p30, magic));
#else
    const double n = nearbyint(v), w = n - o, t = fmin(fmax(w, -(double)lim), (double)lim), d = (v - n) + (w - t);
    h = (int)t;
    l = (int)nearbyint(d * 0x1p30);
#endif
    f = (float)d;
    return fabs(d) <= 1.0;
}

// Charge X in units of 2^-63, |q| < 1.
HSMA_HD void fx_split_charge(int64_t X, int &h, uint32_t &l, float &f)
{
    h = (int)(X >> 32);
    l = (uint32_t)X;
    f = (float)X * 0x1p-63f;
}

// One charge's share of a tile's tally: |q| in units 2^-14 (of |q| < 1, rounded
// down) and, from bit 23, one for a charge that is not zero.  A tile of at most
// 256 sources fits the word.
HSMA_HD uint32_t fx_charge_tally(float fq, bool nonzero)
{
    return (uint32_t)(fabsf(fq) * 16384.f) + (nonzero ? 1u << 23 : 0u);
}

// Whether a tile's charges keep FP64 accuracy in these formats; tally: the sum
// of fx_charge_tally, largest: the largest |q| in the same units 2^-14.
//
// The tally counts without the largest charge, which a target may skip (its own
// slot, or a source at the target): the others must be 3/8 on average, or add up
// to 16 and to a twelfth each.  Rms error of such a target's sums, fixed point
// against the FP64 loop (random positions, near pairs left out; potential, field):
//   256 charges +-1       0.12, 0.44     64  0.24, 0.74     16  0.42, 0.84     2  0.80, 0.97
//   256 normal charges    0.42, 0.74     64  0.70, 1.19     16  1.13, 1.26 (mostly refused)
//   1 and 255 charges +-1/4, 1/8         0.13, 0.60 and 1.04, 1.27 (refused)
//   1 and 255 charges +-1/16             3.1, 3.9 (refused)
// (the FP64 loop rounds its running sum at every source, the integers never do,
// which is what the accuracy of many unlike charges comes from).  Tiles of 256
// normal charges pass while their largest is below 4.8 sigma (all but four in
// 10^4): the scale, a power of two, is then below twelve times their mean.
HSMA_HD bool fx_charges_fit(uint32_t tally, uint32_t largest)
{
    const uint32_t nonzero = tally >> 23;
    if (nonzero == 0u) return true;
    const uint32_t others = (tally & 0x7fffffu) - largest, each = (nonzero - 1u) << 14;
    return 8u * others >= 3u * each || (others >= 16u << 14 && 12u * others >= each);
}

// How often the scale of a direct sum is halved below the one that brings the
// coordinates into range; slo..thi: the boxes of its sources and targets, near:
// kFxNearR at that scale in the units of the coordinates.
//
// V has 51 bits after the point, so q / r^3 is coarse at the largest distances
// (r = 2 to 3.5): at targets away from the sources the fields of neutral charges
// had five to thirty times the rms error of the FP64 loop.  A smaller scale
// brings such pairs nearer, and the near radius, which has them summed natively,
// grows with it.  So it is halved while near pairs stay below 0.2% (of points
// spread evenly over the two boxes).  A cube that both share has 0.1% (side 2 at
// the largest scale) to 0.85% (side 1) and is never halved: eight times the near
// pairs cost half the speed there (20011 sources x 3001 targets in a unit cube
// 529 -> 786 us).  Cubes that touch at a corner are halved once, those far apart
// three times.
HSMA_HD int fx_halvings(const float (&slo)[3], const float (&shi)[3], const float (&tlo)[3], const float (&thi)[3],
                        float near)
{
    int k = 0;
    for (; k < 8; ++k) {
        near *= 2.f;
        float share = 0.5236f;  // of a cube, for the ball
        for (int c = 0; c < 3; ++c) {
            const float ls = shi[c] - slo[c], lt = thi[c] - tlo[c];
            // the part of either box within `near` of the other, and how much
            // of the other is as near to a point there
            const float os = fminf(shi[c], thi[c] + near) - fmaxf(slo[c], tlo[c] - near);
            const float ot = fminf(thi[c], shi[c] + near) - fmaxf(tlo[c], slo[c] - near);
            const float s = os < 0.f ? 0.f : (os < ls ? os / ls : 1.f) * (2.f * near < lt ? 2.f * near / lt : 1.f);
            const float t = ot < 0.f ? 0.f : (ot < lt ? ot / lt : 1.f) * (2.f * near < ls ? 2.f * near / ls : 1.f);
            share *= fminf(s, t);
        }
        if (!(share <= 0.002f)) break;
    }
    return k;
}

// dh, dl: source minus target.  The distance^2 in units 2^-60.
HSMA_HD uint64_t fx_distance2(const int (&dh)[3], const int (&dl)[3])
{
    const uint64_t a = (uint64_t)((int64_t)dh[0] * dh[0]) + (uint64_t)((int64_t)dh[1] * dh[1]) +
                       (uint64_t)((int64_t)dh[2] * dh[2]);
    const int64_t b = (int64_t)dh[0] * dl[0] + (int64_t)dh[1] * dl[1] + (int64_t)dh[2] * dl[2];
    return a + (uint64_t)(b >> 29);
}

// Whether a pair at this distance^2 is nearer than kFxNearR.  fx_distance2
// leaves out sum dl^2 (below eight units), so that two points within a unit of
// the high words can get a small negative number: its high word, all ones,
// becomes the smallest here.  (No true distance^2 reaches it: at most 12 2^60.)
HSMA_HD bool fx_near(uint64_t A) { return (uint32_t)(A >> 32) + 1u < (uint32_t)(kFxNearA >> 32) + 1u; }

struct FxPair {
    int64_t q0;        // q y, units 2^-59
    int64_t x;         // q y (3 e/2 + 15 e^2/8), the same units
    uint64_t P;        // y^2, units 2^-56
    float y, ef;       // y; e in units 2^-52
};

// near: 1/r is put to 0.
HSMA_HD FxPair fx_inverse(uint64_t A, bool near, int qh, uint32_t ql)
{
    FxPair r;
    const uint32_t a0 = (uint32_t)A, a1 = (uint32_t)(A >> 32);
    const float s = fmaf((float)a1, 0x1p-28f, (float)a0 * 0x1p-60f);
    float y = near ? 0.f : fx_rsqrt(s);
    y = fmaf(0.5f * y, fmaf(-s * y, y, 1.f), y);
    r.y = y;
    const int Y = fx_f2i(y * 0x1p28f);
    r.P = (uint64_t)(uint32_t)Y * (uint32_t)Y;
    // (A P - 2^116) / 2^32 in 64 bits, wrapping: -e in units 2^-84
    const uint32_t b0 = (uint32_t)r.P, b1 = (uint32_t)(r.P >> 32);
    uint64_t acc = fx_mulhi16(a0, b0) + (uint64_t)a1 * b0 + (uint64_t)a0 * b1;
    acc += (uint64_t)(a1 * b1) << 32;
    const int64_t ne = (int64_t)acc;
    r.ef = -(float)(int)(ne >> 32);
    const int E3 = fx_f2i(r.ef * (1.875f * 0x1p-52f) * r.ef) - (int)((ne + (ne >> 1)) >> 32);
    r.q0 = (int64_t)qh * Y + (int64_t)(((uint64_t)ql * (uint32_t)Y) >> 32);
    const int qc = (int)((r.q0 + 0x80000000LL) >> 32);
    r.x = ((int64_t)qc * E3) >> 20;
    return r;
}

HSMA_HD void fx_add_potential(FxSums &s, const FxPair &r, float fq)
{
    const int sign = (int)(r.q0 >> 63);
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(s.p0), "+r"(s.p1), "+r"(s.p2)
        : "r"((uint32_t)r.q0), "r"((uint32_t)((uint64_t)r.q0 >> 32)), "r"(sign));
#else
    const uint64_t old = ((uint64_t)s.p1 << 32) | s.p0, now = old + (uint64_t)r.q0;
    s.p2 += sign + (now < old ? 1 : 0);
    s.p0 = (uint32_t)now;
    s.p1 = (uint32_t)(now >> 32);
#endif
    s.px += r.x;
    // 1/r has 3 e^2 / 8 where a third of the 1/r^3 correction has 5 e^2 / 8
    s.pf = fmaf(fq * r.y, r.ef * r.ef * -0x1p-47f, s.pf);
}

// qsign: 0 or -1, the sign of qh; df: dl 2^-30 in FP32.
HSMA_HD void fx_add_field(FxSums &s, const FxPair &r, const int (&dh)[3], const float (&df)[3], int qsign, float fq)
{
    // V = (q0 + x) P / 2^64, rounded: units 2^(64 - 59 - 56) = 2^-51
    const uint64_t Q = (uint64_t)(r.q0 + r.x);
    const uint32_t q0 = (uint32_t)Q, q1 = (uint32_t)(Q >> 32), b0 = (uint32_t)r.P, b1 = (uint32_t)(r.P >> 32);
    const uint64_t t1 = (uint64_t)q0 * b1, t2 = (uint64_t)q1 * b0;
    const uint64_t m = (uint64_t)fx_mulhi16(q0, b0) + (uint32_t)t1 + (uint32_t)t2 + 0x80000000ull;
    const int64_t V = (int64_t)(int)q1 * (int64_t)(int)b1 + (int64_t)(t1 >> 32) + (int64_t)(t2 >> 32) +
                      (int64_t)(m >> 32) - (int64_t)(uint32_t)(qsign & (int)b0);
    const int vh = (int)(V >> 32);
    const uint32_t vl = (uint32_t)V;
    const float fv = fq * (r.y * r.y) * fmaf(r.y, r.ef * (1.5f * 0x1p-52f), r.y);  // V in FP32
    s.vl += vl;
    for (int c = 0; c < 3; ++c) {
        const int64_t hh = (int64_t)vh * dh[c];
        const uint64_t t = (uint64_t)vl * ((uint32_t)dh[c] ^ 0x80000000u);
#ifdef __CUDA_ARCH__
        uint32_t lo = (uint32_t)s.g1[c], hi = (uint32_t)((uint64_t)s.g1[c] >> 32);
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, 0;\n\t"
            "add.cc.u32 %1, %1, %5;\n\taddc.u32 %2, %2, %6;"
            : "+r"(s.g0[c]), "+r"(lo), "+r"(hi)
            : "r"((uint32_t)t), "r"((uint32_t)(t >> 32)), "r"((uint32_t)hh), "r"((uint32_t)((uint64_t)hh >> 32)));
        s.g1[c] = (int64_t)(((uint64_t)hi << 32) | lo);
#else
        const uint32_t old = s.g0[c];
        s.g0[c] = old + (uint32_t)t;
        s.g1[c] += hh + (int64_t)(t >> 32) + (s.g0[c] < old ? 1 : 0);
#endif
        s.gf[c] = fmaf(fv, df[c], s.gf[c]);
    }
}

// The sums in scaled units, in FP64.
HSMA_HD double fx_potential(const FxSums &s)
{
    const double hi = (double)(int64_t)(((uint64_t)(uint32_t)s.p2 << 32) | s.p1);
    return fma(hi, 0x1p-27, fma((double)s.p0, 0x1p-59, fma((double)s.px, 0x1p-59 / 3.0, (double)s.pf * 0x1p-59)));
}

HSMA_HD double fx_field(const FxSums &s, int c, double gf)
{
    // minus 2^31 sum(vl), in units 2^-81
    const uint32_t lo = s.g0[c] - (uint32_t)(s.vl << 31);
    const int64_t hi = s.g1[c] - (int64_t)(s.vl >> 1) - (lo > s.g0[c] ? 1 : 0);
    return fma((double)hi, 0x1p-49, fma((double)lo, 0x1p-81, gf * 0x1p-30));
}

}  // namespace hsma
