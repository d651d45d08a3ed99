// FP64 exponential, sine and cosine with few FP64 instructions (the FP64 pipe has 2
// lanes per SM and clock): tables (2^(j/64), 256 points of the circle) and short
// Taylor polynomials of the reduced argument, table indices taken from the low
// bits of a magic-number addition (Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989; the
// same for sin and cos by angle addition): about 33 FP64 instructions per complex
// exponential, against about 80 for exp and sincos.
#pragma once

namespace gbs {

struct Gf64Tables {         // each value as a double and its rounding error
    double2 exp2[64];         // 2^(j/64)
    double2 sn[256], cs[256]; // sin, cos of 2 pi j / 256
};

constexpr double kMagic = 6755399441055744.0;  // 1.5 2^52

// e^a for a in [-700, 700] (below, e^-700): one rounding above the reduced
// argument's, the table's own rounding error added back.
__device__ __forceinline__ double exp_tab64(double a, const Gf64Tables &T) {
    if (a > 700.0) return exp(a);
    a = a < -700.0 ? -700.0 : a;
    const double t = fma(a, 0x1.71547652b82fep+6, kMagic);  // 64 / ln 2
    const int n = __double2loint(t);
    const double nf = t - kMagic;
    // ln 2 / 64 in a 36-bit piece (products with |n| < 2^17 exact) and the rest
    double r = fma(nf, -0x1.62e42fefap-7, a);
    r = fma(nf, -0x1.cf79abc9e3b3ap-46, r);
    double p = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    p = fma(p, r, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r * r, r);  // e^r - 1; r^7 / 5040 < 2^-64
    const double2 s = T.exp2[n & 63];
    const double v = s.x + fma(s.x, p, s.y);
    return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

// (sin a, cos a) for |a| < 2.5e4 (table as above), else sincos.
__device__ __forceinline__ void sincos_tab64(double a, const Gf64Tables &T, double &sn, double &cs) {
    if (!(fabs(a) < 2.5e4)) {
        sincos(a, &sn, &cs);
        return;
    }
    const double t = fma(a, 0x1.45f306dc9c883p+5, kMagic);  // 256 / (2 pi)
    const int n = __double2loint(t);
    const double nf = t - kMagic;
    // 2 pi / 256 in a 33-bit piece (products with |n| < 2^20 exact) and the rest
    double r = fma(nf, -0x1.921fb544p-6, a);
    r = fma(nf, -0x1.0b4611a626331p-40, r);
    const double q = r * r;
    double ps = fma(q, -1.0 / 5040.0, 1.0 / 120.0);
    ps = fma(ps, q, -1.0 / 6.0);
    const double s = fma(ps, r * q, r);  // sin r; r^9 / 9! < 2^-69 r
    double pc = fma(q, -1.0 / 720.0, 1.0 / 24.0);
    pc = fma(pc, q, -0.5) * q;           // cos r - 1; r^8 / 8! < 2^-65
    const double2 S = T.sn[n & 255], C = T.cs[n & 255];
    sn = S.x + fma(C.x, s, fma(S.x, pc, S.y));
    cs = C.x + fma(-S.x, s, fma(C.x, pc, C.y));
}

// The tables (host; k_gf.cu).
Gf64Tables make_gf64_tables();

}  // namespace gbs
