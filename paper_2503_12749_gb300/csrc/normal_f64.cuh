// Two FP64 standard normals from four random words (Box-Muller on 53-bit
// uniforms), written for a chip whose FP64 pipe is narrow (2 lanes per SM and
// clock against 128 FP32 and integer lanes): a sampler that calls log, sqrt and
// sincospi is bound by about 90 FP64 instructions per pair.  Here the argument
// reductions are exact integer arithmetic, the polynomials of the reduced
// arguments double-float on the FP32 pipe (they are small corrections: 46 bits of
// them are beyond the 53rd bit of the result), and FP64 only adds the parts and
// polishes the root: 17 FP64 instructions per pair, samples included.  Measured
// (ms, with the samples' stores): N = 1000, 32768 trajectories as digit tiles
// 5.08 -> 1.13, N = 700, 20001 as FP32 tiles 2.60 -> 0.60, N = 16, 16384 0.116 ->
// 0.028.  Errors against 113-bit arithmetic, relative to the radius, 1e6 random
// pairs: root mean square 5.69e-17, largest 3.12e-16 (log, sqrt and sincospi: 5.93e-17,
// 3.12e-16).
//   -2 ln u:  u = m 2^E, t = round(4096 / centre of m's 1/512 interval),
//             r = m t / 4096 - 1 exactly (64-bit integers, |r| < 2^-9.6),
//             -2 ln u = -2 E ln 2 + 2 ln(t / 4096) - 2 ln(1 + r)
//             (table-driven logarithm, Tang, "Table-driven implementation of the
//             logarithm function in IEEE floating-point arithmetic", ACM TOMS
//             16, 1990); the table's last entry makes the constant exactly 0
//             next to u = 1, so the result keeps its relative accuracy there;
//   sin, cos of 2 pi v: v to the nearest 1/4096 of the circle by its leading
//             bits, the rest theta (|theta| <= 2^-10.3) by angle addition with a
//             quarter-wave table;
//   root:     FP32 root, its residual in FP32, one Newton step in FP64.
// u and v are the doubles RN(i + 1/2) 2^-53 of 53-bit integers i.
#pragma once

#include <cmath>
#include <cstdint>

#include "dfloat.cuh"

namespace gbs {

struct NormTab {
    struct Log {
        double hi;   // 2 ln(t / 4096), rounded to a multiple of 2^-40
        float lo;    // the rest
        uint32_t t;
    } lg[512];
    struct Exp {
        double hi;   // 2 e ln 2 with ln 2 cut at 2^-41: exact
        float lo, pad;
    } ex[56];
    struct Sin {
        double v;    // sin(2 pi j / 4096)
        float h, l;  // the same as a double-float
    } sn[1025];
    float sn_err[1028];  // sin(2 pi j / 4096) - sn[j].v
};

// Host: the tables, from long double (wider than double on both hosts).
inline void fill_norm_tab(NormTab &T) {
    const long double ln2x2 = 1.386294361119890618834464242916353136L;
    const long double cut = 1099511627776.0L;  // 2^40
    const long double hi1 = std::rint(ln2x2 * cut) / cut;
    for (int j = 0; j < 512; ++j) {
        const long double c = 1.0L + (j + 0.5L) / 512.0L;
        const long double t = j == 511 ? 2048.0L : std::rint(4096.0L / c);
        const long double v = j == 511 ? -ln2x2 : 2.0L * std::log(t / 4096.0L);
        const long double hi = std::rint(v * cut) / cut;
        T.lg[j].t = (uint32_t)t;
        T.lg[j].hi = (double)hi;
        T.lg[j].lo = (float)(v - hi);
    }
    for (int e = 0; e < 56; ++e) {
        T.ex[e].hi = (double)(e * hi1);
        T.ex[e].lo = (float)(e * (ln2x2 - hi1));
        T.ex[e].pad = 0.0f;
    }
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int j = 1025; j < 1028; ++j) T.sn_err[j] = 0.0f;
    for (int j = 0; j <= 1024; ++j) {
        const long double v = j <= 512 ? std::sin(pi * j / 2048.0L) : std::cos(pi * (1024 - j) / 2048.0L);
        T.sn[j].v = (double)v;
        T.sn[j].h = (float)v;
        T.sn[j].l = (float)(v - (long double)T.sn[j].h);
        T.sn_err[j] = (float)(v - (long double)T.sn[j].v);
    }
}

namespace nrm {

// float -> double on the integer pipe (zero and normal numbers).
__device__ __forceinline__ double f2d(float x) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t hi = ((b & 0x7fffffffu) >> 3) + 0x38000000u;
    return (b << 1) ? __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29)) : 0.0;
}

// A positive normal double in float's range as a double-float (53 -> 24 + 24
// bits), on the integer pipe.
__device__ __forceinline__ df d2df(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t b = ((hi - 0x38000000u) << 3) | (lo >> 29);  // truncated
    // the low 29 bits, in units of 2^-52 of the leading bit's weight
    const float unit = __uint_as_float((b & 0x7f800000u) - (52u << 23));
    return {__uint_as_float(b), (float)(int)(lo & 0x1fffffffu) * unit};
}

// The 54-bit integer 2 i + 1 of the words' 53-bit integer i, or where the double
// i + 1/2 rounds (i >= 2^52) twice its rounding to even.
__device__ __forceinline__ uint64_t uniform54(uint32_t a, uint32_t b) {
    const uint64_t i = ((uint64_t)(a >> 5) << 26) | (b >> 6);
    return (i >> 52) ? 2 * (i + (i & 1u)) : 2 * i + 1;
}

__device__ __forceinline__ void normals(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        const NormTab &T, double &w1, double &w2) {
    // ---- W = -2 ln u, u = v 2^-54 = (mant 2^-52) 2^E
    const uint64_t v = uniform54(c0, c1);
    const int lz = __clzll((long long)v);  // 9 (u = 1) .. 63
    const uint64_t mant = lz >= 11 ? v << (lz - 11) : v >> (11 - lz);  // exact
    const int nE = lz - 9;                 // -E
    const NormTab::Log g = T.lg[(mant >> 43) & 511u];
    const NormTab::Exp k = T.ex[nE];
    const int64_t ri = (int64_t)(mant * g.t);  // r 2^64 (mod 2^64: the 1 drops out)
    const uint64_t ra = (uint64_t)(ri < 0 ? -ri : ri);
    const int rz = __clzll((long long)ra);     // 64 when r = 0
    const uint64_t rn = ra << (rz & 63);       // leading bit at 63
    const uint32_t sgn = ri < 0 ? 0x80000000u : 0u;
    // 2 r as a double (truncated to 53 bits), r as a double-float
    const uint64_t rb = ((uint64_t)(1023 - rz) << 52) + ((rn >> 11) & 0xfffffffffffffull);
    double r2d = __longlong_as_double((long long)(rb | ((uint64_t)sgn << 32)));
    const float sc = __uint_as_float(((uint32_t)(127 - 24 - rz) << 23) | sgn);  // 2^-(rz + 24)
    df r = {(float)(int)(uint32_t)(rn >> 40) * sc,
            (float)(int)((uint32_t)(rn >> 16) & 0xffffffu) * (sc * 0x1p-24f)};
    if (ra == 0) {
        r2d = 0.0;
        r = {0.0f, 0.0f};
    }
    // 2 (ln(1 + r) - r) = r^2 (-1 + 2 r / 3 - r^2 / 2 + 2 r^3 / 5 - r^4 / 3)
    const float x = r.hi;
    const float p = x * x * fmaf(x, fmaf(x, -1.0f / 3.0f, 0.4f), -0.5f);
    const df two3 = {0x1.555556p-1f, -0x1.555556p-26f};
    df q = df_add_f(df_mul(r, two3), p);
    q = df_add_f(q, -1.0f);
    const df corr = df_mul(df_mul(r, r), q);
    const df sm = df_add_f(df_neg(corr), g.lo + k.lo);
    // the small parts first (their roundings lie below 2^-62): one rounding of W
    const double W = (k.hi + g.hi) + ((f2d(sm.hi) + f2d(sm.lo)) - r2d);
    // ---- rho = sqrt(W)
    const df wd = d2df(W);
    const float y = rsqrtf(wd.hi);
    const float s0 = wd.hi * y;
    const float c = (fmaf(-s0, s0, wd.hi) + wd.lo) * (0.5f * y);
    double rho = f2d(s0) + f2d(c);
    rho = fma(fma(-rho, rho, W), f2d(0.5f * y), rho);
    if (nE == 0) rho = 0.0;  // u = 1
    // ---- sin, cos of 2 pi u2
    const uint64_t a = uniform54(c2, c3);
    const uint32_t j = (uint32_t)((a + (1ull << 41)) >> 42);
    const int64_t rem = (int64_t)(a - ((uint64_t)j << 42));
    const df xr = df_fast_two_sum((float)(int)(rem >> 18) * 262144.0f,
                                  (float)(int)((uint32_t)rem & 0x3ffffu));
    const df two_pi = {0x1.921fb6p-52f, -0x1.777a5cp-77f};  // 2 pi 2^-54
    const df th = df_mul(xr, two_pi);
    const float t2 = th.hi * th.hi;
    const float e2 = fmaf(2.0f * th.hi, th.lo, fmaf(th.hi, th.hi, -t2));
    const df s = df_fast_two_sum(th.hi, fmaf(th.hi * t2, fmaf(t2, 1.0f / 120.0f, -1.0f / 6.0f), th.lo));
    const df cm = df_fast_two_sum(-0.5f * t2, fmaf(t2 * t2, 1.0f / 24.0f, -0.5f * e2));
    const uint32_t js = j & 1023u, jc = 1024u - js;
    const NormTab::Sin S = T.sn[js], C = T.sn[jc];
    const df Sf = {S.h, S.l}, Cf = {C.h, C.l};
    const df bs = df_add(df_mul(Cf, s), df_mul(Sf, cm));
    const df bc = df_sub(df_mul(Cf, cm), df_mul(Sf, s));
    const double sb = S.v + (f2d(bs.hi) + f2d(bs.lo + T.sn_err[js]));
    const double cb = C.v + (f2d(bc.hi) + f2d(bc.lo + T.sn_err[jc]));
    // quadrant j / 1024: (sin, cos) = (s, c), (c, -s), (-s, -c), (-c, s)
    const bool odd = (j & 1024u) != 0;
    const double sv = odd ? cb : sb, cv = odd ? sb : cb;
    const uint32_t fs = (j & 2048u) << 20, fc = ((j + 1024u) & 2048u) << 20;
    w1 = rho * __hiloint2double(__double2hiint(cv) ^ (int)fc, __double2loint(cv));
    w2 = rho * __hiloint2double(__double2hiint(sv) ^ (int)fs, __double2loint(sv));
}

}  // namespace nrm
}  // namespace gbs
