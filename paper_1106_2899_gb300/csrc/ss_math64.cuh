// ss_math64.cuh -- Box-Muller pairs in FP64 from the 24-bit lattice of the draws.
//
// The FP64 pipe of this GPU takes 64 cycles per warp instruction and SM
// partition, and general log, sqrt and sincos are about 85 FP64 instructions a
// pair.  The arguments here are integers of 24 bits, so range reduction is exact
// integer work and a table leaves short polynomials: 32 FP64 instructions a pair
// (9 logarithm, 7 square root, 14 sine and cosine, 2 products).
//
// The tables are computed at compile time in double-double arithmetic (Dekker's
// products, Knuth's sums) from the Taylor and artanh series, and rounded once.
#pragma once
#include <stdint.h>

namespace ssk {

// ------------------------------------------------ compile-time arithmetic ---
struct DD {
    double h, l;
};
constexpr DD dd_sum(double a, double b) {
    const double s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
constexpr DD dd_norm(double h, double l) {
    const double s = h + l;
    return {s, l - (s - h)};
}
constexpr DD dd_prod(double a, double b) {
    const double ca = 134217729.0 * a, cb = 134217729.0 * b;
    const double ah = ca - (ca - a), bh = cb - (cb - b), al = a - ah, bl = b - bh, p = a * b;
    return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD dd_add(DD a, DD b) {
    const DD s = dd_sum(a.h, b.h);
    return dd_norm(s.h, s.l + (a.l + b.l));
}
constexpr DD dd_mul(DD a, DD b) {
    const DD p = dd_prod(a.h, b.h);
    return dd_norm(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_div(DD a, double b) {
    const double q = a.h / b;
    const DD p = dd_prod(q, b);
    return dd_norm(q, ((a.h - p.h) - p.l + a.l) / b);
}
constexpr DD kPiDD = {3.14159265358979323846, 1.2246467991473532e-16};  // pi

// ---------------------------------------------------------------- tables ----
constexpr int kTrigBits = 10;  // sine and cosine at multiples of 2 pi / 1024
constexpr int kLogBits = 10;   // logarithm at 1024 centres of [1, 2)
// centres from this one on stand for half their value, so that every tabulated
// logarithm is small (between -ln sqrt 2 and ln sqrt 2)
constexpr int kLogHalf = 424;

struct TrigTable {
    double c[1 << kTrigBits], s[1 << kTrigBits];  // -cos, -sin of 2 pi j / 1024
};
constexpr TrigTable make_trig() {
    TrigTable t{};
    constexpr int n = 1 << kTrigBits, q = n / 8;
    // first eighth by Taylor series, the rest by symmetry
    for (int j = 0; j <= q; ++j) {
        const DD x = dd_mul(kPiDD, {2.0 * j / n, 0.0}), x2 = dd_mul(x, x);
        DD c = {1.0, 0.0}, s = x, tc = {1.0, 0.0}, ts = x;
        for (int k = 1; k <= 12; ++k) {
            tc = dd_div(dd_mul(tc, x2), -(2.0 * k - 1.0) * (2.0 * k));
            ts = dd_div(dd_mul(ts, x2), -(2.0 * k) * (2.0 * k + 1.0));
            c = dd_add(c, tc);
            s = dd_add(s, ts);
        }
        const double cv = c.h, sv = s.h;
        const int quarter = n / 4;
        for (int r = 0; r < 4; ++r) {  // angle + r quarter turns: (c, s) -> (-s, c)
            const double rc = r == 0 ? cv : (r == 1 ? -sv : (r == 2 ? -cv : sv));
            const double rs = r == 0 ? sv : (r == 1 ? cv : (r == 2 ? -sv : -cv));
            t.c[(j + r * quarter) % n] = -rc;
            t.s[(j + r * quarter) % n] = -rs;
            // the mirror image at a quarter turn less the angle: (c, s) -> (s, c)
            const double mc = r == 0 ? sv : (r == 1 ? -cv : (r == 2 ? -sv : cv));
            const double ms = r == 0 ? cv : (r == 1 ? sv : (r == 2 ? -cv : -sv));
            t.c[(quarter - j + r * quarter) % n] = -mc;
            t.s[(quarter - j + r * quarter) % n] = -ms;
        }
    }
    return t;
}

struct LogTable {
    double inv[1 << kLogBits];  // 1 / centre in 24 bits: its product with an argument is exact
    double l[1 << kLogBits];    // 2 ln inv (+ 2 ln 2 from kLogHalf on)
    double e[26];               // -2 (e - 24) ln 2
};
// ln x of x near 1 by 2 artanh((x - 1) / (x + 1))
constexpr DD dd_log_near1(double x) {
    const double num = x - 1.0, den = x + 1.0;
    const DD d = dd_sum(x, 1.0);
    const double q0 = num / den;
    const DD p = dd_prod(q0, d.h);
    const DD z = dd_norm(q0, ((num - p.h) - p.l - q0 * d.l) / den);
    const DD z2 = dd_mul(z, z);
    DD sum = {0.0, 0.0}, t = z;
    for (int k = 0; k < 24; ++k) {
        sum = dd_add(sum, dd_div(t, 2.0 * k + 1.0));
        t = dd_mul(t, z2);
    }
    return {2.0 * sum.h, 2.0 * sum.l};
}
constexpr LogTable make_log() {
    LogTable t{};
    constexpr int n = 1 << kLogBits;
    const DD ln2a = dd_log_near1(1.4142135623730951), ln2b = dd_log_near1(1.4142135623730949);
    // ln 2 = ln a + ln b + ln(2 / (a b)), the last factor 1 to a few 1e-16
    const DD ab = dd_prod(1.4142135623730951, 1.4142135623730949);
    const double rest = ((2.0 - ab.h) - ab.l) / 2.0;
    const DD ln2 = dd_add(dd_add(ln2a, ln2b), {rest, 0.0});
    for (int e = 0; e < 26; ++e) {
        const DD v = dd_mul(ln2, {-2.0 * (e - 24), 0.0});
        t.e[e] = v.h;
    }
    for (int i = 0; i < n; ++i) {
        // centre of [1 + i/n, 1 + (i+1)/n); exactly 1 and 2 in the outer intervals
        const double c = i == 0 ? 1.0 : (i == n - 1 ? 2.0 : 1.0 + (i + 0.5) / n);
        const double inv = (double)(float)(1.0 / c);
        t.inv[i] = inv;
        const double y = i >= kLogHalf ? 2.0 * inv : inv;  // 1 / the centre, or 1 / half the centre
        const DD ly = dd_log_near1(y);
        t.l[i] = 2.0 * ly.h;
    }
    return t;
}

__device__ constexpr TrigTable kTrig = make_trig();
__device__ constexpr LogTable kLog = make_log();

// -2 ln(n / 2^24) of n = 1 .. 2^24, and its square root.
__device__ __forceinline__ double radius_lattice(uint32_t n) {
    const int z = __clz((int)n), e = 31 - z;
    const uint32_t f = n << z << 1;  // fraction of n / 2^e
    const double m = __hiloint2double((int)(0x3ff00000u | (f >> 12)), (int)(f << 20));
    const int i = (int)(f >> (32 - kLogBits));
    const double r = fma(m, __ldg(&kLog.inv[i]), -1.0);  // exact, |r| < 2^-10
    const double base = __ldg(&kLog.e[e + (i >= kLogHalf)]) + __ldg(&kLog.l[i]);
    // -2 ln(1 + r) = -2 r + r^2 - 2/3 r^3 + 1/2 r^4 - 2/5 r^5
    const double q = fma(r, fma(r, fma(r, -0.4, 0.5), -2.0 / 3.0), 1.0);
    const double L = base + fma(-2.0, r, (r * r) * q);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(L));
    // one Newton step for sqrt and 1/(2 sqrt) together, then the residual
    const double t = L * y, h = 0.5 * y;
    const double d = fma(-t, h, 0.5);
    const double t1 = fma(t, d, t), h1 = fma(h, d, h);
    const double s = fma(fma(-t1, t1, L), h1, t1);
    return n == 1u << 24 ? 0.0 : s;
}

// Box-Muller pair from two words, as box_muller<double>: radius of n = hi24(wa) + 1,
// cosine and sine of the angle pi (2 k / 2^24 - 1), k = hi24(wb).
__device__ __forceinline__ void box_muller_lattice(uint32_t wa, uint32_t wb, double& n_cos, double& n_sin) {
    constexpr int S = 24 - kTrigBits;
    const double rad = radius_lattice((wa >> 8) + 1u);
    const uint32_t k = wb >> 8, j = (k + (1u << (S - 1))) >> S;
    // the remainder as a double (2^52 + 2^51 added and taken off), times 2 pi / 2^24
    const int lo = (int)k - (int)(j << S);
    const double x = (__hiloint2double(0x43380000 + (lo >> 31), lo) - 6755399441055744.0) * (6.28318530717958647693 / 16777216.0);
    const double c = __ldg(&kTrig.c[j & ((1 << kTrigBits) - 1)]), s = __ldg(&kTrig.s[j & ((1 << kTrigBits) - 1)]);
    const double x2 = x * x;
    const double sx = fma(x * x2, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x);
    const double cx = x2 * fma(x2, 1.0 / 24.0, -0.5);  // cos x - 1
    n_cos = rad * (c + fma(c, cx, -(s * sx)));
    n_sin = rad * (s + fma(s, cx, c * sx));
}

}  // namespace ssk
