// es_log64.cuh -- natural logarithm in FP64 for the node fields, by table (P. T. P. Tang, "Table-driven implementation
// of the logarithm function in IEEE floating-point arithmetic", ACM Trans. Math. Software 16(4), 1990).
//
// x = 2^e m with m in [0.707, 1.414); the leading 7 bits of the significand pick c ~ 1/m, r = c m - 1 is at most 2^-7, and
// ln x = e ln 2 - ln c + ln(1 + r) with the series of ln(1 + r) to r^8 (the next term is under 2^-59 of r).  ln 2 and the
// table's -ln c are sums of a multiple of 2^-42 and a small rest, so that e ln 2 - ln c is exact but for the rests, which
// join the series: one rounding of the result's size is left (a face takes the difference of two logarithms over as
// little as 1/50 of their size, so that their last bit is the flux's sixth).  Beside 1 (c = 1, e = 0) the result is the
// series alone, so small logarithms keep their relative accuracy.  12 instructions on the FP64 pipe (the exponent's double and
// the rests are put together on the integer and FP32 pipes) against about 27 of the library's log(): four logarithms at each of a
// tile's nodes, halo included, were 7% of the 2D stage's FP64 instructions.
// Checked against the logarithm in more than 64 bits on the GPU (es_selftest_log): within 1 ulp.
#pragma once
#include <cuda_runtime.h>

#include "es_bits.cuh"

namespace es {
namespace log64 {

// sums of two doubles (T. J. Dekker, Numer. Math. 18, 1971), for the constants
struct DD {
    double h, l;
};
constexpr DD renorm(double h, double l) {
    const double s = h + l;
    return {s, l - (s - h)};
}
constexpr DD add(DD a, DD b) {
    const double s = a.h + b.h, t = s - a.h;
    return renorm(s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l));
}
constexpr double head(double x) {                            // the leading 26 bits
    const double t = 134217729.0 * x;
    return t - (t - x);
}
constexpr DD mul(DD a, DD b) {
    const double p = a.h * b.h, ah = head(a.h), bh = head(b.h), al = a.h - ah, bl = b.h - bh;
    return renorm(p, (((ah * bh - p) + ah * bl + al * bh) + al * bl) + (a.h * b.l + a.l * b.h));
}
constexpr DD div(DD a, DD b) {
    const double q = a.h / b.h;
    const DD r = add(a, mul({-q, 0.0}, b));
    return renorm(q, (r.h + r.l) / b.h);
}
// ln c = 2 artanh f, f = (c - 1)/(c + 1), |f| <= 1/3: the series to f^81
constexpr DD ln(double c) {
    const DD f = div(add({c, 0.0}, {-1.0, 0.0}), add({c, 0.0}, {1.0, 0.0})), u = mul(f, f);
    DD s = {0.0, 0.0};
    for (int k = 40; k >= 0; --k) s = add(mul(s, u), div({1.0, 0.0}, {2.0 * k + 1.0, 0.0}));
    const DD y = mul(f, s);
    return {2.0 * y.h, 2.0 * y.l};
}
// the multiple of 2^-42 next to x (|x| < 512: beside 1536 an ulp is 2^-42), and the rest of a sum
constexpr double coarse(double x) { return (x + 1536.0) - 1536.0; }
constexpr double rest(DD x) { return (x.h - coarse(x.h)) + x.l; }

constexpr DD LN2 = ln(2.0);
constexpr double LN2_HI = coarse(LN2.h), LN2_LO = rest(LN2);

struct Table {
    double c[128], hi[128];              // c ~ 1/m and -ln c
    float lo[128];
};
constexpr Table make_table() {
    Table t{};
    for (int i = 0; i < 128; ++i) {
        const double m = (1.0 + (i + 0.5) / 128.0) * (i >= 53 ? 0.5 : 1.0);
        const bool one = i == 0 || i == 127;
        t.c[i] = one ? 1.0 : 1.0 / m;
        const DD y = one ? DD{0.0, 0.0} : ln(t.c[i]);
        t.hi[i] = -coarse(y.h);
        t.lo[i] = float(-rest(y));
    }
    return t;
}
static __device__ const Table TABLE = make_table();

static __device__ __noinline__ double other(double x) { return log(x); }

}  // namespace log64

// ln x for positive normal x; other arguments take log()
__device__ __forceinline__ double log_tab(double x) {
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return log64::other(x);
    const int i = (hi >> 13) & 127;
    const int up = i >= 53;                                       // m/2 in [0.707, 1)
    const int e = (hi >> 20) - 1023 + up;
    const double m = __hiloint2double((hi & 0xfffff) | (up ? 0x3fe00000 : 0x3ff00000), __double2loint(x));
    const double r = fma(m, __ldg(&log64::TABLE.c[i]), -1.0);
    double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(r, p, -1.0 / 6.0);
    p = fma(r, p, 1.0 / 5.0);
    p = fma(r, p, -1.0 / 4.0);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    const double de = bits::widen(float(e));
    const double base = fma(de, log64::LN2_HI, __ldg(&log64::TABLE.hi[i]));       // exact
    const double low = bits::widen(fmaf(float(e), float(log64::LN2_LO), __ldg(&log64::TABLE.lo[i])));   // (2^-43: FP32 will do)
    return base + (r + fma(r * r, p, low));
}

}  // namespace es
