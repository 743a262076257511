// es_log64.cuh -- natural logarithm in FP64 for the node fields, by table (P. T. P. Tang, "Table-driven implementation
// of the logarithm function in IEEE floating-point arithmetic", ACM Trans. Math. Software 16(4), 1990).
//
// x = 2^e m with m in [0.71, 1.42); the leading 7 bits of the significand pick c ~ 1/m, r = c m - 1 is at most 2^-7, and
// ln x = e ln 2 - ln c + ln(1 + r) with the series of ln(1 + r) to r^8 (the next term is under 2^-59 of r).  Beside 1
// (c = 1, e = 0) the result is the series alone, so small logarithms keep their relative accuracy.  11 instructions on
// the FP64 pipe (the exponent's double is put together on the integer and FP32 pipes) against about 27 of the library's
// log(): four logarithms at each of a tile's nodes, halo included, were 7% of the 2D stage's FP64 instructions.
// Checked against log() on the GPU (es_selftest_log).
#pragma once
#include <cuda_runtime.h>

#include "es_bits.cuh"

namespace es {

struct LogTable {
    double c[128], lnc[128];             // c ~ 1/m and -ln c
};

constexpr double log_series(double c) {  // ln c = 2 artanh((c - 1)/(c + 1)), |.| <= 0.18
    const double f = (c - 1.0) / (c + 1.0), u = f * f;
    double s = 0.0;
    for (int k = 24; k >= 0; --k) s = s * u + 1.0 / (2 * k + 1);
    return 2.0 * f * s;
}
constexpr LogTable make_log_table() {
    LogTable t{};
    for (int i = 0; i < 128; ++i) {
        const double m = (1.0 + (i + 0.5) / 128.0) * (i >= 53 ? 0.5 : 1.0);
        t.c[i] = i == 0 || i == 127 ? 1.0 : 1.0 / m;
        t.lnc[i] = i == 0 || i == 127 ? 0.0 : -log_series(t.c[i]);
    }
    return t;
}
static __device__ const LogTable LOG_TABLE = make_log_table();

static __device__ __noinline__ double log_other(double x) { return log(x); }
// ln x for positive normal x; other arguments take log()
__device__ __forceinline__ double log_tab(double x) {
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return log_other(x);
    const int i = (hi >> 13) & 127;
    const int up = i >= 53;                                       // m/2 in [0.71, 1)
    const int e = (hi >> 20) - 1023 + up;
    const double m = __hiloint2double((hi & 0xfffff) | (up ? 0x3fe00000 : 0x3ff00000), __double2loint(x));
    const double r = fma(m, __ldg(&LOG_TABLE.c[i]), -1.0);
    double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(r, p, -1.0 / 6.0);
    p = fma(r, p, 1.0 / 5.0);
    p = fma(r, p, -1.0 / 4.0);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    const double base = fma(bits::widen(float(e)), 0.69314718055994530942, __ldg(&LOG_TABLE.lnc[i]));
    return base + fma(r * r, p, r);
}

}  // namespace es
