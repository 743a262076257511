// es_device.cuh -- device-side physics of the ES van der Waals scheme (sm_103a).
//
// Everything here runs inside the library's own kernels.  Formulas follow the
// paper's sections noted at each function, written in general van der Waals
// units (a, b, R, cv): p = rho R T/(1 - b rho) - a rho^2, e = cv T - a rho.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "es_vdw.h"

namespace es {

// ----------------------------------------------------------------- constants
struct Gas {
    double a, b, R, cv, delta;   // delta = R / cv
    double iR, idelta, icv;      // 1/R, 1/delta, 1/cv (set with the others)
};

inline void gas_reciprocals(Gas& g) {
    g.iR = 1.0 / g.R;
    g.idelta = 1.0 / g.delta;
    g.icv = 1.0 / g.cv;
}

// Reciprocal, quotient and reciprocal square root for finite, normal, positive arguments (the reciprocal also for
// negative ones): all the kernels' divisors are positive physical quantities or sums of them.  The FP64 pipe
// issues at 1/64 of the FP32 rate and bounds every kernel that uses these, so each is counted in its
// instructions.  The hardware's approximations have relative errors below 2^-22; one third-order step
// y <- y (1 + e + e^2), e = 1 - b y (Householder's iteration of order two for 1/y - b) leaves e^3 < 2^-65 in three
// instructions, where two Newton steps take four.  The quotient needs only a Newton-refined reciprocal
// (e^2 < 2^-44): its correction q <- q + y (a - b q) squares that error again (Markstein, IBM J. Res. Develop.
// 34(1), 1990), five instructions instead of seven.  Checked against IEEE division (es_selftest_division).
__device__ __forceinline__ double rcp_nr(double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = fma(-b, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double div_nr(double a, double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    y = fma(y, fma(-b, y, 1.0), y);
    const double q = a * y;
    return fma(fma(-b, q, a), y, q);
}
// 1/sqrt(x): y <- y (1 + e/2 + 3 e^2/8), e = 1 - x y^2, the same order (five instructions; sqrt(x) = x rsqrt_nr(x)
// is one more, against about ten of the library's correctly rounded square root)
__device__ __forceinline__ double rsqrt_nr(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Sixth-order EC combination weights alpha_{3,m}, m = 1, 2, 3 (Sec. 3.1:
// sum m alpha = 1, sum m^3 alpha = sum m^5 alpha = 0).
__device__ __forceinline__ double ec_alpha(int m) {
    return m == 1 ? 1.5 : (m == 2 ? -0.3 : 1.0 / 30.0);
}

// --------------------------------------------------------- MR-WENO5 (Sec. 3.3)
// Multi-resolution WENO on the nested stencils {0}, {-1,0,1}, {-2..2} (Zhu & Shu
// framework) reconstructing the value at x_{i+1/2} from point values treated as
// cell averages.  g1, g2, g3 = linear weights of the 1-, 3-, 5-point stencils.
struct Weno {
    double g1, g2, g3;     // linear weights
    double g12, ig22;      // g1/(g1+g2), (g1+g2)/g2
    double ig3;            // 1/g3
    double eps;
    double sign_tol;       // relative round-off size under which a plain jump counts as zero
    // derived (weno_coefficients): the candidates of the FP64 reconstruction as coefficients of the data's
    // differences, and the linear weights over g3
    double h1, h2;         // g1/g3, g2/g3
    double q2;             // (g2/g3) p2 - (g2/g3) w0 = q2 (d_- + 2 d_+)
    double q3[4];          // p3 - w0 = q3 . (the four differences of the stencil)
    double eps4;           // eps/4
};

// p2 = (q_2 - g12 w0)/ig22^-1 and p3 = (q_3 - g1 w0 - g2 p2)/g3 with the 3- and 5-point interface values
// q_2 - w0 = (d1 + 2 d2)/6 and q_3 - w0 = (-2 d0 + 11 d1 + 24 d2 - 3 d3)/60
inline void weno_coefficients(Weno& w) {
    w.h1 = w.g1 * w.ig3;
    w.h2 = w.g2 * w.ig3;
    w.q2 = w.h2 * w.ig22 / 6.0;
    const double p2 = w.g2 * w.ig22 / 6.0;
    w.q3[0] = -2.0 / 60.0 * w.ig3;
    w.q3[1] = (11.0 / 60.0 - p2) * w.ig3;
    w.q3[2] = (24.0 / 60.0 - 2.0 * p2) * w.ig3;
    w.q3[3] = -3.0 / 60.0 * w.ig3;
    w.eps4 = 0.25 * w.eps;
}

// --------------------------------------------------------- index helpers
__device__ __forceinline__ int wrap_index(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

// Decomposition of a possibly-ghost index along one direction into at most two
// interior indices with weights and a period count:
//   periodic: value(i) = value(i mod n) + q * period
//   outflow : value(i) = 2 value(boundary) - value(mirror)   (odd reflection)
struct GhostTerms {
    int idx[2];
    double w[2];
    int nterm;
    int q;         // period count (periodic only)
};

// Walls and symmetry planes: the end of a direction that mirrors the mesh and the state.
__device__ __forceinline__ bool end_mirrored(int bc, bool lo) {
    return bc == ES_BC_REFLECT || (bc == ES_BC_SYMMETRY_LO && lo);
}

// `tangential`: a coordinate or mesh-velocity component along the boundary plane, which a
// mirroring end mirrors (value of the mirror node) instead of reflecting oddly.
__device__ __forceinline__ GhostTerms ghost_terms(int i, int n, int bc, bool tangential = false) {
    GhostTerms g;
    g.q = 0;
    if (i >= 0 && i < n) {
        g.idx[0] = i; g.w[0] = 1.0; g.nterm = 1;
    } else if (bc == ES_BC_PERIODIC) {
        int r = wrap_index(i, n);
        g.q = (i - r) / n;
        g.idx[0] = r; g.w[0] = 1.0; g.nterm = 1;
    } else {
        // the mirror index is clamped to the mesh: nodes that far out only
        // occur in the unused tail of a ragged tile and must stay in bounds
        int m = i < 0 ? -i : 2 * (n - 1) - i;
        m = m < 0 ? 0 : (m > n - 1 ? n - 1 : m);
        if (tangential && end_mirrored(bc, i < 0)) {
            g.idx[0] = m; g.w[0] = 1.0; g.nterm = 1;
        } else {
            g.idx[0] = i < 0 ? 0 : n - 1; g.w[0] = 2.0; g.idx[1] = m; g.w[1] = -1.0; g.nterm = 2;
        }
    }
    return g;
}

// State index for ghosts: periodic wrap, outflow copy of the boundary node, mirror node at a
// wall or symmetry end (the caller negates the normal momentum there).
__device__ __forceinline__ int state_index(int i, int n, int bc) {
    if (i >= 0 && i < n) return i;
    if (bc == ES_BC_PERIODIC) return wrap_index(i, n);
    if (end_mirrored(bc, i < 0)) {
        int m = i < 0 ? -i : 2 * (n - 1) - i;
        return m < 0 ? 0 : (m > n - 1 ? n - 1 : m);
    }
    return i < 0 ? 0 : n - 1;
}

// ------------------------------------------------------------- reductions
// Atomic max / min of non-negative doubles through their ordered bit patterns.
__device__ __forceinline__ void atomic_max_pos(unsigned long long* addr, double v) {
    if (!(v >= 0.0)) v = __longlong_as_double(0x7ff0000000000000ULL);   // NaN -> +inf
    atomicMax(addr, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void atomic_min_pos(unsigned long long* addr, double v) {
    if (!(v >= 0.0)) v = 0.0;
    atomicMin(addr, (unsigned long long)__double_as_longlong(v));
}

// Device error word: first error code wins; the node index is kept with it.
struct DevStatus {
    int code;
    int index;
};

__device__ __forceinline__ void raise_error(DevStatus* st, int code, int index) {
    if (atomicCAS(&st->code, 0, code) == 0) st->index = index;
}

}  // namespace es
