// es_flux64.cuh -- node fields, two-point fluxes and face dissipation of the FP64 operator, in D = 1, 2, 3 dimensions.
//
// The FP64 pipe bounds the kernels that use these (two lanes per clock on an SM: one warp instruction takes as long
// as 64 issue slots), so what counts is the number of FP64 instructions, additions and multiplications alike, and
// everything that the integer and FP32 pipes can do is free beside them.  Three things follow:
//   * means are sums: a node stores HALF of every field that a face reads as the arithmetic mean of its two nodes
//     (halving is exact), so {a} = a_l/2 + a_r/2 is one addition instead of an addition and a multiplication;
//   * quantities are formed in the products that the formulas need, not in the ones the paper prints (the ratio
//     {a}/{a}^ln instead of 1/{a}^ln, p/rho instead of p, A = J xi_t {rho} + n . {rho v} once for both of its uses);
//   * comparisons against constants, sign tests and minima of non-negative values use the bits of the numbers, and
//     the sign switch's round-off test is decided in FP32 bounds wherever those are clear;
//   * the logarithms come from a table (es_log64.cuh), and the differences of the entropy variables that every face's
//     reconstruction starts from are formed once per pair of neighbours.
// Every product that feeds an addition is written as fma() or __dmul_rn(), so that the compiler has no choice of which
// product to fuse and the tile shapes of a kernel give the same bits.  (The 1D line shared by four warps, es_stage.cu, adds
// a face's waves in another order than face_dissipation.)
// Instructions on the FP64 pipe at a 2D pair: 140 before this form, 78 now; at a 2D face: about 1000 and 600.
#pragma once
#include <cuda_runtime.h>

#include "es_device.cuh"
#include "es_log64.cuh"

namespace es {
namespace flux64 {

// node fields: planes of a tile's shared memory (1D/2D) or of global memory (3D)
template <int D>
struct Slots {
    enum {
        RHO,        // rho/2
        T,          // T/2
        OM,         // (1 - b rho)/2
        IOM,        // 1/(1 - b rho)
        G,          // g/2, g = R/(1 - b rho) - a rho/T
        ART,        // a rho/(2T)
        E0,         // |v|^2/(4T) + a rho/T
        RP,         // rho/(2p)
        W0, WE,     // half of the entropy variables V_1 and V_{D+2} = -1/T
        LNR, LNOM, LNT, LNRP,   // logarithms of rho, 1 - b rho, T and rho/p
        V,          // v_k/2
        VT = V + D, // v_k/(2T), half of the entropy variables between V_1 and V_{D+2}
        RV = VT + D,// rho v_k/2
        COUNT = RV + D
    };
};

// ------------------------------------------------------------ bits
// x > 0 (also +infinity; false for NaN), without a comparison on the FP64 pipe
__device__ __forceinline__ bool positive(double x) {
    return (unsigned long long)(__double_as_longlong(x) - 1LL) < 0x7ff0000000000000ULL;
}
// x/2 exactly, by its exponent (zeros, subnormals and values next to them by multiplication)
__device__ __forceinline__ double half(double x) {
    const int hi = __double2hiint(x);
    const int e = hi & 0x7ff00000;
    if (e > 0x00100000 && e != 0x7ff00000) return __hiloint2double(hi - 0x00100000, __double2loint(x));
    return (hi << 1) == 0 && __double2loint(x) == 0 ? x : 0.5 * x;
}
// the smaller of two non-negative numbers, by their ordered bits
__device__ __forceinline__ double min_pos(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
}
// |x| truncated to a float (20 significand bits): below |x| by at most 2^-20 |x|; 0 below the floats' range
__device__ __forceinline__ float abs_f(double x) {
    const int hi = __double2hiint(x) & 0x7fffffff;
    const int v = hi < 0x38100000 ? 0 : (hi >= 0x47f00000 ? 0x7f800000 : (hi - 0x38000000) << 3);
    return __int_as_float(v);
}

// ------------------------------------------------------------ logarithmic mean
// With f = (a_l - a_r)/(a_l + a_r) and u = f^2: {a}/{a}^ln = artanh(f)/f = 1 + u/3 + u^2/5 + u^3/7 + ... and its
// reciprocal 1 - u/3 - 4 u^2/45 - 44 u^3/945 - ...  Below |f| = 1e-2 (tested on the leading bits of f) the next terms,
// u^4/9 and 0.03 u^4, are under 2^-56; above it [[ln a]] = 2 artanh(f) from the nodes' logarithms keeps its digits.
// (Logarithms formed only where a face needs them cost the nodes nothing, but the tiles on a shock then took 40% longer
// than the others, and 200^2 nodes are one wave of tiles: 202 -> 260 us per stage.)
constexpr int F_SERIES = 0x3f847ae1;                                  // 1e-2
// {a}/{a}^ln
__device__ __forceinline__ double mean_over_logmean(double f, double lnl, double lnr) {
    if ((__double2hiint(f) & 0x7fffffff) < F_SERIES) {
        const double u = f * f;
        return fma(u, fma(u, fma(u, 1.0 / 7.0, 1.0 / 5.0), 1.0 / 3.0), 1.0);
    }
    return div_nr(lnl - lnr, f + f);
}
// {a}^ln/{a}
__device__ __forceinline__ double logmean_over_mean(double f, double lnl, double lnr) {
    if ((__double2hiint(f) & 0x7fffffff) < F_SERIES) {
        const double u = f * f;
        return fma(u, fma(u, fma(u, -44.0 / 945.0, -4.0 / 45.0), -1.0 / 3.0), 1.0);
    }
    return div_nr(f + f, lnl - lnr);
}

// ------------------------------------------------------------ node
// Fields of a node from its density, momentum and energy; st(slot, value) stores them.  `parts` (a constant, or the same
// for a warp): which of them, so that several warps can share a node's logarithms; PLAIN leaves V_1/2 without its
// logarithms in W0 (v1_logs adds them).  false: inadmissible
// (rho > 0, 1 - b rho > 0, T > 0, p > 0; the condition R T - 2 a rho (1 - b rho)^2 > 0 enters at the faces).
enum { LOG_RHO = 1, LOG_OM = 2, LOG_T = 4, LOG_RP = 8, PLAIN = 16, ALL = 32 };
__device__ __forceinline__ double v1_logs(double w0, double lnr, double lnom, double lnT, const Gas& G) {
    return fma(-0.5 * G.cv, lnT, fma(-0.5 * G.R, lnom - lnr, w0));
}
template <int D, class ST>
__device__ __forceinline__ bool node_fields(const double* JU, double J, const Gas& G, ST st, int parts = ALL) {
    using SL = Slots<D>;
    const double iJ = rcp_nr(J);
    const double ihJ = half(iJ);
    const double rho = JU[0] * iJ;
    const double r = half(rho);
    const double irho = rcp_nr(rho);
    double m[D], v[D], hke = 0.0;                          // halves; |v|^2/4
#pragma unroll
    for (int k = 0; k < D; ++k) {
        m[k] = JU[1 + k] * ihJ;
        v[k] = m[k] * irho;
        hke = k == 0 ? v[k] * v[k] : fma(v[k], v[k], hke);
    }
    const double E = JU[D + 1] * iJ;
    // T = (E/rho - |v|^2/2 + a rho)/cv
    const double T = fma(-2.0, hke, fma(E, irho, G.a * rho)) * G.icv;
    const double om = fma(-G.b, rho, 1.0);
    const double iom = rcp_nr(om);
    const double iT = rcp_nr(T);
    const double hRiom = (0.5 * G.R) * iom;
    const double art = __dmul_rn(G.a * r, iT);             // a rho/(2T)
    const double E0 = fma(2.0, art, hke * iT);
    const double prho = fma(2.0 * hRiom, T, -(G.a * rho));  // p/rho
    double lnr = 0.0, lnT = 0.0, lnom = 0.0;
    if (parts & (LOG_RHO | ALL)) st(SL::LNR, lnr = log_tab(rho));
    if (parts & (LOG_OM | ALL)) st(SL::LNOM, lnom = G.b > 0.0 ? log_tab(om) : 0.0);
    if (parts & (LOG_T | ALL)) st(SL::LNT, lnT = log_tab(T));
    if (parts & (LOG_RP | ALL)) st(SL::LNRP, -log_tab(prho));
    if (parts & (PLAIN | ALL)) {
        st(SL::RHO, r);
        st(SL::T, half(T));
        st(SL::OM, half(om));
        st(SL::IOM, iom);
        st(SL::G, hRiom - art);
        st(SL::ART, art);
        st(SL::E0, E0);
        st(SL::RP, half(rcp_nr(prho)));
        // V_1 = (e + p/rho)/T - s - |v|^2/(2T) with s = cv ln T + R ln((1 - b rho)/rho)
        const double w0 = fma(0.5, G.cv, hRiom) - E0;
        st(SL::W0, parts & ALL ? v1_logs(w0, lnr, lnom, lnT, G) : w0);
        st(SL::WE, -half(iT));
#pragma unroll
        for (int k = 0; k < D; ++k) {
            st(SL::V + k, v[k]);
            st(SL::VT + k, v[k] * iT);
            st(SL::RV + k, m[k]);
        }
    }
    return positive(rho) && positive(om) && positive(T) && positive(prho);
}

// ------------------------------------------------------------ two-point flux
// EC flux of Sec. 3.1 contracted with the means n, xt of the metrics and J xi_t:
//   F = {J xi_t} U~ + sum_j {J xi_k/x_j} F~_j
// with U~, F~_j from the explicit solution of eq. linear_U / linear_F in general units (D U~_1 = {rho}(Rb/Pi - a/{T})
// + {g}, U~_{1+m} = {v_m} U~_1, ...).  out[D + 1] is a QUARTER of the energy component (Tl Tr from the halved
// temperatures; the combination's weights carry the 4).
template <int D>
__device__ __forceinline__ void pair_flux(const double* S, int NB, int l, int r, const double* n, double xt,
                                          const Gas& G, double* out) {
    using SL = Slots<D>;
    auto L = [&](int f) { return S[f * NB + l]; };
    auto R = [&](int f) { return S[f * NB + r]; };
    auto mean = [&](int f) { return L(f) + R(f); };
    const double rl = L(SL::RHO), rr = R(SL::RHO), Tl = L(SL::T), Tr = R(SL::T);
    const double rm = rl + rr, Tm = Tl + Tr;
    const double ir = rcp_nr(rm), iT = rcp_nr(Tm);         // 1/{rho}, 1/{T}
    const double Fr = mean_over_logmean((rl - rr) * ir, L(SL::LNR), R(SL::LNR));
    const double FT = mean_over_logmean((Tl - Tr) * iT, L(SL::LNT), R(SL::LNT));
    const double aiT = __dmul_rn(G.a, iT);
    const double coef = fma(G.R * G.b, L(SL::IOM) * R(SL::IOM), -aiT);
    double D1 = fma(G.R, Fr * ir, coef) - aiT;
    if (G.b > 0.0) {
        const double ol = L(SL::OM), orr = R(SL::OM);
        const double io = rcp_nr(ol + orr);
        const double Fo = mean_over_logmean((ol - orr) * io, L(SL::LNOM), R(SL::LNOM));
        D1 = fma(G.R * G.b, Fo * io, D1);
    }
    const double iD = rcp_nr(D1);
    const double g = mean(SL::G);
    double vm[D];
    double A = xt * rm, B = xt, nv = 0.0;                  // J xi_t {rho} + n . {rho v}; J xi_t + n . {v}; n . {v/T}
    double sv = fma(G.cv, FT, -mean(SL::E0));              // {v/T} . {v} - B0, B0 = {|v|^2/T}/2 - cv {T}/{T}^ln + 2a {rho/T}
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const double vT = mean(SL::VT + k);
        vm[k] = mean(SL::V + k);
        A = fma(n[k], mean(SL::RV + k), A);
        B = fma(n[k], vm[k], B);
        nv = k == 0 ? n[k] * vT : fma(n[k], vT, nv);
        sv = fma(vT, vm[k], sv);
    }
    const double Q = fma(coef, A, g * B) * iD;             // the density component
    const double P = rm * Tm * g;
    out[0] = Q;
#pragma unroll
    for (int k = 0; k < D; ++k) out[1 + k] = fma(vm[k], Q, n[k] * P);
    // 1/{1/T} = Tl Tr/{T}
    out[D + 1] = fma(mean(SL::ART), A, fma(sv, Q, P * nv)) * (Tl * Tr * iT);
}

// Half of the entropy variables' jump V_r - V_l
template <int D>
__device__ __forceinline__ void entropy_jump(const double* S, int NB, int l, int r, double* dV) {
    using SL = Slots<D>;
#pragma unroll
    for (int m = 0; m < D + 2; ++m) {
        const int f = m == 0 ? SL::W0 : (m == D + 1 ? SL::WE : SL::VT + m - 1);
        dV[m] = S[f * NB + r] - S[f * NB + l];
    }
}

// ------------------------------------------------------------ MR-WENO5 (Sec. 3.3)
// One side's reconstruction as numerator and denominator of (w_{i+1/2} - w_i)/2: d0..d3 are HALF the differences of the
// five stencil values w_{-2} .. w_2 in order, k1 = min(d1^2, d2^2) + eps/4 the first indicator.  Everything is formed from
// differences (the indicators ignore a constant added to the data).  With S = d1 + d2, Dd = d2 - d1 (first and second
// difference of the 3-point stencil), G = (d0 + d3) - S and E = (d3 - d0) - 3 Dd (the odd and even parts that only
// the 5-point stencil sees): beta_2 = 13/12 Dd^2 + S^2/4 and the quartic's integrals collect to
//   beta_3 - beta_2 = E (4405/4032 E - 11/60 Dd) + G (89/320 G - S/12),
// the difference that tau needs, without cancellation.  Halved differences make every indicator a quarter, so that
// with k = (beta + eps)/4 and t = |k_3 - k_1| + |k_3 - k_2| the weights g (1 + tau/(beta + eps)) are g (1 + t^2/k); over
// the common denominator k1 k2 k3 they are g (k1 k2 k3 + t^2 k k'), taken over g_3.
__device__ __forceinline__ void weno_side(double d0, double d1, double d2, double d3, double k1, const Weno& c,
                                          double& num, double& den) {
    const double s = d1 + d2, dd = d2 - d1;
    const double g = (d0 + d3) - s;
    const double e = fma(-3.0, dd, d3 - d0);
    const double k2 = fma(0.25 * s, s, fma((13.0 / 12.0) * dd, dd, c.eps4));
    const double q = fma(e, fma(4405.0 / 4032.0, e, (-11.0 / 60.0) * dd), g * fma(89.0 / 320.0, g, (-1.0 / 12.0) * s));
    const double k3 = k2 + q;
    const double t = fabs(k3 - k1) + fabs(q);
    const double tt = t * t;
    const double k12 = k1 * k2, k123 = k12 * k3;
    const double y1 = fma(tt, k2 * k3, k123);
    const double y2 = fma(tt, k1 * k3, k123);
    const double y3 = fma(tt, k12, k123);
    const double p2 = c.q2 * fma(2.0, d2, d1);
    const double p3 = fma(c.q3[0], d0, fma(c.q3[1], d1, fma(c.q3[2], d2, c.q3[3] * d3)));
    num = fma(y2, p2, y3 * p3);
    den = fma(c.h1, y1, fma(c.h2, y2, y3));
}

// (w^+ - w^-)/2 at the face between the third and fourth of six values, from half their five differences
__device__ __forceinline__ double weno_jump(const double* d, const Weno& c) {
    const double s1 = fma(d[1], d[1], c.eps4), s2 = fma(d[2], d[2], c.eps4), s3 = fma(d[3], d[3], c.eps4);
    double nm, dm, np, dp;
    weno_side(d[0], d[1], d[2], d[3], min_pos(s1, s2), c, nm, dm);
    weno_side(d[4], d[3], d[2], d[1], min_pos(s2, s3), c, np, dp);   // mirrored: the numerator changes sign
    return fma(-np, rcp_nr(dp), fma(-nm, rcp_nr(dm), d[2]));
}

// ------------------------------------------------------------ frame of a face
// rows of the rotation T's momentum block: the normal n/L and the tangents (Sec. 3.3); 3D: theta = atan2(n_2, n_1)
// (0 when |(n_1, n_2)| <= 1e-12 |n|, the rounding of metrics that vanish exactly), phi = atan2(n_3, |(n_1, n_2)|)
template <int D>
struct Frame {
    double L;
    double e[D][D];
};
template <int D>
__device__ __forceinline__ Frame<D> face_frame(const double* n) {
    Frame<D> f;
    if constexpr (D == 1) {
        f.L = fabs(n[0]);
        f.e[0][0] = __double2hiint(n[0]) < 0 ? -1.0 : 1.0;
    } else if constexpr (D == 2) {
        const double q = fma(n[0], n[0], n[1] * n[1]);
        const double iL = rsqrt_nr(q);
        f.L = q * iL;
        f.e[0][0] = n[0] * iL;
        f.e[0][1] = n[1] * iL;
        f.e[1][0] = -f.e[0][1];
        f.e[1][1] = f.e[0][0];
    } else {
        const double q12 = fma(n[0], n[0], n[1] * n[1]);
        const double q = fma(n[2], n[2], q12);
        const double iL = rsqrt_nr(q);
        double ct = 1.0, st = 0.0, r12;
        if (q12 > 1e-24 * q) {
            const double ir = rsqrt_nr(q12);
            ct = n[0] * ir;
            st = n[1] * ir;
            r12 = q12 * ir;
        } else {
            r12 = sqrt(q12);
        }
        const double cp = r12 * iL, sp = n[2] * iL;
        f.L = q * iL;
        f.e[0][0] = cp * ct;
        f.e[0][1] = cp * st;
        f.e[0][2] = sp;
        f.e[1][0] = -st;
        f.e[1][1] = ct;
        f.e[1][2] = 0.0;
        f.e[2][0] = -sp * ct;
        f.e[2][1] = -sp * st;
        f.e[2][2] = cp;
    }
    return f;
}

// ------------------------------------------------------------ face dissipation
// -1/2 Lambda T^{-1} R Y [[W]]^WENO at the face between nodes l and r (Sec. 3.3, eq. HOstable): R = R~ S in the frame of
// the face normal, W = R^T T V at the six stencil nodes.  The state and the scales of a face:
template <int D>
struct Face {
    Frame<D> fr;
    double vr[D];               // {v} in the frame: normal, tangential
    double c, H;                // sound speed, (E + p)/rho
    double hm;                  // H less the entropy wave's last entry
    double sA, sE, sT;          // scales of the acoustic, entropy and shear waves
    double sAc, Lam;
};
// rho = {rho}^ln, v = {v}, p = {rho}^ln/{rho/p}^ln; n, xtf the means of the nodes' metrics and J xi_t
template <int D>
__device__ __forceinline__ Face<D> face_state(const double* S, int NB, int l, int r, const double* n, double xtf,
                                              const Gas& G, DevStatus* st, int gidx) {
    using SL = Slots<D>;
    auto at = [&](int f, int q) { return S[f * NB + q]; };
    Face<D> f;
    double rho;
    {
        const double al = at(SL::RHO, l), ar = at(SL::RHO, r);
        const double m = al + ar;
        rho = m * logmean_over_mean((al - ar) * rcp_nr(m), at(SL::LNR, l), at(SL::LNR, r));
    }
    double prho;                                            // p/rho = 1/{rho/p}^ln
    {
        const double al = at(SL::RP, l), ar = at(SL::RP, r);
        const double im = rcp_nr(al + ar);
        prho = mean_over_logmean((al - ar) * im, at(SL::LNRP, l), at(SL::LNRP, r)) * im;
    }
    const double arho = G.a * rho;
    const double z = fma(G.a, rho, prho);
    const double om = fma(-G.b, rho, 1.0);
    const double iom = rcp_nr(om);
    const double RT = z * om;
    const double c2 = fma((1.0 + G.delta) * z, iom, -2.0 * arho);
    const double w = fma(-2.0 * arho, om, z);               // (R T - 2 a rho (1 - b rho)^2)/(1 - b rho)
    if (!positive(c2) || !positive(w) || !positive(om)) raise_error(st, ES_ERR_INADMISSIBLE, gidx);
    const double ic = rsqrt_nr(c2);
    f.c = __dmul_rn(c2, ic);
    f.fr = face_frame<D>(n);
    double vm[D];
#pragma unroll
    for (int k = 0; k < D; ++k) vm[k] = at(SL::V + k, l) + at(SL::V + k, r);
    double v2 = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        f.vr[a] = f.fr.e[a][0] * vm[0];
#pragma unroll
        for (int k = 1; k < D; ++k)
            if (!(a == 1 && k == 2)) f.vr[a] = fma(f.fr.e[a][k], vm[k], f.vr[a]);
        v2 = a == 0 ? f.vr[a] * f.vr[a] : fma(f.vr[a], f.vr[a], v2);
    }
    // H = (E + p)/rho = cv T - a rho + |v|^2/2 + p/rho, cv T = R T/delta
    f.H = fma(0.5, v2, fma(RT, G.idelta, fma(-G.a, rho, prho)));
    f.hm = __dmul_rn(c2 * om, G.idelta);
    // the scales: S_acoustic = sqrt(rho T/2)/c, S_entropy = sqrt(rho T) sqrt(delta z/w)/c, S_shear = sqrt(rho T)
    const double rT = rho * (RT * G.iR);
    f.sT = rT * rsqrt_nr(rT);
    const double sTc = f.sT * ic;
    f.sA = 0.70710678118654752440 * sTc;
    const double dz = G.delta * z;
    f.sE = sTc * (dz * rsqrt_nr(dz * w));
    f.Lam = fma(f.fr.L, f.c, fabs(fma(f.fr.L, f.vr[0], xtf)));
    f.sAc = f.sA * f.c;
    return f;
}

// W = R^T T d for one difference d of the entropy variables: with A = d_1 + v . d_v + H d_E and B = d_n + v_n d_E,
// W_acoustic = S (A -+ c B), W_entropy = S (A - hm d_E), W_shear = S (d_t + v_t d_E).  MASK: the waves wanted
template <int D>
__device__ __forceinline__ void project(const Face<D>& f, const double* d, double* W, unsigned mask = ~0u) {
    constexpr int NC = D + 2;
    double rv[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        rv[a] = f.fr.e[a][0] * d[1];
#pragma unroll
        for (int k = 1; k < D; ++k)
            if (!(a == 1 && k == 2)) rv[a] = fma(f.fr.e[a][k], d[1 + k], rv[a]);
    }
    const double dE = d[NC - 1];
    double A = fma(f.H, dE, d[0]);
#pragma unroll
    for (int a = 0; a < D; ++a) A = fma(f.vr[a], rv[a], A);
    const double B = fma(f.vr[0], dE, rv[0]);
    const double sa = f.sA * A;
    if (mask & 1u) W[0] = fma(-f.sAc, B, sa);
    if (mask & 2u) W[1] = __dmul_rn(f.sE, fma(-f.hm, dE, A));
#pragma unroll
    for (int a = 1; a < D; ++a)
        if (mask & (2u << a)) W[1 + a] = __dmul_rn(f.sT, fma(f.vr[a], dE, rv[a]));
    if (mask & (1u << (NC - 1))) W[NC - 1] = fma(f.sAc, B, sa);
}

// The sign switch takes a plain jump within sign_tol of sum_a |R_am| (|(TV_l)_a| + |(TV_r)_a|), the size of the terms
// that form W_m, for round-off of zero.  That size lies between the FP32 bounds below (the terms of V_1 and V_E, which
// dominate it, and those plus a bound on the velocity terms); only a jump between them needs it.
struct SwitchBounds {
    float vs, es, qs, vsum, c, tol, H, vc, hm;
};
template <int D>
__device__ __forceinline__ SwitchBounds switch_bounds(const Face<D>& f, const double* S, int NB, int l, int r,
                                                      const Weno& Wc) {
    using SL = Slots<D>;
    auto at = [&](int k, int q) { return abs_f(S[k * NB + q]); };
    SwitchBounds b;
    b.vs = at(SL::W0, l) + at(SL::W0, r);
    b.es = at(SL::WE, l) + at(SL::WE, r);
    b.qs = b.vsum = 0.0f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        b.qs += at(SL::VT + k, l) + at(SL::VT + k, r);
        b.vsum += abs_f(f.vr[k]);
    }
    b.c = abs_f(f.c);
    b.tol = abs_f(Wc.sign_tol) * 1.00001f;
    b.H = abs_f(f.H);
    b.vc = abs_f(f.vr[0]) * b.c;
    b.hm = abs_f(f.hm);
    return b;
}
// is the jump j of wave m zero: 0 no, 1 yes, 2 between the bounds (or out of FP32's range)
template <int D>
__device__ __forceinline__ int jump_is_zero(const SwitchBounds& b, const Face<D>& f, int m, double j) {
    const bool shear = m >= 2 && m <= D;
    // |last entry of R| >= | |H| - |rest| |, <= |H| + |rest|
    const float rest = m == 1 ? b.hm : b.vc;
    const float scale = abs_f(m == 1 ? f.sE : (shear ? f.sT : f.sA)) * b.tol;
    float lo, hi;
    if (shear) {
        lo = scale * ((abs_f(f.vr[m < D + 1 ? m - 1 : 0]) + b.c) * b.es);
        hi = lo + scale * b.qs;
    } else {
        lo = scale * (b.vs + fabsf(b.H - rest) * b.es);
        hi = scale * (b.vs + (b.H + rest) * b.es + (b.vsum + b.c) * b.qs);
    }
    const float ja = abs_f(j);
    // (factors: truncation and rounding of the FP32 values; bounds that leave FP32's range, in units of extreme size, decide
    // nothing)
    if ((__double_as_longlong(j) << 1) == 0) return 1;
    if (__float_as_uint(hi) - 0x0da24260u >= 0x7e967699u - 0x0da24260u) return b.tol == 0.0f ? 0 : 2;   // not in [1e-30, 1e38)
    if (ja * 1.0001f < lo * 0.99f) return 1;
    return ja > hi * 1.001f ? 0 : 2;
}
// the size itself
template <int D>
__device__ __forceinline__ double jump_size(const Face<D>& f, const double* S, int NB, int l, int r, int m) {
    using SL = Slots<D>;
    auto at = [&](int k, int q) { return S[k * NB + q]; };
    double tv[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        double tl = 0.0, tr = 0.0;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            tl = fma(f.fr.e[a][k], at(SL::VT + k, l), tl);
            tr = fma(f.fr.e[a][k], at(SL::VT + k, r), tr);
        }
        tv[a] = fabs(tl) + fabs(tr);
    }
    const double e2 = fabs(at(SL::WE, l)) + fabs(at(SL::WE, r));
    if (m >= 2 && m <= D)                                   // velocity round-off scales with |v_t| + c
        return f.sT * fma(fabs(f.vr[m < D + 1 ? m - 1 : 0]) + f.c, e2, tv[m < D + 1 ? m - 1 : 0]);
    double common = fabs(at(SL::W0, l)) + fabs(at(SL::W0, r));
#pragma unroll
    for (int a = 1; a < D; ++a) common = fma(fabs(f.vr[a]), tv[a], common);
    const double vn = f.vr[0];
    const double u = m == 0 ? vn - f.c : (m == 1 ? vn : vn + f.c);
    const double h = m == 0 ? fma(-vn, f.c, f.H) : (m == 1 ? f.H - f.hm : fma(vn, f.c, f.H));
    return (m == 1 ? f.sE : f.sA) * fma(fabs(u), tv[0], fma(fabs(h), e2, common));
}
// Y [[W]]^WENO: kept where the reconstruction's jump has the sign of the plain jump j (a NaN jump is dropped)
__device__ __forceinline__ double switched(double jw, double j) {
    const bool keep = (__double2hiint(jw) ^ __double2hiint(j)) >= 0 && (__double2hiint(jw) & 0x7fffffff) <= 0x7ff00000;
    return keep ? jw : 0.0;
}

// F += the dissipation of the face between nodes l and l + step, from the entropy variables' jumps between neighbours
// along the line (JB[c * NJ + jq + o] = half of V_{l+o+1} - V_{l+o}, o = -2 .. 2).  They are halved, and with them W
// and its reconstructed jump, so Lambda/2 becomes Lambda.
template <int D>
__device__ __forceinline__ void face_dissipation(const double* S, int NB, int l, int step, const double* n, double xtf,
                                                 const Gas& G, const Weno& Wc, const double* JB, int NJ, int jq, double* F,
                                                 DevStatus* st, int gidx) {
    constexpr int NC = D + 2;
    const int r = l + step;
    const Face<D> f = face_state<D>(S, NB, l, r, n, xtf, G, st, gidx);
    double dW[NC][5];
#pragma unroll
    for (int o = 0; o < 5; ++o) {
        double d[NC], W[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) d[m] = JB[m * NJ + jq + o - 2];
        project<D>(f, d, W);
#pragma unroll
        for (int m = 0; m < NC; ++m) dW[m][o] = W[m];
    }
    bool zero[NC];
    unsigned open = 0u;
    {
        const SwitchBounds b = switch_bounds<D>(f, S, NB, l, r, Wc);
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int is = jump_is_zero<D>(b, f, m, dW[m][2]);
            zero[m] = is == 1;
            open |= is == 2 ? 1u << m : 0u;
        }
    }
    if (open != 0u) {
#pragma unroll
        for (int m = 0; m < NC; ++m)
            if ((open >> m) & 1u) zero[m] = fabs(dW[m][2]) <= Wc.sign_tol * jump_size<D>(f, S, NB, l, r, m);
    }
    double y[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        // a wave whose plain jump is zero adds nothing whatever its reconstruction: the shear waves of a uniform flow,
        // every wave of a constant state
        y[m] = 0.0;
        if (!zero[m]) y[m] = switched(weno_jump(dW[m], Wc), dW[m][2]);
    }
    const double h = -f.Lam, vn = f.vr[0];
    const double y0 = __dmul_rn(f.sA, y[0]), y1 = __dmul_rn(f.sE, y[1]), y4 = __dmul_rn(f.sA, y[NC - 1]);
    const double i0 = (y0 + y4) + y1;
    const double qc = f.c * (y4 - y0);
    double in[D];                                            // the momentum increment in the frame
    in[0] = fma(vn, i0, qc);
    double iE = fma(vn, qc, fma(f.H, i0, -(f.hm * y1)));
#pragma unroll
    for (int a = 1; a < D; ++a) {
        const double ys = __dmul_rn(f.sT, y[1 + a]);
        in[a] = fma(f.vr[a], i0, ys);
        iE = fma(f.vr[a], ys, iE);
    }
    F[0] = fma(h, i0, F[0]);
#pragma unroll
    for (int k = 0; k < D; ++k) {
        double t = f.fr.e[0][k] * in[0];
#pragma unroll
        for (int a = 1; a < D; ++a)
            if (!(a == 1 && k == 2)) t = fma(f.fr.e[a][k], in[a], t);
        F[1 + k] = fma(h, t, F[1 + k]);
    }
    F[NC - 1] = fma(h, iE, F[NC - 1]);
}

}  // namespace flux64
}  // namespace es
