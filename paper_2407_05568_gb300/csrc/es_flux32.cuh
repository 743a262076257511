// es_flux32.cuh -- two-point fluxes, entropy jumps and face dissipation of the mixed form's FP32 arithmetic, in D = 2, 3
// dimensions, on node values in registers.
//
// The kernels that use these are bound by the instructions they issue (73% of the issue slots busy, 7400 instructions a
// node in 2D before this form), so, as in the FP64 form: nodes keep HALF of every field that a face reads as the mean of
// its two nodes, quantities are formed in the products that the formulas need, the jump of the entropy variables takes
// the means of the pair flux between the same nodes, and MR-WENO5 works on halved differences.  Reciprocals and
// reciprocal square roots are the hardware's approximations (1 and 2 ulp; subnormal arguments count as zero).
#pragma once
#include <cuda_runtime.h>

#include "es_internal.h"
#include "es_mixed_device.cuh"

namespace es {
namespace flux32 {

using mixed::GasF;

__device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsq(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// {a}/{a}^ln = artanh(f)/f and its reciprocal from f = (a_l - a_r)/(a_l + a_r), u = f^2: for |f| < 0.2 the next terms of
// the series, u^5/11 and 0.022 u^5, are under 1e-8
__device__ __forceinline__ float artanh_far(float f) { return 0.5f * logf((1.0f + f) * rcp(1.0f - f)) * rcp(f); }
__device__ __forceinline__ float mean_over_logmean(float f) {
    if (fabsf(f) < 0.2f) {
        const float u = f * f;
        return fmaf(u, fmaf(u, fmaf(u, fmaf(u, 1.0f / 9.0f, 1.0f / 7.0f), 1.0f / 5.0f), 1.0f / 3.0f), 1.0f);
    }
    return artanh_far(f);
}
__device__ __forceinline__ float logmean_over_mean(float f) {
    if (fabsf(f) < 0.2f) {
        const float u = f * f;
        return fmaf(u, fmaf(u, fmaf(u, fmaf(u, -428.0f / 14175.0f, -44.0f / 945.0f), -4.0f / 45.0f), -1.0f / 3.0f), 1.0f);
    }
    return rcp(artanh_far(f));
}

// ------------------------------------------------------------ nodes
// what a pair flux reads of a node, halved (iom = 1/(1 - b rho) is not): g = R/(1 - b rho) - a rho/T, art = a rho/T,
// E0 = |v|^2/(2T) + 2 a rho/T
template <int D>
struct Node {
    float rho, T, iom, E0, g, art;
    float v[D], vT[D], rv[D];
};
// what the entropy variables' jump reads besides: the low parts of the double-float rho, T, v (halved) and 1/T
template <int D>
struct NodeLow {
    float rho, T, iT;
    float v[D];
};

template <int D>
struct PairMeans {
    float rm, Tm, iT;           // {rho}, {T}, 1/{T}
    float coef;                 // R b/Pi - a/{T}
    float det;                  // the determinant of Theorem 3.1: d[[V_1]]/d[[rho]]
    float x;                    // cv {T}/{T}^ln - {|v|^2/T}/2 - 2 a {rho/T}
    float v[D];                 // {v_k}
};
template <int D>
__device__ __forceinline__ PairMeans<D> pair_means(const Node<D>& l, const Node<D>& r, const GasF& G) {
    PairMeans<D> p;
    p.rm = l.rho + r.rho;
    p.Tm = l.T + r.T;
    const float ir = rcp(p.rm);
    p.iT = rcp(p.Tm);
    const float dr = l.rho - r.rho;
    const float Fr = mean_over_logmean(dr * ir);
    const float FT = mean_over_logmean((l.T - r.T) * p.iT);
    const float aiT = G.a * p.iT;
    p.coef = fmaf(G.Rb * l.iom, r.iom, -aiT);
    p.det = fmaf(G.R, Fr * ir, p.coef) - aiT;
    if (G.b > 0.0f) {
        const float io = rcp(fmaf(-G.b, p.rm, 1.0f));       // {1 - b rho}
        p.det = fmaf(G.Rb, mean_over_logmean(-G.b * dr * io) * io, p.det);
    }
    p.x = fmaf(G.cv, FT, -(l.E0 + r.E0));
#pragma unroll
    for (int k = 0; k < D; ++k) p.v[k] = l.v[k] + r.v[k];
    return p;
}

// EC flux of Sec. 3.1 contracted with the means n, xt of the metrics and J xi_t (es_flux64.cuh's formulas); the energy
// component is a QUARTER
template <int D>
__device__ __forceinline__ void pair_flux(const Node<D>& l, const Node<D>& r, const PairMeans<D>& p, const float* n,
                                          float xt, float* out) {
    const float iD = rcp(p.det);
    const float g = l.g + r.g;
    float A = xt * p.rm, B = xt, nv = 0.0f, sv = p.x;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float vT = l.vT[k] + r.vT[k];
        A = fmaf(n[k], l.rv[k] + r.rv[k], A);
        B = fmaf(n[k], p.v[k], B);
        nv = fmaf(n[k], vT, nv);
        sv = fmaf(vT, p.v[k], sv);
    }
    const float Q = fmaf(p.coef, A, g * B) * iD;
    const float P = p.rm * p.Tm * g;
    out[0] = Q;
#pragma unroll
    for (int k = 0; k < D; ++k) out[1 + k] = fmaf(p.v[k], Q, n[k] * P);
    out[D + 1] = fmaf(l.art + r.art, A, fmaf(sv, Q, P * nv)) * (l.T * r.T * p.iT);
}

// Half of the entropy variables' jump V_r - V_l (eq. jumpV in general units):
//   [[V_1]] = det [[rho]] - ([[T]] x + sum_m {v_m} [[v_m]])/{T},  [[V_{1+m}]] = ([[v_m]] - {v_m/T} [[T]])/{T},
//   [[V_E]] = [[T]]/(T_l T_r), with the jumps from the double-float node values
template <int D>
__device__ __forceinline__ void entropy_jump(const Node<D>& l, const Node<D>& r, const NodeLow<D>& ll,
                                             const NodeLow<D>& rl, const PairMeans<D>& p, float* dV) {
    const float dr = (r.rho - l.rho) + (rl.rho - ll.rho);
    const float dT = (r.T - l.T) + (rl.T - ll.T);
    float t = dT * p.x;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float dv = (r.v[k] - l.v[k]) + (rl.v[k] - ll.v[k]);
        t = fmaf(p.v[k], dv, t);
        dV[1 + k] = fmaf(-(l.vT[k] + r.vT[k]), dT, dv) * p.iT;
    }
    dV[0] = fmaf(-p.iT, t, p.det * dr);
    dV[D + 1] = dT * (ll.iT * rl.iT);
}

// ------------------------------------------------------------ MR-WENO5 (Sec. 3.3)
struct WenoC {
    float h1, h2, q2, q3[4], eps4, tol;      // Weno's derived coefficients, and the sign switch's tolerance
};
inline WenoC weno_floats(const Weno& w) {
    WenoC c;
    c.h1 = float(w.h1);
    c.h2 = float(w.h2);
    c.q2 = float(w.q2);
    for (int k = 0; k < 4; ++k) c.q3[k] = float(w.q3[k]);
    c.eps4 = float(w.eps4);
    c.tol = float(w.sign_tol);
    return c;
}

// (w_{i+1/2} - w_i)/2 from half the differences of the five stencil values (es_flux64.cuh's weno_side); the weights
// g (1 + t^2/k) keep their quotients, which do not overflow where products of indicators would
__device__ __forceinline__ float weno_side(float d0, float d1, float d2, float d3, float k1, const WenoC& c) {
    const float s = d1 + d2, dd = d2 - d1;
    const float g = (d0 + d3) - s;
    const float e = fmaf(-3.0f, dd, d3 - d0);
    const float k2 = fmaf(0.25f * s, s, fmaf((13.0f / 12.0f) * dd, dd, c.eps4));
    const float q = fmaf(e, fmaf(4405.0f / 4032.0f, e, (-11.0f / 60.0f) * dd),
                         g * fmaf(89.0f / 320.0f, g, (-1.0f / 12.0f) * s));
    const float k3 = fmaxf(k2 + q, c.eps4);                  // (beta_3 >= 0 up to rounding)
    const float t = fabsf(k3 - k1) + fabsf(q);
    const float tt = t * t;
    const float y1 = fmaf(tt, rcp(k1), 1.0f), y2 = fmaf(tt, rcp(k2), 1.0f), y3 = fmaf(tt, rcp(k3), 1.0f);
    const float p2 = c.q2 * fmaf(2.0f, d2, d1);
    const float p3 = fmaf(c.q3[0], d0, fmaf(c.q3[1], d1, fmaf(c.q3[2], d2, c.q3[3] * d3)));
    return fmaf(y2, p2, y3 * p3) * rcp(fmaf(c.h1, y1, fmaf(c.h2, y2, y3)));
}

// Y [[w]]^WENO / 2 at the face between the third and fourth of six values, from half their five differences
__device__ __forceinline__ float weno_jump(const float* d, const WenoC& c) {
    const float s1 = fmaf(d[1], d[1], c.eps4), s2 = fmaf(d[2], d[2], c.eps4), s3 = fmaf(d[3], d[3], c.eps4);
    const float m = weno_side(d[0], d[1], d[2], d[3], fminf(s1, s2), c);
    const float p = weno_side(d[4], d[3], d[2], d[1], fminf(s2, s3), c);      // mirrored: changes sign
    const float jw = d[2] - (m + p);
    return jw * d[2] > 0.0f ? jw : 0.0f;
}

// ------------------------------------------------------------ face
template <int D>
struct Face {
    float e[D][D];              // rows of the rotation's momentum block: normal, tangents
    float vr[D];                // {v} in the frame
    float c, H, hm;             // sound speed, (E + p)/rho, H less the entropy wave's last entry
    float sA, sE, sT, sAc;      // scales of the acoustic, entropy and shear waves, sA c
    float Lam;
};
// rho, rp = rho/p of the two nodes (halved), v = {v}, n, xtf the means of the metrics and J xi_t
template <int D>
__device__ __forceinline__ Face<D> face_state(float rl, float rr, float pl, float pr, const float* v, const float* n,
                                              float xtf, const GasF& G, DevStatus* st) {
    Face<D> f;
    const float rm = rl + rr;
    const float rho = rm * logmean_over_mean((rl - rr) * rcp(rm));
    const float ip = rcp(pl + pr);
    const float prho = mean_over_logmean((pl - pr) * ip) * ip;       // p/rho
    const float arho = G.a * rho;
    const float z = prho + arho;
    const float om = fmaf(-G.b, rho, 1.0f);
    const float RT = z * om;
    const float c2 = fmaf((1.0f + G.delta) * z, rcp(om), -2.0f * arho);
    const float w = fmaf(-2.0f * arho, om, z);               // (R T - 2 a rho (1 - b rho)^2)/(1 - b rho)
    if (!(c2 > 0.0f) || !(w > 0.0f) || !(om > 0.0f)) raise_error(st, ES_ERR_INADMISSIBLE, 0);
    const float ic = rsq(c2);
    f.c = c2 * ic;
    float L;
    if constexpr (D == 2) {
        const float q = fmaf(n[0], n[0], n[1] * n[1]);
        const float iL = rsq(q);
        L = q * iL;
        f.e[0][0] = n[0] * iL;
        f.e[0][1] = n[1] * iL;
        f.e[1][0] = -f.e[0][1];
        f.e[1][1] = f.e[0][0];
    } else {
        // theta = atan2(n_2, n_1) (0 where (n_1, n_2) is the rounding of metrics that vanish), phi = atan2(n_3, .)
        const float q12 = fmaf(n[0], n[0], n[1] * n[1]);
        const float q = fmaf(n[2], n[2], q12);
        const float iL = rsq(q);
        L = q * iL;
        float ct = 1.0f, sn = 0.0f, r12 = 0.0f;
        if (q12 > 1e-24f * q) {
            const float ir = rsq(q12);
            ct = n[0] * ir;
            sn = n[1] * ir;
            r12 = q12 * ir;
        }
        const float cp = r12 * iL, sp = n[2] * iL;
        f.e[0][0] = cp * ct;
        f.e[0][1] = cp * sn;
        f.e[0][2] = sp;
        f.e[1][0] = -sn;
        f.e[1][1] = ct;
        f.e[1][2] = 0.0f;
        f.e[2][0] = -sp * ct;
        f.e[2][1] = -sp * sn;
        f.e[2][2] = cp;
    }
    float v2 = 0.0f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        f.vr[a] = f.e[a][0] * v[0];
#pragma unroll
        for (int k = 1; k < D; ++k)
            if (!(a == 1 && k == 2)) f.vr[a] = fmaf(f.e[a][k], v[k], f.vr[a]);
        v2 = fmaf(f.vr[a], f.vr[a], v2);
    }
    f.H = fmaf(0.5f, v2, fmaf(RT, G.idelta, prho - arho));
    f.hm = c2 * om * G.idelta;
    const float rT = rho * (RT * G.iR);
    f.sT = rT * rsq(rT);
    const float sTc = f.sT * ic;
    f.sA = 0.70710678f * sTc;
    const float dz = G.delta * z;
    f.sE = sTc * (dz * rsq(dz * w));
    f.sAc = f.sA * f.c;
    f.Lam = fmaf(L, f.c, fabsf(fmaf(L, f.vr[0], xtf)));
    return f;
}

// a difference of the entropy variables in the frame: rv the rotated momentum part, A = d_1 + v . d_v + H d_E,
// B = d_n + v_n d_E
template <int D>
struct Rotated {
    float rv[D], A, B;
};
template <int D>
__device__ __forceinline__ Rotated<D> rotate(const Face<D>& f, const float* d) {
    Rotated<D> r;
    r.A = fmaf(f.H, d[D + 1], d[0]);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        r.rv[a] = f.e[a][0] * d[1];
#pragma unroll
        for (int k = 1; k < D; ++k)
            if (!(a == 1 && k == 2)) r.rv[a] = fmaf(f.e[a][k], d[1 + k], r.rv[a]);
        r.A = fmaf(f.vr[a], r.rv[a], r.A);
    }
    r.B = fmaf(f.vr[0], d[D + 1], r.rv[0]);
    return r;
}
// sizes of the terms that form the face's plain jump d of each wave (over its scale S)
template <int D>
__device__ __forceinline__ void term_sizes(const Face<D>& f, const float* d, const Rotated<D>& r, float* size) {
    const float dE = fabsf(d[D + 1]), vn = f.vr[0], vc = vn * f.c;
    float common = fabsf(d[0]);
#pragma unroll
    for (int a = 1; a < D; ++a) common = fmaf(fabsf(f.vr[a]), fabsf(r.rv[a]), common);
    const float rn = fabsf(r.rv[0]);
    size[0] = fmaf(fabsf(vn - f.c), rn, fmaf(fabsf(f.H - vc), dE, common));
    size[1] = fmaf(fabsf(vn), rn, fmaf(fabsf(f.H - f.hm), dE, common));
#pragma unroll
    for (int a = 1; a < D; ++a) size[1 + a] = fmaf(fabsf(f.vr[a]) + f.c, dE, fabsf(r.rv[a]));   // velocity round-off ~ |v_t| + c
    size[D + 1] = fmaf(fabsf(vn + f.c), rn, fmaf(fabsf(f.H + vc), dE, common));
}

// F += -Lambda R (Y [[W]]^WENO / 2) for the waves' values y
template <int D>
__device__ __forceinline__ void add_increment(const Face<D>& f, const float* y, float* F) {
    const float vn = f.vr[0], h = -f.Lam;
    const float y0 = f.sA * y[0], y1 = f.sE * y[1], y4 = f.sA * y[D + 1];
    const float i0 = y0 + y1 + y4;
    const float qc = f.c * (y4 - y0);
    float in[D];
    in[0] = fmaf(vn, i0, qc);
    float iE = fmaf(vn, qc, fmaf(f.H, i0, -f.hm * y1));
#pragma unroll
    for (int a = 1; a < D; ++a) {
        const float ys = f.sT * y[1 + a];
        in[a] = fmaf(f.vr[a], i0, ys);
        iE = fmaf(f.vr[a], ys, iE);
    }
    F[0] = fmaf(h, i0, F[0]);
#pragma unroll
    for (int k = 0; k < D; ++k) {
        float t = f.e[0][k] * in[0];
#pragma unroll
        for (int a = 1; a < D; ++a)
            if (!(a == 1 && k == 2)) t = fmaf(f.e[a][k], in[a], t);
        F[1 + k] = fmaf(h, t, F[1 + k]);
    }
    F[D + 1] = fmaf(h, iE, F[D + 1]);
}

}  // namespace flux32
}  // namespace es
