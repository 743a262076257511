// es_mixed_device.cuh -- device functions of the mixed-precision form (FP32 pipe, double-float state and primitive jumps) in
// 1D, shared by the tiled stage kernel and the batched persistent kernel (see es_stage_mixed.cu for the design), and the
// displacement at a node in 1D and 2D.
#pragma once
#include <cuda_runtime.h>

#include "es_device.cuh"
#include "es_df.cuh"
#include "es_internal.h"

namespace es {
namespace mixed {

enum FieldF {
    G_RHO, G_V1, G_T, G_IT, G_OM, G_IOM, G_G, G_RT, G_VT1, G_V2T, G_RV1, G_RP,
    G_RHOL, G_V1L, G_TL,          // low parts of rho, v, T (double-float)
    G_N1X, G_XT1,
    G_COUNT
};

template <int BX, int NT>
struct TileF {
    static constexpr int NB = BX + 6;
    static constexpr int NC = 3;
    static constexpr int NP = 3 * BX + 6;
    static constexpr int NF = BX + 1;
    static constexpr int PAIR_FLOATS = NP * NC;            // also holds the displacement and the mesh velocity
    // entropy-variable jumps between neighbours (box positions q, q + 1), shared by the faces whose stencils contain them
    static constexpr int NJ = BX + 5;
    static constexpr size_t SMEM =
        sizeof(float) * (size_t(G_COUNT) * NB + PAIR_FLOATS + NF * (NC + 1) + size_t(NJ) * NC);
    static_assert(NT >= BX && NT % 32 == 0 && PAIR_FLOATS >= 2 * NB, "threads cover the tile");
};

struct GasF {
    float a, b, R, cv, delta, Rb, icv, iR, idelta;
};

struct WenoF {
    float g1, g2, g3, g12, ig22, ig3, eps, sign_tol;
};

// reciprocal logarithmic mean 1/{a}^ln from the relative jump f = (a_l - a_r)/(a_l + a_r):
// [[ln a]] = ln((1 + f)/(1 - f)) = 2 artanh(f); series of artanh(f)/f for |f| < 0.05
__device__ __forceinline__ float inv_log_mean_j(float al, float ar, float d) {
    // d = a_l - a_r, passed in when known to more digits than al - ar
    const float s = al + ar;
    const float is = 1.0f / s;
    const float f = d * is;
    if (fabsf(f) < 0.05f) {
        const float u = f * f;
        const float F = 1.0f + u * (1.0f / 3.0f + u * (1.0f / 5.0f + u * (1.0f / 7.0f + u * (1.0f / 9.0f))));
        return 2.0f * F * is;
    }
    return log1pf(2.0f * f / (1.0f - f)) / d;
}

__device__ __forceinline__ float inv_log_mean_f(float al, float ar) { return inv_log_mean_j(al, ar, al - ar); }

__device__ __forceinline__ float mr_weno5_f(float wm2, float wm1, float w0, float wp1, float wp2, const WenoF& c) {
    const float q2 = (-wm1 + 5.0f * w0 + 2.0f * wp1) * (1.0f / 6.0f);
    const float q3 = (2.0f * wm2 - 13.0f * wm1 + 47.0f * w0 + 27.0f * wp1 - 3.0f * wp2) * (1.0f / 60.0f);
    const float p1 = w0;
    const float p2 = (q2 - c.g12 * p1) * c.ig22;
    const float p3 = (q3 - c.g1 * p1 - c.g2 * p2) * c.ig3;
    const float dl = w0 - wm1, dr = wp1 - w0;
    const float b1 = fminf(dl * dl, dr * dr);
    const float s2a = wm1 - 2.0f * w0 + wp1, s2b = wp1 - wm1;
    const float b2 = (13.0f / 12.0f) * s2a * s2a + 0.25f * s2b * s2b;
    const float o1 = 0.5f * (wp1 - wm1), o2 = 0.5f * (wp2 - wm2);
    // even part relative to w0 (beta ignores a constant added to the data)
    const float a1 = 0.5f * ((wp1 - w0) + (wm1 - w0)), a2 = 0.5f * ((wp2 - w0) + (wm2 - w0));
    const float c3 = (o2 - 2.0f * o1) * (1.0f / 6.0f);
    const float c1 = (34.0f * o1 - 5.0f * o2) * (1.0f / 24.0f);
    const float c4 = (a2 - 4.0f * a1) * (1.0f / 12.0f);
    const float c2 = (12.0f * a1 - a2) * 0.125f;
    const float b3 = c1 * (c1 + 0.5f * c3) + c2 * ((13.0f / 3.0f) * c2 + 4.2f * c4) + (3129.0f / 80.0f) * c3 * c3
                   + (87617.0f / 140.0f) * c4 * c4;
    const float t = 0.5f * (fabsf(b3 - b1) + fabsf(b3 - b2));
    const float tau = t * t;
    const float w1 = c.g1 * (1.0f + tau / (b1 + c.eps));
    const float w2 = c.g2 * (1.0f + tau / (b2 + c.eps));
    const float w3 = c.g3 * (1.0f + tau / (b3 + c.eps));
    return (w1 * p1 + w2 * p2 + w3 * p3) / (w1 + w2 + w3);
}

__device__ __forceinline__ void pair_flux_f(const float* S, int NB, int l, int r, float nx, float xt, const GasF& G,
                                            float* out) {
    const float rl = S[G_RHO * NB + l], rr = S[G_RHO * NB + r];
    const float Tl = S[G_T * NB + l], Tr = S[G_T * NB + r];
    const float rho_m = 0.5f * (rl + rr);
    const float T_m = 0.5f * (Tl + Tr);
    const float iT_m = 0.5f * (S[G_IT * NB + l] + S[G_IT * NB + r]);
    const float drho = (rl - rr) + (S[G_RHOL * NB + l] - S[G_RHOL * NB + r]);
    const float ilr = inv_log_mean_j(rl, rr, drho);
    const float ilT = inv_log_mean_j(Tl, Tr, (Tl - Tr) + (S[G_TL * NB + l] - S[G_TL * NB + r]));
    const float Pinv = S[G_IOM * NB + l] * S[G_IOM * NB + r];
    const float iTa = 1.0f / T_m;
    const float coef = G.Rb * Pinv - G.a * iTa;
    float D = G.R * ilr + coef - G.a * iTa;
    if (G.b > 0.0f) D += G.Rb * inv_log_mean_j(S[G_OM * NB + l], S[G_OM * NB + r], -G.b * drho);
    const float iD = 1.0f / D;
    const float g_m = 0.5f * (S[G_G * NB + l] + S[G_G * NB + r]);
    const float rT_m = 0.5f * (S[G_RT * NB + l] + S[G_RT * NB + r]);
    const float v2T_m = 0.5f * (S[G_V2T * NB + l] + S[G_V2T * NB + r]);
    const float vm1 = 0.5f * (S[G_V1 * NB + l] + S[G_V1 * NB + r]);
    const float vT1 = 0.5f * (S[G_VT1 * NB + l] + S[G_VT1 * NB + r]);
    const float rv1 = 0.5f * (S[G_RV1 * NB + l] + S[G_RV1 * NB + r]);
    const float U1 = (rho_m * coef + g_m) * iD;
    const float F11 = (rv1 * coef + g_m * vm1) * iD;
    const float P = rho_m * T_m * g_m;
    const float B0 = 0.5f * v2T_m - G.cv * T_m * ilT + 2.0f * G.a * rT_m;
    const float iiT = 1.0f / iT_m;
    const float Q1 = xt * U1 + nx * F11;
    const float sv = vT1 * vm1;
    out[0] = Q1;
    out[1] = vm1 * Q1 + nx * P;
    out[2] = (G.a * rT_m * (xt * rho_m + nx * rv1) + (sv - B0) * Q1 + P * nx * vT1) * iiT;
}

// Entropy-variable jump V_j - V_i written as the jump decomposition of Sec. 3.1
// (eq. jumpV) in general units, with every mean taken between nodes i and j:
//   [[V_1]] = [[rho]] (R/{rho}^ln + R b/{1-b rho}^ln + R b/Pi - 2a/{T})
//           + [[T]] (-c_v/{T}^ln + (2a {rho/T} + {|v|^2/T}/2)/{T}) - sum_m {v_m}[[v_m]]/{T}
//   [[V_{1+m}]] = ([[v_m]] - {v_m/T}[[T]])/{T},   [[V_E]] = [[T]]/(T_i T_j)
__device__ __forceinline__ void entropy_jump(const float* S, int NB, int i, int j, const GasF& G, float* dV) {
    const float ri = S[G_RHO * NB + i], rj = S[G_RHO * NB + j];
    const float Ti = S[G_T * NB + i], Tj = S[G_T * NB + j];
    // jumps from the double-float node values: exact hi difference plus lo difference
    const float dr = (rj - ri) + (S[G_RHOL * NB + j] - S[G_RHOL * NB + i]);
    const float dT = (Tj - Ti) + (S[G_TL * NB + j] - S[G_TL * NB + i]);
    const float iTa = 2.0f / (Ti + Tj);
    float crho = G.R * inv_log_mean_j(ri, rj, -dr) + G.Rb * S[G_IOM * NB + i] * S[G_IOM * NB + j] - 2.0f * G.a * iTa;
    if (G.b > 0.0f) crho += G.Rb * inv_log_mean_j(S[G_OM * NB + i], S[G_OM * NB + j], G.b * dr);
    const float rT = 0.5f * (S[G_RT * NB + i] + S[G_RT * NB + j]);
    const float v2T = 0.5f * (S[G_V2T * NB + i] + S[G_V2T * NB + j]);
    const float cT = -G.cv * inv_log_mean_j(Ti, Tj, -dT) + (2.0f * G.a * rT + 0.5f * v2T) * iTa;
    const float v1i = S[G_V1 * NB + i], v1j = S[G_V1 * NB + j];
    const float dv1 = (v1j - v1i) + (S[G_V1L * NB + j] - S[G_V1L * NB + i]);
    float kin = 0.5f * (v1i + v1j) * dv1;
    dV[1] = (dv1 - 0.5f * (S[G_VT1 * NB + i] + S[G_VT1 * NB + j]) * dT) * iTa;
    dV[0] = dr * crho + dT * cT - kin * iTa;
    dV[2] = dT * S[G_IT * NB + i] * S[G_IT * NB + j];
}

// the face state of eq. HOstable's dissipation: log-mean density and pressure ratio, T, c, the sign of the face normal of
// length L, normal velocity, and the scalings of R^T T
struct FaceF {
    float c, cs, vn, mid, sA, sE, Lam, Hm, Hp;
};

__device__ __forceinline__ FaceF face_state_f(const float* S, int NB, int l, float nx, float xtf, const GasF& G,
                                              DevStatus* st) {
    FaceF f;
    const int r = l + 1;
    const float ilr = inv_log_mean_f(S[G_RHO * NB + l], S[G_RHO * NB + r]);
    const float rho = 1.0f / ilr;
    const float ilrp = inv_log_mean_f(S[G_RP * NB + l], S[G_RP * NB + r]);
    const float p = rho * ilrp;
    const float om = 1.0f - G.b * rho;
    const float T = (p + G.a * rho * rho) * om * ilr * G.iR;
    const float iom = 1.0f / om;
    const float c2 = (1.0f + G.delta) * G.R * T * iom * iom - 2.0f * G.a * rho;
    const float dcrit = G.R * T - 2.0f * G.a * rho * om * om;
    if (!(c2 > 0.0f) || !(dcrit > 0.0f) || !(om > 0.0f)) raise_error(st, ES_ERR_INADMISSIBLE, 0);
    const float c = sqrtf(c2);
    const float vm1 = 0.5f * (S[G_V1 * NB + l] + S[G_V1 * NB + r]);
    const float L = fabsf(nx);
    const float cs = nx > 0.0f ? 1.0f : -1.0f;
    const float vn = cs * vm1;
    const float E = rho * (G.cv * T - G.a * rho) + 0.5f * rho * (vn * vn);
    const float H = (E + p) * ilr;
    f.c = c;
    f.cs = cs;
    f.vn = vn;
    f.mid = H - c2 * om * G.idelta;
    const float ic2 = 1.0f / c2;
    f.sA = sqrtf(0.5f * rho * T * ic2);
    f.sE = sqrtf(G.R * G.delta * rho * T * T * ic2 / dcrit);
    f.Lam = fabsf(xtf + L * vn) + L * c;
    f.Hm = H - vn * c;
    f.Hp = H + vn * c;
    return f;
}

__device__ __forceinline__ void face_dissipation_f(const float* S, int NB, int l, float nx, float xtf, const GasF& G,
                                                   const WenoF& Wc, float* out, DevStatus* st, const float* JB, int NJ,
                                                   int jq) {
    const FaceF fs = face_state_f(S, NB, l, nx, xtf, G, st);
    const float c = fs.c, cs = fs.cs, vn = fs.vn, mid = fs.mid;
    const float sA = fs.sA, sE = fs.sE, Lam = fs.Lam, Hm = fs.Hm, Hp = fs.Hp;

    // W_j - W_l = R^T T (V_j - V_l) at nodes l-2 .. l+3 (zero at l itself); V_j - V_l is the sum
    // of the neighbour jumps between them (JB[c][jq + q] = V_{q+1} - V_q along the line, the
    // face's left node at jq + 0)
    float W[6][3];
    float aTV[3];
    float cum[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        W[2][m] = 0.0f;
        cum[m] = 0.0f;
    }
#pragma unroll
    for (int o = 3; o < 6; ++o)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            cum[m] += JB[m * NJ + jq + (o - 3)];
            W[o][m] = cum[m];
        }
#pragma unroll
    for (int m = 0; m < 3; ++m) cum[m] = 0.0f;
#pragma unroll
    for (int o = 1; o >= 0; --o)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            cum[m] -= JB[m * NJ + jq + (o - 2)];
            W[o][m] = cum[m];
        }
#pragma unroll
    for (int o = 0; o < 6; ++o) {
        if (o == 2) continue;
        float dV[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) dV[m] = W[o][m];
        const float V0 = dV[0], V1 = cs * dV[1], V2 = dV[2];
        W[o][0] = sA * (V0 + (vn - c) * V1 + Hm * V2);
        W[o][1] = sE * (V0 + vn * V1 + mid * V2);
        W[o][2] = sA * (V0 + (vn + c) * V1 + Hp * V2);
        if (o == 3) {
            aTV[0] = fabsf(V0);
            aTV[1] = fabsf(V1);
            aTV[2] = fabsf(V2);
        }
    }
    float scl[3];
    scl[0] = sA * (aTV[0] + fabsf(vn - c) * aTV[1] + fabsf(Hm) * aTV[2]);
    scl[1] = sE * (aTV[0] + fabsf(vn) * aTV[1] + fabsf(mid) * aTV[2]);
    scl[2] = sA * (aTV[0] + fabsf(vn + c) * aTV[1] + fabsf(Hp) * aTV[2]);
    float y[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        // (no test for a zero wave here: with products that the compiler may fuse its branch changes the last digits, and it
        // gained 15% of a batch that had not developed)
        float j = W[3][m];
        if (fabsf(j) <= Wc.sign_tol * scl[m]) j = 0.0f;
        const float wmin = mr_weno5_f(W[0][m], W[1][m], W[2][m], W[3][m], W[4][m], Wc);
        const float wplu = mr_weno5_f(W[5][m], W[4][m], W[3][m], W[2][m], W[1][m], Wc);
        const float jw = wplu - wmin;
        const bool keep = (jw > 0.0f && j > 0.0f) || (jw < 0.0f && j < 0.0f);
        y[m] = keep ? jw : 0.0f;
    }
    const float h = -0.5f * Lam;
    const float y0 = sA * y[0], y1 = sE * y[1], y2 = sA * y[2];
    out[0] = h * (y0 + y1 + y2);
    out[1] = h * cs * ((vn - c) * y0 + vn * y1 + (vn + c) * y2);
    out[2] = h * (Hm * y0 + mid * y1 + Hp * y2);
}

__device__ __forceinline__ void load_node_f(float* S, int NB, int b, const StageParams& P, const GasF& G, int gi) {
    const int idx = state_index(gi, P.n1, P.bc[0]);
    const size_t N = P.fcs;                                 // component stride
    const size_t LO = P.fps;                                // offset of the lo plane of JU
    // primitive state in double-float arithmetic
    const df iJ = df_recip({P.fJs[idx], P.fJs[P.fpsJ + idx]});
    const df rho = df_mul({P.fJUs[idx], P.fJUs[LO + idx]}, iJ);
    const df m1 = df_mul({P.fJUs[N + idx], P.fJUs[LO + N + idx]}, iJ);
    const df E = df_mul({P.fJUs[2 * N + idx], P.fJUs[LO + 2 * N + idx]}, iJ);
    const df irho = df_recip(rho);
    const df v1 = df_mul(m1, irho);
    const df ke = df_mul_f(df_mul(v1, v1), 0.5f);
    // T = (E/rho - |v|^2/2 + a rho) / cv
    const df e = df_add(df_mul(E, irho), {-ke.hi, -ke.lo});
    const df Td = df_mul_f(df_add(e, df_mul_f(rho, G.a)), G.icv);
    const float r = rho.hi, T = Td.hi;
    const float om = 1.0f - G.b * r;
    const float iom = 1.0f / om;
    const float p = r * G.R * T * iom - G.a * r * r;
    const float iT = 1.0f / T;
    // what the node arithmetic needs; R T - 2 a rho (1 - b rho)^2 > 0 enters through the face states
    if (!(r > 0.0f) || !(om > 0.0f) || !(T > 0.0f) || !(p > 0.0f)) raise_error(P.status, ES_ERR_INADMISSIBLE, idx);
    S[G_RHO * NB + b] = r;
    S[G_RHOL * NB + b] = rho.lo;
    S[G_V1 * NB + b] = v1.hi;
    S[G_V1L * NB + b] = v1.lo;
    S[G_T * NB + b] = T;
    S[G_TL * NB + b] = Td.lo;
    S[G_IT * NB + b] = iT;
    S[G_OM * NB + b] = om;
    S[G_IOM * NB + b] = iom;
    S[G_G * NB + b] = G.R * iom - G.a * r * iT;
    S[G_RT * NB + b] = r * iT;
    S[G_VT1 * NB + b] = v1.hi * iT;
    S[G_V2T * NB + b] = 2.0f * ke.hi * iT;
    S[G_RV1 * NB + b] = m1.hi;
    S[G_RP * NB + b] = r / p;
}

// FP32 displacement and mesh velocity at a possibly-ghost node: periodic wrap
// (the displacement is periodic), outflow odd reflection
template <int DIM>
__device__ __forceinline__ void stage_disp(const StageParams& P, int gi, int gj, float cdt, float* ds, float* xd) {
    const size_t N = P.fcs;
    if (gi >= 0 && gi < P.n1 && (DIM == 1 || (gj >= 0 && gj < P.n2))) {     // interior: plain loads
        const size_t id = size_t(DIM == 2 ? gj : 0) * P.n1 + gi;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const float xdk = P.fxdot ? P.fxdot[k * N + id] : 0.0f;
            ds[k] = P.fdisp[k * N + id] + cdt * xdk;
            xd[k] = xdk;
        }
        return;
    }
    const GhostTerms ti = ghost_terms(gi, P.n1, P.bc[0]);
    GhostTerms tj;
    if (DIM == 2) tj = ghost_terms(gj, P.n2, P.bc[1]);
    else { tj.idx[0] = 0; tj.w[0] = 1.0; tj.nterm = 1; tj.q = 0; }
    float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
    for (int a = 0; a < ti.nterm; ++a)
        for (int c = 0; c < tj.nterm; ++c) {
            const float w = float(ti.w[a] * tj.w[c]);
            const size_t id = size_t(tj.idx[c]) * P.n1 + ti.idx[a];
            for (int k = 0; k < DIM; ++k) {
                const float xdk = P.fxdot ? P.fxdot[k * N + id] : 0.0f;
                acc[0][k] += w * (P.fdisp[k * N + id] + cdt * xdk);
                acc[1][k] += w * xdk;
            }
        }
    ds[0] = acc[0][0];
    xd[0] = acc[1][0];
    if (DIM == 2) {
        ds[1] = acc[0][1];
        xd[1] = acc[1][1];
    }
}


// One tile of the fused operator + RK stage in 1D (mixed form): the tile at i0 is staged with its halo in shared memory
// S / PB / FB / JB (TileF layout), then pair fluxes, face fluxes, divergence and the RK combination follow.  Called by the
// tiled kernel (one tile per CTA) and by the batched kernel (a loop over the chunks of one problem per CTA).
template <int BX, int NT>
__device__ __forceinline__ void stage_tile_mixed(float* smemf, const StageParams& P, int i0, float dt, const GasF& G,
                                                 const WenoF& Wc) {
    using TL = TileF<BX, NT>;
    constexpr int NB = TL::NB, NC = TL::NC;
    float* S = smemf;
    float* PB = smemf + G_COUNT * NB;
    float* FB = PB + TL::PAIR_FLOATS;
    float* JB = FB + TL::NF * (NC + 1);
    const int tid = threadIdx.x;
    const float cdt = P.fcst * dt;
    for (int b = tid; b < NB; b += NT) {
        const int gi = i0 - 3 + b;
        float ds[2], xd[2];
        stage_disp<1>(P, gi, 0, cdt, ds, xd);
        load_node_f(S, NB, b, P, G, gi);
        S[G_N1X * NB + b] = 1.0f;
        S[G_XT1 * NB + b] = -xd[0];
    }
    __syncthreads();

    for (int t = tid; t < TL::NP; t += NT) {
        int m, q;
        if (t < BX + 1) { m = 1; q = 2 + t; }
        else if (t < 2 * BX + 3) { m = 2; q = 1 + (t - BX - 1); }
        else { m = 3; q = t - 2 * BX - 3; }
        const int l = q, r = l + m;
        const float nx = 0.5f * (S[G_N1X * NB + l] + S[G_N1X * NB + r]);
        const float xt = 0.5f * (S[G_XT1 * NB + l] + S[G_XT1 * NB + r]);
        float f[NC];
        pair_flux_f(S, NB, l, r, nx, xt, G, f);
#pragma unroll
        for (int c = 0; c < NC; ++c) PB[c * TL::NP + t] = f[c];
    }
    if (P.diss) {
        // neighbour jumps V_{q+1} - V_q, q = 0 .. BX+4 (eq. jumpV); in a tile whose pairs leave enough threads, on the
        // warps after the pairs'
        constexpr int JOFF = (TL::NP + 31) / 32 * 32 + TL::NJ <= NT ? (TL::NP + 31) / 32 * 32 : 0;
        for (int t = JOFF ? (tid + NT - JOFF) % NT : tid; t < TL::NJ; t += NT) {
            float dV[NC];
            entropy_jump(S, NB, t, t + 1, G, dV);
#pragma unroll
            for (int c = 0; c < NC; ++c) JB[c * TL::NJ + t] = dV[c];
        }
    }
    __syncthreads();
    for (int t = tid; t < TL::NF; t += NT) {
        const int q = 2 + t;
        float F[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) F[c] = 0.0f;
        float FJ = 0.0f;
#pragma unroll
        for (int m = 1; m <= 3; ++m) {
            const int off = m == 1 ? 0 : (m == 2 ? BX + 1 : 2 * BX + 3);
            const float al = float(ec_alpha(m));
            for (int s = 0; s < m; ++s) {
                const int qq = q - s;
                const int pi = off + (qq - (3 - m));
#pragma unroll
                for (int c = 0; c < NC; ++c) F[c] += al * PB[c * TL::NP + pi];
                FJ += al * 0.5f * (S[G_XT1 * NB + qq] + S[G_XT1 * NB + qq + m]);
            }
        }
        bool jump = P.diss;
        if (P.diss) {
            // between two nodes of equal state no wave has a jump and the dissipation is zero whatever the rest of
            // the stencil (eq. sign switch): most faces of a tube whose waves have not reached its ends.  The face
            // state's own check is then the node's.
            const float* jl = JB + q;
            jump = jl[0] != 0.0f || jl[TL::NJ] != 0.0f || jl[2 * TL::NJ] != 0.0f;
            if (!jump) {
                const float RT = G.R * S[G_T * NB + q], ar = 2.0f * G.a * S[G_RHO * NB + q];
                const float om = S[G_OM * NB + q], iom = S[G_IOM * NB + q];
                if (!((1.0f + G.delta) * RT * iom * iom > ar) || !(RT > ar * om * om))
                    raise_error(P.status, ES_ERR_INADMISSIBLE, 0);
            }
        }
        if (jump) {
            const float nx = 0.5f * (S[G_N1X * NB + q] + S[G_N1X * NB + q + 1]);
            const float xtf = 0.5f * (S[G_XT1 * NB + q] + S[G_XT1 * NB + q + 1]);
            float d[NC];
            face_dissipation_f(S, NB, q, nx, xtf, G, Wc, d, P.status, JB, TL::NJ, q);
#pragma unroll
            for (int c = 0; c < NC; ++c) F[c] += d[c];
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) FB[c * TL::NF + t] = F[c];
        FB[NC * TL::NF + t] = FJ;
    }
    __syncthreads();
    float acc[NC + 1];
#pragma unroll
    for (int c = 0; c <= NC; ++c) acc[c] = 0.0f;
    if (tid < BX) {
        const float inv = P.finv_dxi[0];
#pragma unroll
        for (int c = 0; c <= NC; ++c) acc[c] -= (FB[c * TL::NF + tid + 1] - FB[c * TL::NF + tid]) * inv;
    }
    __syncthreads();

    const int gi = i0 + tid;
    if (tid < BX && gi < P.n1) {
        const size_t N = P.fcs;
        const size_t idx = size_t(gi);
        const size_t LO = P.fps;
        if (P.mode == 1) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                P.fJUo[c * N + idx] = acc[c];
                P.fJUo[LO + c * N + idx] = 0.0f;
            }
            P.fJo[idx] = acc[NC];
            P.fJo[P.fpsJ + idx] = 0.0f;
        } else {
            // a_s U^n + b_s (U^s + dt L) in double-float (a_s, b_s are 0, 1, 3/4, 1/4, 1/3, 2/3)
            const float ca = P.fca, cb = P.fcb;
            const float ca_lo = P.fca_lo, cb_lo = P.fcb_lo;
            // all operands loaded before the first store: as far as the compiler knows a store may alias a
            // later load, which would serialise one round trip per component
            df Un[NC + 1], Us[NC + 1];
#pragma unroll
            for (int c = 0; c <= NC; ++c) {
                const float* un = c < NC ? P.fJUn + c * N : P.fJn;
                const float* us = c < NC ? P.fJUs + c * N : P.fJs;
                const size_t lo = c < NC ? LO : P.fpsJ;
                Us[c] = {us[idx], us[lo + idx]};
                Un[c] = ca != 0.0f ? df{un[idx], un[lo + idx]} : df{0.0f, 0.0f};
            }
#pragma unroll
            for (int c = 0; c <= NC; ++c) {
                float* uo = c < NC ? P.fJUo + c * N : P.fJo;
                const size_t lo = c < NC ? LO : P.fpsJ;
                const df inc = df_add_f(Us[c], dt * acc[c]);
                df outv = df_mul(inc, {cb, cb_lo});
                if (ca != 0.0f) outv = df_add(outv, df_mul(Un[c], {ca, ca_lo}));
                uo[idx] = outv.hi;
                uo[lo + idx] = outv.lo;
                if (c == NC && !(outv.hi > 0.0f)) raise_error(P.status, ES_ERR_MESH, int(idx));
            }
        }
    }
}

// float copies of the gas and WENO constants of a launch
__device__ __forceinline__ GasF gas_f(const StageParams& P) {
    GasF G;
    G.a = P.fgas[0];
    G.b = P.fgas[1];
    G.R = P.fgas[2];
    G.cv = P.fgas[3];
    G.delta = P.fgas[4];
    G.Rb = P.fgas[5];
    G.icv = P.fgas[6];
    G.iR = P.fgas[7];
    G.idelta = P.fgas[8];
    return G;
}

__device__ __forceinline__ WenoF weno_f(const StageParams& P) {
    WenoF W;
    W.g1 = P.fweno[0];
    W.g2 = P.fweno[1];
    W.g3 = P.fweno[2];
    W.g12 = P.fweno[3];
    W.ig22 = P.fweno[4];
    W.ig3 = P.fweno[5];
    W.eps = P.fweno[6];
    W.sign_tol = P.fweno[7];
    return W;
}

}  // namespace mixed
}  // namespace es
