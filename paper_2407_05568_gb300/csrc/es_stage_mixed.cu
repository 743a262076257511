// es_stage_mixed.cu -- the fused operator + SSP-RK3 stage in the mixed-precision form.
//
// GB300 runs FP32 about 70 times faster than FP64 (2 FP64 FMA lanes per SM per
// clock), and an FP64 -> FP32 conversion costs as much as an FP64 FMA.  This
// form therefore keeps the per-stage work entirely on the FP32 pipe:
//   * the state JU, J is stored as compensated pairs of floats (hi, lo), value
//     hi + lo with a 48-bit significand, in two planes [2][...] (hi plane first);
//     the primitive state (rho, v, T) and the RK combination are evaluated in
//     double-float arithmetic (error-free sums and products built from FP32
//     FMA), so the jumps of rho, v and T between neighbouring nodes keep their
//     digits even where they are far below the FP32 resolution of the values
//     (near smooth extrema); everything else is plain FP32 on the hi parts;
//   * the mesh enters as an FP32 displacement d = x - (x_00 + i dxi_1, y_00 + j dxi_2)
//     and an FP32 mesh velocity, converted from the FP64 mesh once per step, so
//     the metric differences delta_k[x] = dxi_k e_k + delta_k[d] lose no digits;
//   * logarithmic means are taken per pair from the relative jump
//     f = (a_l - a_r)/(a_l + a_r) (a series for |f| < 0.2 in 2D and 3D, es_flux32.cuh,
//     and 0.05 in 1D, the logarithm otherwise), which is accurate to FP32 rounding of
//     the result even for nearly equal states;
//   * the entropy variables never appear as absolute values (V_1 is O(c_v) =
//     O(200) and its jumps are O(h)): the dissipation works on the jumps
//     V_j - V_i written exactly as the jump decomposition of Sec. 3.1
//     (eq. jumpV, general units), and MR-WENO5 is applied to W_j - W_i, which
//     it reconstructs exactly as it would W_j (the reconstruction commutes with
//     adding a constant).
// What stays FP64 is the once-per-step mesh conversion and the mesh
// redistribution kernels.
#include <cuda_runtime.h>

#include "es_flux32.cuh"
#include "es_mixed_device.cuh"

namespace es {

namespace {

using namespace mixed;

// ------------------------------------------------------------ 2D tile
// Shared memory of a tile: a box with a 3-node halo.  Node values that are read together lie in one float4, so that a
// pair or face takes a node in a few 16-byte loads; the box's row pitch is odd, which spreads the 16-byte columns of a
// xi_2 line over the banks as it does those of a xi_1 line.
template <int BX, int BY, int NT>
struct Tile2 {
    static constexpr int GX = (BX + 6) | 1;                  // row pitch
    static constexpr int GY = BY + 6;
    static constexpr int NB = GX * GY;
    static constexpr int NP1 = BY * (3 * BX + 6), NP2 = BX * (3 * BY + 6), NP = NP1 > NP2 ? NP1 : NP2;
    static constexpr int NJ1 = BY * (BX + 5), NJ2 = BX * (BY + 5), NJ = NJ1 > NJ2 ? NJ1 : NJ2;
    static constexpr int NF1 = BY * (BX + 1), NF2 = BX * (BY + 1), NF = NF1 > NF2 ? NF1 : NF2;
    // float4: (rho, T, 1/(1 - b rho), E0), (v1, v2, v1/T, v2/T), (rho v1, rho v2, g, a rho/T), (low rho, low T, 1/T, rho/p),
    // (n1, n2 of xi_1, n1, n2 of xi_2); float2: (low v1, low v2), (J xi_t of xi_1, xi_2); halves but 1/(1 - b rho), 1/T
    static constexpr int NODE_FLOATS = 5 * 4 + 2 * 2;
    static constexpr int PAIR_FLOATS = 4 * NP > 4 * NB ? 4 * NP : 4 * NB;      // also holds the coordinates
    static constexpr size_t SMEM = sizeof(float) * (size_t(NODE_FLOATS) * NB + PAIR_FLOATS + 4 * NJ + 5 * NF);
    static_assert(NT >= BX * BY && NT % 32 == 0, "threads cover the tile");
};

struct TileViews {
    float4 *a, *b, *c, *l, *n, *pairs, *jumps, *faces;
    float2 *vl, *xt;
    float* facesJ;
};
template <class TL>
__device__ __forceinline__ TileViews views(float* sm) {
    TileViews v;
    float4* q = reinterpret_cast<float4*>(sm);
    v.a = q;
    v.b = q + TL::NB;
    v.c = q + 2 * TL::NB;
    v.l = q + 3 * TL::NB;
    v.n = q + 4 * TL::NB;
    v.pairs = q + 5 * TL::NB;
    v.jumps = v.pairs + TL::PAIR_FLOATS / 4;
    v.faces = v.jumps + TL::NJ;
    v.vl = reinterpret_cast<float2*>(v.faces + TL::NF);
    v.xt = v.vl + TL::NB;
    v.facesJ = reinterpret_cast<float*>(v.xt + TL::NB);
    return v;
}

__device__ __forceinline__ flux32::Node<2> node_at(const TileViews& v, int q) {
    const float4 a = v.a[q], b = v.b[q], c = v.c[q];
    flux32::Node<2> n;
    n.rho = a.x;
    n.T = a.y;
    n.iom = a.z;
    n.E0 = a.w;
    n.v[0] = b.x;
    n.v[1] = b.y;
    n.vT[0] = b.z;
    n.vT[1] = b.w;
    n.rv[0] = c.x;
    n.rv[1] = c.y;
    n.g = c.z;
    n.art = c.w;
    return n;
}
__device__ __forceinline__ flux32::NodeLow<2> low_at(const TileViews& v, int q) {
    const float4 l = v.l[q];
    const float2 w = v.vl[q];
    flux32::NodeLow<2> n;
    n.rho = l.x;
    n.T = l.y;
    n.iT = l.z;
    n.v[0] = w.x;
    n.v[1] = w.y;
    return n;
}

// node (gi, gj) of the state into box position b: the primitive state in double-float arithmetic, the rest in float
__device__ __forceinline__ void load_node2(const TileViews& tv, int b, const StageParams& P, const GasF& G, int gi,
                                           int gj) {
    const int idx = state_index(gj, P.n2, P.bc[1]) * P.n1 + state_index(gi, P.n1, P.bc[0]);
    const size_t N = P.fcs, LO = P.fps;
    const df iJ = df_recip({P.fJs[idx], P.fJs[P.fpsJ + idx]});
    const df rho = df_mul({P.fJUs[idx], P.fJUs[LO + idx]}, iJ);
    const df m1 = df_mul({P.fJUs[N + idx], P.fJUs[LO + N + idx]}, iJ);
    const df m2 = df_mul({P.fJUs[2 * N + idx], P.fJUs[LO + 2 * N + idx]}, iJ);
    const df E = df_mul({P.fJUs[3 * N + idx], P.fJUs[LO + 3 * N + idx]}, iJ);
    const df irho = df_recip(rho);
    const df v1 = df_mul(m1, irho), v2 = df_mul(m2, irho);
    const df ke = df_mul_f(df_add(df_mul(v1, v1), df_mul(v2, v2)), 0.5f);
    // T = (E/rho - |v|^2/2 + a rho) / cv
    const df e = df_add(df_mul(E, irho), {-ke.hi, -ke.lo});
    const df Td = df_mul_f(df_add(e, df_mul_f(rho, G.a)), G.icv);
    const float r = rho.hi, T = Td.hi;
    const float om = 1.0f - G.b * r;
    const float iom = flux32::rcp(om), iT = flux32::rcp(T);
    const float ar = G.a * r;
    const float prho = G.R * T * iom - ar;                   // p/rho
    // R T - 2 a rho (1 - b rho)^2 > 0 enters through the face states
    if (!(r > 0.0f) || !(om > 0.0f) || !(T > 0.0f) || !(prho > 0.0f)) raise_error(P.status, ES_ERR_INADMISSIBLE, idx);
    const float hiT = 0.5f * iT, art = ar * hiT;             // a rho/(2T)
    tv.a[b] = make_float4(0.5f * r, 0.5f * T, iom, fmaf(ke.hi, hiT, 2.0f * art));
    tv.b[b] = make_float4(0.5f * v1.hi, 0.5f * v2.hi, v1.hi * hiT, v2.hi * hiT);
    tv.c[b] = make_float4(0.5f * m1.hi, 0.5f * m2.hi, fmaf(0.5f * G.R, iom, -art), art);
    tv.l[b] = make_float4(0.5f * rho.lo, 0.5f * Td.lo, iT, 0.5f * flux32::rcp(prho));
    tv.vl[b] = make_float2(0.5f * v1.lo, 0.5f * v2.lo);
}

// geometry of direction k in the box: first node of a line, node step, metrics
template <int GX>
__device__ __forceinline__ int line_base(int k, int line) {
    return k == 0 ? (3 + line) * GX : 3 + line;
}
__device__ __forceinline__ float2 normal_at(const TileViews& v, int k, int q) {
    return reinterpret_cast<const float2*>(v.n)[2 * q + k];
}
__device__ __forceinline__ float xt_at(const TileViews& v, int k, int q) {
    return reinterpret_cast<const float*>(v.xt)[2 * q + k];
}

// The tile of nodes at (i0, j0): the box is staged in shared memory, then per direction the pairs (by their reach m: those
// with m = 1 also give the neighbour jumps of the entropy variables), the faces and the divergence, and the Shu-Osher
// combination.  SPLIT: two lanes of a warp share a face, lane 0 the u - c and entropy waves, lane 1 the u + c and shear
// waves, each its own reconstructions and sign switch, for tiles with twice the threads of their faces.
template <int BX, int BY, int NT, bool SPLIT>
__device__ __forceinline__ void stage_tile2(float* smemf, const StageParams& P, int i0, int j0, float dt, const GasF& G,
                                            const flux32::WenoC& Wc) {
    using TL = Tile2<BX, BY, NT>;
    constexpr int GX = TL::GX, NB = TL::NB;
    const TileViews tv = views<TL>(smemf);
    const int tid = threadIdx.x;
    const float cdt = P.fcst * dt;
    const float idx1 = P.finv_dxi[0], idx2 = P.finv_dxi[1];
    float* XS = reinterpret_cast<float*>(tv.pairs);          // displacement and mesh velocity, two components each
    float* XD = XS + 2 * NB;
    for (int t = tid; t < (BX + 6) * TL::GY; t += NT) {
        const int ii = t % (BX + 6), jj = t / (BX + 6);
        const int b = jj * GX + ii;
        const int gi = i0 - 3 + ii, gj = j0 - 3 + jj;
        float ds[2], xd[2];
        stage_disp<2>(P, gi, gj, cdt, ds, xd);
        XS[b] = ds[0];
        XD[b] = xd[0];
        XS[NB + b] = ds[1];
        XD[NB + b] = xd[1];
        if ((ii >= 3 && ii < 3 + BX) || (jj >= 3 && jj < 3 + BY)) load_node2(tv, b, P, G, gi, gj);
    }
    __syncthreads();
    for (int t = tid; t < (BX + 6) * TL::GY; t += NT) {
        const int ii = t % (BX + 6), jj = t / (BX + 6);
        const int b = jj * GX + ii;
        float4 n = make_float4(0.5f, 0.0f, 0.0f, 0.5f);
        float2 x = make_float2(0.0f, 0.0f);
        // 6th-order differences: h_m = alpha_m/2, and half the metrics
        constexpr float h1 = 0.75f, h2 = -0.15f, h3 = 1.0f / 60.0f;
        auto diff = [&](const float* f, int s) {
            return fmaf(h1, f[s] - f[-s], fmaf(h2, f[2 * s] - f[-2 * s], h3 * (f[3 * s] - f[-3 * s])));
        };
        if (jj >= 3 && jj < 3 + BY) {            // J dxi_1/dx = (1 + d2[d_y]/dxi_2, -d2[d_x]/dxi_2)
            n.x = fmaf(0.5f * idx2, diff(XS + NB + b, GX), 0.5f);
            n.y = -0.5f * idx2 * diff(XS + b, GX);
            x.x = -fmaf(XD[b], n.x, XD[NB + b] * n.y);
        }
        if (ii >= 3 && ii < 3 + BX) {            // J dxi_2/dx = (-d1[d_y]/dxi_1, 1 + d1[d_x]/dxi_1)
            n.z = -0.5f * idx1 * diff(XS + NB + b, 1);
            n.w = fmaf(0.5f * idx1, diff(XS + b, 1), 0.5f);
            x.y = -fmaf(XD[b], n.z, XD[NB + b] * n.w);
        }
        tv.n[b] = n;
        tv.xt[b] = x;
    }
    __syncthreads();

    float acc[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    const int tx = tid % BX, ty = tid / BX;
    // one copy of the direction pipeline for both directions (its code is fetched once)
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const int nlines = k == 0 ? BY : BX, LB = k == 0 ? BX : BY, step = k == 0 ? 1 : GX;
        const int per_line = 3 * LB + 6;
        const int c1 = nlines * (LB + 5), c2 = c1 + nlines * (LB + 2), c3 = c2 + nlines * (LB + 3);
        for (int t = tid; t < c3; t += NT) {
            const int m = t < c1 ? 1 : (t < c2 ? 2 : 3);
            const int u = m == 1 ? t : (m == 2 ? t - c1 : t - c2);
            // (division by constants)
            const int line = m == 1 ? (k == 0 ? u / (BX + 5) : u / (BY + 5))
                                    : (m == 2 ? (k == 0 ? u / (BX + 2) : u / (BY + 2))
                                              : (k == 0 ? u / (BX + 3) : u / (BY + 3)));
            const int pos = u - line * (LB + (m == 1 ? 5 : m));
            const int q = m == 2 ? pos + 1 : pos;
            const int l = line_base<GX>(k, line) + q * step, r = l + m * step;
            const flux32::Node<2> nl = node_at(tv, l), nr = node_at(tv, r);
            const flux32::PairMeans<2> p = flux32::pair_means<2>(nl, nr, G);
            float f[4];
            if (m == 1) {
                flux32::entropy_jump<2>(nl, nr, low_at(tv, l), low_at(tv, r), p, f);
                tv.jumps[u] = make_float4(f[0], f[1], f[2], f[3]);
                if (q < 2 || q > LB + 2) continue;
            }
            const float2 a = normal_at(tv, k, l), b = normal_at(tv, k, r);
            const float n[2] = {a.x + b.x, a.y + b.y};
            flux32::pair_flux<2>(nl, nr, p, n, xt_at(tv, k, l) + xt_at(tv, k, r), f);
            tv.pairs[line * per_line + (m == 1 ? q - 2 : (m == 2 ? LB + 1 : 2 * LB + 3) + pos)] =
                make_float4(f[0], f[1], f[2], f[3]);
        }
        __syncthreads();
        const int nfaces = nlines * (LB + 1);
        const int lane = tid & 31;
        // SPLIT: lanes (2 p, 2 p + 1) share face p; the trip count is uniform per warp (the halves exchange
        // values), and a lane past the last face works on the last face and stores nothing
        for (int ub = SPLIT ? tid - lane : tid; ub < (SPLIT ? 2 * nfaces : nfaces); ub += NT) {
            const int u = SPLIT ? ub + lane : ub;
            const bool active = !SPLIT || u < 2 * nfaces;
            const int t = SPLIT ? (active ? (u >> 1) : nfaces - 1) : u;
            const bool second = SPLIT && (u & 1);
            const int line = k == 0 ? t / (BX + 1) : t / (BY + 1);
            const int q = 2 + t - line * (LB + 1);
            const int l = line_base<GX>(k, line) + q * step, r = l + step;
            // the 6th-order combination of the pairs (the energy component is a quarter)
            float F[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            {
                const float4* pb = tv.pairs + line * per_line + q;
                const int o2 = LB + 1 - 1, o3 = 2 * LB + 3;      // pairs of reach m start at q = 3 - m
                const float4 p1 = pb[-2], p2a = pb[o2 - 1], p2b = pb[o2], p3a = pb[o3 - 2], p3b = pb[o3 - 1], p3c = pb[o3];
                constexpr float a1 = 1.5f, a2 = -0.3f, a3 = 1.0f / 30.0f;
                F[0] = fmaf(a1, p1.x, fmaf(a2, p2a.x + p2b.x, a3 * (p3a.x + p3b.x + p3c.x)));
                F[1] = fmaf(a1, p1.y, fmaf(a2, p2a.y + p2b.y, a3 * (p3a.y + p3b.y + p3c.y)));
                F[2] = fmaf(a1, p1.z, fmaf(a2, p2a.z + p2b.z, a3 * (p3a.z + p3b.z + p3c.z)));
                F[3] = 4.0f * fmaf(a1, p1.w, fmaf(a2, p2a.w + p2b.w, a3 * (p3a.w + p3b.w + p3c.w)));
            }
            const float xl = xt_at(tv, k, l), xr = xt_at(tv, k, r);
            // sum_m alpha_m sum of the pairs' mean J xi_t, collected by node
            constexpr float b3 = 1.0f / 30.0f, b2 = -0.3f + b3, b1 = 1.5f + b2;
            const float FJ = fmaf(b1, xl + xr, fmaf(b2, xt_at(tv, k, l - step) + xt_at(tv, k, r + step),
                                                    b3 * (xt_at(tv, k, l - 2 * step) + xt_at(tv, k, r + 2 * step))));
            if (P.diss) {
                const float2 na = normal_at(tv, k, l), nb = normal_at(tv, k, r);
                const float n[2] = {na.x + nb.x, na.y + nb.y};
                const float4 vl = tv.b[l], vr = tv.b[r];
                const float v[2] = {vl.x + vr.x, vl.y + vr.y};
                const flux32::Face<2> f =
                    flux32::face_state<2>(tv.a[l].x, tv.a[r].x, tv.l[l].w, tv.l[r].w, v, n, xl + xr, G, P.status);
                float y[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                const float4* jb = tv.jumps + line * (LB + 5) + q - 2;
                if constexpr (SPLIT) {
                    float Wa[5], Wb[5], sz[4];
                    const float sc = second ? f.sAc : -f.sAc, Sb = second ? f.sT : f.sE, Db = second ? f.vr[1] : -f.hm;
#pragma unroll
                    for (int o = 0; o < 5; ++o) {
                        const float4 j = jb[o];
                        const float d[4] = {j.x, j.y, j.z, j.w};
                        const flux32::Rotated<2> R = flux32::rotate<2>(f, d);
                        Wa[o] = fmaf(sc, R.B, f.sA * R.A);
                        Wb[o] = Sb * fmaf(Db, d[3], second ? R.rv[1] : R.A);
                        if (o == 2) flux32::term_sizes<2>(f, d, R, sz);
                    }
                    float ya = 0.0f, yb = 0.0f;
                    if (!(fabsf(Wa[2]) <= Wc.tol * (f.sA * (second ? sz[3] : sz[0])))) ya = flux32::weno_jump(Wa, Wc);
                    if (!(fabsf(Wb[2]) <= Wc.tol * (Sb * (second ? sz[2] : sz[1])))) yb = flux32::weno_jump(Wb, Wc);
                    const float oa = __shfl_xor_sync(0xffffffffu, ya, 1), ob = __shfl_xor_sync(0xffffffffu, yb, 1);
                    y[0] = second ? oa : ya;
                    y[1] = second ? ob : yb;
                    y[2] = second ? yb : ob;
                    y[3] = second ? ya : oa;
                } else {
                    float W[4][5], sz[4];
#pragma unroll
                    for (int o = 0; o < 5; ++o) {
                        const float4 j = jb[o];
                        const float d[4] = {j.x, j.y, j.z, j.w};
                        const flux32::Rotated<2> R = flux32::rotate<2>(f, d);
                        const float sa = f.sA * R.A;
                        W[0][o] = fmaf(-f.sAc, R.B, sa);
                        W[1][o] = f.sE * fmaf(-f.hm, d[3], R.A);
                        W[2][o] = f.sT * fmaf(f.vr[1], d[3], R.rv[1]);
                        W[3][o] = fmaf(f.sAc, R.B, sa);
                        if (o == 2) flux32::term_sizes<2>(f, d, R, sz);
                    }
                    // a wave whose plain jump is round-off adds nothing whatever its reconstruction
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float S = m == 1 ? f.sE : (m == 2 ? f.sT : f.sA);
                        if (!(fabsf(W[m][2]) <= Wc.tol * (S * sz[m]))) y[m] = flux32::weno_jump(W[m], Wc);
                    }
                }
                flux32::add_increment<2>(f, y, F);
            }
            if (active && !second) {
                tv.faces[t] = make_float4(F[0], F[1], F[2], F[3]);
                tv.facesJ[t] = FJ;
            }
        }
        __syncthreads();
        if (tid < BX * BY) {
            const int fm = (k == 0 ? ty : tx) * (LB + 1) + (k == 0 ? tx : ty);
            const float inv = k == 0 ? idx1 : idx2;
            const float4 a = tv.faces[fm], b = tv.faces[fm + 1];
            acc[0] = fmaf(a.x - b.x, inv, acc[0]);
            acc[1] = fmaf(a.y - b.y, inv, acc[1]);
            acc[2] = fmaf(a.z - b.z, inv, acc[2]);
            acc[3] = fmaf(a.w - b.w, inv, acc[3]);
            acc[4] = fmaf(tv.facesJ[fm] - tv.facesJ[fm + 1], inv, acc[4]);
        }
        // (the next direction's pairs and jumps are not read here, and its faces are written after a barrier)
    }

    const int gi = i0 + tx, gj = j0 + ty;
    if (tid >= BX * BY || gi >= P.n1 || gj >= P.n2) return;
    const size_t N = P.fcs, idx = size_t(gj) * P.n1 + gi, LO = P.fps;
    if (P.mode == 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            P.fJUo[c * N + idx] = acc[c];
            P.fJUo[LO + c * N + idx] = 0.0f;
        }
        P.fJo[idx] = acc[4];
        P.fJo[P.fpsJ + idx] = 0.0f;
        return;
    }
    // a_s U^n + b_s (U^s + dt L) in double-float (a_s, b_s are 0, 1, 3/4, 1/4, 1/3, 2/3); all operands loaded before the
    // first store (as far as the compiler knows a store may alias a later load)
    const float ca = P.fca, cb = P.fcb;
    df Un[5], Us[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const float* un = c < 4 ? P.fJUn + c * N : P.fJn;
        const float* us = c < 4 ? P.fJUs + c * N : P.fJs;
        const size_t lo = c < 4 ? LO : P.fpsJ;
        Us[c] = {us[idx], us[lo + idx]};
        Un[c] = ca != 0.0f ? df{un[idx], un[lo + idx]} : df{0.0f, 0.0f};
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        float* uo = c < 4 ? P.fJUo + c * N : P.fJo;
        const size_t lo = c < 4 ? LO : P.fpsJ;
        df v = df_mul(df_add_f(Us[c], dt * acc[c]), {cb, P.fcb_lo});
        if (ca != 0.0f) v = df_add(v, df_mul(Un[c], {ca, P.fca_lo}));
        uo[idx] = v.hi;
        uo[lo + idx] = v.lo;
        if (c == 4 && !(v.hi > 0.0f)) raise_error(P.status, ES_ERR_MESH, int(idx));
    }
}

// resident CTAs per SM the register allocation must allow: 5 x 160 or 4 x 192 threads, 2 x 384 (two lanes per face), 1 x 608
template <int BX, int BY, int NT, bool SPLIT>
__global__ void __launch_bounds__(NT, NT <= 160 ? 5 : (NT <= 192 ? 4 : (NT <= 384 ? 2 : 1)))
    stage_kernel_mixed2(StageParams P) {
    extern __shared__ float4 smem4[];
    const int ntx = (P.n1 + BX - 1) / BX;
    const int i0 = (blockIdx.x % ntx) * BX, j0 = (blockIdx.x / ntx) * BY;
    const double dtd = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && dtd == 0.0) return;               // finished run: leave the state untouched
    flux32::WenoC W;
    W.h1 = P.fwc[0];
    W.h2 = P.fwc[1];
    W.q2 = P.fwc[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) W.q3[k] = P.fwc[3 + k];
    W.eps4 = P.fwc[7];
    W.tol = P.fwc[8];
    stage_tile2<BX, BY, NT, SPLIT>(reinterpret_cast<float*>(smem4), P, i0, j0, float(dtd), gas_f(P), W);
}

template <int BX, int NT>
__global__ void __launch_bounds__(NT, 2) stage_kernel_mixed1(StageParams P) {
    extern __shared__ float smemf[];
    const double dtd = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && dtd == 0.0) return;
    stage_tile_mixed<BX, NT>(smemf, P, blockIdx.x * BX, float(dtd), gas_f(P), weno_f(P));
}

template <int BX, int BY, int NT, bool SPLIT = false>
cudaError_t prepare_tile_f() {
    return cudaFuncSetAttribute(stage_kernel_mixed2<BX, BY, NT, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(Tile2<BX, BY, NT>::SMEM));
}

template <int BX, int BY, int NT, bool SPLIT = false>
cudaError_t launch_tile_f(const StageParams& P, cudaStream_t s) {
    const int tiles = (P.n1 + BX - 1) / BX * ((P.n2 + BY - 1) / BY);
    stage_kernel_mixed2<BX, BY, NT, SPLIT><<<tiles, NT, Tile2<BX, BY, NT>::SMEM, s>>>(P);
    return cudaGetLastError();
}

// 1D tiles: 254 nodes, a node per thread, or 58 with the same 256 threads, one thread per pair or jump, for lines that the
// smaller tiles cover in one wave of two CTAs per SM: there a stage is the length of one tile's dependent phases, which
// take three rounds of pairs and two of jumps with 254 nodes.  Stages of 40 to 17632 nodes, launch to launch: 8.3 -> 6.3 us,
// the same bits; a second wave would bring the short tile to 8.3, where the other stays up to 30000 nodes.
constexpr int LINE_BX = 254, SHORT_BX = 58, LINE_NT = 256;
using LineTile = TileF<LINE_BX, LINE_NT>;
using ShortTile = TileF<SHORT_BX, LINE_NT>;

}  // namespace

// 2D shapes: 20 x 8 nodes with 384 threads, two lanes per face (twice the warps of the 192-thread
// shape: small meshes are latency bound), 25 x 6 with 192 (175 faces; 8 x 34 = 272 tiles fill
// 200 x 200 at two CTAs per SM in one wave), 20 x 8 with 192 (180 faces), 20 x 14 with 608, two lanes
// per face (10 x 15 = 150 tiles: one CTA on each SM at 200 x 200, less halo per node), and 16 x 8 with 160
// (more CTAs for small meshes)
cudaError_t stage_prepare_mixed(int dim) {
    if (dim == 1)
        return cudaFuncSetAttribute(stage_kernel_mixed1<LINE_BX, LINE_NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    int(LineTile::SMEM));      // (the short tile's 11 KB need no attribute)
    cudaError_t e = prepare_tile_f<20, 8, 384, true>();
    if (e == cudaSuccess) e = prepare_tile_f<25, 6, 192>();
    if (e == cudaSuccess) e = prepare_tile_f<20, 8, 192>();
    if (e == cudaSuccess) e = prepare_tile_f<20, 14, 608, true>();
    if (e == cudaSuccess) e = prepare_tile_f<16, 8, 160>();
    return e;
}

cudaError_t launch_stage_mixed(const StageParams& P, int nsm, cudaStream_t s) {
    if (P.dim == 1) {
        if (P.n1 <= 2 * nsm * SHORT_BX)
            stage_kernel_mixed1<SHORT_BX, LINE_NT><<<(P.n1 + SHORT_BX - 1) / SHORT_BX, LINE_NT, ShortTile::SMEM, s>>>(P);
        else
            stage_kernel_mixed1<LINE_BX, LINE_NT><<<(P.n1 + LINE_BX - 1) / LINE_BX, LINE_NT, LineTile::SMEM, s>>>(P);
        return cudaGetLastError();
    }
    switch (P.tile) {
        case 1: return launch_tile_f<25, 6, 192>(P, s);
        case 2: return launch_tile_f<20, 8, 192>(P, s);
        case 3: return launch_tile_f<20, 14, 608, true>(P, s);
        case 4: return launch_tile_f<16, 8, 160>(P, s);
        default: return launch_tile_f<20, 8, 384, true>(P, s);
    }
}

}  // namespace es
