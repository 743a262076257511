// es_stage.cu -- fused semi-discrete ES operator + SSP-RK3 stage, FP64 form.
//
// One CTA owns a BX x BY tile of nodes (BY = 1 in 1D).  It stages a box with
// a 3-node halo in shared memory (the reach of the 6-point pair stencil and of
// WENO5), computes per node the primitive state, logarithms and entropy
// variables once, the metrics of the stage mesh (Sec. 3.2, eq. SCLCoeff and
// VCLCoeff), then per direction:
//   pair fluxes F(U_q, U_{q+m}), m = 1..3 (Sec. 3.1, eq. ECfluxMM), shared
//   by the faces that use them,
//   face fluxes = the 6th-order combination (eq. ECFlux_curv_2p, GCL_flux)
//   plus the ES dissipation (eq. HOstable) with MR-WENO5 on the scaled
//   entropy variables,
//   the divergence (eq. semi_U, semi_J),
// and finally the Shu-Osher SSP-RK3 combination.  Nothing but the inputs and
// the outputs touches global memory.
#include <cuda_runtime.h>

#include "es_device.cuh"
#include "es_flux64.cuh"
#include "es_internal.h"

namespace es {

// shared-memory field slots (each NB doubles): the node fields, then per direction half of the metrics and J xi_t
template <int DIM>
struct Slot {
    static constexpr int N1 = flux64::Slots<DIM>::COUNT;                // DIM metric components, then J xi_t
    static constexpr int N2 = N1 + DIM + 1;
    static constexpr int COUNT = DIM == 2 ? N2 + DIM + 1 : N2;
};

template <int DIM, int BX, int BY, int NT>
struct Tile {
    static constexpr int GX = BX + 6;
    static constexpr int GY = DIM == 2 ? BY + 6 : 1;
    static constexpr int NB = GX * GY;
    static constexpr int NC = DIM + 2;
    static constexpr int ROWP = 3 * BX + 6;                 // pairs per xi_1 line
    static constexpr int COLP = 3 * BY + 6;                 // pairs per xi_2 line
    static constexpr int NP1 = (DIM == 2 ? BY : 1) * ROWP;
    static constexpr int NP2 = DIM == 2 ? BX * COLP : 0;
    static constexpr int NP = NP1 > NP2 ? NP1 : NP2;
    static constexpr int NF1 = (DIM == 2 ? BY : 1) * (BX + 1);
    static constexpr int NF2 = DIM == 2 ? BX * (BY + 1) : 0;
    static constexpr int NF = NF1 > NF2 ? NF1 : NF2;
    // Joint schedule (2D, when shared memory allows): the pairs of both directions in one phase
    // and their faces in the next (two block barriers per stage instead of six, and the faces
    // dealt to the warps as one pool of NF1 + NF2).  Otherwise pairs and faces go direction by
    // direction.
    static constexpr size_t FIELDS = sizeof(double) * size_t(Slot<DIM>::COUNT) * NB;
    static constexpr int PAIRJ = ((NP1 + NP2) * NC > 4 * NB) ? (NP1 + NP2) * NC : 4 * NB;
    // entropy-variable jumps between neighbours along each line (box positions q, q + 1)
    static constexpr int NJ1 = (DIM == 2 ? BY : 1) * (BX + 5);
    static constexpr int NJ2 = DIM == 2 ? BX * (BY + 5) : 0;
    static constexpr size_t SMEM_JOINT =
        FIELDS + sizeof(double) * (size_t(PAIRJ) + size_t(NF1 + NF2) * (NC + 1) + size_t(NJ1 + NJ2) * NC);
    static constexpr bool JOINT = DIM == 2 && SMEM_JOINT <= 227 * 1024;
    // pair and face buffers: per-component strides and the offset of direction 2's entries
    static constexpr int PS = JOINT ? NP1 + NP2 : NP;
    static constexpr int FS = JOINT ? NF1 + NF2 : NF;
    static constexpr int JS = JOINT ? NJ1 + NJ2 : (NJ1 > NJ2 ? NJ1 : NJ2);
    static constexpr int POFF2 = JOINT ? NP1 : 0;
    static constexpr int FOFF2 = JOINT ? NF1 : 0;
    static constexpr int PAIR_DOUBLES = JOINT ? PAIRJ : ((NP * NC > 4 * NB) ? NP * NC : 4 * NB);   // also holds coords
    static constexpr size_t SMEM =
        FIELDS + sizeof(double) * (size_t(PAIR_DOUBLES) + size_t(FS) * (NC + 1) + size_t(JS) * NC);
    static constexpr int THREADS = NT;
    static_assert(NT >= BX * (DIM == 2 ? BY : 1) && NT % 32 == 0, "threads cover the tile");
};

// ----------------------------------------------------------- node loader
template <int DIM>
__device__ __forceinline__ void load_node(double* S, int NB, int b, const StageParams& P, int gi, int gj) {
    const int si = state_index(gi, P.n1, P.bc[0]);
    const int sj = DIM == 2 ? state_index(gj, P.n2, P.bc[1]) : 0;
    const int idx = sj * P.n1 + si;
    const size_t N = size_t(P.n1) * P.n2;
    double JU[DIM + 2];
#pragma unroll
    for (int c = 0; c < DIM + 2; ++c) JU[c] = P.JUs[c * N + idx];
    // at a wall or symmetry end the ghost is the mirror node with the normal momentum negated
    if ((gi < 0 || gi >= P.n1) && end_mirrored(P.bc[0], gi < 0)) JU[1] = -JU[1];
    if (DIM == 2 && (gj < 0 || gj >= P.n2) && end_mirrored(P.bc[1], gj < 0)) JU[DIM] = -JU[DIM];
    const bool ok = flux64::node_fields<DIM>(JU, P.Js[idx], P.gas, [&](int f, double v) { S[f * NB + b] = v; });
    if (!ok) raise_error(P.status, ES_ERR_INADMISSIBLE, idx);
}

// stage coordinates x^n + c dt xdot and mesh velocity at a possibly-ghost node
template <int DIM>
__device__ __forceinline__ void stage_coords(const StageParams& P, int gi, int gj, double cdt, double* xs,
                                             double* xd) {
    const size_t N = size_t(P.n1) * P.n2;
    // per component k: a wall or symmetry end mirrors the components along it (tangential) and
    // reflects the normal one; the other ends treat every component alike
    for (int k = 0; k < DIM; ++k) {
        const GhostTerms ti = ghost_terms(gi, P.n1, P.bc[0], k != 0);
        GhostTerms tj;
        if (DIM == 2) tj = ghost_terms(gj, P.n2, P.bc[1], k != 1);
        else { tj.idx[0] = 0; tj.w[0] = 1.0; tj.nterm = 1; tj.q = 0; }
        double as = 0.0, ad = 0.0;
        for (int a = 0; a < ti.nterm; ++a)
            for (int c = 0; c < tj.nterm; ++c) {
                const double w = ti.w[a] * tj.w[c];
                const size_t id = size_t(tj.idx[c]) * P.n1 + ti.idx[a];
                const double xdk = P.xdot ? P.xdot[k * N + id] : 0.0;
                as = fma(w, fma(cdt, xdk, P.xn[k * N + id]), as);
                ad = fma(w, xdk, ad);
            }
        const int per = k == 0 ? ti.q : tj.q;
        xs[k] = per != 0 ? fma(double(per), P.period[k], as) : as;
        xd[k] = ad;
    }
}

// geometry of direction k in the box: lines, interior nodes per line, pairs per line, node step
// and the metric slots
template <int DIM, int BX, int BY>
struct DirGeo {
    int k, nlines, LB, per_line, step, fN;       // fN: the slot of the direction's first metric component
    __device__ __forceinline__ explicit DirGeo(int kk) : k(kk) {
        nlines = k == 0 ? (DIM == 2 ? BY : 1) : BX;
        LB = k == 0 ? BX : BY;
        per_line = 3 * LB + 6;
        step = k == 0 ? 1 : BX + 6;
        fN = k == 0 ? Slot<DIM>::N1 : Slot<DIM>::N2;
    }
    __device__ __forceinline__ int base(int line) const {
        return k == 0 ? (DIM == 2 ? (3 + line) * (BX + 6) : 0) : 3 + line;
    }
};

// ---- C: pair flux P_m(q) = F(U_q, U_{q+m}), q = 3-m .. LB+2, item t of direction d; stored at
// PB[c * ps + out]
template <int DIM, int BX, int BY>
__device__ __forceinline__ void pair_item(const double* S, int NB, const DirGeo<DIM, BX, BY>& d, int t, const Gas& G,
                                          double* PB, int ps, int out) {
    const int line = t / d.per_line, kk = t % d.per_line;
    int m, q;
    if (kk < d.LB + 1) { m = 1; q = 2 + kk; }
    else if (kk < 2 * d.LB + 3) { m = 2; q = 1 + (kk - d.LB - 1); }
    else { m = 3; q = kk - 2 * d.LB - 3; }
    const int l = d.base(line) + q * d.step, r = l + m * d.step;
    double n[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) n[c] = S[(d.fN + c) * NB + l] + S[(d.fN + c) * NB + r];
    const double xt = S[(d.fN + DIM) * NB + l] + S[(d.fN + DIM) * NB + r];
    double f[DIM + 2];
    flux64::pair_flux<DIM>(S, NB, l, r, n, xt, G, f);
#pragma unroll
    for (int c = 0; c < DIM + 2; ++c) PB[c * ps + out] = f[c];
}
// the entropy variables' jump between box positions q and q + 1 of a line, q = 0 .. LB+4, item t; at JB[c * js + out]
template <int DIM, int BX, int BY>
__device__ __forceinline__ void jump_item(const double* S, int NB, const DirGeo<DIM, BX, BY>& d, int t, double* JB,
                                          int js, int out) {
    const int l = d.base(t / (d.LB + 5)) + t % (d.LB + 5) * d.step;
    double f[DIM + 2];
    flux64::entropy_jump<DIM>(S, NB, l, l + d.step, f);
#pragma unroll
    for (int c = 0; c < DIM + 2; ++c) JB[c * js + out] = f[c];
}

// ---- D: face flux at q+1/2, q = 2 .. LB+2 (box coordinates), item t of direction d: the 6th-order
// combination of the direction's pairs (which start at PB[c * ps + poff]) plus the dissipation;
// stored at FB[c * fs + out]
template <int DIM, int BX, int BY>
__device__ __forceinline__ void face_item(const double* S, int NB, const DirGeo<DIM, BX, BY>& d, int t,
                                          const StageParams& P, const double* PB, int ps, int poff, const double* JB,
                                          int js, int joff, double* FB, int fs, int out) {
    constexpr int NC = DIM + 2;
    const int line = t / (d.LB + 1), f = t % (d.LB + 1);
    const int q = 2 + f;
    const int pbase = poff + line * d.per_line;
    double F[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) F[c] = 0.0;
    const int base = d.base(line);
#pragma unroll
    for (int m = 1; m <= 3; ++m) {
        const int off = m == 1 ? 0 : (m == 2 ? d.LB + 1 : 2 * d.LB + 3);
        const double al = ec_alpha(m);
        for (int s = 0; s < m; ++s) {
            const int qq = q - s;                       // left node of the pair
            const int pi = pbase + off + (qq - (3 - m));
#pragma unroll
            for (int c = 0; c < NC; ++c) F[c] = fma(c == NC - 1 ? 4.0 * al : al, PB[c * ps + pi], F[c]);   // (a quarter of the energy)
        }
    }
    // sum_m alpha_m sum of the pairs' mean J xi_t, collected by node
    const double* XT = S + (d.fN + DIM) * NB + base + q * d.step;        // halves
    const double a3 = ec_alpha(3), a2 = ec_alpha(2) + a3, a1 = ec_alpha(1) + a2;
    const double FJ = fma(a1, XT[0] + XT[d.step],
                          fma(a2, XT[-d.step] + XT[2 * d.step], a3 * (XT[-2 * d.step] + XT[3 * d.step])));
    if (P.diss) {
        const int l = base + q * d.step, r = l + d.step;
        double n[DIM];
#pragma unroll
        for (int c = 0; c < DIM; ++c) n[c] = S[(d.fN + c) * NB + l] + S[(d.fN + c) * NB + r];
        flux64::face_dissipation<DIM>(S, NB, l, d.step, n, XT[0] + XT[d.step], P.gas, P.weno, JB, js,
                                      joff + line * (d.LB + 5) + q, F, P.status, 0);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) FB[c * fs + out] = F[c];
    FB[NC * fs + out] = FJ;
}

template <int DIM, int BX, int BY, int NT>
__global__ void __launch_bounds__(NT, 1)
stage_kernel_fp64(StageParams P) {
    using TL = Tile<DIM, BX, BY, NT>;
    constexpr int GX = TL::GX, NB = TL::NB, NC = TL::NC;
    extern __shared__ double smem[];
    double* S = smem;                                   // COUNT * NB
    double* PB = smem + Slot<DIM>::COUNT * NB;                   // pair buffer (also the coordinates)
    double* FB = PB + TL::PAIR_DOUBLES;                 // face buffer (NC + 1) * FS
    double* JB = FB + (NC + 1) * TL::FS;                // entropy-variable jumps NC * JS
    const int tid = threadIdx.x;
    const int ntx = (P.n1 + BX - 1) / BX;
    const int i0 = (blockIdx.x % ntx) * BX;
    const int j0 = DIM == 2 ? (blockIdx.x / ntx) * BY : 0;
    const double dt = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && dt == 0.0) return;               // finished run: leave the state untouched
    const double cdt = P.cst * dt;
    const Gas& G = P.gas;

    // ---- A: coordinates of the whole box, node data of the cross-shaped halo
    double* XS = PB;            // DIM * NB
    double* XD = PB + 2 * NB;   // DIM * NB
    for (int b = tid; b < NB; b += TL::THREADS) {
        const int ii = b % GX, jj = b / GX;
        const int gi = i0 - 3 + ii, gj = j0 - 3 + jj;
        double xs[2], xd[2];
        stage_coords<DIM>(P, gi, DIM == 2 ? gj : 0, cdt, xs, xd);
        XS[b] = xs[0];
        XD[b] = xd[0];
        if (DIM == 2) {
            XS[NB + b] = xs[1];
            XD[NB + b] = xd[1];
        }
        const bool in_x = ii >= 3 && ii < 3 + BX;
        const bool in_y = DIM == 1 || (jj >= 3 && jj < 3 + BY);
        if (in_x || in_y) load_node<DIM>(S, NB, b, P, gi, gj);
    }
    __syncthreads();

    // ---- B: metrics of the stage mesh (eq. SCLCoeff degenerate to 2D, eq. VCLCoeff)
    for (int b = tid; b < NB; b += TL::THREADS) {
        const int ii = b % GX, jj = b / GX;
        if (DIM == 1) {
            S[Slot<DIM>::N1 * NB + b] = 0.5;
            S[(Slot<DIM>::N1 + 1) * NB + b] = -0.5 * XD[b];
        } else {
            if (jj >= 3 && jj < 3 + BY) {          // xi_1 lines: J dxi_1/dx = (d2 y, -d2 x)/dxi_2
                double dy = 0.0, dx = 0.0;
#pragma unroll
                for (int m = 1; m <= 3; ++m) {
                    const double h = 0.5 * ec_alpha(m);
                    dx = fma(h, XS[b + m * GX] - XS[b - m * GX], dx);
                    dy = fma(h, XS[NB + b + m * GX] - XS[NB + b - m * GX], dy);
                }
                const double h = 0.5 * P.inv_dxi[1];
                const double nx = dy * h, ny = -dx * h;          // halves
                S[Slot<DIM>::N1 * NB + b] = nx;
                S[(Slot<DIM>::N1 + 1) * NB + b] = ny;
                S[(Slot<DIM>::N1 + 2) * NB + b] = -fma(XD[b], nx, XD[NB + b] * ny);
            }
            if (ii >= 3 && ii < 3 + BX) {          // xi_2 lines: J dxi_2/dx = (-d1 y, d1 x)/dxi_1
                double dy = 0.0, dx = 0.0;
#pragma unroll
                for (int m = 1; m <= 3; ++m) {
                    const double h = 0.5 * ec_alpha(m);
                    dx = fma(h, XS[b + m] - XS[b - m], dx);
                    dy = fma(h, XS[NB + b + m] - XS[NB + b - m], dy);
                }
                const double h = 0.5 * P.inv_dxi[0];
                const double nx = -dy * h, ny = dx * h;          // halves
                S[Slot<DIM>::N2 * NB + b] = nx;
                S[(Slot<DIM>::N2 + 1) * NB + b] = ny;
                S[(Slot<DIM>::N2 + 2) * NB + b] = -fma(XD[b], nx, XD[NB + b] * ny);
            }
        }
    }
    __syncthreads();

    double acc[NC + 1];
#pragma unroll
    for (int c = 0; c <= NC; ++c) acc[c] = 0.0;
    const int tx = tid % BX, ty = tid / BX;

    // ---- C, D, E: pairs, faces and the divergence at the interior node (tx, ty)
    if constexpr (TL::JOINT) {
        // a warp may hold items of both directions: the direction is data (one code path), not a branch
        for (int t = tid; t < TL::NP1 + TL::NP2; t += TL::THREADS) {
            const bool two = t >= TL::NP1;
            pair_item<DIM, BX, BY>(S, NB, DirGeo<DIM, BX, BY>(two ? 1 : 0), two ? t - TL::NP1 : t, G, PB, TL::PS, t);
        }
        for (int t = tid; t < TL::NJ1 + TL::NJ2; t += TL::THREADS) {
            const bool two = t >= TL::NJ1;
            jump_item<DIM, BX, BY>(S, NB, DirGeo<DIM, BX, BY>(two ? 1 : 0), two ? t - TL::NJ1 : t, JB, TL::JS, t);
        }
        __syncthreads();
        for (int t = tid; t < TL::NF1 + TL::NF2; t += TL::THREADS) {
            const bool two = t >= TL::NF1;
            face_item<DIM, BX, BY>(S, NB, DirGeo<DIM, BX, BY>(two ? 1 : 0), two ? t - TL::NF1 : t, P, PB, TL::PS,
                                   two ? TL::POFF2 : 0, JB, TL::JS, two ? TL::NJ1 : 0, FB, TL::FS, t);
        }
        __syncthreads();
        if (tid < BX * BY) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int LB = k == 0 ? BX : BY;
                const int fm = (k == 0 ? 0 : TL::FOFF2) + (k == 0 ? ty : tx) * (LB + 1) + (k == 0 ? tx : ty);
                const double inv = P.inv_dxi[k];
#pragma unroll
                for (int c = 0; c <= NC; ++c) acc[c] = fma(FB[c * TL::FS + fm] - FB[c * TL::FS + fm + 1], inv, acc[c]);
            }
        }
    } else {
#pragma unroll 1
        for (int k = 0; k < DIM; ++k) {
            const DirGeo<DIM, BX, BY> d(k);
            for (int t = tid; t < d.nlines * d.per_line; t += TL::THREADS)
                pair_item<DIM, BX, BY>(S, NB, d, t, G, PB, TL::PS, t);
            for (int t = tid; t < d.nlines * (d.LB + 5); t += TL::THREADS)
                jump_item<DIM, BX, BY>(S, NB, d, t, JB, TL::JS, t);
            __syncthreads();
            for (int t = tid; t < d.nlines * (d.LB + 1); t += TL::THREADS)
                face_item<DIM, BX, BY>(S, NB, d, t, P, PB, TL::PS, 0, JB, TL::JS, 0, FB, TL::FS, t);
            __syncthreads();
            if (tid < BX * (DIM == 2 ? BY : 1)) {
                const int line = k == 0 ? ty : tx;
                const int pos = k == 0 ? tx : ty;
                const int fm = line * (d.LB + 1) + pos;           // face pos - 1/2
                const double inv = P.inv_dxi[k];
#pragma unroll
                for (int c = 0; c <= NC; ++c) acc[c] = fma(FB[c * TL::FS + fm] - FB[c * TL::FS + fm + 1], inv, acc[c]);
            }
            __syncthreads();
        }
    }

    // ---- F: Shu-Osher combination (or the bare right-hand side)
    const int gi = i0 + tx, gj = j0 + ty;
    if (tid < BX * (DIM == 2 ? BY : 1) && gi < P.n1 && (DIM == 1 || gj < P.n2)) {
        const size_t N = size_t(P.n1) * P.n2;
        const size_t idx = size_t(DIM == 2 ? gj : 0) * P.n1 + gi;
        if (P.mode == 1) {
#pragma unroll
            for (int c = 0; c < NC; ++c) P.JUo[c * N + idx] = acc[c];
            P.Jo[idx] = acc[NC];
        } else {
            // all operands loaded before the first store (a store may alias a later load as far as the compiler
            // knows, which would serialise one round trip per component)
            double un[NC], us[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                un[c] = P.JUn[c * N + idx];
                us[c] = P.JUs[c * N + idx];
            }
            const double Jn = P.Jn[idx];
            const double Js = P.Js[idx];
#pragma unroll
            for (int c = 0; c < NC; ++c) P.JUo[c * N + idx] = fma(P.ca, un[c], P.cb * fma(dt, acc[c], us[c]));
            const double Jnew = fma(P.ca, Jn, P.cb * fma(dt, acc[NC], Js));
            P.Jo[idx] = Jnew;
            if (!(Jnew > 0.0)) raise_error(P.status, ES_ERR_MESH, int(idx));
        }
    }
}

// --------------------------------------------------------- short 1D lines
// A 1D line with few nodes is one warp's chain of dependent work, whatever its width: each of an SM's four schedulers
// issues one FP64 warp instruction per 64 cycles, so a tile of 8 nodes whose face phase runs on one warp (about 800
// instructions from load to store) takes 27 us, and a tile of 254 nodes on one SM 62 us.  Here a tile of 8 nodes is
// shared by the four warps of a CTA, one per scheduler: the node fields with one logarithm each, then the pairs on one
// warp beside the entropy variables' jumps on another, then one wave of the faces per warp (two lanes a face, one
// reconstruction each) beside the EC combination on the fourth, about 300 instructions.
constexpr int LINE = 8;                       // nodes of a tile
constexpr int LINE_NB = LINE + 6, LINE_NP = 3 * LINE + 6, LINE_NF = LINE + 1, LINE_NJ = LINE + 5;
static_assert(LINE_NP <= 32 && 2 * LINE_NF <= 32 && LINE_NB <= 32, "a phase is one pass of a warp");

__global__ void __launch_bounds__(128) stage_line_fp64(StageParams P) {
    using SL = flux64::Slots<1>;
    constexpr int XT = SL::COUNT;             // half of J xi_t (the metric is 1)
    constexpr int NB = LINE_NB;
    __shared__ double S[(SL::COUNT + 1) * NB];
    __shared__ double PB[3 * LINE_NP], JB[3 * LINE_NJ];
    __shared__ double FB[4][3][LINE_NF];      // a wave's dissipation per warp, and the EC flux
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i0 = blockIdx.x * LINE;
    const int n = P.n1;
    const double dt = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && dt == 0.0) return;     // finished run: leave the state untouched
    const Gas& G = P.gas;

    // ---- A: node fields, a logarithm per warp
    if (lane < NB) {
        const int gi = i0 - 3 + lane;
        const int si = state_index(gi, n, P.bc[0]);
        double JU[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) JU[c] = P.JUs[size_t(c) * n + si];
        if ((gi < 0 || gi >= n) && end_mirrored(P.bc[0], gi < 0)) JU[1] = -JU[1];
        const int parts = warp == 0 ? flux64::LOG_RHO : (warp == 1 ? flux64::LOG_OM | flux64::PLAIN
                                                         : (warp == 2 ? flux64::LOG_T : flux64::LOG_RP));
        const bool ok = flux64::node_fields<1>(JU, P.Js[si], G, [&](int f, double v) { S[f * NB + lane] = v; }, parts);
        if (!ok && warp == 0) raise_error(P.status, ES_ERR_INADMISSIBLE, si);
        if (warp == 0) {
            double xd = 0.0;
            if (P.xdot) {
                const GhostTerms t = ghost_terms(gi, n, P.bc[0]);
                xd = t.w[0] * P.xdot[t.idx[0]];
                if (t.nterm > 1) xd = fma(t.w[1], P.xdot[t.idx[1]], xd);
            }
            S[XT * NB + lane] = -0.5 * xd;
        }
    }
    __syncthreads();

    // ---- C: pairs on warp 0; the entropy variables and their jumps on warp 1
    if (warp == 0 && lane < LINE_NP) {
        int m, q;
        if (lane < LINE + 1) { m = 1; q = 2 + lane; }
        else if (lane < 2 * LINE + 3) { m = 2; q = lane - LINE; }
        else { m = 3; q = lane - 2 * LINE - 3; }
        const double one = 1.0;
        double f[3];
        flux64::pair_flux<1>(S, NB, q, q + m, &one, S[XT * NB + q] + S[XT * NB + q + m], G, f);
#pragma unroll
        for (int c = 0; c < 3; ++c) PB[c * LINE_NP + lane] = f[c];
    } else if (warp == 1) {
        if (lane < NB)
            S[SL::W0 * NB + lane] = flux64::v1_logs(S[SL::W0 * NB + lane], S[SL::LNR * NB + lane],
                                                    S[SL::LNOM * NB + lane], S[SL::LNT * NB + lane], G);
        __syncwarp();
        if (lane < LINE_NJ) {
            double d[3];
            flux64::entropy_jump<1>(S, NB, lane, lane + 1, d);
#pragma unroll
            for (int c = 0; c < 3; ++c) JB[c * LINE_NJ + lane] = d[c];
        }
    }
    __syncthreads();

    // ---- D: faces q + 1/2, q = 2 .. LINE + 2: wave `warp` of each (two lanes: the reconstructions from the left and from
    // the right), and on the last warp the 6th-order combination of the pairs
    double FJ = 0.0;
    if (warp == 3) {
        if (lane < LINE_NF) {
            double F[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int m = 1; m <= 3; ++m) {
                const int off = m == 1 ? 0 : (m == 2 ? LINE + 1 : 2 * LINE + 3);
                const double al = ec_alpha(m);
#pragma unroll
                for (int s = 0; s < m; ++s)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        F[c] = fma(c == 2 ? 4.0 * al : al, PB[c * LINE_NP + off + lane + m - 1 - s], F[c]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) FB[3][c][lane] = F[c];
        }
    } else if (P.diss) {
        const int face = lane >> 1 < LINE_NF ? lane >> 1 : LINE_NF - 1;         // (idle lanes repeat the last face)
        const bool right = lane & 1;
        const int l = 2 + face;
        const double one = 1.0;
        const flux64::Face<1> f =
            flux64::face_state<1>(S, NB, l, l + 1, &one, S[XT * NB + l] + S[XT * NB + l + 1], G, P.status, 0);
        double d[5];
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            const double dv[3] = {JB[l + o - 2], JB[LINE_NJ + l + o - 2], JB[2 * LINE_NJ + l + o - 2]};
            double W[3] = {0.0, 0.0, 0.0};
            flux64::project<1>(f, dv, W, 1u << warp);
            d[o] = warp == 0 ? W[0] : (warp == 1 ? W[1] : W[2]);
        }
        const flux64::SwitchBounds b = flux64::switch_bounds<1>(f, S, NB, l, l + 1, P.weno);
        const int is = flux64::jump_is_zero<1>(b, f, warp, d[2]);
        bool zero = is == 1;
        if (is == 2) zero = fabs(d[2]) <= P.weno.sign_tol * flux64::jump_size<1>(f, S, NB, l, l + 1, warp);
        double y = 0.0;
        if (__any_sync(0xffffffffu, !zero)) {
            const double s2 = fma(d[2], d[2], P.weno.eps4);
            const double sx = right ? d[3] : d[1];
            double num, den;
            flux64::weno_side(right ? d[4] : d[0], sx, d[2], right ? d[1] : d[3],
                              flux64::min_pos(fma(sx, sx, P.weno.eps4), s2), P.weno, num, den);
            const double part = num * rcp_nr(den);
            const double other = __shfl_xor_sync(0xffffffffu, part, 1);
            if (!zero)
                y = -f.Lam * ((warp == 1 ? f.sE : f.sA) * flux64::switched(d[2] - (part + other), d[2]));
        }
        const double vn = f.vr[0], c = warp == 0 ? -f.c : (warp == 1 ? 0.0 : f.c);
        if (!right && lane >> 1 < LINE_NF) {
            FB[warp][0][face] = y;
            FB[warp][1][face] = f.fr.e[0][0] * ((vn + c) * y);
            FB[warp][2][face] = (warp == 1 ? f.H - f.hm : fma(vn, c, f.H)) * y;
        }
    }
    __syncthreads();

    // ---- E: divergence and the Shu-Osher combination on warp 0, a face per lane
    if (warp != 0) return;
    double F[4] = {0.0, 0.0, 0.0, 0.0};
    if (lane < LINE_NF) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            F[c] = P.diss ? FB[3][c][lane] + ((FB[0][c][lane] + FB[2][c][lane]) + FB[1][c][lane]) : FB[3][c][lane];
        // sum_m alpha_m sum of the pairs' mean J xi_t, collected by node
        const double* X = S + XT * NB + 2 + lane;
        const double a3 = ec_alpha(3), a2 = ec_alpha(2) + a3, a1 = ec_alpha(1) + a2;
        FJ = fma(a1, X[0] + X[1], fma(a2, X[-1] + X[2], a3 * (X[-2] + X[3])));
    }
    F[3] = FJ;
    double acc[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = (F[c] - __shfl_down_sync(0xffffffffu, F[c], 1)) * P.inv_dxi[0];
    const int gi = i0 + lane;
    if (lane >= LINE || gi >= n) return;
    if (P.mode == 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) P.JUo[size_t(c) * n + gi] = acc[c];
        P.Jo[gi] = acc[3];
        return;
    }
    double un[4], us[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        un[c] = c < 3 ? P.JUn[size_t(c) * n + gi] : P.Jn[gi];
        us[c] = c < 3 ? P.JUs[size_t(c) * n + gi] : P.Js[gi];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double v = fma(P.ca, un[c], P.cb * fma(dt, acc[c], us[c]));
        if (c < 3) P.JUo[size_t(c) * n + gi] = v;
        else {
            P.Jo[gi] = v;
            if (!(v > 0.0)) raise_error(P.status, ES_ERR_MESH, gi);
        }
    }
}

// ----------------------------------------------------------------- launch
template <int DIM, int BX, int BY, int NT>
static cudaError_t prepare_tile() {
    return cudaFuncSetAttribute(stage_kernel_fp64<DIM, BX, BY, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(Tile<DIM, BX, BY, NT>::SMEM));
}

template <int DIM, int BX, int BY, int NT>
static cudaError_t launch_tile(const StageParams& P, cudaStream_t s) {
    using TL = Tile<DIM, BX, BY, NT>;
    const int ntx = (P.n1 + BX - 1) / BX;
    const int nty = DIM == 2 ? (P.n2 + BY - 1) / BY : 1;
    stage_kernel_fp64<DIM, BX, BY, NT><<<ntx * nty, NT, TL::SMEM, s>>>(P);
    return cudaGetLastError();
}

// 2D shapes: 32 x 8 nodes with 288 threads (= the 32 x 9 faces of xi_2), 25 x 11 with 384
// (25 x 12 = 300 faces; 8 x 19 = 152 tiles cover 200 x 200 in one wave on 152 SMs), 16 x 16
// with 288 (272 faces), 32 x 12 with 416 (416 faces; less halo per node), 20 x 10 with 224.  A mesh that 20 x 10 tiles
// cover in one wave has five shapes of its own, 64 to 200 nodes: a launch there is the time of one tile on its SM's FP64
// pipe, so the smallest tile whose tiles the SMs can hold wins (a
// Riemann stage, us: 64 x 64 74 with 8 x 8 nodes against 137 with 20 x 10, 120 x 120 83 with 12 x 8 against 139, 140 x 140
// 114 with 20 x 8 against 138; the shapes of larger meshes take at least the last).  Above one wave 20 x 10 nodes and less
// cost more halo than they balance (170 x 170: 166 us in one wave; 200 x 200: 192 against 176 with 25 x 11).
// All 2D shapes give the same bits.  1D: by the line's length (launch_stage_fp64); the 62- and 254-node tiles give the same
// bits, the 8-node line adds the waves of a face in another order.
static bool small_mesh(const StageParams& P, int nsm) { return (P.n1 + 19) / 20 * ((P.n2 + 9) / 10) <= nsm; }
cudaError_t stage_prepare_fp64(int dim) {
    if (dim == 1) {
        cudaError_t e1 = prepare_tile<1, 254, 1, 256>();
        return e1 == cudaSuccess ? prepare_tile<1, 62, 1, 128>() : e1;
    }
    cudaError_t e = prepare_tile<2, 32, 8, 288>();
    if (e == cudaSuccess) e = prepare_tile<2, 25, 11, 384>();
    if (e == cudaSuccess) e = prepare_tile<2, 16, 16, 288>();
    if (e == cudaSuccess) e = prepare_tile<2, 32, 12, 416>();
    if (e == cudaSuccess) e = prepare_tile<2, 20, 10, 224>();
    if (e == cudaSuccess) e = prepare_tile<2, 8, 8, 128>();
    if (e == cudaSuccess) e = prepare_tile<2, 12, 8, 128>();
    if (e == cudaSuccess) e = prepare_tile<2, 16, 8, 160>();
    if (e == cudaSuccess) e = prepare_tile<2, 20, 8, 192>();
    return e;
}

cudaError_t launch_stage_fp64(const StageParams& P, int nsm, cudaStream_t s) {
    if (P.dim == 1) {
        // measured per stage launch (us), 8-node lines / 62-node tiles / 254-node tiles: 200 nodes 16.4 / 28.7 / 61.5,
        // 1600 20.5 / 28.7 / 62.5, 6400 49.2 / 28.7 / 63.5, 25600 164 / 47.2 / 61.5, 102400 621 / 176 / 172.  A line is
        // spread over an SM's four schedulers, so it pays while an SM has two of them or fewer (152 SMs x 2 x 8 nodes);
        // 62-node tiles (faces, pairs and nodes two, six and two full warps of four) while the 254-node ones, which
        // repeat less of the halo, leave SMs idle
        if (P.n1 <= 2 * nsm * LINE) {
            stage_line_fp64<<<(P.n1 + LINE - 1) / LINE, 128, 0, s>>>(P);
            return cudaGetLastError();
        }
        if ((long long)P.n1 * 152 <= 65536LL * nsm) return launch_tile<1, 62, 1, 128>(P, s);     // (431 nodes per SM)
        return launch_tile<1, 254, 1, 256>(P, s);
    }
    if (small_mesh(P, nsm)) {
        switch (P.tile) {
            case 1: return launch_tile<2, 12, 8, 128>(P, s);
            case 2: return launch_tile<2, 16, 8, 160>(P, s);
            case 3: return launch_tile<2, 20, 8, 192>(P, s);
            case 4: return launch_tile<2, 20, 10, 224>(P, s);
            default: return launch_tile<2, 8, 8, 128>(P, s);
        }
    }
    switch (P.tile) {
        case 1: return launch_tile<2, 25, 11, 384>(P, s);
        case 2: return launch_tile<2, 16, 16, 288>(P, s);
        case 3: return launch_tile<2, 32, 12, 416>(P, s);
        case 4: return launch_tile<2, 20, 10, 224>(P, s);
        default: return launch_tile<2, 32, 8, 288>(P, s);
    }
}

}  // namespace es
