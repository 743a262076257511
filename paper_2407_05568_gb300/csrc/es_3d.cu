// es_3d.cu -- the ES operator, SSP-RK3 stage and mesh redistribution in three dimensions (FP64).
//
// A 3D tile with a 3-node halo in every direction holds (BX+6)(BY+6)(BZ+6) nodes: in FP64
// that is several times the shared memory of an SM for any useful tile, so the 3D path is
// split by direction instead:
//   k3_coords   stage coordinates x^n + c dt xdot on the mesh extended by 3 ghosts (Sec. 3.2)
//   k3_deriv    delta_l[x_p] there (the inner differences of eq. SCLCoeff)
//   k3_metric   J dxi_k/dx_j = (delta_m[delta_l[x_p] x_q] - delta_l[delta_m[x_p] x_q])/(dxi_l dxi_m)
//               for (k, l, m), (j, p, q) cyclic (eq. SCLCoeff), on each direction's nodes plus
//               3 ghosts along xi_k
//   k3_nodes    primitive state, logarithms and entropy variables of every node, once
//   k3_dir<K>   per xi_K: pencils of LB nodes x W lines staged in shared memory; pair fluxes
//               (eq. ECfluxMM), the 6th-order combination (eq. ECFlux_curv_2p, GCL_flux), the ES
//               dissipation with the theta/phi rotation (eq. HOstable, Sec. 3.3) and the
//               divergence, accumulated over the directions; the last direction applies the
//               Shu-Osher combination.
// The mesh redistribution (Sec. 4) uses 3D monitor, filter, Jacobi and limiter kernels and
// shares the elementwise kernels of the 1D/2D path.
#include <cuda_runtime.h>

#include "es_3d.h"
#include "es_3d_filter.cuh"
#include "es_3d_grid.cuh"
#include "es_device.cuh"
#include "es_flux64.cuh"
#include "es_internal.h"
#include "es_mesh64.cuh"

namespace es {

// node fields of the 3D path (global planes and shared-memory slots), and the direction's metrics (shared memory only)
using SL3 = flux64::Slots<3>;
constexpr int F3_COUNT = SL3::COUNT;
constexpr int G_N = F3_COUNT;              // halves of the three metric components, then of J xi_t
constexpr int G_XT = G_N + 3;
constexpr int S3_COUNT = G_XT + 1;

// stride of direction k in a [n3][n2][n1] field
__device__ __forceinline__ size_t stride3(const Grid3& g, int k) {
    return k == 0 ? 1 : (k == 1 ? size_t(g.n[0]) : size_t(g.n[0]) * g.n[1]);
}

// index of the node at offset s (|s| = 1) along direction k from in-mesh node id (position i_k),
// ghosts by copy / wrap: the neighbour can leave the mesh along k only
__device__ __forceinline__ size_t nb_index(const Grid3& g, size_t id, int ik, int k, int s) {
    const int j = state_index(ik + s, g.n[k], g.bc[k]);
    return id + (long long)(j - ik) * (long long)stride3(g, k);
}

// coordinate component `comp` of that neighbour: wrap with the period shift, or odd reflection
// about the boundary node (2 x_b - x_{b -+ 1}), the one-direction case of the ghost rule
__device__ __forceinline__ double nb_coord(const Grid3& g, const double* f, size_t id, int ik, int k, int s,
                                           int comp) {
    const int n = g.n[k];
    const int j = ik + s;
    const long long st = (long long)stride3(g, k);
    if (j >= 0 && j < n) return f[id + (long long)s * st];
    if (g.bc[k] == ES_BC_PERIODIC) {
        const int r = j < 0 ? j + n : j - n;
        double v = f[id + (long long)(r - ik) * st];
        if (comp == k) v += (j < 0 ? -1.0 : 1.0) * g.period[k];
        return v;
    }
    const int b = j < 0 ? 0 : n - 1, m = j < 0 ? 1 : n - 2;
    if (comp != k && end_mirrored(g.bc[k], j < 0)) return f[id + (long long)(m - ik) * st];
    return 2.0 * f[id + (long long)(b - ik) * st] - f[id + (long long)(m - ik) * st];
}

// sqrt(x), x >= 0 (or NaN): x rsqrt_nr(x) where x is normal and not huge, six FP64 instructions
__device__ __forceinline__ double sqrt_pos(double x) {
    const unsigned h = unsigned(__double2hiint(x));
    return h - 0x03000000u < 0x7a000000u ? x * rsqrt_nr(x) : sqrt(x);
}

__device__ __forceinline__ double block_min(double v) {
    __shared__ double sh[32];
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = threadIdx.x < nw ? sh[threadIdx.x] : 1e300;
    if (w == 0)
        for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    return v;
}

// ================================================================ metrics
// stage coordinates on the extended grid
__global__ void k3_coords(Grid3 g, const double* xn, const double* xdot, double cst, const double* dt_dev,
                          double dt_host, double* XE) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const int E1 = g.n[0] + 6, E2 = g.n[1] + 6, E3 = g.n[2] + 6;
    const size_t NE = size_t(E1) * E2 * E3;
    const double cdt = cst * (dt_dev ? *dt_dev : dt_host);
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < NE; e += size_t(gridDim.x) * blockDim.x) {
        const int e1 = int(e % E1), e2 = int((e / E1) % E2), e3 = int(e / (size_t(E1) * E2));
        const int i1 = e1 - 3, i2 = e2 - 3, i3 = e3 - 3;
        if (inside3(g, i1, i2, i3, 0)) {
            const size_t id = idx3(g, i1, i2, i3);
            for (int c = 0; c < 3; ++c) XE[c * NE + e] = xdot ? xn[c * N + id] + cdt * xdot[c * N + id] : xn[c * N + id];
            continue;
        }
        for (int c = 0; c < 3; ++c)
            XE[c * NE + e] = ghost_value3(g, xn + c * N, xdot ? xdot + c * N : nullptr, cdt, i1, i2, i3, c);
    }
}

// The products of eq. SCLCoeff's cross form, once per node: D[3 l + j] = delta_l[x_p] x_q with
// p = (j + 1) % 3, q = (j + 2) % 3 (delta_l undivided; 0 where the xi_l index is not interior).
// Each is differenced by two directions' metrics, which therefore read the same rounded value.
__global__ void k3_deriv(Grid3 g, const double* XE, double* D) {
    const int E1 = g.n[0] + 6, E2 = g.n[1] + 6, E3 = g.n[2] + 6;
    const size_t NE = size_t(E1) * E2 * E3;
    const size_t st[3] = {1, size_t(E1), size_t(E1) * E2};
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < NE; e += size_t(gridDim.x) * blockDim.x) {
        const int ee[3] = {int(e % E1), int((e / E1) % E2), int(e / (size_t(E1) * E2))};
        const double x[3] = {XE[e], XE[NE + e], XE[2 * NE + e]};
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const bool ok = ee[l] >= 3 && ee[l] < g.n[l] + 3;
            double dl[3];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                double s = 0.0;
                if (ok) {
#pragma unroll
                    for (int m = 1; m <= 3; ++m)
                        s += 0.5 * ec_alpha(m) * (XE[p * NE + e + m * st[l]] - XE[p * NE + e - m * st[l]]);
                }
                dl[p] = s;
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) D[(3 * l + j) * NE + e] = dl[(j + 1) % 3] * x[(j + 2) % 3];
        }
    }
}

// Half of J dxi_k/dx_j (a face takes the mean of two nodes as a sum) on direction k's grid (n_k + 6 nodes along xi_k, interior across); the direction is a template
// parameter (no run-time indexing of the grid's arrays)
template <int k>
__global__ void k3_metric(Grid3 g, const double* D, double* NKo) {
    const int E1 = g.n[0] + 6, E2 = g.n[1] + 6;
    const size_t NE = size_t(E1) * E2 * (g.n[2] + 6);
    int m1 = g.n[0], m2 = g.n[1], m3 = g.n[2];
    if (k == 0) m1 += 6;
    else if (k == 1) m2 += 6;
    else m3 += 6;
    const size_t M = size_t(m1) * m2 * m3;
    const int l = (k + 1) % 3, m = (k + 2) % 3;
    const double scale = 0.5 * (g.inv_dxi[l] * g.inv_dxi[m]);
    const double h[3] = {0.5 * ec_alpha(1) * scale, 0.5 * ec_alpha(2) * scale, 0.5 * ec_alpha(3) * scale};
    const size_t stl = l == 0 ? 1 : (l == 1 ? size_t(E1) : size_t(E1) * E2);
    const size_t stm = m == 0 ? 1 : (m == 1 ? size_t(E1) : size_t(E1) * E2);
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < M; t += size_t(gridDim.x) * blockDim.x) {
        const int a1 = int(t % m1), a2 = int((t / m1) % m2), a3 = int(t / (size_t(m1) * m2));
        // extended-grid position: the metric grid already carries the 3 ghosts along xi_k
        const size_t e = eidx(g, a1 + (k == 0 ? 0 : 3), a2 + (k == 1 ? 0 : 3), a3 + (k == 2 ? 0 : 3));
        for (int j = 0; j < 3; ++j) {
            const double* Pl = D + (3 * l + j) * NE;      // delta_l[x_p] x_q
            const double* Pm = D + (3 * m + j) * NE;      // delta_m[x_p] x_q
            double A = 0.0;
#pragma unroll
            for (int a = 1; a <= 3; ++a) {
                const size_t sm = a * stm, sl = a * stl;
                A = fma(h[a - 1], Pl[e + sm] - Pl[e - sm], A);
                A = fma(-h[a - 1], Pm[e + sl] - Pm[e - sl], A);
            }
            NKo[j * M + t] = A;
        }
    }
}

// ================================================================ node fields
__global__ void k3_nodes(Grid3 g, Gas G, const double* JU, const double* J, double* NF, DevStatus* st) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    for (size_t id = blockIdx.x * size_t(blockDim.x) + threadIdx.x; id < N; id += size_t(gridDim.x) * blockDim.x) {
        const double U[5] = {JU[id], JU[N + id], JU[2 * N + id], JU[3 * N + id], JU[4 * N + id]};
        const bool ok = flux64::node_fields<3>(U, J[id], G, [&](int f, double v) { NF[f * N + id] = v; });
        if (!ok) raise_error(st, ES_ERR_INADMISSIBLE, int(id));
    }
}

// ================================================================ direction flux
struct Dir3Params {
    Grid3 g;
    Gas gas;
    Weno weno;
    int diss;
    const double* NF;         // node fields [F3_COUNT][N]
    const double* NK;         // metrics of this direction [3][M]
    const double* xdot;       // nullable
    double* RH;               // accumulated right-hand sides [6][N]
    int first, last;
    int mode;                 // last direction: 0 RK combination, 1 right-hand sides out
    double ca, cb;
    double dt_host;
    const double* dt_dev;
    const double *JUn, *Jn, *JUs, *Js;
    double *JUo, *Jo;
    DevStatus* status;
};

template <int LB, int W>
struct Pencil {
    static constexpr int LS = (LB + 6) | 1;             // node stride of a line (odd: no bank conflicts)
    static constexpr int NB = W * LS;
    static constexpr int PL = 3 * LB + 6;               // pairs per line
    static constexpr int NP = W * PL;
    static constexpr int NF = W * (LB + 1);             // faces
    static constexpr int NJ = W * (LB + 5);             // entropy-variable jumps between neighbours
    static constexpr size_t SMEM = sizeof(double) * (size_t(S3_COUNT) * NB + 5 * NP + 6 * NF + 5 * NJ);
};

template <int K, int LB, int W, int NT>
__global__ void __launch_bounds__(NT, W >= 16 ? 1 : (NT <= 96 ? 3 : 2)) k3_dir(Dir3Params P) {
    using PC = Pencil<LB, W>;
    constexpr int LS = PC::LS, NB = PC::NB, NP = PC::NP, NFc = PC::NF;
    extern __shared__ double smem[];
    double* S = smem;
    double* PB = S + S3_COUNT * NB;
    double* FB = PB + 5 * NP;
    double* JB = FB + 6 * NFc;
    const Grid3& g = P.g;
    const int tid = threadIdx.x;
    const int nk = g.n[K];
    // transverse indices: A (W consecutive lines) and B
    const int nA = K == 0 ? g.n[1] : g.n[0];
    const int nB = K == 2 ? g.n[1] : g.n[2];
    const int nseg = (nk + LB - 1) / LB;
    const int ngA = (nA + W - 1) / W;
    const int seg = blockIdx.x % nseg;
    const int grp = blockIdx.x / nseg;
    const int a0 = (grp % ngA) * W;
    const int b = grp / ngA;
    if (b >= nB) return;
    const int s0 = seg * LB;
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const double dt = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && P.dt_dev && dt == 0.0) return;   // finished run: leave the state untouched
    const int M1 = g.n[0] + (K == 0 ? 6 : 0), M2 = g.n[1] + (K == 1 ? 6 : 0), M3 = g.n[2] + (K == 2 ? 6 : 0);
    const size_t M = size_t(M1) * M2 * M3;

    // ---- A: node fields and metrics of the pencils (3 ghosts along xi_K)
    for (int t = tid; t < W * (LB + 6); t += NT) {
        int line, q;
        if (K == 0) { line = t / (LB + 6); q = t % (LB + 6); }
        else { q = t / W; line = t % W; }
        int a = a0 + line;
        if (a > nA - 1) a = nA - 1;                          // ragged group: a valid line, not written
        const int s = s0 + q - 3;                            // along xi_K, possibly a ghost
        const int ss = state_index(s, nk, g.bc[K]);
        int i1, i2, i3, j1, j2, j3;
        if (K == 0) { i1 = ss; i2 = a; i3 = b; }
        else if (K == 1) { i1 = a; i2 = ss; i3 = b; }
        else { i1 = a; i2 = b; i3 = ss; }
        const size_t id = idx3(g, i1, i2, i3);
        const int bx = line * LS + q;
        double v[F3_COUNT];                                  // all loads in flight before the stores
#pragma unroll
        for (int f = 0; f < F3_COUNT; ++f) v[f] = P.NF[f * N + id];
#pragma unroll
        for (int f = 0; f < F3_COUNT; ++f) S[f * NB + bx] = v[f];
        if ((s < 0 || s >= nk) && end_mirrored(g.bc[K], s < 0)) {     // wall / symmetry ghost
            S[(SL3::V + K) * NB + bx] = -S[(SL3::V + K) * NB + bx];
            S[(SL3::VT + K) * NB + bx] = -S[(SL3::VT + K) * NB + bx];
            S[(SL3::RV + K) * NB + bx] = -S[(SL3::RV + K) * NB + bx];
        }
        // metrics: the metric grid holds s in [-3, n_K + 3); the tail of a ragged pencil is clamped
        int se = s + 3;
        se = se < 0 ? 0 : (se > nk + 5 ? nk + 5 : se);
        if (K == 0) { j1 = se; j2 = a; j3 = b; }
        else if (K == 1) { j1 = a; j2 = se; j3 = b; }
        else { j1 = a; j2 = b; j3 = se; }
        const size_t mi = (size_t(j3) * M2 + j2) * M1 + j1;
        const double nx = P.NK[mi], ny = P.NK[M + mi], nz = P.NK[2 * M + mi];
        S[G_N * NB + bx] = nx;
        S[(G_N + 1) * NB + bx] = ny;
        S[(G_N + 2) * NB + bx] = nz;
        double xt = 0.0;
        if (P.xdot) {
            // mesh velocity at the node: wrap, odd reflection, or at a wall / symmetry end the
            // mirror image (components along the plane mirrored, the normal one reflected)
            double xd[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const GhostTerms tk = ghost_terms(s, nk, g.bc[K], c != K);
                for (int u = 0; u < tk.nterm; ++u) {
                    int k1 = i1, k2 = i2, k3 = i3;
                    if (K == 0) k1 = tk.idx[u];
                    else if (K == 1) k2 = tk.idx[u];
                    else k3 = tk.idx[u];
                    xd[c] += tk.w[u] * P.xdot[c * N + idx3(g, k1, k2, k3)];
                }
            }
            xt = -fma(xd[0], nx, fma(xd[1], ny, xd[2] * nz));
        }
        S[G_XT * NB + bx] = xt;
    }
    __syncthreads();

    // ---- C: pair fluxes F(U_q, U_{q+m}), m = 1..3, q = 3-m .. LB+2 along each line, and the entropy variables' jumps
    // between neighbours, q = 0 .. LB+4
    for (int t = tid; t < NP; t += NT) {
        const int line = t / PC::PL, kk = t % PC::PL;
        int m, q;
        if (kk < LB + 1) { m = 1; q = 2 + kk; }
        else if (kk < 2 * LB + 3) { m = 2; q = 1 + (kk - LB - 1); }
        else { m = 3; q = kk - 2 * LB - 3; }
        const int l = line * LS + q, r = l + m;
        double n[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) n[c] = S[(G_N + c) * NB + l] + S[(G_N + c) * NB + r];
        double f[5];
        flux64::pair_flux<3>(S, NB, l, r, n, S[G_XT * NB + l] + S[G_XT * NB + r], P.gas, f);
#pragma unroll
        for (int c = 0; c < 5; ++c) PB[c * NP + t] = f[c];
    }
    for (int t = tid; t < PC::NJ; t += NT) {
        const int l = t / (LB + 5) * LS + t % (LB + 5);
        double f[5];
        flux64::entropy_jump<3>(S, NB, l, l + 1, f);
#pragma unroll
        for (int c = 0; c < 5; ++c) JB[c * PC::NJ + t] = f[c];
    }
    __syncthreads();

    // ---- D: face fluxes at q+1/2, q = 2 .. LB+2
    for (int t = tid; t < NFc; t += NT) {
        const int line = t / (LB + 1), f = t % (LB + 1);
        const int q = 2 + f;
        const int pbase = line * PC::PL;
        const int base = line * LS;
        double F[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int m = 1; m <= 3; ++m) {
            const int off = m == 1 ? 0 : (m == 2 ? LB + 1 : 2 * LB + 3);
            const double al = ec_alpha(m);
            for (int s = 0; s < m; ++s) {
                const int qq = q - s;
                const int pi = pbase + off + (qq - (3 - m));
#pragma unroll
                for (int c = 0; c < 5; ++c) F[c] = fma(c == 4 ? 4.0 * al : al, PB[c * NP + pi], F[c]);   // (a quarter of the energy)
            }
        }
        // sum_m alpha_m sum of the pairs' mean J xi_t, collected by node
        const double* XT = S + G_XT * NB + base + q;            // halves
        const double a3 = ec_alpha(3), a2 = ec_alpha(2) + a3, a1 = ec_alpha(1) + a2;
        const double FJ = fma(a1, XT[0] + XT[1], fma(a2, XT[-1] + XT[2], a3 * (XT[-2] + XT[3])));
        if (P.diss) {
            const int l = base + q;
            double n[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) n[c] = S[(G_N + c) * NB + l] + S[(G_N + c) * NB + l + 1];
            flux64::face_dissipation<3>(S, NB, l, 1, n, XT[0] + XT[1], P.gas, P.weno, JB, PC::NJ,
                                        line * (LB + 5) + q, F, P.status, 0);
        }
#pragma unroll
        for (int c = 0; c < 5; ++c) FB[c * NFc + t] = F[c];
        FB[5 * NFc + t] = FJ;
    }
    __syncthreads();

    // ---- E: divergence at the pencil's nodes, accumulated over the directions; the last
    // direction writes the right-hand sides or the Shu-Osher combination
    const double inv = g.inv_dxi[K];
    for (int t = tid; t < W * LB; t += NT) {
        int line, pos;
        if (K == 0) { line = t / LB; pos = t % LB; }
        else { pos = t / W; line = t % W; }
        const int a = a0 + line, s = s0 + pos;
        if (a >= nA || s >= nk) continue;
        int i1, i2, i3;
        if (K == 0) { i1 = s; i2 = a; i3 = b; }
        else if (K == 1) { i1 = a; i2 = s; i3 = b; }
        else { i1 = a; i2 = b; i3 = s; }
        const size_t id = idx3(g, i1, i2, i3);
        const int fm = line * (LB + 1) + pos;
        // every global operand of the node is loaded before the first global store (a store may alias a later
        // load as far as the compiler knows, which would serialise one round trip per component)
        double rh[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        double un[6], us[6];
        if (!P.first) {
#pragma unroll
            for (int c = 0; c < 6; ++c) rh[c] = P.RH[c * N + id];
        }
        const bool combine = P.last && P.mode != 1;
        if (combine) {
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                un[c] = P.JUn[c * N + id];
                us[c] = P.JUs[c * N + id];
            }
            un[5] = P.Jn[id];
            us[5] = P.Js[id];
        }
        double acc[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            // (explicit: every pencil shape fuses the same product)
            acc[c] = fma(FB[c * NFc + fm] - FB[c * NFc + fm + 1], inv, rh[c]);
        }
        if (!P.last) {
#pragma unroll
            for (int c = 0; c < 6; ++c) P.RH[c * N + id] = acc[c];
        } else if (P.mode == 1) {
#pragma unroll
            for (int c = 0; c < 5; ++c) P.JUo[c * N + id] = acc[c];
            P.Jo[id] = acc[5];
        } else {
#pragma unroll
            for (int c = 0; c < 5; ++c) P.JUo[c * N + id] = fma(P.ca, un[c], P.cb * fma(dt, acc[c], us[c]));
            const double Jnew = fma(P.ca, un[5], P.cb * fma(dt, acc[5], us[5]));
            P.Jo[id] = Jnew;
            if (!(Jnew > 0.0)) raise_error(P.status, ES_ERR_MESH, int(id));
        }
    }
}

// pencil shapes (nodes along xi_K x lines, threads >= faces): 16 x 16 / 288 (one CTA per SM by
// shared memory), 16 x 8 / 160 (two CTAs per SM: one CTA's loads overlap the other's arithmetic),
// 16 x 4 / 96 (three CTAs per SM), 32 x 4 / 160 (two per SM, 19% halo nodes instead of 38%)
template <int K, int LB, int W, int NT>
static cudaError_t dir_prepare_shape() {
    return cudaFuncSetAttribute(k3_dir<K, LB, W, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(Pencil<LB, W>::SMEM));
}

template <int K>
static cudaError_t dir_prepare() {
    cudaError_t e = dir_prepare_shape<K, 16, 16, 288>();
    if (e == cudaSuccess) e = dir_prepare_shape<K, 16, 8, 160>();
    if (e == cudaSuccess) e = dir_prepare_shape<K, 16, 4, 96>();
    if (e == cudaSuccess) e = dir_prepare_shape<K, 32, 4, 160>();
    return e;
}

template <int K, int LB, int W, int NT>
static cudaError_t dir_launch_shape(const Dir3Params& P, cudaStream_t s) {
    const Grid3& g = P.g;
    const int nA = K == 0 ? g.n[1] : g.n[0];
    const int nB = K == 2 ? g.n[1] : g.n[2];
    const long long blocks = (long long)((g.n[K] + LB - 1) / LB) * ((nA + W - 1) / W) * nB;
    k3_dir<K, LB, W, NT><<<unsigned(blocks), NT, Pencil<LB, W>::SMEM, s>>>(P);
    return cudaGetLastError();
}

template <int K>
static cudaError_t dir_launch(const Dir3Params& P, int shape, cudaStream_t s) {
    switch (shape) {
        case 1: return dir_launch_shape<K, 16, 8, 160>(P, s);
        case 2: return dir_launch_shape<K, 16, 4, 96>(P, s);
        case 3: return dir_launch_shape<K, 32, 4, 160>(P, s);
        default: return dir_launch_shape<K, 16, 16, 288>(P, s);
    }
}

// ================================================================ CFL (eq. cfl)
// max_i sum_k (|J xi_{k,t} + n_k . v| + |n_k| c) / (J dxi_k), J xi_{k,t} = -xdot . n_k (eq. VCLCoeff), from the
// node fields and metrics of x^n; xdot = nullptr is a mesh at rest.  The maximum goes to d->red[slot].
// Bound by the FP64 pipe: 60 instructions a node (library square roots, FP64 maxima and J xi_t apart from n . v: 95).
__global__ void k3_cfl(Grid3 g, Gas G, const double* NF, const double* J, const double* NK0, const double* NK1,
                       const double* NK2, const double* xdot, int slot, DevScalars* d) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const size_t M[3] = {size_t(g.n[0] + 6) * g.n[1] * g.n[2], size_t(g.n[0]) * (g.n[1] + 6) * g.n[2],
                         size_t(g.n[0]) * g.n[1] * (g.n[2] + 6)};
    const double* NK[3] = {NK0, NK1, NK2};
    const double c2f = 2.0 * (1.0 + G.delta) * G.R, a4 = 4.0 * G.a;
    double mx = 0.0;
    for (unsigned id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i1 = int(id % unsigned(g.n[0])), r12 = int(id / unsigned(g.n[0]));
        const int i2 = r12 % g.n[1], i3 = r12 / g.n[1];
        // the node fields and metrics are halves
        const double r = NF[SL3::RHO * N + id], hT = NF[SL3::T * N + id], iom = NF[SL3::IOM * N + id];
        double v[3] = {NF[SL3::V * N + id], NF[(SL3::V + 1) * N + id], NF[(SL3::V + 2) * N + id]};
        if (xdot) {                                           // half the velocity relative to the mesh
#pragma unroll
            for (int k = 0; k < 3; ++k) v[k] = fma(-0.5, xdot[k * N + id], v[k]);
        }
        const double c2 = fma(c2f * hT, iom * iom, -a4 * r);
        const double hc = c2 > 0.0 ? 0.5 * sqrt_pos(c2) : 0.0;
        double tot = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int m1 = g.n[0] + (k == 0 ? 6 : 0), m2 = g.n[1] + (k == 1 ? 6 : 0);
            const size_t mi = (size_t(i3 + (k == 2 ? 3 : 0)) * m2 + i2 + (k == 1 ? 3 : 0)) * m1 + i1 + (k == 0 ? 3 : 0);
            const double n0 = NK[k][mi], n1 = NK[k][M[k] + mi], n2 = NK[k][2 * M[k] + mi];
            const double nv = fma(n2, v[2], fma(n1, v[1], n0 * v[0])), nn = fma(n2, n2, fma(n1, n1, n0 * n0));
            tot = fma(fma(sqrt_pos(nn), hc, fabs(nv)), g.inv_dxi[k], tot);
        }
        mx = max_bits(mx, c2 > 0.0 ? 4.0 * tot * rcp_nr(J[id]) : 1e300);
    }
    block_max_bits<1>(&mx);
    if (threadIdx.x == 0) atomic_max_pos(&d->red[slot], mx);
}

// ================================================================ init
__global__ void k3_init_J(Grid3 g, const double* x, double* J) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    for (size_t id = blockIdx.x * size_t(blockDim.x) + threadIdx.x; id < N; id += size_t(gridDim.x) * blockDim.x) {
        const int ii[3] = {int(id % g.n[0]), int((id / g.n[0]) % g.n[1]), int(id / (size_t(g.n[0]) * g.n[1]))};
        double Dm[3][3];                                     // Dm[c][k] = delta_k[x_c] / dxi_k
        for (int c = 0; c < 3; ++c)
            for (int k = 0; k < 3; ++k) {
                double s = 0.0;
#pragma unroll
                for (int m = 1; m <= 3; ++m) {
                    int p[3] = {ii[0], ii[1], ii[2]}, q[3] = {ii[0], ii[1], ii[2]};
                    p[k] += m;
                    q[k] -= m;
                    s += 0.5 * ec_alpha(m) * (ghost_value3(g, x + c * N, nullptr, 0.0, p[0], p[1], p[2], c) -
                                              ghost_value3(g, x + c * N, nullptr, 0.0, q[0], q[1], q[2], c));
                }
                Dm[c][k] = s * g.inv_dxi[k];
            }
        J[id] = Dm[0][0] * (Dm[1][1] * Dm[2][2] - Dm[1][2] * Dm[2][1]) -
                Dm[0][1] * (Dm[1][0] * Dm[2][2] - Dm[1][2] * Dm[2][0]) +
                Dm[0][2] * (Dm[1][0] * Dm[2][1] - Dm[1][1] * Dm[2][0]);
    }
}

// ================================================================ mesh (Sec. 4)
// squares of the difference quotients' factors per direction: (1/(2 dxi))^2 and (1/dxi^2)^2
struct MonScale3 {
    double d1[3], d2[3];
};

// raw monitor terms (eq. van der Waalsmonitor, or the smooth-test monitor): central first and second differences, whose
// factors multiply the squares; maxima by their ordered bits.  Bound by the FP64 pipe: about 30 instructions a node for
// the van der Waals monitor and 45 with the two square roots of the other, where both forms' sums, differences divided
// one by one and FP64 maxima were 91 (140 us at 96^3).
template <bool SMOOTH>
__global__ void k3_mon_terms(Grid3 g, MonScale3 sc, int kappa, const double* rhoF, const double* GF, double* t0, double* t1,
                             double* t2, DevScalars* d) {
    const unsigned N = unsigned(g.n[0]) * g.n[1] * g.n[2];
    double mx[3] = {0.0, 0.0, 0.0};
    for (unsigned id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i1 = int(id % unsigned(g.n[0])), r = int(id / unsigned(g.n[0]));
        const int ii[3] = {i1, r % g.n[1], r / g.n[1]};
        const double* f2 = SMOOTH ? rhoF : GF;               // the field of the second differences
        const double c0 = f2[id];
        double v0 = 0.0, v1 = 0.0, v2 = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const size_t ip = nb_index(g, id, ii[k], k, 1), im = nb_index(g, id, ii[k], k, -1);
            const double a = rhoF[ip] - rhoF[im];
            v0 = fma(sc.d1[k] * a, a, v0);
            const double fp = f2[ip], fm = f2[im];
            if (!SMOOTH && kappa >= 2) {
                const double b = fp - fm;
                v1 = fma(sc.d1[k] * b, b, v1);
            }
            const double c = fma(-2.0, c0, fp) + fm;
            v2 = fma(sc.d2[k] * c, c, v2);
        }
        if (SMOOTH) {
            v0 = sqrt_pos(v0);
            v2 = sqrt_pos(v2);
        }
        t0[id] = v0;
        t1[id] = v1;
        t2[id] = v2;
        mx[0] = max_bits(mx[0], v0);
        mx[1] = max_bits(mx[1], v1);
        mx[2] = max_bits(mx[2], v2);
    }
    block_max_bits<3>(mx);
    if (threadIdx.x == 0) {
        atomic_max_pos(&d->red[RED_MON0], mx[0]);
        atomic_max_pos(&d->red[RED_MON1], mx[1]);
        atomic_max_pos(&d->red[RED_MON2], mx[2]);
    }
}

// Coordinate component c of a boundary node that does not move: every component on an outflow
// end, the normal one on a wall or symmetry end (the node slides along the plane).
__device__ __forceinline__ bool fixed3(const Grid3& g, const int* ii, int c) {
    bool f = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (g.bc[k] == ES_BC_PERIODIC) continue;
        const bool lo = ii[k] == 0, hi = ii[k] == g.n[k] - 1;
        if (!lo && !hi) continue;
        const bool mir = end_mirrored(g.bc[k], lo);
        f = f || !mir || c == k;
    }
    return f;
}

// The sweeps' normalised weights of a node's neighbours (-xi_1, +xi_1, -xi_2, ...): the first sweep forms them from omega,
// the others read them.
struct SweepWeights3 {
    double* a[6];
};

// Jacobi sweep k (no warm start in 3D: sweep 0 reads x_n and writes xa, sweep k reads
// buf[(k - 1) % 2] and writes buf[k % 2]); with `check` the last block to finish compares the
// grid's max change with eps and latches convergence, after which the remaining sweeps return.
// A sweep that formed the weights again took 78 FP64 instructions a node (119 us at 96^3, bound by the FP64 pipe); with
// stored weights it is 18 and the traffic of 12 doubles a node bounds it.
template <bool FIRST, bool CHG>
__global__ void k3_jacobi(Grid3 g, const double* omega, SweepWeights3 W, double r2, double r3, const double* xin,
                          double* xout, DevScalars* d, double eps) {
    if (d->conv) return;
    const unsigned N = unsigned(g.n[0]) * g.n[1] * g.n[2];
    const int st[3] = {1, g.n[0], g.n[0] * g.n[1]};
    double chg = 0.0;
    for (unsigned id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i1 = int(id % unsigned(g.n[0])), r = int(id / unsigned(g.n[0]));
        const int ii[3] = {i1, r % g.n[1], r / g.n[1]};
        double a[6];
        if (FIRST) {
            const double w0 = omega[id];
            double sum = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const double w = w0 + omega[nb_index(g, id, ii[k], k, 2 * q - 1)];
                    a[2 * k + q] = k == 0 ? w : w * (k == 1 ? r2 : r3);
                }
            sum = ((a[0] + a[1]) + (a[2] + a[3])) + (a[4] + a[5]);
            const double is = rcp_nr(sum);
            // the first is 1 less the others: their sum is 1 to one rounding and a sweep adds no drift to the coordinates
#pragma unroll
            for (int m = 1; m < 6; ++m) a[m] *= is;
            a[0] = 1.0 - ((a[1] + (a[2] + a[3])) + (a[4] + a[5]));
#pragma unroll
            for (int m = 0; m < 6; ++m) W.a[m][id] = a[m];
        } else {
#pragma unroll
            for (int m = 0; m < 6; ++m) a[m] = W.a[m][id];
        }
        const bool in = inside3(g, ii[0], ii[1], ii[2], 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double* x = xin + size_t(c) * N;
            double v = 0.0;
            if (in) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    v = fma(a[2 * k + 1], x[id + st[k]], k == 0 ? a[0] * x[id - 1] : fma(a[2 * k], x[id - st[k]], v));
            } else if (fixed3(g, ii, c)) {
                v = x[id];
            } else {
                for (int k = 0; k < 3; ++k)
                    v = fma(a[2 * k + 1], nb_coord(g, x, id, ii[k], k, 1, c),
                            fma(a[2 * k], nb_coord(g, x, id, ii[k], k, -1, c), v));
            }
            if (CHG) chg = max_bits(chg, fabs(v - x[id]));
            xout[size_t(c) * N + id] = v;
        }
    }
    if (CHG) {
        block_max_bits<1>(&chg);
        if (threadIdx.x == 0) {
            atomic_max_pos(&d->red[RED_JAC], chg);
            __threadfence();
            const unsigned int ticket = atomicAdd(&d->done, 1u);
            if (ticket == gridDim.x - 1) {
                const double c = __longlong_as_double((long long)atomicAdd(&d->red[RED_JAC], 0ULL));
                if (c < eps) d->conv = 1;
                d->red[RED_JAC] = 0ULL;
                d->done = 0u;
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&d->sweeps, 1);
}

// Delta_gamma over all nodes and directions (Sec. 4): the spacing to the neighbour that a node moves towards over twice its
// displacement; the division only where it lowers the minimum so far (a node that moves less than half of its spacing, as
// nearly all do, is three FP64 instructions a direction)
__global__ void k3_limiter(Grid3 g, const double* xn, const double* xa, const double* xb, DevScalars* d) {
    const unsigned N = unsigned(g.n[0]) * g.n[1] * g.n[2];
    const double* xit = d->sweeps == 0 ? xn : (((d->sweeps - 1) & 1) ? xb : xa);
    double m = 1.0;
    for (unsigned id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i1 = int(id % unsigned(g.n[0])), r = int(id / unsigned(g.n[0]));
        const int ii[3] = {i1, r % g.n[1], r / g.n[1]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double* x = xn + size_t(k) * N;
            const double x0 = x[id], dx = xit[size_t(k) * N + id] - x0;
            if (__double_as_longlong(dx) << 1 == 0) continue;                        // +-0
            const bool back = __double2hiint(dx) < 0;
            const double xb1 = nb_coord(g, x, id, ii[k], k, back ? -1 : 1, k);
            const double gap = back ? x0 - xb1 : xb1 - x0, a = fabs(dx);
            if (gap < m * (LIMIT_TEST * a)) m = fmin(m, div_nr(gap, 2.0 * a));
        }
    }
    m = block_min(m);
    if (threadIdx.x == 0) atomic_min_pos(&d->red[RED_GAMMA], m);
}

// ================================================================ host side
cudaError_t d3_alloc(Ctx3* d) {
    const Grid3& g = d->g;
    d->N = size_t(g.n[0]) * g.n[1] * g.n[2];
    d->NE = size_t(g.n[0] + 6) * (g.n[1] + 6) * (g.n[2] + 6);
    for (int k = 0; k < 3; ++k) d->NKk[k] = d->N / g.n[k] * (g.n[k] + 6);
    cudaError_t e = cudaMalloc((void**)&d->XE, sizeof(double) * 3 * d->NE);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d->D, sizeof(double) * 9 * d->NE);
    for (int k = 0; k < 3 && e == cudaSuccess; ++k) e = cudaMalloc((void**)&d->NK[k], sizeof(double) * 3 * d->NKk[k]);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d->NF, sizeof(double) * F3_COUNT * d->N);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d->RH, sizeof(double) * 6 * d->N);
    if (e == cudaSuccess && d->mixed) e = cudaMalloc((void**)&d->XD, sizeof(float) * 3 * d->NE);
    return e;
}

void d3_free(Ctx3* d) {
    if (!d) return;
    void* b[] = {d->XE, d->D, d->NK[0], d->NK[1], d->NK[2], d->NF, d->RH, d->XD};
    for (void* p : b)
        if (p) cudaFree(p);
}

cudaError_t d3_prepare() {
    cudaError_t e = dir_prepare<0>();
    if (e == cudaSuccess) e = dir_prepare<1>();
    if (e == cudaSuccess) e = dir_prepare<2>();
    return e;
}

int d3_init_J(const Ctx3* d, const double* x, void* J, cudaStream_t s, cudaError_t* err) {
    int n = 1;
    if (d->mixed) {                                   // FP64 J into the scratch, then split
        k3_init_J<<<d->grid, 256, 0, s>>>(d->g, x, d->RH);
        n += d3f_init_J(const_cast<Ctx3*>(d), d->RH, J, s);
    } else {
        k3_init_J<<<d->grid, 256, 0, s>>>(d->g, x, (double*)J);
    }
    *err = cudaGetLastError();
    return *err == cudaSuccess ? n : -1;
}

// metrics of x_s = xn + cst dt xdot for the three directions
static int enqueue_metrics(Ctx3* d, const double* xn, const double* xdot, double cst, const double* dt_dev,
                           double dt_host, cudaStream_t s, const Stage3* inc = nullptr) {
    if (d->mixed) return d3f_metrics(d, xn, xdot, cst, dt_dev, dt_host, s, inc);
    const int G = d->grid;
    k3_coords<<<G, 256, 0, s>>>(d->g, xn, cst != 0.0 ? xdot : nullptr, cst, dt_dev, dt_host, d->XE);
    k3_deriv<<<G, 256, 0, s>>>(d->g, d->XE, d->D);
    k3_metric<0><<<G, 256, 0, s>>>(d->g, d->D, d->NK[0]);
    k3_metric<1><<<G, 256, 0, s>>>(d->g, d->D, d->NK[1]);
    k3_metric<2><<<G, 256, 0, s>>>(d->g, d->D, d->NK[2]);
    return 5;
}

int d3_stage(Ctx3* d, const Stage3& a0, DevStatus* st, cudaStream_t s, cudaError_t* err) {
    int n = 0;
    Stage3 a = a0;
    if (d->mixed && a.xdot && !a.xd_ready) {       // the mixed kernels read xdot on the extended mesh as floats
        n += d3f_form_xd(d, a.xdot, s);
        a.xd_ready = 1;
    }
    if (!a.reuse) {
        n += enqueue_metrics(d, a.xn, a.xdot, a.cst, a.dt_dev, a.dt_host, s, a.xe_incr ? &a : nullptr);
        if (d->mixed) n += d3f_nodes(d, a.JUs, a.Js, st, s);
        else {
            k3_nodes<<<d->grid, 256, 0, s>>>(d->g, d->gas, (const double*)a.JUs, (const double*)a.Js, d->NF, st);
            ++n;
        }
    }
    if (d->mixed) {
        const int m = d3f_directions(d, a, st, s, err);
        return m < 0 ? -1 : n + m;
    }
    Dir3Params P;
    P.g = d->g;
    P.gas = d->gas;
    P.weno = d->weno;
    P.diss = d->diss;
    P.NF = d->NF;
    P.xdot = a.xdot;
    P.RH = d->RH;
    P.mode = a.mode;
    P.ca = a.ca;
    P.cb = a.cb;
    P.dt_host = a.dt_host;
    P.dt_dev = a.dt_dev;
    P.JUn = (const double*)a.JUn;
    P.Jn = (const double*)a.Jn;
    P.JUs = (const double*)a.JUs;
    P.Js = (const double*)a.Js;
    P.JUo = (double*)a.JUo;
    P.Jo = (double*)a.Jo;
    P.status = st;
    cudaError_t e = cudaGetLastError();
    for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
        P.NK = d->NK[k];
        P.first = k == 0;
        P.last = k == 2;
        e = k == 0 ? dir_launch<0>(P, d->shape, s) : (k == 1 ? dir_launch<1>(P, d->shape, s) : dir_launch<2>(P, d->shape, s));
        ++n;
    }
    *err = e;
    return e == cudaSuccess ? n : -1;
}

int d3_cfl(Ctx3* d, const void* JU, const void* J, const double* x, DevScalars* dv, cudaStream_t s,
           cudaError_t* err) {
    int n = enqueue_metrics(d, x, nullptr, 0.0, nullptr, 0.0, s);
    if (d->mixed) {
        n += d3f_nodes(d, JU, J, &dv->status, s);
        n += d3f_cfl(d, J, nullptr, RED_CFL, dv, s);
    } else {
        k3_nodes<<<d->grid, 256, 0, s>>>(d->g, d->gas, (const double*)JU, (const double*)J, d->NF, &dv->status);
        k3_cfl<<<d->grid, 256, 0, s>>>(d->g, d->gas, d->NF, (const double*)J, d->NK[0], d->NK[1], d->NK[2], nullptr,
                                       RED_CFL, dv);
        n += 2;
    }
    *err = cudaGetLastError();
    return *err == cudaSuccess ? n : -1;
}

int d3_cfl_moving(Ctx3* d, const void* J, const double* xdot, DevScalars* dv, cudaStream_t s, cudaError_t* err) {
    int n;
    if (d->mixed) {
        n = d3f_cfl(d, J, xdot, RED_CFL2, dv, s);
    } else {
        k3_cfl<<<d->grid, 256, 0, s>>>(d->g, d->gas, d->NF, (const double*)J, d->NK[0], d->NK[1], d->NK[2], xdot,
                                       RED_CFL2, dv);
        n = 1;
    }
    *err = cudaGetLastError();
    return *err == cudaSuccess ? n : -1;
}

int d3_mesh(Ctx3* d, const void* JU, const void* J, const double* xn, double* xdot, DevScalars* dv,
            cudaStream_t s, cudaError_t* err, bool xe_current) {
    if (d->mixed) return d3f_mesh(d, JU, J, xn, xdot, dv, s, err, xe_current);   // FP32 pipe (es_3d_mixed.cu)
    const int G = d->grid;
    // the elementwise kernels of the 1D/2D path see the 3D mesh as N nodes in a row
    GridParams flat;
    flat.dim = 3;
    flat.n1 = int(d->N);
    flat.n2 = 1;
    flat.bc[0] = flat.bc[1] = ES_BC_PERIODIC;
    flat.inv_dxi[0] = flat.inv_dxi[1] = 1.0;
    flat.period[0] = flat.period[1] = 0.0;
    grid_floats(flat);
    int n = 0;
    launch_mon_fields(flat, d->gas, JU, J, d->rhoF, d->GF, false, G, s);
    MonScale3 sc;
    for (int k = 0; k < 3; ++k) {
        const double h = d->g.inv_dxi[k];
        sc.d1[k] = 0.25 * h * h;
        sc.d2[k] = (h * h) * (h * h);
    }
    if (d->mon.kind == ES_MONITOR_SMOOTH)
        k3_mon_terms<true><<<G, 256, 0, s>>>(d->g, sc, d->mon.kappa, d->rhoF, d->GF, d->t0, d->t1, d->t2, dv);
    else
        k3_mon_terms<false><<<G, 256, 0, s>>>(d->g, sc, d->mon.kappa, d->rhoF, d->GF, d->t0, d->t1, d->t2, dv);
    k_mon_omega<<<G, 256, 0, s>>>(flat, d->mon, d->t0, d->t1, d->t2, dv, d->om0);
    n += 3;
    double* om = d->om0;
    double* other = d->om1;
    for (int k = 0; k < d->filter_passes; ++k) {
        launch_filter3(d->g, om, other, d->nsm, s);
        ++n;
        double* t = om;
        om = other;
        other = t;
    }
    // the monitor's fields and the filter's other buffer are free: the sweeps' weights
    const SweepWeights3 W = {{d->t0, d->t1, d->t2, d->rhoF, d->GF, other}};
    const double h1 = d->g.inv_dxi[0], h2 = d->g.inv_dxi[1], h3 = d->g.inv_dxi[2];
    const double r2 = (h2 / h1) * (h2 / h1), r3 = (h3 / h1) * (h3 / h1);
    const bool check = d->eps > 0.0;
    for (int k = 0; k < d->sweeps; ++k) {
        const double* xin = k == 0 ? xn : ((k & 1) ? d->xa : d->xb);
        double* xout = (k & 1) ? d->xb : d->xa;
        if (k == 0) {
            if (check) k3_jacobi<true, true><<<G, 256, 0, s>>>(d->g, om, W, r2, r3, xin, xout, dv, d->eps);
            else k3_jacobi<true, false><<<G, 256, 0, s>>>(d->g, om, W, r2, r3, xin, xout, dv, d->eps);
        } else {
            if (check) k3_jacobi<false, true><<<G, 256, 0, s>>>(d->g, om, W, r2, r3, xin, xout, dv, d->eps);
            else k3_jacobi<false, false><<<G, 256, 0, s>>>(d->g, om, W, r2, r3, xin, xout, dv, d->eps);
        }
        ++n;
    }
    k3_limiter<<<G, 256, 0, s>>>(d->g, xn, d->xa, d->xb, dv);
    k_velocity<<<G, 256, 0, s>>>(flat, xn, d->xa, d->xb, dv, xdot);
    n += 2;
    *err = cudaGetLastError();
    return *err == cudaSuccess ? n : -1;
}

}  // namespace es
