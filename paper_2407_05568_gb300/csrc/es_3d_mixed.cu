// es_3d_mixed.cu -- the mixed-precision form of the 3D path: the direction kernels on the FP32 pipe.
//
// As in the 1D/2D mixed form, the state is kept as double-float pairs (hi + lo float planes), the
// primitive state rho, v, T of every node carries a low part so that jumps between neighbours
// keep their digits, the two-point fluxes and MR-WENO5 run in float, and the dissipation works on
// entropy-variable jumps from the jump decomposition of Sec. 3.1 (eq. jumpV) shared by the faces
// of a line (es_flux32.cuh, D = 3).  The node fields are computed once per node in double-float arithmetic and stored
// as floats (with the low parts), and the metrics are the cross-form metrics of es_3d.cu formed in double-float and
// rounded to float.  The right-hand sides are accumulated over the
// three directions in float and the Shu-Osher combination is done in double-float.
#include <cuda.h>            // CUtensorMap (the encoder is fetched from the driver at run time)
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <string.h>

#include "es_3d.h"
#include "es_bits.cuh"
#include "es_3d_filter.cuh"
#include "es_3d_grid.cuh"
#include "es_device.cuh"
#include "es_flux32.cuh"
#include "es_internal.h"
#include "es_mesh_f32.h"
#include "es_mixed_device.cuh"

namespace es {
namespace mixed3 {

using mixed::df;
using mixed::df_add;
using mixed::df_add_f;
using mixed::df_diff;
using mixed::df_second_diff;
using mixed::df_mul;
using mixed::df_mul_f;
using mixed::df_recip;
using mixed::fast_two_sum;
using mixed::two_sum;
using mixed::GasF;

// Float node fields (global planes), in the order of the direction kernels' float4: halves of rho, T, v, v/T, rho v,
// g = R/(1 - b rho) - a rho/T, a rho/T, E0 = |v|^2/(2T) + 2 a rho/T, rho/p and of the low parts of the double-float rho, T,
// v (the faces and pairs read means of two nodes, then one addition); 1/(1 - b rho) and 1/T whole.
enum FieldM {
    M_RHO, M_T, M_IOM, M_E0, M_V1, M_V2, M_V3, M_G, M_VT1, M_VT2, M_VT3, M_ART, M_RV1, M_RV2, M_RV3, M_RP,
    M_RHOL, M_TL, M_IT, M_V1L, M_V2L, M_V3L,
    MF_COUNT
};
static_assert(MF_COUNT <= 23, "the float node fields reuse the FP64 node-field buffer");

// ---------------------------------------------------------------- node fields
// From the double-float state (JU: hi plane [5][N] then lo plane; J: hi then lo) in double-float
// arithmetic on the FP32 pipe (as the 2D mixed tile does), stored as floats with the low parts of
// rho, v, T.
__global__ void k3_nodes_f(Grid3 g, GasF G, const float* JU, const float* J, float* NF, DevStatus* st) {
    const int N = g.n[0] * g.n[1] * g.n[2];
    const size_t P = size_t(N), LO = 5 * P;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const df iJ = df_recip({J[id], J[P + id]});
        const df rho = df_mul({JU[id], JU[LO + id]}, iJ);
        const df E = df_mul({JU[4 * P + id], JU[LO + 4 * P + id]}, iJ);
        const df irho = df_recip(rho);
        df m[3], v[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            m[c] = df_mul({JU[(1 + c) * P + id], JU[LO + (1 + c) * P + id]}, iJ);
            v[c] = df_mul(m[c], irho);
        }
        const df ke = df_mul_f(df_add(df_add(df_mul(v[0], v[0]), df_mul(v[1], v[1])), df_mul(v[2], v[2])), 0.5f);
        // T = (E/rho - |v|^2/2 + a rho) / cv
        const df e = df_add(df_mul(E, irho), {-ke.hi, -ke.lo});
        const df Td = df_mul_f(df_add(e, df_mul_f(rho, G.a)), G.icv);
        const float r = rho.hi, Tf = Td.hi;
        const float om = 1.0f - G.b * r;
        const float iom = flux32::rcp(om), iT = flux32::rcp(Tf);
        const float ar = G.a * r;
        const float prho = G.R * Tf * iom - ar;              // p/rho
        if (!(r > 0.0f) || !(om > 0.0f) || !(Tf > 0.0f) || !(prho > 0.0f)) raise_error(st, ES_ERR_INADMISSIBLE, id);
        const float hiT = 0.5f * iT, art = ar * hiT;
        NF[M_RHO * P + id] = 0.5f * r;
        NF[M_RHOL * P + id] = 0.5f * rho.lo;
        NF[M_T * P + id] = 0.5f * Tf;
        NF[M_TL * P + id] = 0.5f * Td.lo;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            NF[(M_V1 + c) * P + id] = 0.5f * v[c].hi;
            NF[(M_V1L + c) * P + id] = 0.5f * v[c].lo;
            NF[(M_VT1 + c) * P + id] = v[c].hi * hiT;
            NF[(M_RV1 + c) * P + id] = 0.5f * m[c].hi;
        }
        NF[M_IT * P + id] = iT;
        NF[M_IOM * P + id] = iom;
        NF[M_G * P + id] = fmaf(0.5f * G.R, iom, -art);
        NF[M_ART * P + id] = art;
        NF[M_E0 * P + id] = fmaf(ke.hi, hiT, 2.0f * art);
        NF[M_RP * P + id] = 0.5f * flux32::rcp(prho);
    }
}

// ---------------------------------------------------------------- direction kernels
// Bound by instruction issue at the occupancy that 96 registers leave (96^3, 32 x 4 pencils: 61 to 63 M warp instructions,
// 54 to 62% of the issue slots busy, the rest waits at the barriers between the phases and on shared memory; DRAM at 20%).
// With means of unhalved scalar fields, whole values W_j - W_l and exact divisions the three directions took 130, 141 and
// 159 us at 96^3; on es_flux32.cuh's forms 72, 89 and 87 us.
struct Dir3FParams {
    Grid3 g;
    GasF gas;
    flux32::WenoC weno;
    int diss;
    const float* NF;          // float node fields [MF_COUNT][N]
    const float* NK;          // metrics of this direction [3][M] (float, from k3f_metric)
    const float* XD;          // the mesh velocity on the extended mesh [3][NE] (nullable: mesh at rest)
    float* RH;                // accumulated right-hand sides [6][N] (float)
    int first, last;
    int tma;                  // xi_2 / xi_3: node fields staged by TMA (persistent grid)
    int mode;
    float ca, cb, ca_lo, cb_lo;
    double dt_host;
    const double* dt_dev;
    const float *JUn, *Jn, *JUs, *Js;   // double-float planes
    float *JUo, *Jo;
    DevStatus* status;
};

// Shared memory of a pencil of W lines: node values that are read together lie in one float4, so that a pair or face takes
// a node in a few 16-byte loads; the lines' pitch is odd, which spreads them over the banks.
template <int LB, int W>
struct PencilF {
    static constexpr int LS = (LB + 6) | 1;
    static constexpr int NB = W * LS;
    static constexpr int PL = 3 * LB + 6;
    static constexpr int NP = W * PL;
    static constexpr int NF = W * (LB + 1);
    static constexpr int NJ = W * (LB + 5);
    // float4: five groups of the node fields and (n, J xi_t), pairs, jumps, faces; float2: the last two node fields;
    // floats: the fifth components and the faces' J xi_t
    static constexpr size_t SMEM = sizeof(float) * (size_t(26) * NB + 5 * NP + 5 * NJ + 6 * NF);
    // TMA staging of the node fields of a xi_2 / xi_3 pencil: [MF_COUNT][LB + 6][W] floats, in 128-byte units
    static constexpr int STG = (W * (LB + 6) * MF_COUNT + 31) / 32 * 32;
    static constexpr size_t STG_BYTES = sizeof(float) * size_t(W) * (LB + 6) * MF_COUNT;
};

struct PencilViews {
    float4 *a, *b, *c, *d, *l, *n, *pairs, *jumps, *faces;
    float2* vl;
    float *pairsE, *jumpsE, *facesE, *facesJ;
};
template <class PC>
__device__ __forceinline__ PencilViews views(float* sm) {
    PencilViews v;
    v.a = reinterpret_cast<float4*>(sm);
    v.b = v.a + PC::NB;
    v.c = v.b + PC::NB;
    v.d = v.c + PC::NB;
    v.l = v.d + PC::NB;
    v.n = v.l + PC::NB;
    v.pairs = v.n + PC::NB;
    v.jumps = v.pairs + PC::NP;
    v.faces = v.jumps + PC::NJ;
    v.vl = reinterpret_cast<float2*>(v.faces + PC::NF);
    v.pairsE = reinterpret_cast<float*>(v.vl + PC::NB);
    v.jumpsE = v.pairsE + PC::NP;
    v.facesE = v.jumpsE + PC::NJ;
    v.facesJ = v.facesE + PC::NF;
    return v;
}
__device__ __forceinline__ flux32::Node<3> node_at(const PencilViews& v, int q) {
    const float4 a = v.a[q], b = v.b[q], c = v.c[q], d = v.d[q];
    flux32::Node<3> n;
    n.rho = a.x;
    n.T = a.y;
    n.iom = a.z;
    n.E0 = a.w;
    n.v[0] = b.x;
    n.v[1] = b.y;
    n.v[2] = b.z;
    n.g = b.w;
    n.vT[0] = c.x;
    n.vT[1] = c.y;
    n.vT[2] = c.z;
    n.art = c.w;
    n.rv[0] = d.x;
    n.rv[1] = d.y;
    n.rv[2] = d.z;
    return n;
}
__device__ __forceinline__ flux32::NodeLow<3> low_at(const PencilViews& v, int q) {
    const float4 l = v.l[q];
    const float2 w = v.vl[q];
    flux32::NodeLow<3> n;
    n.rho = l.x;
    n.T = l.y;
    n.iT = l.z;
    n.v[0] = l.w;
    n.v[1] = w.x;
    n.v[2] = w.y;
    return n;
}

// ---------------------------------------------------------------- TMA staging
// The xi_2 and xi_3 kernels run persistent: a CTA takes pencils p, p + gridDim.x, ... and, while it
// computes one, the tensor-memory accelerator copies the next pencil's node fields (a box of W lines
// along xi_1 x (LB + 6) nodes along xi_k x all MF_COUNT field planes, one cp.async.bulk.tensor) into
// the staging buffer.  The box starts at xi_1 = a0, a multiple of W >= 4 floats (16 bytes), and the
// field planes have a row pitch of n1 floats, a multiple of 4 (checked when the map is built); the
// box may reach past the mesh along xi_k and xi_1, where the copy fills zeros: those nodes are the
// ghosts and the clamped lines, which the fill phase takes by plain loads or from the clamped line.
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// bounded wait for the phase of the given parity; false when it did not complete in 2^20 polls
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity) {
    const uint32_t a = smem_u32(bar);
    for (int i = 0; i < (1 << 20); ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// one thread: the copy of pencil (a0, b, s0) into stg, completing on bar
template <int K, int LB>
__device__ __forceinline__ void stage_pencil(float* stg, const CUtensorMap* map, unsigned long long* bar,
                                             uint32_t bytes, int a0, int b, int s0) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");    // the fill phase's reads of stg come first
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    const int c1 = K == 1 ? s0 - 3 : b, c2 = K == 1 ? b : s0 - 3;
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(stg)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(a0), "r"(c1), "r"(c2), "r"(0), "r"(smem_u32(bar))
        : "memory");
}

template <int K, int LB, int W, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k3_dir_f(const __grid_constant__ Dir3FParams P,
                                                     const __grid_constant__ CUtensorMap tmap) {
    using PC = PencilF<LB, W>;
    constexpr int LS = PC::LS, NFc = PC::NF;
    extern __shared__ __align__(128) float smf[];
    __shared__ __align__(8) unsigned long long bar;
    const bool tma = K != 0 && P.tma;
    float* STG = smf;
    const PencilViews pv = views<PC>(smf + (tma ? PC::STG : 0));
    const Grid3& g = P.g;
    const int tid = threadIdx.x;
    const int nk = g.n[K];
    const int nA = K == 0 ? g.n[1] : g.n[0];
    const int nB = K == 2 ? g.n[1] : g.n[2];
    const int nseg = (nk + LB - 1) / LB;
    const int ngA = (nA + W - 1) / W;
    const int total = nseg * ngA * nB;
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const double dtd = P.dt_dev ? *P.dt_dev : P.dt_host;
    if (P.mode == 0 && P.dt_dev && dtd == 0.0) return;   // finished run
    const float dt = float(dtd);
    const int M1 = g.n[0] + (K == 0 ? 6 : 0), M2 = g.n[1] + (K == 1 ? 6 : 0), M3 = g.n[2] + (K == 2 ? 6 : 0);
    const size_t M = size_t(M1) * M2 * M3;
    const int M1e = g.n[0] + 6, M2e = g.n[1] + 6, M3e = g.n[2] + 6;     // the extended mesh (3 ghosts each way)
    const GasF& G = P.gas;
    const uint32_t stg_bytes = uint32_t(PC::STG_BYTES);
    if (tma) {
        if (tid == 0) {
            mbar_init(&bar);
            if (int(blockIdx.x) < total) {
                const int p = blockIdx.x, grp = p / nseg;
                stage_pencil<K, LB>(STG, &tmap, &bar, stg_bytes, (grp % ngA) * W, grp / ngA, (p % nseg) * LB);
            }
        }
        __syncthreads();
    }

    int iter = 0;
    for (int pen = blockIdx.x; pen < total; pen += tma ? int(gridDim.x) : total, ++iter) {   // plain: once
        const int seg = pen % nseg;
        const int grp = pen / nseg;
        const int a0 = (grp % ngA) * W;
        const int b = grp / ngA;
        const int s0 = seg * LB;
        if (tma) {
            // every thread waits for the copy itself (the acquire makes it visible); the CTA leaves together if
            // it did not arrive
            const bool ok = mbar_wait(&bar, uint32_t(iter & 1));
            if (!__syncthreads_and(ok)) {
                if (tid == 0) {
                    raise_error(P.status, ES_ERR_TIMEOUT, pen);
                    mbar_wait(&bar, uint32_t(iter & 1));         // the copy in flight, once more with the limit
                }
                return;
            }
        }

        // ---- A: node fields and metrics of the pencils
        for (int t = tid; t < W * (LB + 6); t += NT) {
            int line, q;
            if (K == 0) { line = t / (LB + 6); q = t % (LB + 6); }
            else { q = t / W; line = t % W; }
            int a = a0 + line;
            if (a > nA - 1) a = nA - 1;
            const int s = s0 + q - 3;
            const int ss = state_index(s, nk, g.bc[K]);
            int i1, i2, i3, j1, j2, j3;
            if (K == 0) { i1 = ss; i2 = a; i3 = b; }
            else if (K == 1) { i1 = a; i2 = ss; i3 = b; }
            else { i1 = a; i2 = b; i3 = ss; }
            const size_t id = idx3(g, i1, i2, i3);
            const int bx = line * LS + q;
            float v[MF_COUNT];                                   // all loads in flight before the stores
            if (tma && s >= 0 && s < nk) {                       // the staged copy: line a - a0 of the box
#pragma unroll
                for (int f = 0; f < MF_COUNT; ++f) v[f] = STG[(f * (LB + 6) + q) * W + (a - a0)];
            } else {
#pragma unroll
                for (int f = 0; f < MF_COUNT; ++f) v[f] = P.NF[f * N + id];
            }
            pv.a[bx] = make_float4(v[0], v[1], v[2], v[3]);
            pv.b[bx] = make_float4(v[4], v[5], v[6], v[7]);
            pv.c[bx] = make_float4(v[8], v[9], v[10], v[11]);
            pv.d[bx] = make_float4(v[12], v[13], v[14], v[15]);
            pv.l[bx] = make_float4(v[16], v[17], v[18], v[19]);
            pv.vl[bx] = make_float2(v[20], v[21]);
            int se = s + 3;
            se = se < 0 ? 0 : (se > nk + 5 ? nk + 5 : se);
            if (K == 0) { j1 = se; j2 = a; j3 = b; }
            else if (K == 1) { j1 = a; j2 = se; j3 = b; }
            else { j1 = a; j2 = b; j3 = se; }
            const size_t mi = (size_t(j3) * M2 + j2) * M1 + j1;
            const float nx = 0.5f * P.NK[mi], ny = 0.5f * P.NK[M + mi], nz = 0.5f * P.NK[2 * M + mi];
            float xt = 0.0f;
            if (P.XD) {     // J xi_{k,t} = -xdot . n_k, xdot from the extended mesh (its ghosts: the coordinates' rule)
                const size_t NE = size_t(M1e) * M2e * M3e;
                size_t e;
                if (K == 0) e = (size_t(b + 3) * M2e + (a + 3)) * M1e + se;
                else if (K == 1) e = (size_t(b + 3) * M2e + se) * M1e + (a + 3);
                else e = (size_t(se) * M2e + (b + 3)) * M1e + (a + 3);
                xt = -(P.XD[e] * nx + P.XD[NE + e] * ny + P.XD[2 * NE + e] * nz);
            }
            pv.n[bx] = make_float4(nx, ny, nz, xt);
        }
        __syncthreads();
        if (tma && tid == 0 && pen + int(gridDim.x) < total) {    // the staging buffer is free: next pencil
            const int p = pen + gridDim.x, gp = p / nseg;
            stage_pencil<K, LB>(STG, &tmap, &bar, stg_bytes, (gp % ngA) * W, gp / ngA, (p % nseg) * LB);
        }

        // ---- B: pair fluxes by their reach m; those with m = 1 also give the neighbour jumps V_{q+1} - V_q,
        // q = 0 .. LB + 4 (eq. jumpV)
        constexpr int c1 = W * (LB + 5), c2 = c1 + W * (LB + 2), c3 = c2 + W * (LB + 3);
        for (int t = tid; t < c3; t += NT) {
            const int m = t < c1 ? 1 : (t < c2 ? 2 : 3);
            const int u = m == 1 ? t : (m == 2 ? t - c1 : t - c2);
            const int line = m == 1 ? u / (LB + 5) : (m == 2 ? u / (LB + 2) : u / (LB + 3));
            const int pos = u - line * (LB + (m == 1 ? 5 : m));
            const int q = m == 2 ? pos + 1 : pos;
            const int l = line * LS + q, r = l + m;
            const flux32::Node<3> nl = node_at(pv, l), nr = node_at(pv, r);
            const flux32::PairMeans<3> p = flux32::pair_means<3>(nl, nr, G);
            float f[5];
            if (m == 1) {
                flux32::entropy_jump<3>(nl, nr, low_at(pv, l), low_at(pv, r), p, f);
                pv.jumps[u] = make_float4(f[0], f[1], f[2], f[3]);
                pv.jumpsE[u] = f[4];
                if (q < 2 || q > LB + 2) continue;
            }
            const float4 na = pv.n[l], nb = pv.n[r];
            const float n[3] = {na.x + nb.x, na.y + nb.y, na.z + nb.z};
            flux32::pair_flux<3>(nl, nr, p, n, na.w + nb.w, f);
            const int o = line * PC::PL + (m == 1 ? q - 2 : (m == 2 ? LB + 1 : 2 * LB + 3) + pos);
            pv.pairs[o] = make_float4(f[0], f[1], f[2], f[3]);
            pv.pairsE[o] = f[4];
        }
        __syncthreads();

        // ---- C: face fluxes
        for (int t = tid; t < NFc; t += NT) {
            const int line = t / (LB + 1);
            const int q = 2 + t - line * (LB + 1);
            const int l = line * LS + q, r = l + 1;
            // the 6th-order combination of the pairs (the energy component is a quarter); pairs of reach m start at
            // q = 3 - m
            constexpr float a1 = 1.5f, a2 = -0.3f, a3 = 1.0f / 30.0f;
            constexpr int o2 = LB, o3 = 2 * LB + 3;
            float F[5];
            {
                const float4* pb = pv.pairs + line * PC::PL + q;
                const float* pe = pv.pairsE + line * PC::PL + q;
                const float4 p1 = pb[-2], p2a = pb[o2 - 1], p2b = pb[o2], p3a = pb[o3 - 2], p3b = pb[o3 - 1], p3c = pb[o3];
                F[0] = fmaf(a1, p1.x, fmaf(a2, p2a.x + p2b.x, a3 * (p3a.x + p3b.x + p3c.x)));
                F[1] = fmaf(a1, p1.y, fmaf(a2, p2a.y + p2b.y, a3 * (p3a.y + p3b.y + p3c.y)));
                F[2] = fmaf(a1, p1.z, fmaf(a2, p2a.z + p2b.z, a3 * (p3a.z + p3b.z + p3c.z)));
                F[3] = fmaf(a1, p1.w, fmaf(a2, p2a.w + p2b.w, a3 * (p3a.w + p3b.w + p3c.w)));
                F[4] = 4.0f * fmaf(a1, pe[-2], fmaf(a2, pe[o2 - 1] + pe[o2], a3 * (pe[o3 - 2] + pe[o3 - 1] + pe[o3])));
            }
            const float4 na = pv.n[l], nb = pv.n[r];
            // sum_m alpha_m sum of the pairs' mean J xi_t, collected by node
            constexpr float b3 = a3, b2 = a2 + b3, b1 = a1 + b2;
            pv.facesJ[t] = fmaf(b1, na.w + nb.w, fmaf(b2, pv.n[l - 1].w + pv.n[r + 1].w, b3 * (pv.n[l - 2].w + pv.n[r + 2].w)));
            if (P.diss) {
                const float n[3] = {na.x + nb.x, na.y + nb.y, na.z + nb.z};
                const float4 vl = pv.b[l], vr = pv.b[r];
                const float v[3] = {vl.x + vr.x, vl.y + vr.y, vl.z + vr.z};
                const flux32::Face<3> f =
                    flux32::face_state<3>(pv.a[l].x, pv.a[r].x, pv.d[l].w, pv.d[r].w, v, n, na.w + nb.w, G, P.status);
                float w[5][5], sz[5], y[5];
                const float4* jb = pv.jumps + line * (LB + 5) + q - 2;
                const float* je = pv.jumpsE + line * (LB + 5) + q - 2;
#pragma unroll
                for (int o = 0; o < 5; ++o) {
                    const float4 j = jb[o];
                    const float d[5] = {j.x, j.y, j.z, j.w, je[o]};
                    const flux32::Rotated<3> R = flux32::rotate<3>(f, d);
                    const float sa = f.sA * R.A;
                    w[0][o] = fmaf(-f.sAc, R.B, sa);
                    w[1][o] = f.sE * fmaf(-f.hm, d[4], R.A);
                    w[2][o] = f.sT * fmaf(f.vr[1], d[4], R.rv[1]);
                    w[3][o] = f.sT * fmaf(f.vr[2], d[4], R.rv[2]);
                    w[4][o] = fmaf(f.sAc, R.B, sa);
                    if (o == 2) flux32::term_sizes<3>(f, d, R, sz);
                }
                // a wave whose plain jump is round-off adds nothing whatever its reconstruction
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    const float S = m == 1 ? f.sE : (m == 2 || m == 3 ? f.sT : f.sA);
                    y[m] = fabsf(w[m][2]) <= P.weno.tol * (S * sz[m]) ? 0.0f : flux32::weno_jump(w[m], P.weno);
                }
                flux32::add_increment<3>(f, y, F);
            }
            pv.faces[t] = make_float4(F[0], F[1], F[2], F[3]);
            pv.facesE[t] = F[4];
        }
        __syncthreads();

        // ---- D: divergence, accumulated in float; the last direction writes double-float results
        const float inv = g.finv[K];
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
            // every global operand of this node is loaded before the first global store (as far as the
            // compiler knows a store may alias a later load, which would serialise one round trip per component)
            float rh[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            float uh[6], ul[6], sh[6], sl[6];
            if (!P.first) {
#pragma unroll
                for (int c = 0; c < 6; ++c) rh[c] = P.RH[c * N + id];
            }
            const bool combine = P.last && P.mode != 1;
            if (combine) {
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    const float* un = c < 5 ? P.JUn + c * N : P.Jn;
                    const float* us = c < 5 ? P.JUs + c * N : P.Js;
                    const size_t lo = c < 5 ? 5 * N : N;
                    sh[c] = us[id];
                    sl[c] = us[lo + id];
                    uh[c] = P.ca != 0.0f ? un[id] : 0.0f;
                    ul[c] = P.ca != 0.0f ? un[lo + id] : 0.0f;
                }
            }
            const float4 fl = pv.faces[fm], fr = pv.faces[fm + 1];
            const float acc[6] = {fmaf(fl.x - fr.x, inv, rh[0]),
                                  fmaf(fl.y - fr.y, inv, rh[1]),
                                  fmaf(fl.z - fr.z, inv, rh[2]),
                                  fmaf(fl.w - fr.w, inv, rh[3]),
                                  fmaf(pv.facesE[fm] - pv.facesE[fm + 1], inv, rh[4]),
                                  fmaf(pv.facesJ[fm] - pv.facesJ[fm + 1], inv, rh[5])};
            if (!P.last) {
#pragma unroll
                for (int c = 0; c < 6; ++c) P.RH[c * N + id] = acc[c];
            } else if (P.mode == 1) {
#pragma unroll
                for (int c = 0; c < 5; ++c) {
                    P.JUo[c * N + id] = acc[c];
                    P.JUo[5 * N + c * N + id] = 0.0f;
                }
                P.Jo[id] = acc[5];
                P.Jo[N + id] = 0.0f;
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    float* uo = c < 5 ? P.JUo + c * N : P.Jo;
                    const size_t lo = c < 5 ? 5 * N : N;
                    const df Un = {uh[c], ul[c]};
                    const df Us = {sh[c], sl[c]};
                    const df inc = df_add_f(Us, dt * acc[c]);
                    df outv = df_mul(inc, {P.cb, P.cb_lo});
                    if (P.ca != 0.0f) outv = df_add(outv, df_mul(Un, {P.ca, P.ca_lo}));
                    uo[id] = outv.hi;
                    uo[lo + id] = outv.lo;
                    if (c == 5 && !(outv.hi > 0.0f)) raise_error(P.status, ES_ERR_MESH, int(id));
                }
            }
        }
        __syncthreads();                                      // the nodes, pairs, jumps and faces are refilled next
    }
}

int g_nsm = 0;                 // SMs of the device (the persistent grids), set by d3f_prepare

template <int K, int LB, int W, int NT, int MINB>
static cudaError_t prep_shape() {
    const size_t smem = PencilF<LB, W>::SMEM + (K != 0 ? sizeof(float) * PencilF<LB, W>::STG : 0);
    return cudaFuncSetAttribute(k3_dir_f<K, LB, W, NT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

template <int K, int LB, int W, int NT, int MINB>
static cudaError_t launch_shape(const Dir3FParams& P, const CUtensorMap& map, cudaStream_t s) {
    const Grid3& g = P.g;
    const int nA = K == 0 ? g.n[1] : g.n[0];
    const int nB = K == 2 ? g.n[1] : g.n[2];
    const long long blocks = (long long)((g.n[K] + LB - 1) / LB) * ((nA + W - 1) / W) * nB;
    const bool tma = K != 0 && P.tma;
    const long long resident = (long long)(g_nsm > 0 ? g_nsm : 1) * MINB;
    const long long grid = tma && blocks > resident ? resident : blocks;
    const size_t smem = PencilF<LB, W>::SMEM + (tma ? sizeof(float) * PencilF<LB, W>::STG : 0);
    k3_dir_f<K, LB, W, NT, MINB><<<unsigned(grid), NT, smem, s>>>(P, map);
    return cudaGetLastError();
}

// pencil shapes of the float kernels: 16 x 16 lines / 288 threads (two CTAs per SM), 32 x 8 / 288,
// 16 x 8 / 160 (four per SM: 96 registers and, with the TMA staging, 50 KB each), 32 x 4 / 160
template <int K>
static cudaError_t prep_dir() {
    cudaError_t e = prep_shape<K, 16, 16, 288, 2>();
    if (e == cudaSuccess) e = prep_shape<K, 32, 8, 288, 2>();
    if (e == cudaSuccess) e = prep_shape<K, 16, 8, 160, 4>();
    if (e == cudaSuccess) e = prep_shape<K, 32, 4, 160, 4>();
    return e;
}

template <int K>
static cudaError_t launch_dir(const Dir3FParams& P, const CUtensorMap& map, int shape, cudaStream_t s) {
    switch (shape) {
        case 1: return launch_shape<K, 32, 8, 288, 2>(P, map, s);
        case 2: return launch_shape<K, 16, 8, 160, 4>(P, map, s);
        case 3: return launch_shape<K, 32, 4, 160, 4>(P, map, s);
        default: return launch_shape<K, 16, 16, 288, 2>(P, map, s);
    }
}

// the driver's tensor-map encoder (fetched once; nullptr if the driver has none)
static PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
        else
            cudaGetLastError();
    }
    return fn;
}

// the tensor map of the float node fields [MF_COUNT][n3][n2][n1] with the box of one xi_k pencil (k = 1, 2):
// W nodes along xi_1, LB + 6 along xi_k, 1 along the third direction, all field planes.  Plain loads (false)
// when n1 is not a multiple of 4 (TMA strides are multiples of 16 bytes) or the encoder refuses.
template <int LB, int W>
static bool build_tmap(Ctx3* d, int k, int shape) {
    const Grid3& g = d->g;
    if (g.n[0] % 4 != 0) return false;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return false;
    CUtensorMap m;
    const cuuint64_t dims[4] = {cuuint64_t(g.n[0]), cuuint64_t(g.n[1]), cuuint64_t(g.n[2]), cuuint64_t(MF_COUNT)};
    const cuuint64_t strides[3] = {cuuint64_t(g.n[0]) * 4, cuuint64_t(g.n[0]) * g.n[1] * 4, cuuint64_t(d->N) * 4};
    const cuuint32_t box[4] = {cuuint32_t(W), cuuint32_t(k == 1 ? LB + 6 : 1), cuuint32_t(k == 2 ? LB + 6 : 1),
                               cuuint32_t(MF_COUNT)};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, d->NF, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return false;
    static_assert(sizeof(CUtensorMap) == sizeof(d->tmap[0][0]), "tensor map size");
    memcpy(d->tmap[k - 1][shape], &m, sizeof(m));
    return true;
}

static bool tmap_for(Ctx3* d, int k, int shape, CUtensorMap* out) {
    if (k == 0 || d->no_tma) return false;
    int& st = d->tmap_state[k - 1][shape];
    if (st == 0) {
        bool ok;
        switch (shape) {
            case 1: ok = build_tmap<32, 8>(d, k, shape); break;
            case 2: ok = build_tmap<16, 8>(d, k, shape); break;
            case 3: ok = build_tmap<32, 4>(d, k, shape); break;
            default: ok = build_tmap<16, 16>(d, k, shape); break;
        }
        st = ok ? 1 : -1;
    }
    if (st != 1) return false;
    memcpy(out, d->tmap[k - 1][shape], sizeof(*out));
    return true;
}

// ---------------------------------------------------------------- metrics in double-float
// The cross-form metrics of eq. SCLCoeff formed as the FP64 path forms them (k3_coords, k3_deriv, k3_metric:
// stage coordinates on the mesh extended by 3 ghosts, the products delta_l[x_p] x_q once per node, and each
// direction's metric from differences of those products), in double-float arithmetic on the FP32 pipe: the
// stage coordinates are split into (hi, lo) floats once and every product and difference keeps a 48-bit
// significand, so the metric is rounded once, to the float the direction kernels read.  On GB300 the FP64
// version of these three kernels took more time than the float direction kernels.
__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, {-b.hi, -b.lo}); }

// acc + h (a - b), the inner step of the differences: the difference of the high parts, its product with h and the sum of
// the high parts are exact, and what they leave is collected in the low part, which is normalised only where the sum is
// used (19 instructions against 28 with a normalised value after each operation; the kernels are bound by them)
__device__ __forceinline__ df df_diff_fma(df acc, float h, df a, df b, bool first) {
    const df d = two_sum(a.hi, -b.hi);
    const float lo = d.lo + (a.lo - b.lo);
    const float p = __fmul_rn(h, d.hi);
    const float e = fmaf(h, lo, fmaf(h, d.hi, -p));
    if (first) return {p, e};
    const df s = two_sum(acc.hi, p);
    return {s.hi, acc.lo + (s.lo + e)};
}

// the coordinates of x_s = xn + cst dt xdot on the extended grid as (hi, lo) planes: XEh [3][NE], XEl [3][NE]
__global__ void k3f_coords(Grid3 g, const double* xn, const double* xdot, double cst, const double* dt_dev,
                           double dt_host, float* XEh, float* XEl) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const unsigned E1 = g.n[0] + 6, E2 = g.n[1] + 6, E3 = g.n[2] + 6;
    const size_t NE = size_t(E1) * E2 * E3;
    const double cdt = cst * (dt_dev ? *dt_dev : dt_host);
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < NE; e += size_t(gridDim.x) * blockDim.x) {
        const unsigned eu = unsigned(e);                      // NE < 2^31 (es_create limits N to 2^30)
        const int i1 = int(eu % E1) - 3, i2 = int((eu / E1) % E2) - 3, i3 = int(eu / (E1 * E2)) - 3;
        const bool in = inside3(g, i1, i2, i3, 0);
        const size_t id = in ? idx3(g, i1, i2, i3) : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double v;
            if (in) v = xdot ? xn[c * N + id] + cdt * xdot[c * N + id] : xn[c * N + id];
            else v = ghost_value3(g, xn + c * N, xdot ? xdot + c * N : nullptr, cdt, i1, i2, i3, c);
            float hi, lo;
            bits::split(v, hi, lo);                          // integer operations, not FP64 conversions
            XEh[c * NE + e] = hi;
            XEl[c * NE + e] = lo;
        }
    }
}

// the mesh velocity on the extended mesh as floats XD [3][NE]: the ghost rule of the coordinates without their
// period shift (a ghost's coordinate is the ghost rule's combination of x^n + c dt xdot plus the shift, so its
// velocity is the same combination of xdot)
__global__ void k3f_xdot_ext(Grid3 g, const double* xdot, float* XD) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const unsigned E1 = g.n[0] + 6, E2 = g.n[1] + 6, E3 = g.n[2] + 6;
    const size_t NE = size_t(E1) * E2 * E3;
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < NE; e += size_t(gridDim.x) * blockDim.x) {
        const unsigned eu = unsigned(e);
        const int i1 = int(eu % E1) - 3, i2 = int((eu / E1) % E2) - 3, i3 = int(eu / (E1 * E2)) - 3;
        const bool in = inside3(g, i1, i2, i3, 0);
        const size_t id = in ? idx3(g, i1, i2, i3) : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c)
            XD[c * NE + e] = float(in ? xdot[c * N + id] : ghost_value3(g, xdot + c * N, nullptr, 0.0, i1, i2, i3, -1));
    }
}

// XE += f dt XD in double-float (f = the change of the stage-time fraction; dt from the device or the host)
__global__ void k3f_coords_add(size_t NE, float* XEh, float* XEl, const float* XD, double f, const double* dt_dev,
                               double dt_host) {
    const float a = float(f * (dt_dev ? *dt_dev : dt_host));
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < 3 * NE; e += size_t(gridDim.x) * blockDim.x) {
        const df v = df_add_f({XEh[e], XEl[e]}, a * XD[e]);
        XEh[e] = v.hi;
        XEl[e] = v.lo;
    }
}

// D[3 l + j] = delta_l[x_p] x_q (p = (j + 1) % 3, q = (j + 2) % 3; delta_l undivided, 0 where the xi_l index is
// not interior) as (hi, lo) planes Dh, Dl [9][NE]
__global__ void k3f_deriv(Grid3 g, const float* XEh, const float* XEl, float* Dh, float* Dl) {
    const unsigned E1 = g.n[0] + 6, E2 = g.n[1] + 6, E3 = g.n[2] + 6;
    const size_t NE = size_t(E1) * E2 * E3;
    const size_t st[3] = {1, size_t(E1), size_t(E1) * E2};
    for (size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x; e < NE; e += size_t(gridDim.x) * blockDim.x) {
        const unsigned eu = unsigned(e);
        const int ee[3] = {int(eu % E1), int((eu / E1) % E2), int(eu / (E1 * E2))};
        const df x[3] = {{XEh[e], XEl[e]}, {XEh[NE + e], XEl[NE + e]}, {XEh[2 * NE + e], XEl[2 * NE + e]}};
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const bool ok = ee[l] >= 3 && ee[l] < g.n[l] + 3;
            df dl[3];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                df acc = {0.0f, 0.0f};
                if (ok) {
#pragma unroll
                    for (int m = 1; m <= 3; ++m) {
                        const size_t up = p * NE + e + m * st[l], dn = p * NE + e - m * st[l];
                        acc = df_diff_fma(acc, float(0.5 * ec_alpha(m)), {XEh[up], XEl[up]}, {XEh[dn], XEl[dn]}, m == 1);
                    }
                }
                dl[p] = fast_two_sum(acc.hi, acc.lo);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const df v = df_mul(dl[(j + 1) % 3], x[(j + 2) % 3]);
                Dh[(3 * l + j) * NE + e] = v.hi;
                Dl[(3 * l + j) * NE + e] = v.lo;
            }
        }
    }
}

// J dxi_k/dx_j on direction k's grid (n_k + 6 nodes along xi_k, interior across), rounded to float [3][M]
// (the direction is a template parameter: no run-time indexing of the grid's arrays)
template <int k>
__global__ void k3f_metric(Grid3 g, const float* Dh, const float* Dl, float* NKo) {
    const unsigned E1 = g.n[0] + 6, E2 = g.n[1] + 6;
    const size_t NE = size_t(E1) * E2 * (g.n[2] + 6);
    unsigned m1 = g.n[0], m2 = g.n[1], m3 = g.n[2];
    if (k == 0) m1 += 6;
    else if (k == 1) m2 += 6;
    else m3 += 6;
    const size_t M = size_t(m1) * m2 * m3;
    const int l = (k + 1) % 3, m = (k + 2) % 3;
    const float scale = float(g.inv_dxi[l] * g.inv_dxi[m]);
    const size_t stl = l == 0 ? 1 : (l == 1 ? size_t(E1) : size_t(E1) * E2);
    const size_t stm = m == 0 ? 1 : (m == 1 ? size_t(E1) : size_t(E1) * E2);
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < M; t += size_t(gridDim.x) * blockDim.x) {
        const unsigned tu = unsigned(t);
        const int a1 = int(tu % m1), a2 = int((tu / m1) % m2), a3 = int(tu / (m1 * m2));
        const size_t e = eidx(g, a1 + (k == 0 ? 0 : 3), a2 + (k == 1 ? 0 : 3), a3 + (k == 2 ? 0 : 3));
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const size_t ol = size_t(3 * l + j) * NE, om = size_t(3 * m + j) * NE;    // delta_l[x_p] x_q, delta_m[...]
            df A = {0.0f, 0.0f};
#pragma unroll
            for (int a = 1; a <= 3; ++a) {
                const float h = float(0.5 * ec_alpha(a));
                const size_t sm = a * stm, sl = a * stl;
                A = df_diff_fma(A, h, {Dh[ol + e + sm], Dl[ol + e + sm]}, {Dh[ol + e - sm], Dl[ol + e - sm]}, a == 1);
                A = df_diff_fma(A, -h, {Dh[om + e + sl], Dl[om + e + sl]}, {Dh[om + e - sl], Dl[om + e - sl]}, false);
            }
            NKo[j * M + t] = (A.hi + A.lo) * scale;
        }
    }
}

// CFL (eq. cfl) from the float node fields and the FP64 metrics: J xi_{k,t} = -xdot . n_k, xdot = nullptr
// is a mesh at rest; the maximum goes to d->red[slot]
__global__ void k3_cfl_f(Grid3 g, Gas Gd, const float* NF, const float* J, const float* NK0, const float* NK1,
                         const float* NK2, const double* xdot, int slot, DevScalars* d) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    const size_t M[3] = {size_t(g.n[0] + 6) * g.n[1] * g.n[2], size_t(g.n[0]) * (g.n[1] + 6) * g.n[2],
                         size_t(g.n[0]) * g.n[1] * (g.n[2] + 6)};
    const float* NK[3] = {NK0, NK1, NK2};
    const float a = float(Gd.a), R = float(Gd.R), delta = float(Gd.delta);
    float mx = 0.0f;
    for (size_t id = blockIdx.x * size_t(blockDim.x) + threadIdx.x; id < N; id += size_t(gridDim.x) * blockDim.x) {
        const int i1 = int(id % g.n[0]), i2 = int((id / g.n[0]) % g.n[1]), i3 = int(id / (size_t(g.n[0]) * g.n[1]));
        const float rho = 2.0f * NF[M_RHO * N + id], T = 2.0f * NF[M_T * N + id], iom = NF[M_IOM * N + id];
        const float v[3] = {2.0f * NF[M_V1 * N + id], 2.0f * NF[M_V2 * N + id], 2.0f * NF[M_V3 * N + id]};
        const float c2 = (1.0f + delta) * R * T * (iom * iom) - 2.0f * a * rho;
        const float c = sqrtf(fmaxf(c2, 0.0f));
        const float iJ = 1.0f / J[id];
        const float vr[3] = {v[0] - (xdot ? float(xdot[id]) : 0.0f), v[1] - (xdot ? float(xdot[N + id]) : 0.0f),
                             v[2] - (xdot ? float(xdot[2 * N + id]) : 0.0f)};      // velocity relative to the mesh
        float tot = 0.0f;
        for (int k = 0; k < 3; ++k) {
            const int m1 = g.n[0] + (k == 0 ? 6 : 0), m2 = g.n[1] + (k == 1 ? 6 : 0);
            const size_t mi = (size_t(i3 + (k == 2 ? 3 : 0)) * m2 + i2 + (k == 1 ? 3 : 0)) * m1 + i1 + (k == 0 ? 3 : 0);
            const float n0 = NK[k][mi], n1 = NK[k][M[k] + mi], n2 = NK[k][2 * M[k] + mi];
            tot += (fabsf(n0 * vr[0] + n1 * vr[1] + n2 * vr[2]) + sqrtf(n0 * n0 + n1 * n1 + n2 * n2) * c) * iJ *
                   g.finv[k];
        }
        if (!(c2 > 0.0f)) tot = 3.0e38f;
        mx = fmaxf(mx, tot);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomic_max_pos(&d->red[slot], double(mx));
}

// J (FP64, from the FP64 kernel) into double-float planes
__global__ void k3_split(const double* a, float* out, size_t n) {
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
        const float hi = float(a[i]);
        out[i] = hi;
        out[n + i] = float(a[i] - double(hi));
    }
}


// ---------------------------------------------------------------- mesh redistribution (Sec. 4)
// On the FP32 pipe, with the Jacobi iteration written for the displacement delta = x - x^n from
// the mesh at t^n.  omega is fixed during the sweeps, so x^[nu+1]_i = sum_nb a_nb x^[nu]_nb with
// a_nb = w_nb / sum_nb w_nb becomes delta^[nu+1]_i = g_i + sum_nb a_nb delta^[nu]_nb, where
// g_i = sum_nb a_nb (x^n_nb - x^n_i) is formed once per solve in double-float from x^n on the
// extended mesh (the stage metrics' coordinates, ghosts with the period shift) and then rounded:
// the sweeps round only the displacement, which is small against the spacing.
// The mixed form has periodic and outflow ends only; every node on an outflow end is fixed, so a
// node that moves has its six neighbours in the mesh or across a periodic end, where delta wraps
// (x shifts by the period, delta does not).

__device__ __forceinline__ void split3(const Grid3& g, int id, int* ii) {
    const int r = id / g.n[0];
    ii[0] = id - r * g.n[0];
    ii[2] = r / g.n[1];
    ii[1] = r - ii[2] * g.n[1];
}

__device__ __forceinline__ int stride3i(const Grid3& g, int k) {
    return k == 0 ? 1 : (k == 1 ? g.n[0] : g.n[0] * g.n[1]);
}

// neighbour at s = +-1 along k, ghosts by copy (outflow) or wrap (periodic)
__device__ __forceinline__ int nb3(const Grid3& g, int id, int ik, int k, int s) {
    const int j = state_index(ik + s, g.n[k], g.bc[k]);
    return id + (j - ik) * stride3i(g, k);
}

__device__ __forceinline__ bool fixed_node3(const Grid3& g, const int* ii) {
    bool f = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) f = f || (g.bc[k] != ES_BC_PERIODIC && (ii[k] == 0 || ii[k] == g.n[k] - 1));
    return f;
}

__device__ __forceinline__ float warp_max_f(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float warp_min_f(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// the raw monitor terms of eq. van der Waalsmonitor (or the smooth-test monitor) from the
// float density and G: central first and second differences along each direction
// rhoF, GF: (hi, lo) float planes of the density and G (k_mon_fields_f); the differences of neighbours
// are taken in double-float arithmetic and then rounded
__global__ void k3f_mon_terms(Grid3 g, MonitorParams mp, const float* rhoF, const float* GF, float* t0, float* t1,
                              float* t2, DevScalars* d) {
    const int N = g.n[0] * g.n[1] * g.n[2];
    float m0 = 0.0f, m1 = 0.0f, m2 = 0.0f;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        int ii[3];
        split3(g, id, ii);
        const df r0 = {rhoF[id], rhoF[N + id]}, G0 = {GF[id], GF[N + id]};
        float gr = 0.0f, gg = 0.0f, lg = 0.0f, lr = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float h = g.finv[k];
            const int ip = nb3(g, id, ii[k], k, 1), im = nb3(g, id, ii[k], k, -1);
            const df rp = {rhoF[ip], rhoF[N + ip]}, rm = {rhoF[im], rhoF[N + im]};
            const df Gp = {GF[ip], GF[N + ip]}, Gm = {GF[im], GF[N + im]};
            const float a = df_diff(rp, rm) * 0.5f * h, b = df_diff(Gp, Gm) * 0.5f * h;
            const float c = df_second_diff(Gp, G0, Gm) * h * h, e = df_second_diff(rp, r0, rm) * h * h;
            gr += a * a;
            gg += b * b;
            lg += c * c;
            lr += e * e;
        }
        float v0, v1, v2;
        if (mp.kind == ES_MONITOR_SMOOTH) {
            v0 = sqrtf(gr);
            v1 = 0.0f;
            v2 = sqrtf(lr);
        } else {
            v0 = gr;
            v1 = mp.kappa >= 2 ? gg : 0.0f;
            v2 = lg;
        }
        t0[id] = v0;
        t1[id] = v1;
        t2[id] = v2;
        m0 = fmaxf(m0, v0);
        m1 = fmaxf(m1, v1);
        m2 = fmaxf(m2, v2);
    }
    m0 = warp_max_f(m0);
    m1 = warp_max_f(m1);
    m2 = warp_max_f(m2);
    if ((threadIdx.x & 31) == 0) {
        atomic_max_pos(&d->red[RED_MON0], double(m0));
        atomic_max_pos(&d->red[RED_MON1], double(m1));
        atomic_max_pos(&d->red[RED_MON2], double(m2));
    }
}

// the sweep coefficients of every node: a_nb for the six neighbours ([6][N], order -xi_1, +xi_1,
// -xi_2, ...) and g ([3][N]); zero at fixed nodes
__global__ void k3f_coeffs(Grid3 g, const float* om, const float* XEh, const float* XEl, float* A, float* Gc) {
    const int N = g.n[0] * g.n[1] * g.n[2];
    const size_t P = size_t(N);
    const size_t NE = size_t(g.n[0] + 6) * (g.n[1] + 6) * (g.n[2] + 6);
    const size_t est[3] = {1, size_t(g.n[0] + 6), size_t(g.n[0] + 6) * (g.n[1] + 6)};
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        int ii[3];
        split3(g, id, ii);
        if (fixed_node3(g, ii)) {
#pragma unroll
            for (int m = 0; m < 6; ++m) A[m * P + id] = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) Gc[c * P + id] = 0.0f;
            continue;
        }
        const float w0 = om[id];
        float w[6], den = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float ih2 = g.finv2[k];
            w[2 * k] = 0.5f * (w0 + om[nb3(g, id, ii[k], k, -1)]) * ih2;
            w[2 * k + 1] = 0.5f * (w0 + om[nb3(g, id, ii[k], k, 1)]) * ih2;
            den += w[2 * k] + w[2 * k + 1];
        }
        const float iden = 1.0f / den;
        // x^n_nb - x^n_i from the extended mesh (ghosts with the period shift), in double-float
        const size_t e = eidx(g, ii[0] + 3, ii[1] + 3, ii[2] + 3);
        df gs[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float am = w[2 * k] * iden, ap = w[2 * k + 1] * iden;
            A[(2 * k) * P + id] = am;
            A[(2 * k + 1) * P + id] = ap;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const size_t o = c * NE + e;
                const df xi = {XEh[o], XEl[o]};
                const df dm = df_sub({XEh[o - est[k]], XEl[o - est[k]]}, xi);
                const df dp = df_sub({XEh[o + est[k]], XEl[o + est[k]]}, xi);
                gs[c] = df_add(gs[c], df_add(df_mul_f(dm, am), df_mul_f(dp, ap)));
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) Gc[c * P + id] = gs[c].hi + gs[c].lo;
    }
}

// Jacobi sweep k on the displacement (sweep 0 starts from delta = 0 and writes da; sweep k reads
// buf[(k - 1) % 2] and writes buf[k % 2]); with `check` the last block to finish compares the
// grid's max change with eps and latches convergence, after which the remaining sweeps return
__global__ void k3f_jacobi(Grid3 g, const float* A, const float* Gc, float* da, float* db, int k, DevScalars* d,
                           int check, double eps) {
    if (d->conv) return;
    const int N = g.n[0] * g.n[1] * g.n[2];
    const size_t P = size_t(N);
    const float* din = k == 0 ? nullptr : (((k - 1) & 1) ? db : da);
    float* dout = (k & 1) ? db : da;
    float chg = 0.0f;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        int ii[3];
        split3(g, id, ii);
        if (fixed_node3(g, ii)) {
#pragma unroll
            for (int c = 0; c < 3; ++c) dout[c * P + id] = 0.0f;
            continue;
        }
        float v[3] = {Gc[id], Gc[P + id], Gc[2 * P + id]};
        if (din) {
#pragma unroll
            for (int kk = 0; kk < 3; ++kk) {
                const float am = A[(2 * kk) * P + id], ap = A[(2 * kk + 1) * P + id];
                const int im = nb3(g, id, ii[kk], kk, -1), ip = nb3(g, id, ii[kk], kk, 1);
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] += am * din[c * P + im] + ap * din[c * P + ip];
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            chg = fmaxf(chg, fabsf(v[c] - (din ? din[c * P + id] : 0.0f)));
            dout[c * P + id] = v[c];
        }
    }
    if (check) {
        chg = warp_max_f(chg);
        __shared__ float sh[32];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (lane == 0) sh[w] = chg;
        __syncthreads();
        if (threadIdx.x == 0) {
            float m = 0.0f;
            for (int i = 0; i < int(blockDim.x + 31) / 32; ++i) m = fmaxf(m, sh[i]);
            atomic_max_pos(&d->red[RED_JAC], double(m));
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

__device__ __forceinline__ const float* sweep_result(const DevScalars* d, const float* da, const float* db) {
    if (d->sweeps == 0) return nullptr;
    return ((d->sweeps - 1) & 1) ? db : da;
}

// Delta_gamma over all nodes and directions (Sec. 4): the spacing to the neighbour the node
// moves towards, over twice its displacement along that direction
__global__ void k3f_limiter(Grid3 g, const float* XEh, const float* XEl, const float* da, const float* db,
                            DevScalars* d) {
    const int N = g.n[0] * g.n[1] * g.n[2];
    const size_t P = size_t(N);
    const size_t NE = size_t(g.n[0] + 6) * (g.n[1] + 6) * (g.n[2] + 6);
    const size_t est[3] = {1, size_t(g.n[0] + 6), size_t(g.n[0] + 6) * (g.n[1] + 6)};
    const float* dl = sweep_result(d, da, db);
    float m = 1.0f;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; dl && id < N; id += gridDim.x * blockDim.x) {
        int ii[3];
        split3(g, id, ii);
        if (fixed_node3(g, ii)) continue;
        const size_t e = eidx(g, ii[0] + 3, ii[1] + 3, ii[2] + 3);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float dx = dl[k * P + id];
            const size_t o = k * NE + e;                       // component k of x^n along direction k
            if (dx < 0.0f)
                m = fminf(m, df_diff({XEh[o], XEl[o]}, {XEh[o - est[k]], XEl[o - est[k]]}) / (-2.0f * dx));
            else if (dx > 0.0f)
                m = fminf(m, df_diff({XEh[o + est[k]], XEl[o + est[k]]}, {XEh[o], XEl[o]}) / (2.0f * dx));
        }
    }
    m = warp_min_f(m);
    if ((threadIdx.x & 31) == 0) atomic_min_pos(&d->red[RED_GAMMA], double(m));
}

// xdot = Delta_gamma delta^[mu] / dt (FP64, the API's array)
__global__ void k3f_velocity(Grid3 g, const float* da, const float* db, DevScalars* d, double* xdot) {
    const int N = g.n[0] * g.n[1] * g.n[2];
    const size_t P = size_t(N);
    const float* dl = sweep_result(d, da, db);
    // Delta_gamma / dt once per block (an FP64 division); the velocity in float, widened from its bits
    __shared__ float fs;
    if (threadIdx.x == 0) {
        const double gam = __longlong_as_double((long long)d->red[RED_GAMMA]);
        const double dt = d->dt;
        fs = dt > 0.0 ? float(gam / dt) : 0.0f;
    }
    __syncthreads();
    const float f = fs;
    for (size_t id = blockIdx.x * size_t(blockDim.x) + threadIdx.x; id < 3 * P; id += size_t(gridDim.x) * blockDim.x)
        xdot[id] = dl ? bits::widen(f * dl[id]) : 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        d->gamma = __longlong_as_double((long long)d->red[RED_GAMMA]);
        d->sweeps_total += d->sweeps;
        d->solves += 1;
    }
}

}  // namespace mixed3

using namespace mixed3;

cudaError_t d3f_prepare() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = prep_dir<0>();
    if (e == cudaSuccess) e = prep_dir<1>();
    if (e == cudaSuccess) e = prep_dir<2>();
    return e;
}

static GasF gasf(const Gas& g) {
    GasF G;
    G.a = float(g.a);
    G.b = float(g.b);
    G.R = float(g.R);
    G.cv = float(g.cv);
    G.delta = float(g.delta);
    G.Rb = float(g.R * g.b);
    G.icv = float(1.0 / g.cv);
    G.iR = float(1.0 / g.R);
    G.idelta = float(g.cv / g.R);
    return G;
}

int d3f_metrics(Ctx3* d, const double* xn, const double* xdot, double cst, const double* dt_dev, double dt_host,
                cudaStream_t s, const Stage3* inc) {
    const int G = d->grid;
    const size_t NE = d->NE;
    float* XEh = (float*)d->XE;                   // [3][NE] doubles hold the (hi, lo) float planes
    float* Dh = (float*)d->D;                     // [9][NE] likewise
    int n = 4;
    if (inc && xdot) {                            // within a step: move the coordinates the buffer holds (d->XD
                                                  // holds xdot: d3_stage formed it)
        k3f_coords_add<<<G, 256, 0, s>>>(NE, XEh, XEh + 3 * NE, d->XD, cst - inc->xe_cst, dt_dev, dt_host);
    } else {
        k3f_coords<<<G, 256, 0, s>>>(d->g, xn, cst != 0.0 ? xdot : nullptr, cst, dt_dev, dt_host, XEh, XEh + 3 * NE);
    }
    k3f_deriv<<<G, 256, 0, s>>>(d->g, XEh, XEh + 3 * NE, Dh, Dh + 9 * NE);
    k3f_metric<0><<<G, 256, 0, s>>>(d->g, Dh, Dh + 9 * NE, (float*)d->NK[0]);
    k3f_metric<1><<<G, 256, 0, s>>>(d->g, Dh, Dh + 9 * NE, (float*)d->NK[1]);
    k3f_metric<2><<<G, 256, 0, s>>>(d->g, Dh, Dh + 9 * NE, (float*)d->NK[2]);
    return n + 1;
}

int d3f_form_xd(Ctx3* d, const double* xdot, cudaStream_t s) {
    k3f_xdot_ext<<<d->grid, 256, 0, s>>>(d->g, xdot, d->XD);
    return 1;
}

int d3f_nodes(Ctx3* d, const void* JU, const void* J, DevStatus* st, cudaStream_t s) {
    k3_nodes_f<<<d->grid, 256, 0, s>>>(d->g, gasf(d->gas), (const float*)JU, (const float*)J, (float*)d->NF, st);
    return 1;
}

int d3f_cfl(Ctx3* d, const void* J, const double* xdot, int slot, DevScalars* dv, cudaStream_t s) {
    k3_cfl_f<<<d->grid, 256, 0, s>>>(d->g, d->gas, (const float*)d->NF, (const float*)J, (const float*)d->NK[0],
                                      (const float*)d->NK[1], (const float*)d->NK[2], xdot, slot, dv);
    return 1;
}

int d3f_init_J(Ctx3* d, const double* Jd, void* J, cudaStream_t s) {
    k3_split<<<d->grid, 256, 0, s>>>(Jd, (float*)J, d->N);
    return 1;
}

int d3f_directions(Ctx3* d, const Stage3& a, DevStatus* st, cudaStream_t s, cudaError_t* err) {
    Dir3FParams P;
    P.g = d->g;
    P.gas = gasf(d->gas);
    P.weno = flux32::weno_floats(d->weno);
    P.diss = d->diss;
    P.NF = (const float*)d->NF;
    P.XD = a.xdot ? d->XD : nullptr;          // d3_stage formed it from a.xdot
    P.RH = (float*)d->RH;
    P.mode = a.mode;
    P.ca = float(a.ca);
    P.cb = float(a.cb);
    P.ca_lo = float(a.ca - double(P.ca));
    P.cb_lo = float(a.cb - double(P.cb));
    P.dt_host = a.dt_host;
    P.dt_dev = a.dt_dev;
    P.JUn = (const float*)a.JUn;
    P.Jn = (const float*)a.Jn;
    P.JUs = (const float*)a.JUs;
    P.Js = (const float*)a.Js;
    P.JUo = (float*)a.JUo;
    P.Jo = (float*)a.Jo;
    P.status = st;
    cudaError_t e = cudaGetLastError();
    int n = 0;
    for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
        P.NK = (const float*)d->NK[k];
        P.first = k == 0;
        P.last = k == 2;
        CUtensorMap map;
        memset(&map, 0, sizeof(map));
        P.tma = tmap_for(d, k, d->shape, &map) ? 1 : 0;
        e = k == 0 ? launch_dir<0>(P, map, d->shape, s)
                   : (k == 1 ? launch_dir<1>(P, map, d->shape, s) : launch_dir<2>(P, map, d->shape, s));
        ++n;
    }
    *err = e;
    return e == cudaSuccess ? n : -1;
}

int d3f_mesh(Ctx3* d, const void* JU, const void* J, const double* xn, double* xdot, DevScalars* dv,
             cudaStream_t s, cudaError_t* err, bool xe_current) {
    const int G = d->grid;
    int n = 0;
    // the sweep coefficients and the limiter read x^n on the extended mesh as double-float planes, which the
    // step's time-step pass has just formed for its metrics (xe_current); otherwise form them here
    float* XEh = (float*)d->XE;
    float* XEl = XEh + 3 * d->NE;
    if (!xe_current) {
        k3f_coords<<<G, 256, 0, s>>>(d->g, xn, nullptr, 0.0, nullptr, 0.0, XEh, XEl);
        ++n;
    }
    // the elementwise kernels of the 1D/2D mixed path see the 3D mesh as N nodes in a row
    GridParams flat;
    flat.dim = 3;
    flat.n1 = int(d->N);
    flat.n2 = 1;
    flat.bc[0] = flat.bc[1] = ES_BC_PERIODIC;
    flat.inv_dxi[0] = flat.inv_dxi[1] = 1.0;
    flat.period[0] = flat.period[1] = 0.0;
    grid_floats(flat);
    float* rho = (float*)d->rhoF;
    float* Gf = (float*)d->GF;
    float* t0 = (float*)d->t0;
    float* t1 = (float*)d->t1;
    float* t2 = (float*)d->t2;
    float* om = (float*)d->om0;
    float* other = (float*)d->om1;
    float* A = (float*)d->xa;                     // [6][N] floats in the [3][N] doubles
    float* da = (float*)d->xb;                    // two [3][N] float displacements
    float* db = da + 3 * d->N;               // (xb holds [3][N] doubles)
    k_mon_fields_f<<<G, 256, 0, s>>>(flat, gas_f32(d->gas), (const float*)JU, (const float*)J, rho, Gf);
    k3f_mon_terms<<<G, 256, 0, s>>>(d->g, d->mon, rho, Gf, t0, t1, t2, dv);
    k_mon_omega_f<<<G, 256, 0, s>>>(flat, d->mon, t0, t1, t2, dv, om);
    n += 3;
    for (int k = 0; k < d->filter_passes; ++k) {
        launch_filter3(d->g, om, other, d->nsm, s);
        ++n;
        float* t = om;
        om = other;
        other = t;
    }
    k3f_coeffs<<<G, 256, 0, s>>>(d->g, om, XEh, XEl, A, d->gc);
    ++n;
    const int check = d->eps > 0.0;
    for (int k = 0; k < d->sweeps; ++k) {
        k3f_jacobi<<<G, 256, 0, s>>>(d->g, A, d->gc, da, db, k, dv, check, d->eps);
        ++n;
    }
    k3f_limiter<<<G, 256, 0, s>>>(d->g, XEh, XEl, da, db, dv);
    k3f_velocity<<<G, 256, 0, s>>>(d->g, da, db, dv, xdot);
    n += 2;
    *err = cudaGetLastError();
    return *err == cudaSuccess ? n : -1;
}

}  // namespace es
