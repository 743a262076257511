// es_mesh64.cu -- the FP64 mesh redistribution of Sec. 4 in 1D and 2D: monitor, low-pass filter, Jacobi sweeps of the
// discretised Winslow equation, movement limiter.
//
// Two regimes.  On a large mesh every kernel is bound by the FP64 pipe (two lanes per clock on an SM), so the kernels
// count FP64 instructions: maxima and sign tests work on the numbers' bits, squares and spacings are folded into
// constants, the filter takes row sums once for the rows that share them, and the sweeps' normalised weights are formed
// by the first sweep and read by the others.  On a small mesh a kernel is one thread's chain of dependent work plus the
// launch, so the filter's passes, and the sweeps with the limiter, are one launch each, on tiles with a halo as wide as
// the number of passes (k_filter_tile, k_sweep_tile).
#include <cuda_runtime.h>

#include "es_aux.h"
#include "es_device.cuh"
#include "es_mesh64.cuh"

namespace es {

// ------------------------------------------------------------ monitor
__device__ __forceinline__ double field_at(const GridParams& g, const double* f, int i, int j) {
    const int si = state_index(i, g.n1, g.bc[0]);
    const int sj = g.dim == 2 ? state_index(j, g.n2, g.bc[1]) : 0;
    return f[size_t(sj) * g.n1 + si];
}

// raw monitor terms and their grid maxima: sum_k of the squared first differences of rho and of G, and of the squared
// second differences of G (eq. van der Waalsmonitor), or the norms of rho's (eq. van der Waalssinmonitor)
// (a template: with a run-time choice the compiler formed the square roots of the other monitor ahead of it)
template <bool SMOOTH>
__global__ void k_mon_terms(GridParams g, MonitorParams mp, const double* __restrict__ rhoF,
                            const double* __restrict__ GF, double* __restrict__ t0, double* __restrict__ t1,
                            double* __restrict__ t2, DevScalars* d) {
    const int N = g.n1 * g.n2;
    const bool two = !SMOOTH && mp.kappa >= 2;
    double mx[3] = {0.0, 0.0, 0.0};
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i = id % g.n1, j = id / g.n1;
        const int xm = state_index(i - 1, g.n1, g.bc[0]) - i, xp = state_index(i + 1, g.n1, g.bc[0]) - i;
        const int ym = g.dim == 2 ? (state_index(j - 1, g.n2, g.bc[1]) - j) * g.n1 : 0;
        const int yp = g.dim == 2 ? (state_index(j + 1, g.n2, g.bc[1]) - j) * g.n1 : 0;
        const double* F = SMOOTH ? rhoF : GF;               // the field of the second differences
        double gr, gg = 0.0, lg;
        {
            const double a = rhoF[id + xp] - rhoF[id + xm];
            gr = (a * g.d1sq[0]) * a;
            const double fp = F[id + xp], fm = F[id + xm];
            if (two) {
                const double b = fp - fm;
                gg = (b * g.d1sq[0]) * b;
            }
            const double s = fma(-2.0, F[id], fp + fm);
            lg = (s * g.d2sq[0]) * s;
        }
        if (g.dim == 2) {
            const double a = rhoF[id + yp] - rhoF[id + ym];
            gr = fma(a * g.d1sq[1], a, gr);
            const double fp = F[id + yp], fm = F[id + ym];
            if (two) {
                const double b = fp - fm;
                gg = fma(b * g.d1sq[1], b, gg);
            }
            const double s = fma(-2.0, F[id], fp + fm);
            lg = fma(s * g.d2sq[1], s, lg);
        }
        if (SMOOTH) {
            gr = sqrt(gr);
            lg = sqrt(lg);
        }
        t0[id] = gr;
        t1[id] = gg;
        t2[id] = lg;
        mx[0] = max_bits(mx[0], gr);
        mx[1] = max_bits(mx[1], gg);
        mx[2] = max_bits(mx[2], lg);
    }
    block_max_bits<3>(mx);
    if (threadIdx.x == 0) {
        atomic_max_pos(&d->red[RED_MON0], mx[0]);
        atomic_max_pos(&d->red[RED_MON1], mx[1]);
        atomic_max_pos(&d->red[RED_MON2], mx[2]);
    }
}

void launch_mon_terms(const GridParams& g, const MonitorParams& mp, const double* rhoF, const double* GF, double* t0,
                      double* t1, double* t2, DevScalars* d, int grid, int block, cudaStream_t s) {
    if (mp.kind == ES_MONITOR_SMOOTH) k_mon_terms<true><<<grid, block, 0, s>>>(g, mp, rhoF, GF, t0, t1, t2, d);
    else k_mon_terms<false><<<grid, block, 0, s>>>(g, mp, rhoF, GF, t0, t1, t2, d);
}

// omega's coefficient alpha_k / max_k (0: the term is dropped)
__device__ __forceinline__ double mon_coef(const MonitorParams& mp, const DevScalars* d, int k) {
    const double M = __longlong_as_double((long long)d->red[RED_MON0 + k]);
    const double w = k == 0 ? mp.w0 : (k == 1 ? mp.w1 : mp.w2);
    return M > 0.0 ? w / M : 0.0;
}
__device__ __forceinline__ double omega_of(double c0, double c1, double c2, double t0, double t1, double t2) {
    const double q = fma(c2, t2, fma(c1, t1, fma(c0, t0, 1.0)));
    return q * rsqrt_nr(q);
}

__global__ void k_mon_omega(GridParams g, MonitorParams mp, const double* __restrict__ t0,
                            const double* __restrict__ t1, const double* __restrict__ t2, const DevScalars* d,
                            double* __restrict__ omega) {
    const int N = g.n1 * g.n2;
    const double c0 = mon_coef(mp, d, 0), c1 = mon_coef(mp, d, 1), c2 = mon_coef(mp, d, 2);
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x)
        omega[id] = omega_of(c0, c1, c2, t0[id], t1[id], t2[id]);
}

// ------------------------------------------------------------ low-pass filter
// omega_i <- sum_{j in {0,+-1}^d} (1/2)^(|j|_1 + d) omega_{i+j}, one pass.  A thread takes FILTER_ROWS rows of a column:
// the row sums (l + r) + 2 c of FILTER_ROWS + 2 rows serve all of them, 6 FP64 instructions a node instead of 12.
constexpr int FILTER_ROWS = 4;
__global__ void k_filter(GridParams g, const double* __restrict__ in, double* __restrict__ out) {
    const int bands = g.dim == 2 ? (g.n2 + FILTER_ROWS - 1) / FILTER_ROWS : 1;
    const int items = g.n1 * bands;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < items; t += gridDim.x * blockDim.x) {
        const int i = t % g.n1, j0 = t / g.n1 * FILTER_ROWS;
        const int im = state_index(i - 1, g.n1, g.bc[0]), ip = state_index(i + 1, g.n1, g.bc[0]);
        if (g.dim == 1) {
            out[i] = 0.25 * fma(2.0, in[i], in[im] + in[ip]);
            continue;
        }
        double s[FILTER_ROWS + 2];
#pragma unroll
        for (int r = 0; r < FILTER_ROWS + 2; ++r) {
            // (rows past the mesh's end are not written; state_index keeps their reads inside)
            const double* row = in + size_t(state_index(min(j0 + r - 1, g.n2), g.n2, g.bc[1])) * g.n1;
            s[r] = fma(2.0, row[i], row[im] + row[ip]);
        }
#pragma unroll
        for (int r = 0; r < FILTER_ROWS; ++r)
            if (j0 + r < g.n2) out[size_t(j0 + r) * g.n1 + i] = 0.0625 * fma(2.0, s[r + 1], s[r] + s[r + 2]);
    }
}

// ------------------------------------------------------------ Jacobi sweeps
// The normalised weights of a node's neighbours (xi_1 +, -, xi_2 +, -): w_{k,+-} = (omega_i + omega_{i +- e_k})/(2
// dxi_k^2) over their sum, from omega (2/dxi_2^2 drops out; r = (dxi_2/dxi_1)^2).  The first is 1 less the others, so that
// their sum is 1 to one rounding and a sweep adds no drift to the coordinates.
__device__ __forceinline__ void sweep_weights(const GridParams& g, double w0, const double* nb, double* a) {
    a[0] = w0 + nb[0];
    a[1] = w0 + nb[1];
    if (g.dim == 1) {
        a[1] *= rcp_nr(a[0] + a[1]);
        a[0] = 1.0 - a[1];
        return;
    }
    a[2] = w0 + nb[2];
    a[3] = w0 + nb[3];
    const double q = rcp_nr(fma(g.ratio, a[0] + a[1], a[2] + a[3]));
    a[1] *= q * g.ratio;
    a[2] *= q;
    a[3] *= q;
    a[0] = (1.0 - a[1]) - (a[2] + a[3]);
}

// Coordinate component c of a boundary node that does not move: every component on an outflow end,
// the normal one on a wall or symmetry end (the node slides along it).
__device__ __forceinline__ bool fixed_coord(const GridParams& g, int i, int j, int c) {
    bool f = false;
    if (g.bc[0] != ES_BC_PERIODIC && (i == 0 || i == g.n1 - 1)) f = !end_mirrored(g.bc[0], i == 0) || c == 0;
    if (g.dim == 2 && g.bc[1] != ES_BC_PERIODIC && (j == 0 || j == g.n2 - 1))
        f = f || !end_mirrored(g.bc[1], j == 0) || c == 1;
    return f;
}

// The coordinate of the neighbour of a MOVING component at offset s (|s| = 1) along direction k: in the mesh, wrapped
// with the period shift, or (c tangential to a wall) mirrored.  (An outflow end's nodes do not move.)
__device__ __forceinline__ double coord_beside(const GridParams& g, const double* x, int id, int pos, int k, int s,
                                               int c) {
    const int n = k == 0 ? g.n1 : g.n2, st = k == 0 ? 1 : g.n1, bc = k == 0 ? g.bc[0] : g.bc[1];
    const int q = pos + s;
    if (q >= 0 && q < n) return x[id + s * st];
    if (bc == ES_BC_PERIODIC) {
        const double v = x[id + (q < 0 ? n - 1 : 1 - n) * st];
        return c == k ? v + (q < 0 ? -1.0 : 1.0) * (k == 0 ? g.period[0] : g.period[1]) : v;
    }
    return x[id - s * st];
}

// The limiter's bound at one node and component: it moves by dx; `room`, the spacing towards the neighbour it moves to.
// gamma = min(gamma, room/(2 |dx|)) over the grid: the quotient is formed, and the grid's minimum lowered, only where it
// can be below what the grid has reached so far (m; reading an older, larger value only costs the quotient).  The test is
// against the bound enlarged by 2^-50: m t is rounded, and where that gives `room` itself the quotient can still be an ulp
// below m, so that the test would let the order of the nodes decide between quotients that close.
__device__ __forceinline__ double grid_limit(const DevScalars* d) {
    return __longlong_as_double((long long)__ldcg(&d->red[RED_GAMMA]));
}
__device__ __forceinline__ double limit_by(double m, double dx, double room, DevScalars* d) {
    const double a = fabs(dx);
    if (room < m * (LIMIT_TEST * a)) {
        const double q = div_nr(room, 2.0 * a);
        if (q < m) {
            atomic_min_pos(&d->red[RED_GAMMA], q);
            m = q;
        }
    }
    return m;
}

// One sweep from xin into xout over the grid.  The first sweep forms the weights from omega and keeps them in w
// (FIRST); the others read them: 8 FP64 instructions a node for both components instead of about 50.  CHG: returns this
// thread's largest change; LIMIT: also lowers RED_GAMMA to the limiter's bound Delta_gamma at every node, from the
// result and x^n = xn.
template <bool FIRST, bool CHG, bool LIMIT>
__device__ __forceinline__ double sweep_nodes(const GridParams& g, const double* __restrict__ omega, const SweepWeights& w,
                                              const double* xin, double* xout, const double* xn, DevScalars* d) {
    const int N = g.n1 * g.n2;
    double chg = 0.0;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i = id % g.n1, j = id / g.n1;
        double m = LIMIT ? grid_limit(d) : 1.0;
        double a[4];
        if (FIRST) {
            const double nb[4] = {field_at(g, omega, i + 1, j), field_at(g, omega, i - 1, j),
                                  g.dim == 2 ? field_at(g, omega, i, j + 1) : 0.0,
                                  g.dim == 2 ? field_at(g, omega, i, j - 1) : 0.0};
            sweep_weights(g, omega[id], nb, a);
            w.w[0][id] = a[0];
            w.w[1][id] = a[1];
            if (g.dim == 2) {
                w.w[2][id] = a[2];
                w.w[3][id] = a[3];
            }
        } else {
            a[0] = w.w[0][id];
            a[1] = w.w[1][id];
            if (g.dim == 2) {
                a[2] = w.w[2][id];
                a[3] = w.w[3][id];
            }
        }
        const bool inside = i > 0 && i < g.n1 - 1 && (g.dim == 1 || (j > 0 && j < g.n2 - 1));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (c >= g.dim) break;
            const double* x = xin + size_t(c) * N;
            double v;
            if (inside) {
                v = fma(a[0], x[id + 1], a[1] * x[id - 1]);
                if (g.dim == 2) v = fma(a[2], x[id + g.n1], fma(a[3], x[id - g.n1], v));
            } else if (fixed_coord(g, i, j, c)) {
                v = x[id];
            } else {
                v = fma(a[0], coord_beside(g, x, id, i, 0, 1, c), a[1] * coord_beside(g, x, id, i, 0, -1, c));
                if (g.dim == 2)
                    v = fma(a[2], coord_beside(g, x, id, j, 1, 1, c), fma(a[3], coord_beside(g, x, id, j, 1, -1, c), v));
            }
            if (CHG) chg = max_bits(chg, fabs(v - x[id]));
            xout[size_t(c) * N + id] = v;
            if (LIMIT) {
                const double* y = xn + size_t(c) * N;
                const double x0 = y[id], dx = v - x0;
                if ((__double_as_longlong(dx) << 1) != 0) {
                    const int s = __double2hiint(dx) < 0 ? -1 : 1;
                    const double to = inside ? y[id + s * (c == 0 ? 1 : g.n1)]
                                             : coord_beside(g, y, id, c == 0 ? i : j, c, s, c);
                    m = limit_by(m, dx, s < 0 ? x0 - to : to - x0, d);
                }
            }
        }
    }
    return chg;
}

// Sweep k of the iteration.  Sweep k >= 1 reads buf[(pick + k - 1) % 2] and writes
// buf[(pick + k) % 2]; sweep 0 reads `first` (x_n or the warm start) and writes buf[dst0].  Once
// the iteration has converged (d->conv) the remaining sweeps return at once.  With `check`, the
// grid-wide max change goes to red[slot]; if `decide`, the last block to finish compares it with eps.
__global__ void k_jacobi(GridParams g, const double* omega, SweepWeights w, const double* first, double* xa, double* xb,
                         int k, int dst0, DevScalars* d, int check, int slot, int decide, double eps, int limit) {
    if (d->conv) return;
    const double* xin;
    double* xout;
    if (k == 0) {
        xin = first;
        xout = dst0 ? xb : xa;
    } else {
        const int src = (d->pick + k - 1) & 1;
        xin = src ? xb : xa;
        xout = src ? xa : xb;
    }
    double chg[1] = {0.0};
    if (limit) {                    // the last sweep without a tolerance: k_limiter's work (first is x^n)
        if (k == 0) sweep_nodes<true, false, true>(g, omega, w, xin, xout, first, d);
        else sweep_nodes<false, false, true>(g, omega, w, xin, xout, first, d);
    } else if (!check) {
        if (k == 0) sweep_nodes<true, false, false>(g, omega, w, xin, xout, nullptr, nullptr);
        else sweep_nodes<false, false, false>(g, omega, w, xin, xout, nullptr, nullptr);
    } else {
        chg[0] = k == 0 ? sweep_nodes<true, true, false>(g, omega, w, xin, xout, nullptr, nullptr)
                        : sweep_nodes<false, true, false>(g, omega, w, xin, xout, nullptr, nullptr);
        block_max_bits<1>(chg);
        if (threadIdx.x == 0) {
            atomic_max_pos(&d->red[slot], chg[0]);
            __threadfence();
            const unsigned int ticket = atomicAdd(&d->done, 1u);
            if (ticket == gridDim.x - 1) {                 // every block's maximum is in
                if (decide) {
                    const double c = __longlong_as_double((long long)atomicAdd(&d->red[slot], 0ULL));
                    if (c < eps) d->conv = 1;
                    d->red[slot] = 0ULL;
                }
                d->done = 0u;
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && (k > 0 || slot == RED_JAC)) atomicAdd(&d->sweeps, 1);
}

// The body of a graph while-loop over the sweeps with a tolerance: sweep k = d->sweeps (the
// same buffers as k_jacobi), and the last block to finish tests the change, counts the sweep
// and sets the loop's condition: another sweep while not converged and fewer than mu sweeps.
__global__ void k_jacobi_loop(GridParams g, const double* omega, SweepWeights w, const double* xn, double* xa,
                              double* xb, DevScalars* d, double eps, int mu, cudaGraphConditionalHandle h) {
    if (d->conv || d->sweeps >= mu) {
        if (blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(h, 0u);
        return;
    }
    const int k = d->sweeps;
    const double* xin;
    double* xout;
    if (k == 0) {
        xin = xn;
        xout = xa;
    } else {
        const int src = (d->pick + k - 1) & 1;
        xin = src ? xb : xa;
        xout = src ? xa : xb;
    }
    double chg[1];
    if (k == 0) chg[0] = sweep_nodes<true, true, false>(g, omega, w, xin, xout, nullptr, nullptr);
    else chg[0] = sweep_nodes<false, true, false>(g, omega, w, xin, xout, nullptr, nullptr);
    block_max_bits<1>(chg);
    if (threadIdx.x == 0) {
        atomic_max_pos(&d->red[RED_JAC], chg[0]);
        __threadfence();
        const unsigned int ticket = atomicAdd(&d->done, 1u);
        if (ticket == gridDim.x - 1) {
            const double c = __longlong_as_double((long long)atomicAdd(&d->red[RED_JAC], 0ULL));
            if (c < eps) d->conv = 1;
            d->red[RED_JAC] = 0ULL;
            d->done = 0u;
            d->sweeps = k + 1;
            cudaGraphSetConditional(h, (d->conv == 0 && k + 1 < mu) ? 1u : 0u);
        }
    }
}

// Delta_gamma: each node moves at most half of the spacing towards its neighbour (Sec. 4)
__global__ void k_limiter(GridParams g, const double* xn, const double* xa, const double* xb, DevScalars* d) {
    const int N = g.n1 * g.n2;
    const double* xit = d->sweeps == 0 ? xn : (((d->pick + d->sweeps - 1) & 1) ? xb : xa);
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const int i = id % g.n1, j = id / g.n1;
        double m = grid_limit(d);
        for (int k = 0; k < g.dim; ++k) {
            const double* y = xn + size_t(k) * N;
            const double x0 = y[id], dx = xit[size_t(k) * N + id] - x0;
            if ((__double_as_longlong(dx) << 1) == 0) continue;
            const int s = __double2hiint(dx) < 0 ? -1 : 1;
            const double to = coord_beside(g, y, id, k == 0 ? i : j, k, s, k);
            m = limit_by(m, dx, s < 0 ? x0 - to : to - x0, d);
        }
    }
}

// ------------------------------------------------------------ small meshes: passes and sweeps on tiles
// A CTA owns bx x by nodes and keeps them with a halo of h nodes in shared memory.  Pass p updates the nodes within
// h - p of the tile, so that after h passes the tile's own nodes are what the whole mesh's passes give.  A halo position
// outside the mesh holds the wrapped node along a periodic direction (and evolves with it) and is unused otherwise: at a
// mesh end the missing neighbour is the end node itself (outflow, monitor fields) or the node inside it (a mirroring end).
struct TileBox {
    int i0, j0, w, h, bx, by, halo, n1, n2;
    bool per1, per2;
    __device__ __forceinline__ TileBox(const GridParams& g, int bx_, int by_, int halo_) : bx(bx_), by(by_), halo(halo_) {
        const int ntx = (g.n1 + bx - 1) / bx;
        i0 = int(blockIdx.x) % ntx * bx - halo;
        j0 = g.dim == 2 ? int(blockIdx.x) / ntx * by - halo : 0;
        w = bx + 2 * halo;
        h = g.dim == 2 ? by + 2 * halo : 1;
        n1 = g.n1;
        n2 = g.n2;
        per1 = g.bc[0] == ES_BC_PERIODIC;
        per2 = g.dim < 2 || g.bc[1] == ES_BC_PERIODIC;
    }
    // is box position (li, lj) a node of the mesh (or its periodic image)
    __device__ __forceinline__ bool live(int li, int lj) const {
        const int gi = i0 + li, gj = j0 + lj;
        return (per1 || (gi >= 0 && gi < n1)) && (per2 || (gj >= 0 && gj < n2));
    }
};
// the positions within dx columns and dy rows of the tile (1D: its line): item t of count()
struct TileRange {
    int w, n, x0, y0;
    __device__ __forceinline__ TileRange(const TileBox& B, int dx, int dy)
        : w(B.bx + 2 * dx), n((B.bx + 2 * dx) * (B.h == 1 ? 1 : B.by + 2 * dy)), x0(B.halo - dx),
          y0(B.h == 1 ? 0 : B.halo - dy) {}
    __device__ __forceinline__ void at(int t, int& li, int& lj) const {
        lj = t / w;
        li = x0 + t - lj * w;
        lj += y0;
    }
};
// offset (in positions) to the neighbour at s along a direction with position q of n
__device__ __forceinline__ int beside(int q, int n, int bc, int s) {
    if (bc == ES_BC_PERIODIC || (s < 0 ? q > 0 : q < n - 1)) return s;
    return end_mirrored(bc, s < 0) ? -s : 0;
}

// omega from the monitor's terms and `passes` filter passes
__global__ void __launch_bounds__(TILE_THREADS) k_filter_tile(GridParams g, MonitorParams mp,
                                                              const double* __restrict__ t0,
                                                              const double* __restrict__ t1,
                                                              const double* __restrict__ t2, const DevScalars* d,
                                                              int passes, int bx, int by, double* __restrict__ out) {
    extern __shared__ double sm[];
    __shared__ double coef[3];
    const TileBox B(g, bx, by, passes);
    const int box = B.w * B.h;
    double* A = sm;
    double* R = sm + box;                                    // row sums
    if (threadIdx.x < 3) coef[threadIdx.x] = mon_coef(mp, d, threadIdx.x);
    __syncthreads();
    const double c0 = coef[0], c1 = coef[1], c2 = coef[2];
    for (int b = threadIdx.x; b < box; b += TILE_THREADS) {
        const int li = b % B.w, lj = b / B.w;
        if (!B.live(li, lj)) continue;
        const size_t id = size_t(state_index(B.j0 + lj, g.n2, g.bc[1])) * g.n1 + state_index(B.i0 + li, g.n1, g.bc[0]);
        A[b] = omega_of(c0, c1, c2, t0[id], t1[id], t2[id]);
    }
    __syncthreads();
    for (int p = 1; p <= passes; ++p) {
        const int dd = passes - p;                           // distance still updated
        const TileRange rows(B, dd, dd + 1), nodes(B, dd, dd);   // row sums one row further out than the pass's nodes
        for (int t = threadIdx.x; t < rows.n; t += TILE_THREADS) {
            int li, lj;
            rows.at(t, li, lj);
            if (!B.live(li, lj)) continue;
            const int b = lj * B.w + li, q = B.i0 + li;
            R[b] = fma(2.0, A[b], A[b + beside(q, g.n1, g.bc[0], -1)] + A[b + beside(q, g.n1, g.bc[0], 1)]);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < nodes.n; t += TILE_THREADS) {
            int li, lj;
            nodes.at(t, li, lj);
            if (!B.live(li, lj)) continue;
            const int b = lj * B.w + li;
            if (g.dim == 1) {
                A[b] = 0.25 * R[b];
                continue;
            }
            const int q = B.j0 + lj;
            A[b] = 0.0625 * fma(2.0, R[b], R[b + B.w * beside(q, g.n2, g.bc[1], -1)] +
                                               R[b + B.w * beside(q, g.n2, g.bc[1], 1)]);
        }
        __syncthreads();
    }
    const int own = bx * (g.dim == 2 ? by : 1);
    for (int t = threadIdx.x; t < own; t += TILE_THREADS) {
        const int li = B.halo + t % bx, lj = g.dim == 2 ? B.halo + t / bx : 0;
        const int i = B.i0 + li, j = B.j0 + lj;
        if (i < g.n1 && j < g.n2) out[size_t(j) * g.n1 + i] = A[lj * B.w + li];
    }
}

// `mu` sweeps from x^n into xout and the limiter's Delta_gamma (into RED_GAMMA)
__global__ void __launch_bounds__(TILE_THREADS) k_sweep_tile(GridParams g, const double* __restrict__ omega,
                                                             const double* __restrict__ xn, double* __restrict__ xout,
                                                             int mu, int bx, int by, DevScalars* d) {
    extern __shared__ double sm[];
    const TileBox B(g, bx, by, mu);
    const int box = B.w * B.h, N = g.n1 * g.n2, nc = g.dim;
    double* X[2] = {sm, sm + nc * box};                      // the iterate and the next one, nc components each
    double* a = sm + 2 * nc * box;                           // weights, 2 nc per node
    double* om = a + 2 * nc * box;
    for (int b = threadIdx.x; b < box; b += TILE_THREADS) {
        const int li = b % B.w, lj = b / B.w;
        if (!B.live(li, lj)) continue;
        const int i = B.i0 + li, j = B.j0 + lj;
        const int si = state_index(i, g.n1, g.bc[0]), sj = g.dim == 2 ? state_index(j, g.n2, g.bc[1]) : 0;
        const size_t id = size_t(sj) * g.n1 + si;
        om[b] = omega[id];
        // a periodic image is shifted by whole periods
        double x = xn[id];
        if (i != si) x = fma(double((i - si) / g.n1), g.period[0], x);
        X[0][b] = x;
        if (nc == 2) {
            double y = xn[N + id];
            if (j != sj) y = fma(double((j - sj) / g.n2), g.period[1], y);
            X[0][box + b] = y;
        }
    }
    __syncthreads();
    for (int s = 0; s < mu; ++s) {
        const int dd = mu - 1 - s;
        const double* x = X[s & 1];
        double* y = X[(s + 1) & 1];
        const TileRange nodes(B, dd, dd);
        for (int t = threadIdx.x; t < nodes.n; t += TILE_THREADS) {
            int li, lj;
            nodes.at(t, li, lj);
            if (!B.live(li, lj)) continue;
            const int b = lj * B.w + li;
            const int i = B.i0 + li, j = B.j0 + lj;
            const int e = beside(i, g.n1, g.bc[0], 1), w = beside(i, g.n1, g.bc[0], -1);
            const int n = nc == 2 ? B.w * beside(j, g.n2, g.bc[1], 1) : 0;
            const int u = nc == 2 ? B.w * beside(j, g.n2, g.bc[1], -1) : 0;
            double q[4];
            if (s == 0) {
                const double nb[4] = {om[b + e], om[b + w], om[b + n], om[b + u]};
                sweep_weights(g, om[b], nb, q);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k < 2 * nc) a[k * box + b] = q[k];
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) q[k] = k < 2 * nc ? a[k * box + b] : 0.0;
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (c >= nc) break;
                const double* z = x + c * box + b;
                double v = fma(q[0], z[e], q[1] * z[w]);
                if (nc == 2) v = fma(q[2], z[n], fma(q[3], z[u], v));
                y[c * box + b] = fixed_coord(g, i, j, c) ? z[0] : v;
            }
        }
        __syncthreads();
    }
    const double* x = X[mu & 1];
    double m = grid_limit(d);
    const int own = bx * (nc == 2 ? by : 1);
    for (int t = threadIdx.x; t < own; t += TILE_THREADS) {
        const int li = B.halo + t % bx, lj = nc == 2 ? B.halo + t / bx : 0;
        const int i = B.i0 + li, j = B.j0 + lj;
        if (i >= g.n1 || j >= g.n2) continue;
        const int id = j * g.n1 + i;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (c >= nc) break;
            const double v = x[c * box + lj * B.w + li];
            xout[size_t(c) * N + id] = v;
            const double* y = xn + size_t(c) * N;
            const double x0 = y[id], dx = v - x0;
            if ((__double_as_longlong(dx) << 1) == 0) continue;
            const int s = __double2hiint(dx) < 0 ? -1 : 1;
            const double to = coord_beside(g, y, id, c == 0 ? i : j, c, s, c);
            m = limit_by(m, dx, s < 0 ? x0 - to : to - x0, d);
        }
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) d->sweeps = mu;
}

// The tile of a small mesh: 20 nodes wide in 2D (32 in 1D), and as tall as lets the tiles fill the SMs once.  False: the
// passes one by one are as fast, or the halo does not fit.  Steps with all `halo` passes (or sweeps) in one launch / pass by
// pass, us:
//   1D, filter: 100 nodes and 5 passes 68 / 73, 64 passes 109 / 153; 14592 nodes (three tiles per SM) 124 / 126, 171 / 208;
//     16000 116 / 113, 200 / 197; 77000 316 / 298, 577 / 402.
//   1D, sweeps: 100 nodes and 5 sweeps 69 / 75, 64 99 / 194; 9728 (two tiles per SM) one sweep 110 / 109, 5 112 / 118; 14592 two
//     126 / 124; 19456 (four per SM) 3 155 / 154, 5 157 / 159, 64 228 / 286; 24320 5 162 / 160, 10 169 / 170, 64 262 / 282; 28000 10
//     171 / 173; 32000 10 177 / 173.
//   2D, filter: 64 x 64 and 5 passes 248 / 254; 200 x 200 547 / 554; 270 x 280 1044 / 1059, 10 passes 1062 / 1084; 9000 x 8 1066 /
//     1084.
//   2D, sweeps: a tile forms the weights and the first sweeps of its halo again.  Tiles of 140 nodes (200 x 100) 10 sweeps 380 / 384;
//     280 (200 x 200) 5 sweeps 555 / 557, 8 565 / 564, 10 574 / 572; 340 (215 x 215) 5 744 / 745, 8 755 / 753; 400 (230 x 230) 5
//     814 / 812; 560 (270 x 280) one 1047 / 1045, 5 1061 / 1057; three tiles per SM (9000 x 8) 8 1093 / 1089.
// (Halos of more than 10 nodes in 2D and 64 in 1D were not measured.)
bool tile_shape(const GridParams& g, int halo, bool sweeps, int nsm, size_t doubles_per_node, int* bx, int* by, size_t* smem) {
    if (halo < 1) return false;
    if (g.dim == 1) {
        *bx = 32;
        *by = 1;
        const int per_sm = !sweeps ? 3 : (halo >= 10 ? 6 : (halo >= 5 ? 4 : 2));
        if (halo > 64 || (g.n1 + *bx - 1) / *bx > per_sm * nsm) return false;
    } else {
        *bx = 20;
        const int ntx = (g.n1 + *bx - 1) / *bx;
        const int rows = nsm / ntx > 0 ? nsm / ntx : 1;      // tiles per column
        int b = (g.n2 + rows - 1) / rows;
        if (b < 4) b = 4;
        *by = b;
        if (halo > 10 || (long long)g.n1 * g.n2 > (long long)nsm * TILE_NODES_PER_SM) return false;
        if (sweeps && (ntx > nsm || *bx * b > 340 || *bx * b * halo > 2000)) return false;
    }
    const size_t box = size_t(*bx + 2 * halo) * (g.dim == 2 ? *by + 2 * halo : 1);
    *smem = sizeof(double) * box * doubles_per_node;
    return *smem <= 200 * 1024;
}

cudaError_t mesh64_prepare() {
    cudaError_t e = cudaFuncSetAttribute(k_filter_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return e;
}

static int tiles(const GridParams& g, int bx, int by) {
    return (g.n1 + bx - 1) / bx * (g.dim == 2 ? (g.n2 + by - 1) / by : 1);
}

bool launch_filter_tile(const GridParams& g, const MonitorParams& mp, const double* t0, const double* t1,
                        const double* t2, const DevScalars* d, int passes, double* omega, int nsm, cudaStream_t s) {
    int bx, by;
    size_t sm;
    if (!tile_shape(g, passes, false, nsm, 2, &bx, &by, &sm)) return false;
    k_filter_tile<<<tiles(g, bx, by), TILE_THREADS, sm, s>>>(g, mp, t0, t1, t2, d, passes, bx, by, omega);
    return true;
}

bool launch_sweep_tile(const GridParams& g, const double* omega, const double* xn, double* xout, int mu, DevScalars* d,
                       int nsm, cudaStream_t s) {
    int bx, by;
    size_t sm;
    if (!tile_shape(g, mu, true, nsm, g.dim == 2 ? 9 : 5, &bx, &by, &sm)) return false;
    k_sweep_tile<<<tiles(g, bx, by), TILE_THREADS, sm, s>>>(g, omega, xn, xout, mu, bx, by, d);
    return true;
}

}  // namespace es
