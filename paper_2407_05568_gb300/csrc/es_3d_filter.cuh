// es_3d_filter.cuh -- the monitor's low-pass filter in 3D, in double and in float.
#pragma once
#include <cuda_runtime.h>

#include "es_3d_grid.cuh"

namespace es {

// omega_i <- sum_{j in {0,+-1}^3} (1/2)^(|j|_1 + 3) omega_{i+j} (Sec. 4), ghosts by copy / wrap.
// The filter is the product of three (1/4, 1/2, 1/4) sums.  Read node by node it is 27 products (in FP64, 48 instructions on
// the FP64 pipe, which bound it: 72 us at 96^3); here the sums are shared: a warp takes 32 nodes along xi_1 and RY lines,
// and marches along xi_3 keeping the last two planes' partial sums, so a node costs the row sums of (RY + 2)/RY lines, a
// column sum and a plane sum, two instructions each, and one scaling: 9 at RY = 2, 8 at RY = 4 (and the segments' ends).
// Neighbours along xi_1 come from the neighbouring lanes (the warp's ends and the mesh's last node load theirs), so there is
// no shared memory and no barrier; the next plane's loads are in flight while a plane is summed.  The weights are powers of
// two, so that the sums without them (l + 2 c + r) have the same bits as with them.  A pass within a step at 96^3: FP64 72 ->
// 17 us, FP32 9.8 -> 8.6.  (Four passes at a time on 16^3 tiles in shared memory, FP32: 9.7 us a pass, bound by the nine
// shared loads a node, and no better on larger meshes.)
template <typename T, int RY>
__global__ void __launch_bounds__(128) k3_filter(Grid3 g, const T* in, T* out, int seg) {
    const int n1 = g.n[0], n2 = g.n[1], n3 = g.n[2];
    const int nb1 = (n1 + 31) / 32, nb2 = (n2 + RY - 1) / RY, nb3 = (n3 + seg - 1) / seg;
    const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= nb1 * nb2 * nb3) return;
    const int i1 = w % nb1 * 32 + lane, j0 = w / nb1 % nb2 * RY, k0 = w / (nb1 * nb2) * seg;
    const int k1 = k0 + seg < n3 ? k0 + seg : n3;
    const int c1 = i1 < n1 ? i1 : n1 - 1;
    const bool lo = lane == 0, hi = lane == 31 || i1 >= n1 - 1;
    const int xr = state_index(c1 + 1, n1, g.bc[0]);
    const int xe = lo ? state_index(c1 - 1, n1, g.bc[0]) : xr;
    int row[RY + 2];
#pragma unroll
    for (int j = 0; j < RY + 2; ++j) row[j] = state_index(j0 + j - 1, n2, g.bc[1]) * n1;

    T v[RY + 2], e[RY + 2], p0[RY], p1[RY];
    const T* pl = in + size_t(state_index(k0 - 1, n3, g.bc[2])) * n1 * n2;
    auto load = [&]() {
#pragma unroll
        for (int j = 0; j < RY + 2; ++j) {
            v[j] = pl[row[j] + c1];
            e[j] = lo || hi ? pl[row[j] + xe] : T(0);
        }
    };
    load();
    for (int k = k0 - 1; k <= k1; ++k) {
        T r[RY + 2];
#pragma unroll
        for (int j = 0; j < RY + 2; ++j) {
            const T up = __shfl_up_sync(0xffffffffu, v[j], 1), dn = __shfl_down_sync(0xffffffffu, v[j], 1);
            const T a = lo ? e[j] : up;
            const T b = hi ? (lo ? pl[row[j] + xr] : e[j]) : dn;
            r[j] = fma(T(2), v[j], a) + b;
        }
        if (k < k1) {
            pl = in + size_t(state_index(k + 1, n3, g.bc[2])) * n1 * n2;
            load();
        }
#pragma unroll
        for (int j = 0; j < RY; ++j) {
            const T c = fma(T(2), r[j + 1], r[j]) + r[j + 2];
            if (k > k0 && i1 < n1 && j0 + j < n2)
                out[(size_t(k - 1) * n2 + j0 + j) * n1 + i1] = (fma(T(2), p1[j], p0[j]) + c) * T(1.0 / 64.0);
            p0[j] = p1[j];
            p1[j] = c;
        }
    }
}

// Node by node, the same sums: 27 loads in flight at once.  On a small mesh a pass is the length of one thread's chain, and
// here it is one load's latency.
template <typename T>
__global__ void __launch_bounds__(128) k3_filter_nodes(Grid3 g, const T* __restrict__ in, T* __restrict__ out) {
    const int n1 = g.n[0], n2 = g.n[1], n12 = n1 * n2;
    const int id = blockIdx.x * 128 + threadIdx.x;
    if (id >= n12 * g.n[2]) return;
    const int r12 = id / n1, i = id - r12 * n1, k = r12 / n2, j = r12 - k * n2;
    const int xm = state_index(i - 1, n1, g.bc[0]) - i, xp = state_index(i + 1, n1, g.bc[0]) - i;
    const int y[3] = {(state_index(j - 1, n2, g.bc[1]) - j) * n1, 0, (state_index(j + 1, n2, g.bc[1]) - j) * n1};
    const int z[3] = {(state_index(k - 1, g.n[2], g.bc[2]) - k) * n12, 0, (state_index(k + 1, g.n[2], g.bc[2]) - k) * n12};
    T c[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        T r[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const T* v = in + (id + y[p] + z[q]);
            r[p] = fma(T(2), v[0], v[xm]) + v[xp];
        }
        c[q] = fma(T(2), r[1], r[0]) + r[2];
    }
    out[id] = (fma(T(2), c[1], c[0]) + c[2]) * T(1.0 / 64.0);
}

// Lines per warp and planes per segment.  A warp's planes follow one another (a load's latency each), so on meshes of up to
// 2^21 nodes short segments and two lines keep the launch short although they sum more planes and rows twice: 16 warps on
// each SM where the mesh gives them, at least 2 planes.  Above, four lines in segments of 4 to 12 planes:
// 200^3 172 and 41 us (two lines 190 and 43).
template <typename T, int RY>
inline void launch_filter3(const Grid3& g, const T* in, T* out, int target, int lo, cudaStream_t s) {
    const int cols = (g.n[0] + 31) / 32 * ((g.n[1] + RY - 1) / RY);
    const int parts = (target + cols - 1) / cols;
    int seg = (g.n[2] + parts - 1) / parts;
    seg = seg < lo ? lo : (seg > 12 ? 12 : seg);
    const int warps = cols * ((g.n[2] + seg - 1) / seg);
    k3_filter<T, RY><<<(warps + 3) / 4, 128, 0, s>>>(g, in, out, seg);
}
// Meshes that the node-by-node kernel filters faster, a pass within a step in us, it / the marching one: FP32 24^3 1.9 / 4.5,
// 48^3 2.2 / 4.5, 64^3 3.8 / 5.0, 80^3 5.8 / 6.9, 96^3 8.6 / 8.6; FP64 24^3 2.8 / 6.1, 44^3 6.6 / 7.3, 48^3 7.7 / 7.3.
template <typename T>
inline void launch_filter3(const Grid3& g, const T* in, T* out, int nsm, cudaStream_t s) {
    const size_t N = size_t(g.n[0]) * g.n[1] * g.n[2];
    if (N <= (sizeof(T) == 4 ? size_t(1) << 19 : size_t(100000)))
        k3_filter_nodes<<<int((N + 127) / 128), 128, 0, s>>>(g, in, out);
    else if (N <= (size_t(1) << 21)) launch_filter3<T, 2>(g, in, out, 16 * nsm, 2, s);
    else launch_filter3<T, 4>(g, in, out, 8 * nsm, 4, s);
}

}  // namespace es
