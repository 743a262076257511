// es_3d_filter.cuh -- the monitor's low-pass filter in 3D, in double and in float.
#pragma once
#include <cuda_runtime.h>

#include "es_3d_grid.cuh"

namespace es {

// omega_i <- sum_{j in {0,+-1}^3} (1/2)^(|j|_1 + 3) omega_{i+j} (Sec. 4), ghosts by copy / wrap.
// The filter is the product of three (1/4, 1/2, 1/4) sums.  Read node by node it is 27 products (in FP64, 48 instructions on
// the FP64 pipe, which bound it: 73 us at 96^3); here the sums are shared: a warp takes 32 nodes along xi_1 and RY lines,
// and marches along xi_3 keeping the last two planes' partial sums, so a node costs the row sums of (RY + 2)/RY lines, a
// column sum and a plane sum, two instructions each, and one scaling: 8 at RY = 4.  Neighbours along xi_1 come from the
// neighbouring lanes (the warp's ends and the mesh's last node load theirs), so there is no shared memory and no barrier;
// the next plane's loads are in flight while a plane is summed.  The weights are powers of two, so that the sums without
// them (l + 2 c + r) have the same bits as with them.  96^3: FP64 73 -> 24 us (FP32 stays at 12: there the loads of one plane after the other bound it).
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

// segments along xi_3: short enough for two warps on each of the 608 schedulers, at least 4 planes (each segment sums two
// planes more), at most 32
template <typename T>
inline void launch_filter3(const Grid3& g, const T* in, T* out, cudaStream_t s) {
    constexpr int RY = 4;
    const int cols = (g.n[0] + 31) / 32 * ((g.n[1] + RY - 1) / RY);
    const int parts = (1216 + cols - 1) / cols;
    int seg = (g.n[2] + parts - 1) / parts;
    seg = seg < 4 ? 4 : (seg > 32 ? 32 : seg);
    const int warps = cols * ((g.n[2] + seg - 1) / seg);
    k3_filter<T, RY><<<(warps + 3) / 4, 128, 0, s>>>(g, in, out, seg);
}

}  // namespace es
