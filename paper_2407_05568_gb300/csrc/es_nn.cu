// es_nn.cu -- kernels of the learned mesh warm start: 3x3 convolution layers with
// BF16 weights and FP32 activations/accumulation, their backward passes, the MSE
// loss and the Adam update.  The network maps the filtered monitor, the
// fundamental derivative and the current mesh (Sec. 4) to the displacement that
// starts the Jacobi iteration; the plain iteration always finishes the solve.
// The FP32 layers run on the tensor cores with their operands split into three bf16
// parts (k_conv_fwd_s3, k_conv_wgrad_s3), the inference path on bf16 operands.
//
// Layout: activations [B][C][H][W] float; weights [Cout][Cin][3][3] bf16; cross-correlation with zero padding:
//   out[co](y, x) = bias[co] + sum_{ci, dy, dx} w[co][ci][dy+1][dx+1] in[ci](y+dy, x+dx).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "es_internal.h"
#include "es_vdw.h"

namespace es {
namespace {

constexpr int TS = 16;            // output tile edge (pixels)
constexpr int HALO = TS + 2;
constexpr int MAXC = 32;          // channel limit

// a sum and its correction products: beside an infinite sum they are products of an infinity with the other operand's
// low parts, which may be zero (NaN)
__device__ __forceinline__ float with_low(float sum, float low) { return isinf(sum) ? sum : sum + low; }
// the same in place: what the sum's rounding leaves stays in `low`
__device__ __forceinline__ void take_low(float& sum, float& low) {
    const float s = with_low(sum, low);
    low += sum - s;
    sum = s;
}
// sum + v with the rounding error collected in `low` (D. E. Knuth, TAOCP 2, 4.2.2)
__device__ __forceinline__ void add_comp(float& sum, float& low, float v) {
    const float s = sum + v, b = s - sum;
    low += (sum - (s - b)) + (v - b);
    sum = s;
}

// out[o] = sum_s partial[s][o] over the strips: RP_GROUPS threads per output take every RP_GROUPS-th strip, and their sums
// are added in order (the same order every time), with the rounding errors: a long image has a thousand strips
constexpr int RP_GROUPS = 16;
__global__ void __launch_bounds__(32 * RP_GROUPS) k_reduce_partials(const float* __restrict__ partial, int nstrips,
                                                                    int len, float* grad_w, float* grad_b, int nout) {
    __shared__ float part[2][RP_GROUPS][32];
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    float s = 0.0f, c = 0.0f;
    if (o < len)
#pragma unroll 4
        for (int k = grp; k < nstrips; k += RP_GROUPS) add_comp(s, c, partial[size_t(k) * len + o]);
    part[0][grp][lane] = s;
    part[1][grp][lane] = c;
    __syncthreads();
    if (grp != 0 || o >= len) return;
    s = c = 0.0f;
#pragma unroll
    for (int k = 0; k < RP_GROUPS; ++k) {
        add_comp(s, c, part[0][k][lane]);
        c += part[1][k][lane];
    }
    s = with_low(s, c);
    if (o < nout) grad_w[o] = s;
    else grad_b[o - nout] = s;
}

__global__ void k_f32_to_bf16(const float* f, __nv_bfloat16* w, size_t n) {
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
        w[i] = __float2bfloat16_rn(f[i]);
}

// loss += mean (pred - target)^2; grad = 2 (pred - target) / n
__global__ void k_mse(const float* pred, const float* tgt, float* grad, float* loss, size_t n) {
    __shared__ float red[32];
    float s = 0.0f;
    const float sc = 2.0f / float(n);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
        const float d = pred[i] - tgt[i];
        grad[i] = sc * d;
        s = fmaf(d, d, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < int(blockDim.x + 31) / 32; ++w) t += red[w];
        atomicAdd(loss, t / float(n));
    }
}

// Adam (Kingma & Ba 2015) on the FP32 master weights; the BF16 copy is the master rounded to nearest
__global__ void k_adam(float* master, __nv_bfloat16* wb, const float* grad, float* m, float* v, int n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = grad[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float w = master[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        master[i] = w;
        if (wb) wb[i] = __float2bfloat16_rn(w);
    }
}

// ---- tensor-core forward (inference): implicit GEMM on mma.sync.m16n8k16 (bf16 in, FP32 accumulate).
// A CTA of 4 warps computes a 16 x 16 pixel tile; warp w owns output rows 4w .. 4w+3 (one m16 tile
// per row, rows of the m16 tile = the 16 pixels of that row), all NPAD output channels (NPAD/8 n8
// tiles).  GEMM: M = pixels, N = Cout, K = 9 Cin ordered k = tap * Cin + ci (padded to 16).  The
// input tile with its halo is staged as bf16 pairs [pixel][ci/2] and the weights as bf16 pairs
// [n][k/2]; the row strides are padded so that the fragment loads of a warp hit 32 distinct banks.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16_16816(float* d, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// IN_NHWC / OUT_NHWC: the layer input / output as bf16 [B][H][W][C] (the context's inference
// buffers between layers: what the next layer's staging would round to anyway) instead of FP32
// [B][C][H][W].  The results are the same either way.
template <int CIN, int NPAD, bool IN_NHWC, bool OUT_NHWC>
__global__ void __launch_bounds__(128) k_conv_fwd_tc(const void* __restrict__ in_,
                                                    const __nv_bfloat16* __restrict__ w,
                                                    const float* __restrict__ bias, void* __restrict__ out_,
                                                    int Cout, int H, int W, int act) {
    constexpr int K = 9 * CIN;
    constexpr int KP = (K + 15) / 16 * 16;
    constexpr int KSW = KP / 2 + 4;                       // words per weight row
    constexpr int PSW = CIN / 2 + (CIN >= 32 ? 4 : 1);    // words per staged pixel
    constexpr int NT = NPAD / 8;
    __shared__ uint32_t ws[NPAD * KSW];
    __shared__ uint32_t xs[HALO * HALO * PSW];
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * TS, y0 = blockIdx.y * TS, b = blockIdx.z;
    const size_t HW = size_t(H) * W;
    for (int idx = tid; idx < NPAD * (KP / 2); idx += 128) {
        const int n = idx / (KP / 2), k0 = 2 * (idx % (KP / 2));
        float v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = k0 + e;
            v[e] = (n < Cout && k < K) ? __bfloat162float(w[(n * CIN + k % CIN) * 9 + k / CIN]) : 0.0f;
        }
        ws[n * KSW + k0 / 2] = pack_bf16(v[0], v[1]);
    }
    if (IN_NHWC) {
        // CIN/2 words per pixel, copied 4 words (16 bytes) at a time when CIN is a multiple of 8
        const uint32_t* inb = reinterpret_cast<const uint32_t*>(in_) + size_t(b) * HW * (CIN / 2);
        constexpr int VW = (CIN % 8 == 0) ? 4 : 1;
        for (int idx = tid; idx < HALO * HALO * (CIN / 2 / VW); idx += 128) {
            const int p = idx / (CIN / 2 / VW), q = idx % (CIN / 2 / VW);
            const int yy = y0 - 1 + p / HALO, xx = x0 - 1 + p % HALO;
            const bool ok = yy >= 0 && yy < H && xx >= 0 && xx < W;
            const size_t o = (size_t(yy) * W + xx) * (CIN / 2) + q * VW;
            if (VW == 4) {
                const uint4 v = ok ? *reinterpret_cast<const uint4*>(inb + o) : make_uint4(0u, 0u, 0u, 0u);
                uint32_t* d = xs + p * PSW + q * 4;
                d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
            } else {
                xs[p * PSW + q] = ok ? inb[o] : 0u;
            }
        }
    } else {
        const float* inb = reinterpret_cast<const float*>(in_) + size_t(b) * CIN * HW;
        for (int idx = tid; idx < HALO * HALO * (CIN / 2); idx += 128) {
            const int p = idx % (HALO * HALO), cw = idx / (HALO * HALO);
            const int yy = y0 - 1 + p / HALO, xx = x0 - 1 + p % HALO;
            float v0 = 0.0f, v1 = 0.0f;
            if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
                const size_t o = size_t(yy) * W + xx;
                v0 = inb[(2 * cw) * HW + o];
                v1 = inb[(2 * cw + 1) * HW + o];
            }
            xs[p * PSW + cw] = pack_bf16(v0, v1);
        }
    }
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    float acc[4][NT][4];
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.0f;
#pragma unroll 2
    for (int s = 0; s < KP / 16; ++s) {
        uint32_t bf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int n = nt * 8 + g;
            bf[nt][0] = ws[n * KSW + s * 8 + t];
            bf[nt][1] = ws[n * KSW + s * 8 + 4 + t];
        }
        const int klo = s * 16 + 2 * t, khi = klo + 8;
        const bool vlo = klo < K, vhi = khi < K;
        const int tlo = klo / CIN, clo = (klo % CIN) / 2, thi = khi / CIN, chi = (khi % CIN) / 2;
        const int olo = (tlo / 3) * HALO + tlo % 3, ohi = (thi / 3) * HALO + thi % 3;
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) {
            const int row = (warp * 4 + mt) * HALO;           // output row of this m16 tile, box coordinates
            uint32_t af[4];
            af[0] = vlo ? xs[(row + olo + g) * PSW + clo] : 0u;
            af[1] = vlo ? xs[(row + olo + g + 8) * PSW + clo] : 0u;
            af[2] = vhi ? xs[(row + ohi + g) * PSW + chi] : 0u;
            af[3] = vhi ? xs[(row + ohi + g + 8) * PSW + chi] : 0u;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc[mt][nt], af, bf[nt]);
        }
    }
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
        const int y = y0 + warp * 4 + mt;
        if (y >= H) continue;
        if (OUT_NHWC) {
            // channel pairs (co, co + 1) as one bf16x2 word; Cout is even here
            uint32_t* ob = reinterpret_cast<uint32_t*>(out_) + size_t(b) * HW * (Cout / 2);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int x = x0 + g + hh * 8;
                    const int co = nt * 8 + 2 * t;
                    if (co < Cout && x < W) {
                        float v0 = acc[mt][nt][2 * hh] + bias[co], v1 = acc[mt][nt][2 * hh + 1] + bias[co + 1];
                        if (act) {
                            v0 = tanhf(v0);
                            v1 = tanhf(v1);
                        }
                        ob[(size_t(y) * W + x) * (Cout / 2) + co / 2] = pack_bf16(v0, v1);
                    }
                }
        } else {
            float* ob = reinterpret_cast<float*>(out_) + size_t(b) * Cout * HW;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int x = x0 + g + (e >= 2 ? 8 : 0);
                    const int co = nt * 8 + 2 * t + (e & 1);
                    if (co < Cout && x < W) {
                        const float v = acc[mt][nt][e] + bias[co];
                        ob[co * HW + size_t(y) * W + x] = act ? tanhf(v) : v;
                    }
                }
        }
    }
}

// ---- FP32 layers and gradients on the tensor cores.  A float is the exact sum of three bf16 numbers (8 significand bits
// each), and the weights are bf16: the correlations (forward, and the input gradient's) are three bf16 products per term,
// the weight gradient, whose operands are both FP32, six (the three of relative size 2^-24 and less are dropped).  On
// mma.sync the CUDA-core kernels' 22 TFLOP/s no longer bound them.  The tensor cores truncate their FP32 sums, so the
// leading products are summed over one tap's channels (forward) or 16 pixels (weight gradient) only and added to the
// result with a rounded FP32 addition; the other products are 2^-8 of these and share one accumulator, over 64 rows at most
// in the weight gradient.
struct Split3 {
    uint32_t v[3];                 // bf16 pairs: leading, middle, last parts
};
// The first two parts are cut to the finite bf16 range: a finite value that would round past it keeps its sum, and an
// infinity (or a NaN) leaves itself as the last part.
__device__ __forceinline__ Split3 split3(float a, float b) {
    constexpr float MAX = 3.38953139e38f;                    // the largest bf16
    Split3 s;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float x = k < 2 ? fminf(fmaxf(a, -MAX), MAX) : a, y = k < 2 ? fminf(fmaxf(b, -MAX), MAX) : b;
        const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        s.v[k] = *reinterpret_cast<const uint32_t*>(&h);
        a -= __uint_as_float(s.v[k] << 16);
        b -= __uint_as_float(s.v[k] & 0xffff0000u);
    }
    return s;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(uint32_t* r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm2_t(uint32_t* r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void zero4(float* d) { d[0] = d[1] = d[2] = d[3] = 0.0f; }

// words (bf16 pairs) per staged pixel of C channels: 16-byte rows at a stride of 20 words spread over all banks
template <int C>
constexpr int pixel_words() {
    return C == 32 ? 20 : 4;
}
// the three parts of C channels of pixels [n] into planes of n pixels; value(c, p) reads channel c of pixel p
template <int C, int THREADS, class F>
__device__ __forceinline__ void stage_split(uint32_t* dst, int n, F value) {
    constexpr int PW = pixel_words<C>(), G = C == 32 ? 4 : 1;           // groups of 8 channels
    for (int k = threadIdx.x; k < G * n; k += THREADS) {
        const int c0 = k / n * 8, p = k % n;
        float x[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) x[c] = c < C ? value(c0 + c, p) : 0.0f;
        uint32_t w[3][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const Split3 s = split3(x[2 * c], x[2 * c + 1]);
#pragma unroll
            for (int q = 0; q < 3; ++q) w[q][c] = s.v[q];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q)
            *reinterpret_cast<uint4*>(dst + (q * n + p) * PW + c0 / 2) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
    }
}

constexpr int C3_THREADS = 256;
template <int CIN, int NPAD>
struct Conv3 {
    // K = 9 taps of CIN channels, 8 at least (zero weights and inputs fill them up)
    static constexpr int CP = CIN == 32 ? 32 : 8;
    static constexpr int K = 9 * CP;                         // 288 or 72
    static constexpr int KP = (K + 15) / 16 * 16;
    static constexpr int KSW = KP / 2 + 4;                   // words per weight row: 148 or 44 (16-byte rows, spread banks)
    static constexpr int PW = pixel_words<CIN>();
    static constexpr int HP = HALO * HALO;
    static constexpr size_t SMEM = sizeof(uint32_t) * (size_t(3) * HP * PW + size_t(NPAD) * KSW);
};

// out = act(bias + w (*) in) for FP32 in and out, or (FLIP) the input gradient's correlation with the flipped, transposed
// weights w[cin][cout][8 - tap].  A CTA of 8 warps computes 16 x 16 pixels, a warp two rows of them (one m16 tile per
// row), all channels.
template <int CIN, int NPAD, bool FLIP>
__global__ void __launch_bounds__(C3_THREADS, 2) k_conv_fwd_s3(const float* __restrict__ in,
                                                              const __nv_bfloat16* __restrict__ w,
                                                              const float* __restrict__ bias, float* __restrict__ out,
                                                              int Cout, int H, int W, int act) {
    using CV = Conv3<CIN, NPAD>;
    constexpr int NT = NPAD / 8, PW = CV::PW, HP = CV::HP, CP = CV::CP;
    extern __shared__ uint4 sm16[];
    uint32_t* xs = reinterpret_cast<uint32_t*>(sm16);        // [3][HALO^2][PW]
    uint32_t* ws = xs + 3 * HP * PW;                         // [NPAD][KSW]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * TS, y0 = blockIdx.y * TS, b = blockIdx.z;
    const size_t HW = size_t(H) * W;
    const float* inb = in + size_t(b) * CIN * HW;
    stage_split<CIN, C3_THREADS>(xs, HP, [&](int c, int p) {
        const int yy = y0 - 1 + p / HALO, xx = x0 - 1 + p % HALO;
        return yy >= 0 && yy < H && xx >= 0 && xx < W ? inb[c * HW + size_t(yy) * W + xx] : 0.0f;
    });
    for (int idx = tid; idx < NPAD * (CV::KP / 2); idx += C3_THREADS) {
        const int n = idx / (CV::KP / 2), k0 = 2 * (idx % (CV::KP / 2));
        uint32_t v = 0u;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int c = (k0 + e) % CP, tap = (k0 + e) / CP;
            if (n < Cout && c < CIN && tap < 9) {
                const __nv_bfloat16 q = FLIP ? w[(size_t(c) * Cout + n) * 9 + 8 - tap] : w[(size_t(n) * CIN + c) * 9 + tap];
                v |= uint32_t(*reinterpret_cast<const uint16_t*>(&q)) << (16 * e);
            }
        }
        ws[n * CV::KSW + k0 / 2] = v;
    }
    __syncthreads();
    // ldmatrix rows: lanes 0..15 the 16 pixels' first 8 channels of a k16 step, lanes 16..31 the next 8 (CP = 8: the next tap's)
    const uint32_t xa = smem_addr(xs), wa = smem_addr(ws);
    const int ap = lane & 15, ah = lane >> 4;
    const int bn = (lane & 7) + ((lane >> 4) << 3), bk = (lane >> 3) & 1;      // weight rows: n, k half
    float acc[2][NT][4], low[2][NT][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            zero4(acc[mt][nt]);
            zero4(low[mt][nt]);
        }
    constexpr int STEPS = CV::KP / 16, FLUSH = CP == 32 ? 2 : 1;               // k16 steps; steps per rounded addition
#pragma unroll 1
    for (int s0 = 0; s0 < STEPS; s0 += FLUSH) {
        float lead[2][NT][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) zero4(lead[mt][nt]);
#pragma unroll
        for (int f = 0; f < FLUSH; ++f) {
            const int s = s0 + f;
            uint32_t bf[NT][2];
            if constexpr (NT == 1) {
                const uint32_t* r = ws + (lane >> 2) * CV::KSW + s * 8 + (lane & 3);
                bf[0][0] = r[0];
                bf[0][1] = r[4];
            } else {
#pragma unroll
                for (int nt = 0; nt < NT; nt += 2) {
                    uint32_t r[4];
                    ldsm4(r, wa + 4u * ((nt * 8 + bn) * CV::KSW + s * 8 + bk * 4));
                    bf[nt][0] = r[0];
                    bf[nt][1] = r[1];
                    bf[nt + 1][0] = r[2];
                    bf[nt + 1][1] = r[3];
                }
            }
            // tap and channel offset of this lane's row (past the last tap: any pixel, its fragments are zeroed below)
            const int k = s * 16 + ah * 8;
            const int tap = min(k / CP, 8), c = k % CP;
            const int off = ((tap / 3) * HALO + tap % 3 + ap) * PW + c / 2;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const uint32_t row = xa + 4u * ((warp * 2 + mt) * HALO * PW + off);
                uint32_t a[3][4];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    ldsm4(a[q], row + 4u * q * HP * PW);
                    if (CV::K % 16 && s == STEPS - 1) a[q][2] = a[q][3] = 0u;      // past the last tap (0 x infinity is NaN)
                }
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    mma_bf16_16816(lead[mt][nt], a[0], bf[nt]);
                    mma_bf16_16816(low[mt][nt], a[1], bf[nt]);
                    mma_bf16_16816(low[mt][nt], a[2], bf[nt]);
                }
            }
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[mt][nt][e] += lead[mt][nt][e];
    }
    const int g = lane >> 2, t = lane & 3;
    float* ob = out + size_t(b) * Cout * HW;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        const int y = y0 + warp * 2 + mt;
        if (y >= H) continue;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int x = x0 + g + (e >= 2 ? 8 : 0), co = nt * 8 + 2 * t + (e & 1);
                if (co < Cout && x < W) {
                    const float v = acc[mt][nt][e] + low[mt][nt][e] + (bias ? bias[co] : 0.0f);
                    ob[co * HW + size_t(y) * W + x] = act ? tanhf(v) : v;
                }
            }
    }
}

// Weight and bias gradients of one strip of tiles (a 16-pixel column, `rows` tiles high, one image): partial[strip] gets
// sum_p g[co](p) in[ci](p + tap) and sum_p g[co](p) over the strip's pixels (reduced over strips by k_reduce_partials).
// GEMM per tap: M = Cout, N = Cin, K = pixels, both operands read from [pixel][channel] planes by transposed
// ldmatrix, so a tap is a pixel offset.  With tanh the gradient through it, g (1 - a^2), is formed while the tile is staged
// and written back (each pixel belongs to one tile).
// Tiles are 16 x 8 pixels in two buffers: the next tile's values are loaded into registers before the current tile's
// products and split into the other buffer after them, so that the loads' latency hides behind the tensor cores.  18 warps
// (9 taps x 2 halves of 32 output channels) spread over the four schedulers as 5, 5, 4, 4 (with a warp per tap, 3, 2, 2, 2,
// and 16 x 16 tiles in one buffer: 920 us instead of 487 us for 32 -> 32 channels at 4 x 512^2).
constexpr int WG_H = 8;           // rows of a tile
template <int CIN, int COUT>
struct Wgrad {
    static constexpr int MT = COUT == 32 ? 2 : 1, NT = CIN == 32 ? 4 : 1;
    static constexpr int THREADS = 32 * 9 * MT;              // a warp per tap and 16 output channels
    static constexpr int PX = pixel_words<CIN>(), PG = pixel_words<COUT>();
    static constexpr int HP = HALO * (WG_H + 2), NP = TS * WG_H;
    static constexpr int NG = (COUT == 32 ? 4 : 1) * NP, NX = (CIN == 32 ? 4 : 1) * HP;    // groups of 8 channels
    static constexpr int GI = (NG + THREADS - 1) / THREADS, XI = (NX + THREADS - 1) / THREADS;
    static constexpr int BUF = 3 * (HP * PX + NP * PG);      // words of a buffer
    static constexpr size_t SMEM = sizeof(uint32_t) * size_t(2) * BUF;
};
// the three parts of 8 channels at word `w` of a plane, planes `plane` words apart
__device__ __forceinline__ void store_split(uint32_t* w, int plane, const float* x) {
    uint32_t v[3][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const Split3 s = split3(x[2 * c], x[2 * c + 1]);
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q][c] = s.v[q];
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(w + q * plane) = make_uint4(v[q][0], v[q][1], v[q][2], v[q][3]);
}
// LONG: strips of more than 64 rows, where the truncated sums of the correction products (2^-8 of the others) are taken into
// the rounded ones every 64 rows.  (A kernel of its own: the code spills eleven more words, 3% of a training step whose
// strips are shorter.)
template <int CIN, int COUT, bool LONG>
__global__ void __launch_bounds__(Wgrad<CIN, COUT>::THREADS, 1)
    k_conv_wgrad_s3(const float* __restrict__ in, float* g, const float* __restrict__ aout, float* __restrict__ partial,
                    int H, int W, int rows) {
    using WG = Wgrad<CIN, COUT>;
    constexpr int NT = WG::NT, PX = WG::PX, PG = WG::PG, HP = WG::HP, NP = WG::NP, TH = WG::THREADS;
    extern __shared__ uint4 sm16[];
    uint32_t* sm = reinterpret_cast<uint32_t*>(sm16);        // two of { [3][HP][PX], [3][NP][PG] }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tap = warp % 9, mt = warp / 9;
    const int x0 = blockIdx.x * TS, b = blockIdx.z;
    const int yb = blockIdx.y * rows * TS;
    const int ye = min(H, yb + rows * TS);                   // the strip's rows
    const size_t HW = size_t(H) * W;
    const float* inb = in + size_t(b) * CIN * HW;
    float* gb = g + size_t(b) * COUT * HW;
    const float* ab = aout ? aout + size_t(b) * COUT * HW : nullptr;

    float gv[WG::GI][8], av[WG::GI][8], xv[WG::XI][8];
    auto load = [&](int y0) {
#pragma unroll
        for (int i = 0; i < WG::GI; ++i) {
            const int k = tid + i * TH, c0 = k / NP * 8, p = k % NP;
            const int yy = y0 + p / TS, xx = x0 + p % TS;
            const bool ok = k < WG::NG && yy < H && xx < W;
            const size_t o = size_t(yy) * W + xx;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                gv[i][c] = ok && c < COUT ? gb[(c0 + c) * HW + o] : 0.0f;
                av[i][c] = ok && c < COUT && ab ? ab[(c0 + c) * HW + o] : 0.0f;
            }
        }
#pragma unroll
        for (int i = 0; i < WG::XI; ++i) {
            const int k = tid + i * TH, c0 = k / HP * 8, p = k % HP;
            const int yy = y0 - 1 + p / HALO, xx = x0 - 1 + p % HALO;
            const bool ok = k < WG::NX && yy >= 0 && yy < H && xx >= 0 && xx < W;
            const size_t o = size_t(ok ? yy : 0) * W + (ok ? xx : 0);
#pragma unroll
            for (int c = 0; c < 8; ++c) xv[i][c] = ok && c < CIN ? inb[(c0 + c) * HW + o] : 0.0f;
        }
    };
    auto store = [&](int y0, uint32_t* buf) {
#pragma unroll
        for (int i = 0; i < WG::GI; ++i) {
            const int k = tid + i * TH, c0 = k / NP * 8, p = k % NP;
            if (k >= WG::NG) break;
            if (ab) {                                        // the gradient through tanh, kept for the input gradient
                const int yy = y0 + p / TS, xx = x0 + p % TS;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    gv[i][c] *= 1.0f - av[i][c] * av[i][c];
                    if (c < COUT && yy < H && xx < W) gb[(c0 + c) * HW + size_t(yy) * W + xx] = gv[i][c];
                }
            }
            store_split(buf + 3 * HP * PX + p * PG + c0 / 2, NP * PG, gv[i]);
        }
#pragma unroll
        for (int i = 0; i < WG::XI; ++i) {
            const int k = tid + i * TH, c0 = k / HP * 8, p = k % HP;
            if (k < WG::NX) store_split(buf + p * PX + c0 / 2, HP * PX, xv[i]);
        }
    };

    float acc[NT][4], low[NT][4], accb[4], lowb[4];
    zero4(accb);
    zero4(lowb);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        zero4(acc[nt]);
        zero4(low[nt]);
    }
    const int ty = tap / 3, tx = tap % 3;
    const uint32_t one[2] = {0x3f803f80u, 0x3f803f80u};      // bf16 ones: the bias gradient as a product
    load(yb);
    store(yb, sm);
    __syncthreads();
    int cur = 0;
    for (int y0 = yb; y0 < ye; y0 += WG_H, cur ^= 1) {
        const bool more = y0 + WG_H < ye;
        if (LONG && (y0 & 63) == 0) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) take_low(acc[nt][e], low[nt][e]);
#pragma unroll
            for (int e = 0; e < 4; ++e) take_low(accb[e], lowb[e]);
        }
        if (more) load(y0 + WG_H);
        const uint32_t xa = smem_addr(sm + cur * WG::BUF), ga = xa + 4u * 3 * HP * PX;
#pragma unroll 1
        for (int row = 0; row < WG_H; ++row) {               // 16 pixels of the sum
            // A: (m, k) = (co, pixel); ldmatrix rows are pixels of 8 channels: matrices (k 0-7 | k 8-15) x (m 0-7 | m 8-15)
            uint32_t a[3][4];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if constexpr (COUT == 32) {
                    const int p = row * TS + (lane & 7) + ((lane >> 4) << 3);
                    ldsm4_t(a[q], ga + 4u * ((q * NP + p) * PG + mt * 8 + ((lane >> 3) & 1) * 4));
                } else {                                     // channels 8..15 of the tile are zero
                    uint32_t h[2];
                    ldsm2_t(h, ga + 4u * ((q * NP + row * TS + (lane & 15)) * PG));
                    a[q][0] = h[0];
                    a[q][2] = h[1];
                    a[q][1] = a[q][3] = 0u;
                }
            }
            // B: (k, n) = (pixel + tap, ci), two n8 tiles at a time
            const int pr = (row + ty) * HALO + tx;
#pragma unroll
            for (int n0 = 0; n0 < NT; n0 += 2) {
                constexpr int NB = NT == 1 ? 1 : 2;
                uint32_t bf[3][2][2];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if constexpr (CIN == 32) {
                        uint32_t v[4];
                        ldsm4_t(v, xa + 4u * ((q * HP + pr + (lane & 15)) * PX + n0 * 4 + (lane >> 4) * 4));
                        bf[q][0][0] = v[0];
                        bf[q][0][1] = v[1];
                        bf[q][1][0] = v[2];
                        bf[q][1][1] = v[3];
                    } else {
                        ldsm2_t(bf[q][0], xa + 4u * ((q * HP + pr + (lane & 15)) * PX));
                    }
                }
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    float* l = low[n0 + n];
                    float lead[4];
                    zero4(lead);
                    mma_bf16_16816(lead, a[0], bf[0][n]);
                    mma_bf16_16816(l, a[0], bf[1][n]);
                    mma_bf16_16816(l, a[1], bf[0][n]);
                    mma_bf16_16816(l, a[1], bf[1][n]);
                    mma_bf16_16816(l, a[0], bf[2][n]);
                    mma_bf16_16816(l, a[2], bf[0][n]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[n0 + n][e] += lead[e];
                }
            }
            if (tap == 4) {
                float lead[4];
                zero4(lead);
                mma_bf16_16816(lead, a[0], one);
                mma_bf16_16816(lowb, a[1], one);
                mma_bf16_16816(lowb, a[2], one);
#pragma unroll
                for (int e = 0; e < 4; ++e) accb[e] += lead[e];
            }
        }
        if (more) store(y0 + WG_H, sm + (cur ^ 1) * WG::BUF);
        __syncthreads();
    }
    constexpr int nout = COUT * CIN * 9;
    const size_t strip = (size_t(b) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    float* part = partial + strip * (nout + COUT);
    const int gq = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int co = mt * 16 + gq + (e >= 2 ? 8 : 0), ci = nt * 8 + 2 * t + (e & 1);
            if (co < COUT && ci < CIN) part[(co * CIN + ci) * 9 + tap] = with_low(acc[nt][e], low[nt][e]);
        }
    if (tap == 4 && t == 0)
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            const int co = mt * 16 + gq + (e >= 2 ? 8 : 0);
            if (co < COUT) part[nout + co] = with_low(accb[e], lowb[e]);
        }
}

int grid_for(size_t n) {
    const size_t g = (n + 255) / 256;
    return int(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

// strip height (tiles) so that the weight-gradient grid holds about 7 blocks per SM (one is resident: with 4 the last of 5
// waves was a fifth full)
int strip_rows(int B, int H, int W) {
    int nsm = 152;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long gx = (W + TS - 1) / TS, ty = (H + TS - 1) / TS;
    const long long want = 7LL * nsm;
    long long gy = (want + B * gx - 1) / (B * gx);
    if (gy < 1) gy = 1;
    if (gy > ty) gy = ty;
    return int((ty + gy - 1) / gy);
}

bool chan_ok(int c) { return c == 2 || c == 4 || c == 32; }

bool shape_ok(int B, int Cin, int Cout, int H, int W) {
    return B > 0 && H > 0 && W > 0 && chan_ok(Cin) && chan_ok(Cout) && (H + TS - 1) / TS <= 65535 &&
           B <= 65535 && (long long)B * MAXC * H * W < (1LL << 40);
}

}  // namespace

namespace {

// the FP32 layers' kernels by their channel counts: f(integral constants Cin, output channels padded to 8 or 32)
template <int C>
struct Int {
    static constexpr int value = C;
};
template <class F>
cudaError_t by_channels(int Cin, int Cout, F f) {
    const bool wide = Cout > 8;
    switch (Cin) {
        case 2: return wide ? f(Int<2>(), Int<32>()) : f(Int<2>(), Int<8>());
        case 4: return wide ? f(Int<4>(), Int<32>()) : f(Int<4>(), Int<8>());
        case 32: return wide ? f(Int<32>(), Int<32>()) : f(Int<32>(), Int<8>());
        default: return cudaErrorInvalidValue;
    }
}
template <bool FLIP>
cudaError_t conv_s3(const float* in, const uint16_t* w, const float* bias, float* out, int B, int Cin, int Cout, int H,
                    int W, int act, cudaStream_t s) {
    return by_channels(Cin, Cout, [&](auto ci, auto np) {
        constexpr int CIN = decltype(ci)::value, NPAD = decltype(np)::value;
        const size_t sm = Conv3<CIN, NPAD>::SMEM;
        const cudaError_t e = cudaFuncSetAttribute(k_conv_fwd_s3<CIN, NPAD, FLIP>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
        if (e != cudaSuccess) return e;
        const dim3 grid((W + TS - 1) / TS, (H + TS - 1) / TS, B);
        k_conv_fwd_s3<CIN, NPAD, FLIP><<<grid, C3_THREADS, sm, s>>>(in, (const __nv_bfloat16*)w, bias, out, Cout, H, W, act);
        return cudaGetLastError();
    });
}
template <int CIN, int COUT, bool LONG>
cudaError_t wgrad_launch_as(dim3 grid, const float* in, float* g, const float* aout, float* partial, int H, int W, int rows,
                            cudaStream_t s) {
    const size_t sm = Wgrad<CIN, COUT>::SMEM;
    const cudaError_t e = cudaFuncSetAttribute(k_conv_wgrad_s3<CIN, COUT, LONG>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
    if (e != cudaSuccess) return e;
    k_conv_wgrad_s3<CIN, COUT, LONG><<<grid, Wgrad<CIN, COUT>::THREADS, sm, s>>>(in, g, aout, partial, H, W, rows);
    return cudaGetLastError();
}
template <int CIN, int COUT>
cudaError_t wgrad_launch(dim3 grid, const float* in, float* g, const float* aout, float* partial, int H, int W, int rows,
                         cudaStream_t s) {
    return rows * TS > 64 ? wgrad_launch_as<CIN, COUT, true>(grid, in, g, aout, partial, H, W, rows, s)
                          : wgrad_launch_as<CIN, COUT, false>(grid, in, g, aout, partial, H, W, rows, s);
}
template <int CIN>
cudaError_t wgrad_by_cout(int Cout, dim3 grid, const float* in, float* g, const float* aout, float* partial, int H, int W,
                          int rows, cudaStream_t s) {
    switch (Cout) {
        case 2: return wgrad_launch<CIN, 2>(grid, in, g, aout, partial, H, W, rows, s);
        case 4: return wgrad_launch<CIN, 4>(grid, in, g, aout, partial, H, W, rows, s);
        default: return wgrad_launch<CIN, 32>(grid, in, g, aout, partial, H, W, rows, s);
    }
}

}  // namespace

template <bool IN_NHWC, bool OUT_NHWC>
cudaError_t conv_tc_launch(const void* in, const __nv_bfloat16* wb, const float* bias, void* out, int B, int Cin,
                           int Cout, int H, int W, int act, cudaStream_t s) {
    dim3 grid((W + TS - 1) / TS, (H + TS - 1) / TS, B);
#define ES_TC(CI, NP) k_conv_fwd_tc<CI, NP, IN_NHWC, OUT_NHWC><<<grid, 128, 0, s>>>(in, wb, bias, out, Cout, H, W, act)
    if (Cout <= 8) {
        switch (Cin) {
            case 2: ES_TC(2, 8); break;
            case 4: ES_TC(4, 8); break;
            case 32: ES_TC(32, 8); break;
            default: return cudaErrorInvalidValue;
        }
    } else {
        switch (Cin) {
            case 2: ES_TC(2, 32); break;
            case 4: ES_TC(4, 32); break;
            case 32: ES_TC(32, 32); break;
            default: return cudaErrorInvalidValue;
        }
    }
#undef ES_TC
    return cudaGetLastError();
}

cudaError_t nn_conv_forward_bf16(const float* in, const uint16_t* w, const float* bias, float* out, int B, int Cin,
                                 int Cout, int H, int W, int act, cudaStream_t s) {
    return conv_tc_launch<false, false>(in, (const __nv_bfloat16*)w, bias, out, B, Cin, Cout, H, W, act, s);
}

cudaError_t nn_conv_forward_bf16_fmt(const void* in, bool in_nhwc, const uint16_t* w, const float* bias, void* out,
                                     bool out_nhwc, int B, int Cin, int Cout, int H, int W, int act, cudaStream_t s) {
    const __nv_bfloat16* wb = (const __nv_bfloat16*)w;
    if (out_nhwc && (Cout & 1)) return cudaErrorInvalidValue;
    if (in_nhwc)
        return out_nhwc ? conv_tc_launch<true, true>(in, wb, bias, out, B, Cin, Cout, H, W, act, s)
                        : conv_tc_launch<true, false>(in, wb, bias, out, B, Cin, Cout, H, W, act, s);
    return out_nhwc ? conv_tc_launch<false, true>(in, wb, bias, out, B, Cin, Cout, H, W, act, s)
                    : conv_tc_launch<false, false>(in, wb, bias, out, B, Cin, Cout, H, W, act, s);
}

}  // namespace es

using namespace es;

extern "C" {

size_t es_nn_workspace_bytes(int B, int Cin, int Cout, int H, int W) {
    if (!shape_ok(B, Cin, Cout, H, W)) return 0;
    const int rows = strip_rows(B, H, W);
    const size_t gx = (W + TS - 1) / TS, gy = ((H + TS - 1) / TS + rows - 1) / rows;
    const size_t strips = size_t(B) * gx * gy;
    const size_t len = size_t(Cout) * Cin * 9 + Cout;
    return sizeof(float) * strips * len;
}

int es_nn_conv_forward(const float* in, const uint16_t* w, const float* bias, float* out, int B, int Cin, int Cout,
                       int H, int W, int act_tanh, void* workspace, size_t workspace_bytes, void* stream) {
    if (!in || !w || !out || !workspace || !shape_ok(B, Cin, Cout, H, W)) return ES_ERR_ARG;
    if (workspace_bytes < sizeof(float) * size_t(Cout) * Cin * 9) return ES_ERR_ARG;
    if (in == out) return ES_ERR_ARG;
    return conv_s3<false>(in, w, bias, out, B, Cin, Cout, H, W, act_tanh, (cudaStream_t)stream) == cudaSuccess ? ES_OK
                                                                                                              : ES_ERR_CUDA;
}

int es_nn_conv_forward_bf16(const float* in, const uint16_t* w, const float* bias, float* out, int B, int Cin,
                            int Cout, int H, int W, int act_tanh, void* stream) {
    if (!in || !w || !bias || !out || !shape_ok(B, Cin, Cout, H, W) || in == out) return ES_ERR_ARG;
    return nn_conv_forward_bf16(in, w, bias, out, B, Cin, Cout, H, W, act_tanh, (cudaStream_t)stream) == cudaSuccess
               ? ES_OK
               : ES_ERR_CUDA;
}

int es_nn_conv_backward(const float* in, const uint16_t* w, const float* out, float* grad_out, float* grad_in,
                        float* grad_w, float* grad_b, int B, int Cin, int Cout, int H, int W, int act_tanh,
                        void* workspace, size_t workspace_bytes, void* stream) {
    if (!in || !w || !grad_out || !grad_w || !grad_b || !workspace || !shape_ok(B, Cin, Cout, H, W))
        return ES_ERR_ARG;
    if (act_tanh && !out) return ES_ERR_ARG;
    if (workspace_bytes < es_nn_workspace_bytes(B, Cin, Cout, H, W)) return ES_ERR_ARG;
    if (grad_in && (grad_in == grad_out || grad_in == in)) return ES_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    float* partial = (float*)workspace;
    const int rows = strip_rows(B, H, W);
    const dim3 grid((W + TS - 1) / TS, ((H + TS - 1) / TS + rows - 1) / rows, B);
    const float* aout = act_tanh ? out : nullptr;            // the gradient through tanh is formed in the same pass
    const cudaError_t e = Cin == 2   ? wgrad_by_cout<2>(Cout, grid, in, grad_out, aout, partial, H, W, rows, s)
                          : Cin == 4 ? wgrad_by_cout<4>(Cout, grid, in, grad_out, aout, partial, H, W, rows, s)
                                     : wgrad_by_cout<32>(Cout, grid, in, grad_out, aout, partial, H, W, rows, s);
    if (e != cudaSuccess) return ES_ERR_CUDA;
    const int nout = Cout * Cin * 9, len = nout + Cout;
    k_reduce_partials<<<(len + 31) / 32, 32 * RP_GROUPS, 0, s>>>(partial, int(grid.x * grid.y * grid.z), len, grad_w, grad_b,
                                                              nout);
    if (grad_in && conv_s3<true>(grad_out, w, nullptr, grad_in, B, Cout, Cin, H, W, 0, s) != cudaSuccess)
        return ES_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? ES_OK : ES_ERR_CUDA;
}

int es_nn_to_bf16(const float* src, uint16_t* dst, int64_t n, void* stream) {
    if (!src || !dst || n <= 0) return ES_ERR_ARG;
    k_f32_to_bf16<<<grid_for(size_t(n)), 256, 0, (cudaStream_t)stream>>>(src, (__nv_bfloat16*)dst, size_t(n));
    return cudaGetLastError() == cudaSuccess ? ES_OK : ES_ERR_CUDA;
}

int es_nn_mse(const float* pred, const float* target, float* grad, float* loss, int64_t n, void* stream) {
    if (!pred || !target || !grad || !loss || n <= 0) return ES_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    k_mse<<<grid_for(size_t(n)), 256, 0, s>>>(pred, target, grad, loss, size_t(n));
    return cudaGetLastError() == cudaSuccess ? ES_OK : ES_ERR_CUDA;
}

int es_nn_adam(float* master, uint16_t* w_bf16, const float* grad, float* m, float* v, int n, float lr, float beta1,
               float beta2, float eps, int step, void* stream) {
    if (!master || !grad || !m || !v || n <= 0 || step < 1 || !(lr >= 0.0f)) return ES_ERR_ARG;
    const float c1 = float(1.0 / (1.0 - pow(double(beta1), double(step))));
    const float c2 = float(1.0 / (1.0 - pow(double(beta2), double(step))));
    k_adam<<<grid_for(size_t(n)), 256, 0, (cudaStream_t)stream>>>(master, (__nv_bfloat16*)w_bf16, grad, m, v, n, lr,
                                                                  beta1, beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? ES_OK : ES_ERR_CUDA;
}

}  // extern "C"
