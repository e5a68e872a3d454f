// What the winner-driven backward kernels share: winner codes of the Sum forms, grad_bias sums, the padded
// copy of grad_y.  The Max / Min channel combine has its kernels in tconv_bwd_idx.cuh, the Sum channel combine
// (one code per output and channel) in tconv_bwd_sum.cuh.
#pragma once
#include "tconv_bwd_idx.cuh"
#include "tconv_common.cuh"

namespace tconv {

// out[i] = sum over chunks (ascending) of partial[chunk][i]
static __global__ void bwd_reduce_partials_kernel(const float* __restrict__ partial, float* __restrict__ out,
                                           size_t len, int chunks) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len) return;
    float s = 0.0f;
    for (int c = 0; c < chunks; ++c) s += partial[(size_t)c * len + i];
    out[i] = s;
}

// ---------------------------------------------------------------------------------- codes
// The 4 winner codes of a quad.  Narrow codes (R*S <= 16): one byte each, argmin
// tap in the low nibble, argmax tap in the high nibble.  WIDE (R*S <= 256): 16 bits each, argmin tap
// in the low byte, argmax tap in the high byte.
template <bool WIDE> struct Codes4 { unsigned lo, hi; };
template <> struct Codes4<false> { unsigned lo; };

// grad_bias partials: grid (K, chunks); partial[chunk][k] = sum of grad_y over the chunk's images
template <typename T>
__global__ void __launch_bounds__(256)
bwd_bias_partial_kernel(Geo g, const T* __restrict__ gy, float* __restrict__ partial, int n_per_chunk) {
    __shared__ float red[256];
    const int k = blockIdx.x, chunk = blockIdx.y;
    const size_t plane = (size_t)g.OH * g.OW;
    const int n_lo = chunk * n_per_chunk, n_hi = min(g.N, n_lo + n_per_chunk);
    float s = 0.0f;
    for (int n = n_lo; n < n_hi; ++n) {
        const T* src = gy + ((size_t)n * g.K + k) * plane;
        for (size_t j = threadIdx.x; j < plane; j += blockDim.x) s += to_f32(src[j]);
    }
    const float t = block_sum(s, red);
    if (threadIdx.x == 0) partial[chunk * g.K + k] = t;
}

// ---------------------------------------------------------------------------------- host side
// Sum forms whose output width is not a multiple of 4 run their code-driven kernels as a layer of
// output width OWP on a copy of grad_y with zero-padded rows (every quad whole, every load an
// aligned vector): the geometry those kernels see, and the bytes of the copy.
inline Geo widened_geo(const Geo& g) {
    Geo q = g;
    q.OW = g.OWP;
    return q;
}
inline size_t padded_gy_bytes(const Geo& g, int esize) {
    if ((g.OW & 3) == 0) return 0;
    return ((size_t)g.N * g.K * g.OH * g.OWP * esize + 255) / 256 * 256;
}

inline size_t bwd_ws_bytes(const Geo& g) {
    // grad_bias partials of the any-shape path; Max / Min combine: the histograms of bwd_idx_gw_kernel
    const size_t bias = (size_t)16 * g.K * sizeof(float) + 256;
    IdxGwPlan p;
    if (g.chan == CH_SUM || !plan_idx_gw(g, &p)) return bias;
    const size_t part = p.part_floats * sizeof(float) + 256;
    return part > bias ? part : bias;
}

__device__ __forceinline__ void store_quad(float* o, const float* v) {
    *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store_quad(__nv_bfloat16* o, const __nv_bfloat16* v) {
    __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(o);
    p[0] = __halves2bfloat162(v[0], v[1]);
    p[1] = __halves2bfloat162(v[2], v[3]);
}

// grad_y with rows padded by zeros to OWP elements: one thread per four of them (one store).
// N=80 K=152 71x142 fp32 (983 MB) took 492 us with one thread and two divisions per element.
template <typename T>
__global__ void __launch_bounds__(256)
pad_grad_kernel(Geo g, const T* __restrict__ gy, T* __restrict__ out, size_t rows, unsigned rpb) {
    const unsigned QPR = (unsigned)g.OWP >> 2, r = threadIdx.x / QPR, q0 = threadIdx.x - r * QPR;
    const unsigned step = QPR < 256 ? QPR : 256;
    if (r >= rpb) return;
    // a block takes rpb whole rows at once (long rows: one, in steps of 256 threads), four times
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const size_t row = ((size_t)blockIdx.x * 4 + u) * rpb + r;
        if (row >= rows) return;
        for (unsigned q = q0; q < QPR; q += step) {
            const T* p = gy + row * g.OW + 4 * q;
            T v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = (int)(4 * q) + j < g.OW ? __ldg(p + j) : zero_of<T>();
            store_quad(out + (row * QPR + q) * 4, v);
        }
    }
}

constexpr int kBwdSmemAttr = 200 * 1024;       // opt-in ceiling set on the kernels

}  // namespace tconv
