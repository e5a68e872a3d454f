// Backward kernels driven by the stored winners.  All are deterministic and use no
// atomics: every accumulator has exactly one writer at a time and a fixed order.
//
// Max / Min channel combine (one int32 winner per output):
//   bwd_idx_gx_kernel   a CTA owns a band of input rows of one image for every channel
//                       in shared memory; outputs are scattered tap by tap (within one tap
//                       two different output pixels never hit the same input element, and
//                       one thread walks all k of its pixel), barriers between taps.
//   bwd_idx_gw_kernel   warp-private histograms over (c, tap); lanes of a warp that hit the
//                       same bin take turns in lane order; per-CTA partials, fixed-order
//                       final sum (bwd_reduce_partials_kernel).  Also grad_bias.
// The Sum channel combine (one code per output and channel) has its kernels in tconv_bwd_sum.cuh.
#pragma once
#include "tconv_common.cuh"

namespace tconv {

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// ---------------------------------------------------------------------------------- idx: grad_x
template <typename T>
__global__ void __launch_bounds__(256)
bwd_idx_gx_kernel(Geo g, const T* __restrict__ gy, const int32_t* __restrict__ idx,
                  T* __restrict__ gx, int THI, int tiles_per_img, unsigned magic) {
    extern __shared__ float tile[];  // [C][THI][W]
    const int n = blockIdx.x / tiles_per_img;
    const int ih0 = (blockIdx.x - n * tiles_per_img) * THI;
    const int rows = min(THI, g.H - ih0);
    const int cstride = THI * g.W;
    for (int e = threadIdx.x; e < g.C * cstride; e += blockDim.x) tile[e] = 0.0f;
    __syncthreads();
    // output rows whose windows can reach the owned input rows
    const int num = ih0 + g.ph - (g.R - 1) * g.dh;
    const int oh_lo = num <= 0 ? 0 : (num + g.sh - 1) / g.sh;
    const int oh_hi = min(g.OH - 1, (ih0 + rows - 1 + g.ph) / g.sh);
    const int npix = (oh_hi - oh_lo + 1) * g.OW;
    const size_t plane = (size_t)g.OH * g.OW;
    for (int tap = 0; tap < g.RS; ++tap) {
        const int r = tap / g.S, s = tap - r * g.S;
        for (int pp = threadIdx.x; pp < npix; pp += blockDim.x) {
            const int orow = pp / g.OW;
            const int oh = oh_lo + orow, ow = pp - orow * g.OW;
            const int ih = oh * g.sh - g.ph + r * g.dh;
            const int iw = ow * g.sw - g.pw + s * g.dw;
            if (ih < ih0 || ih >= ih0 + rows || iw < 0 || iw >= g.W) continue;
            const size_t base = (size_t)n * g.K * plane + (size_t)oh * g.OW + ow;
            float* dst = tile + (ih - ih0) * g.W + iw;
#pragma unroll 4
            for (int k = 0; k < g.K; ++k) {
                const unsigned id = (unsigned)idx[base + (size_t)k * plane];
                const unsigned c = magic ? __umulhi(id, magic) : id;  // id / RS (magic 0: RS == 1)
                if ((int)(id - c * g.RS) == tap) dst[c * cstride] += to_f32(gy[base + (size_t)k * plane]);
            }
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < g.C * rows * g.W; e += blockDim.x) {
        const int c = e / (rows * g.W);
        const int rem = e - c * rows * g.W;
        gx[((size_t)n * g.C + c) * g.H * g.W + (size_t)ih0 * g.W + rem] =
            from_f32<T>(tile[c * cstride + rem]);
    }
}

// Second form of the same kernel for R*S <= 15: a thread reads the winners of its pixel once
// (batches of independent loads) and keeps only their taps, 4 bits each, in registers (blocks of
// 64 output channels).  In the phase of tap t it finds the channels whose winner is t with a few
// bit operations and touches only those: it reloads their winner (for the input channel) and
// their grad_y, the loads of the next match in flight while the current one is accumulated.
constexpr int kIdxGxKB = 8;    // output channels per staging round of bwd_idx_gx2_kernel
// RST: taps of the window when known at compile time (9: the tap loop unrolls and the targets of
// the nine phases are computed once per pixel), 0: taken from the descriptor.
template <typename T, int RST>
__global__ void __launch_bounds__(256)
bwd_idx_gx2_kernel(Geo g, const T* __restrict__ gy, const int32_t* __restrict__ idx,
                   T* __restrict__ gx, int THI, int tiles_per_img, unsigned magic) {
    constexpr int KB = kIdxGxKB;     // output channels staged per round
    constexpr int NOFF = RST > 0 ? RST : 1;
    extern __shared__ float tile[];  // [C][THI][W] | gs[KB][256] | cs[KB][256]
    const int n = blockIdx.x / tiles_per_img;
    const int ih0 = (blockIdx.x - n * tiles_per_img) * THI;
    const int rows = min(THI, g.H - ih0);
    const int cstride = THI * g.W;
    // thread-private columns: gradient and winning channel of the round's output channels
    float* gs = tile + (size_t)g.C * cstride + threadIdx.x;
    unsigned* cs = reinterpret_cast<unsigned*>(tile + (size_t)g.C * cstride + KB * 256) + threadIdx.x;
    for (int e = threadIdx.x; e < g.C * cstride; e += blockDim.x) tile[e] = 0.0f;
    const int num = ih0 + g.ph - (g.R - 1) * g.dh;
    const int oh_lo = num <= 0 ? 0 : (num + g.sh - 1) / g.sh;
    const int oh_hi = min(g.OH - 1, (ih0 + rows - 1 + g.ph) / g.sh);
    const int npix = (oh_hi - oh_lo + 1) * g.OW;
    const size_t plane = (size_t)g.OH * g.OW;
    const size_t img = (size_t)n * g.K * plane + (size_t)oh_lo * g.OW;   // first contributing pixel, k = 0
    __syncthreads();
    for (int pp0 = 0; pp0 < npix; pp0 += blockDim.x) {
        const int pp = pp0 + threadIdx.x;
        const bool live = pp < npix;
        const int orow = live ? pp / g.OW : 0;
        const int oh = oh_lo + orow, ow = live ? pp - orow * g.OW : 0;
        // element of the tile that tap t of this pixel reaches, -1 if outside the CTA's band
        auto target = [&](int tap) {
            const int r = tap / g.S, sx = tap - r * g.S;
            const int ih = oh * g.sh - g.ph + r * g.dh;
            const int iw = ow * g.sw - g.pw + sx * g.dw;
            return (live && ih >= ih0 && ih < ih0 + rows && iw >= 0 && iw < g.W) ? (ih - ih0) * g.W + iw : -1;
        };
        int off[NOFF];
        if constexpr (RST > 0) {
#pragma unroll
            for (int tap = 0; tap < RST; ++tap) off[tap] = target(tap);
        }
        const int32_t* ip = idx + img + pp;
        const T* gp = gy + img + pp;
        for (int kb0 = 0; kb0 < g.K; kb0 += KB, ip += (size_t)KB * plane, gp += (size_t)KB * plane) {
            const int kn = min(KB, g.K - kb0);
            // one round: KB winners and gradients of this pixel, all loads independent; the taps
            // stay in registers as 4-bit fields (15 marks "no channel here"), channel and gradient
            // go to the thread's shared-memory columns so that the phases below touch no global memory
            unsigned id[KB];
            float gv[KB];
#pragma unroll
            for (int i = 0; i < KB; ++i) {
                const bool ok = live && i < kn;
                id[i] = ok ? (unsigned)__ldg(ip + (size_t)i * plane) : 0xffffffffu;
                gv[i] = ok ? to_f32(__ldg(gp + (size_t)i * plane)) : 0.0f;
            }
            unsigned taps4[KB / 8];
#pragma unroll
            for (int wq = 0; wq < KB / 8; ++wq) {
                unsigned packed = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const unsigned v = id[wq * 8 + i];
                    const unsigned c = magic ? __umulhi(v, magic) : v;
                    const unsigned tap = (v == 0xffffffffu) ? 15u : (v - c * g.RS);
                    packed |= tap << (4 * i);
                    cs[(wq * 8 + i) * 256] = c;
                    gs[(wq * 8 + i) * 256] = gv[wq * 8 + i];
                }
                taps4[wq] = packed;
            }
            auto phase = [&](int tap, int o) {
                if (o >= 0) {
                    float* dst = tile + o;
                    const unsigned pat = 0x11111111u * (unsigned)tap;
#pragma unroll
                    for (int wq = 0; wq < KB / 8; ++wq) {
                        unsigned z = taps4[wq] ^ pat;       // nibble == 0 where the tap matches
                        z |= z >> 1;
                        z |= z >> 2;
                        unsigned m = ~z & 0x11111111u;      // bit 4*i set where nibble i matches
                        while (m) {
                            const int kk = wq * 8 + ((__ffs(m) - 1) >> 2);
                            m &= m - 1;
                            dst[cs[kk * 256] * cstride] += gs[kk * 256];
                        }
                    }
                }
                __syncthreads();   // inside one phase distinct pixels hit distinct inputs; phases are ordered
            };
            if constexpr (RST > 0) {
#pragma unroll
                for (int tap = 0; tap < RST; ++tap) phase(tap, off[tap]);
            } else {
                for (int tap = 0; tap < g.RS; ++tap) phase(tap, target(tap));
            }
        }
    }
    for (int e = threadIdx.x; e < g.C * rows * g.W; e += blockDim.x) {
        const int c = e / (rows * g.W);
        const int rem = e - c * rows * g.W;
        gx[((size_t)n * g.C + c) * g.H * g.W + (size_t)ih0 * g.W + rem] =
            from_f32<T>(tile[c * cstride + rem]);
    }
}

// ---------------------------------------------------------------------------------- idx: grad_w, grad_bias
template <typename T>
__global__ void __launch_bounds__(256)
bwd_idx_gw_kernel(Geo g, const T* __restrict__ gy, const int32_t* __restrict__ idx,
                  float* __restrict__ partial_w, float* __restrict__ partial_b, int n_per_chunk) {
    extern __shared__ float bins[];  // [8 warps][C*RS], then 256 floats for the bias sum
    const int CRS = g.C * g.RS;
    const int k = blockIdx.x, chunk = blockIdx.y;
    const int warp = threadIdx.x >> 5;
    float* mine = bins + warp * CRS;
    float* red = bins + 8 * CRS;
    for (int e = threadIdx.x; e < 8 * CRS; e += blockDim.x) bins[e] = 0.0f;
    __syncthreads();
    const int plane = g.OH * g.OW;
    const int n_lo = chunk * n_per_chunk, n_hi = min(g.N, n_lo + n_per_chunk);
    const unsigned lt = lanemask_lt();
    float bsum = 0.0f;
    // items of the chunk in a fixed order: (image, block of 256 pixels); the winners and gradients of
    // the next PF items are requested before the current ones are binned
    constexpr int PF = 4;
    const int blocks_per_img = (plane + 255) / 256;
    const int items = (n_hi - n_lo) * blocks_per_img;
    auto fetch = [&](int it, int& id, float& gv) {
        const int nn = it / blocks_per_img, p = (it - nn * blocks_per_img) * 256 + (int)threadIdx.x;
        const bool valid = it < items && p < plane;
        const size_t at = ((size_t)(n_lo + nn) * g.K + k) * plane + p;
        // an out-of-range lane takes a bin of its own so that it matches nobody
        id = valid ? __ldg(idx + at) : -1 - (int)threadIdx.x;
        gv = valid ? to_f32(__ldg(gy + at)) : 0.0f;
    };
    int idq[PF];
    float gq[PF];
#pragma unroll
    for (int u = 0; u < PF; ++u) fetch(u, idq[u], gq[u]);
    for (int it0 = 0; it0 < items; it0 += PF) {
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            if (it0 + u >= items) break;
            const int id = idq[u];
            const float gv = gq[u];
            fetch(it0 + u + PF, idq[u], gq[u]);
            const bool valid = id >= 0;
            bsum += gv;
            const unsigned same = __match_any_sync(0xffffffffu, id);
            const int rank = __popc(same & lt);
            const int maxrank = __reduce_max_sync(0xffffffffu, rank);
            for (int rr = 0; rr <= maxrank; ++rr) {
                if (rank == rr && valid) mine[id] += gv;
                __syncwarp();
            }
        }
    }
    __syncthreads();
    float* out = partial_w + ((size_t)chunk * g.K + k) * CRS;
    for (int b = threadIdx.x; b < CRS; b += blockDim.x) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += bins[w * CRS + b];
        out[b] = s;
    }
    const float tb = block_sum(bsum, red);
    if (threadIdx.x == 0) partial_b[chunk * g.K + k] = tb;
}

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
    // partial histograms of the Max / Min combine: at most 16 chunks of [K][C*RS + 1] floats; Sum forms
    // (any-shape kernels): 16 chunks of grad_bias partials
    if (g.chan == CH_SUM) return (size_t)16 * g.K * sizeof(float) + 256;
    return (size_t)16 * g.K * ((size_t)g.C * g.RS + 1) * sizeof(float) + 256;
}

// grad_y with rows padded by zeros to OWP elements: one thread per padded element.
template <typename T>
__global__ void __launch_bounds__(256)
pad_grad_kernel(Geo g, const T* __restrict__ gy, T* __restrict__ out) {
    const size_t total = (size_t)g.N * g.K * g.OH * g.OWP;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int ow = (int)(i % g.OWP);
    const size_t row = i / g.OWP;
    out[i] = ow < g.OW ? gy[row * g.OW + ow] : zero_of<T>();
}

constexpr size_t kBwdSmemLimit = 160 * 1024;   // planning budget per CTA
constexpr int kBwdSmemAttr = 200 * 1024;       // opt-in ceiling set on the kernels

// Plans for the winner-driven kernels; false when the shape does not fit (the caller then
// uses the any-shape kernels).
inline bool plan_idx_gx(const Geo& g, int* THI, size_t* smem) {
    const size_t row = (size_t)g.C * g.W * sizeof(float);
    if (row == 0 || row > kBwdSmemLimit) return false;
    int t = (int)(kBwdSmemLimit / row);
    if (t > g.H) t = g.H;
    // keep at least ~2 CTAs per SM worth of tiles when the batch is small, but never bands so thin
    // that most scanned rows are halo
    const int halo = (g.R - 1) * g.dh;
    while ((t + 1) / 2 >= 2 * halo && (t + 1) / 2 >= 4 && (size_t)g.N * ((g.H + t - 1) / t) < 296) t = (t + 1) / 2;
    if (t < g.H && t < 2 * halo) return false;  // too much redundant scanning
    *THI = t;
    *smem = row * t;
    return true;
}

inline bool plan_idx_gw(const Geo& g, int* chunks, size_t* smem) {
    const size_t bins = (size_t)8 * g.C * g.RS * sizeof(float) + 256 * sizeof(float);
    if (bins > kBwdSmemLimit) return false;
    int ch = (296 + g.K - 1) / g.K;
    if (ch > 16) ch = 16;
    if (ch > g.N) ch = g.N;
    if (ch < 1) ch = 1;
    *chunks = ch;
    *smem = bins;
    return true;
}

}  // namespace tconv
