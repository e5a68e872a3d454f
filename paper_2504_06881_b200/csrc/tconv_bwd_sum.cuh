// Backward of the Sum channel combine (layers (i), (ii), compound, parallel): two kernels over the winner
// codes and one that finishes their partial sums.
//
//   bwd_sum_gx_kernel   a CTA owns one input channel of a tile of outputs of one image (or of several
//                       small images); a thread owns 4 adjacent output pixels and walks the output
//                       channels k.  It adds coef * g into its private per-tap accumulators, which a
//                       gather over the taps turns into grad_x at the end.  For grad_alpha / grad_beta
//                       the inputs of its windows sit beside the accumulators, so the input of a winner
//                       is read through the address of its accumulator; with the winning weight it gives
//                       the branch value as the forward rounded it, and g * (x + w) is summed over the
//                       warp per k.
//   bwd_sum_edges_kernel  where an image is cut into tiles: adds the (overlapping) input regions the
//                       tiles' outputs reach.
//   bwd_sum_gw_kernel   a warp owns one (k, c) pair and a share of its (image, pixel) items; every
//                       lane keeps a private histogram of g over the *pair* of winning taps, so that
//                       an item costs one shared-memory read-modify-write for both branches.
//   bwd_sum_finish_kernel  sums the partials in a fixed order and applies alpha / beta.
//
// No atomics; every accumulator has one writer and a fixed order.
#pragma once
#include <cstring>
#include <type_traits>

#include "tconv_bwd.cuh"

namespace tconv {

// ---------------------------------------------------------------------------------- plans
constexpr int kSgThreads = 256;         // most threads of a grad_x CTA: one quad each
constexpr int kSgKB = 8;                // output channels per stage of coefficients and weights
constexpr size_t kSgSmem = 112 * 1024;  // two CTAs per SM (other windows than 3 x 3)
constexpr int kSgSmemAttr = 214 * 1024; // opt-in ceiling: accumulators of kBwdSmemAttr and their stages

struct SumGxPlan {
    int threads;
    int imgs;                      // images per CTA (> 1: whole images of a small map)
    int TR, TQ;                    // output rows and quads per row of a tile
    int nrow, ncol;                // tiles of an image
    int ER, EC;                    // input rows and columns the outputs of a tile reach
    unsigned ctas;                 // tiles of all images (without the channels)
    size_t smem;
};

struct SumGwPlan {
    int flat;                      // items run over the flattened (image, quad) space
    int blocks;                    // an image is whole blocks of 128 quads, and so are the shares
    int splits;                    // shares of a pair's items
    int per;                       // quads (flat) or rounds of 32 quads per share
    int pairs;                     // 1: one table over the pair of winners, 0: one table per branch
    int nbins;                     // bins of a lane's tables
    unsigned grid;
    size_t smem;
};

// Stage of eight output channels' operands: weights [channel][tap], {alpha, beta} behind them, then (parallel) the
// weights of the max branch.  Both tables and the two stages start at multiples of 256 bytes, so that a winner's
// weight is addressed by putting tap * 4 into the low byte.  (Single-branch layers have none of them.)
struct SumStage {
    int coef, w2, stride, bytes;       // offsets of {alpha, beta} and w2, distance of the two stages, bytes of both
};
__host__ __device__ inline SumStage sum_stage(int mode, int RS) {
    SumStage t;
    t.coef = two_branch(mode) ? kSgKB * RS * 4 : 0;
    const int len = t.coef + kSgKB * 8;
    t.w2 = mode == TCONV_PARALLEL ? (len + 255) / 256 * 256 : 0;
    const int all = mode == TCONV_PARALLEL ? t.w2 + kSgKB * RS * 4 : len;
    t.stride = (all + 255) / 256 * 256;
    t.bytes = two_branch(mode) ? t.stride + all : 0;
    return t;
}

// Picks the tile of outputs with the least work: lanes (idle ones included) times output channels, and
// the input region a tile leaves for the final sum.
inline bool plan_sum_gx(const Geo& g, SumGxPlan* best) {
    const bool ab = two_branch(g.mode), k3 = g.R == 3 && g.S == 3;
    const size_t group = (size_t)g.RS * 256 * (ab ? 8 : 4);     // accumulators (and window inputs) of 64 threads
    const int halo_h = (g.R - 1) * g.dh, halo_w = (g.S - 1) * g.dw, QPR = (g.OW + 3) / 4;
    int most = kSgThreads;
    const size_t stages = sum_stage(g.mode, g.RS).bytes;
    while (most > 64 && most / 64 * group + stages > kSgSmem) most -= 64;
    if (most / 64 * group > kBwdSmemAttr) return false;
    double best_cost = -1.0;
    for (int ncol = 1; ncol <= QPR; ++ncol) {
        SumGxPlan p;
        p.TQ = (QPR + ncol - 1) / ncol;
        if (p.TQ > most) continue;
        p.ncol = (QPR + p.TQ - 1) / p.TQ;
        if (p.ncol != ncol) continue;
        if (p.TQ < 4 && ncol > 1) break;
        const int rows = most / p.TQ < g.OH ? most / p.TQ : g.OH;
        p.nrow = (g.OH + rows - 1) / rows;
        p.TR = (g.OH + p.nrow - 1) / p.nrow;                    // even bands
        p.nrow = (g.OH + p.TR - 1) / p.TR;
        p.imgs = 1;
        if (p.nrow * ncol == 1) {
            int im = most / (p.TR * p.TQ);
            if (im > g.N) im = g.N;
            // (a thread addresses the codes of its CTA's images with a 32-bit count of quads)
            const double per_img = (double)g.K * g.C * g.OH * g.OW;
            while (im > 1 && per_img * im > 1.6e10) --im;
            // small batches: as many CTAs as the SMs can take before a CTA takes a second image
            while (im > 1 && (double)((g.N + im - 1) / im) * g.C < 148.0) --im;
            const int groups = (g.N + im - 1) / im;             // even groups
            p.imgs = (g.N + groups - 1) / groups;
        }
        p.ER = (p.TR - 1) * g.sh + halo_h + 1;
        p.EC = (p.TQ * 4 - 1) * g.sw + halo_w + 1;
        p.threads = (p.TR * p.TQ * p.imgs + 31) / 32 * 32;
        const double ctas = (double)((g.N + p.imgs - 1) / p.imgs) * p.nrow * ncol;
        if (ctas * g.C > 2.0e9) continue;
        p.ctas = (unsigned)ctas;
        p.smem = (k3 ? kSgThreads / 64 : (p.threads + 63) / 64) * group + stages;
        const double per_sm = ctas * g.C / 148.0;
        const double cost = ctas * (4.0 * p.threads * g.K + (p.nrow * ncol > 1 ? 2.0 * p.ER * p.EC : 0.0)) * (per_sm < 1.0 ? 1.0 / per_sm : 1.0);
        if (best_cost < 0.0 || cost < best_cost) { best_cost = cost; *best = p; }
    }
    return best_cost >= 0.0;
}

inline bool plan_sum_gw(const Geo& g, SumGwPlan* p) {
    const long pairs = (long)g.K * g.C;
    const long nq = (long)g.OH * ((g.OW + 3) / 4), rpi = nq / 32;
    p->flat = nq % 32 != 0;
    const long items = p->flat ? g.N * nq : g.N * rpi;
    const long least = p->flat ? 256 : 8;              // a share is at least eight rounds
    // one table over the pair of winners while it is small and a pair's items outweigh clearing and
    // summing it (RS * RS columns against one access per item saved)
    const bool two = two_branch(g.mode);
    p->pairs = two && g.RS <= 9 && (double)g.N * nq * 4 / 32 >= 2.0 * g.RS * g.RS;
    p->nbins = p->pairs ? g.RS * g.RS : two ? 2 * g.RS : g.RS;
    p->smem = (size_t)4 * p->nbins * 32 * sizeof(float);
    if (p->smem > kBwdSmemAttr) return false;
    long per_sm = (long)((227 * 1024) / (p->smem + 1024)) * 4;
    if (per_sm > 32) per_sm = 32;
    const long slots = 148 * per_sm;
    // among the counts that fill the SMs the one whose last round of resident warps is fullest
    long most = items / least;
    if (most < 1) most = 1;
    if (most > 64) most = 64;
    long s = 1;
    double best = -1.0;
    for (long c = 1; c <= most; ++c) {
        const long w = pairs * c, rounds = (w + slots - 1) / slots;
        const double eff = (double)w / (double)(rounds * slots);
        if (eff > best + 0.02) { best = eff; s = c; }
        if (best > 0.92) break;
    }
    p->per = (int)((items + s - 1) / s);
    p->blocks = !p->flat && rpi % 4 == 0;
    // (Blocks: rounded up behind the search, up to a third longer where shares are short, yet no slower than the shares of
    // the search in whole rounds: 3 -> 16 channels 32x32 N=64 fp32 compound 43 of 12 rounds 6.5 us, 57 of 9 7.5.  A search
    // over the rounded lengths ends at fewer and longer or more and shorter ones, up to 12 % slower.)
    if (p->blocks) p->per = (p->per + 3) / 4 * 4;
    p->splits = (int)((items + p->per - 1) / p->per);
    p->grid = (unsigned)((pairs * p->splits + 3) / 4);
    return true;
}

// Both plans of a layer; the search above is host work of some microseconds, so the last few are kept
// per host thread (they depend on nothing but the geometry).
struct SumPlans {
    Geo g;
    int esize;
    SumGxPlan gx;
    SumGwPlan gw;
    int ok;      // the layer fits both kernels
};
inline const SumPlans& sum_plans(const Geo& g, int esize) {
    constexpr int kKept = 32;
    static thread_local SumPlans kept[kKept];
    static thread_local int used = 0, next = 0;
    for (int i = 0; i < used; ++i)
        if (kept[i].esize == esize && memcmp(&kept[i].g, &g, sizeof(Geo)) == 0) return kept[i];
    SumPlans& p = kept[next];
    p.g = g;
    p.esize = esize;
    // 31-bit counts: quads of all images (a share's last round may end past them), positions of a map, images x channels
    p.ok = (double)g.N * g.OH * g.OWP < 8.0e9 && (double)g.OH * g.OWP < 2.1e9 && (double)g.H * g.W < 2.1e9 &&
           (double)g.N * g.C < 2.0e9 && plan_sum_gx(g, &p.gx) && plan_sum_gw(g, &p.gw);
    next = (next + 1) % kKept;
    if (used < kKept) ++used;
    return p;
}
// Partial sums of a call: [grad_w histograms | grad_alpha, grad_beta rows | input regions of the tiles].
inline size_t sum_part_gw_bytes(const Geo& g, const SumGwPlan& p) {
    return ((size_t)p.splits * g.K * g.C * 2 * g.RS * sizeof(float) + 255) / 256 * 256;
}
inline size_t sum_part_ab_bytes(const Geo& g, const SumGxPlan& p) {
    return two_branch(g.mode) ? ((size_t)p.ctas * g.K * g.C * 2 * sizeof(float) + 255) / 256 * 256 : 0;
}
inline size_t sum_part_gx_bytes(const Geo& g, const SumGxPlan& p) {
    return p.nrow * p.ncol > 1 ? ((size_t)p.ctas * g.C * p.ER * p.EC * sizeof(float) + 255) / 256 * 256 : 0;
}
// Images of 2^32 gradients or of 2^32 quads of winners and more.
inline bool sum_far(const Geo& g) {
    return (double)g.OH * g.OW * g.K > 4.2e9 || (double)g.OH * g.OW * g.K * g.C > 1.6e10;
}
// Bytes of all partial sums; 0 when the layer does not fit the kernels.  g: widened to whole quads.
inline size_t sum_ws_bytes(const Geo& g, int esize) {
    const SumPlans& p = sum_plans(g, esize);
    return p.ok ? sum_part_gw_bytes(g, p.gw) + sum_part_ab_bytes(g, p.gx) + sum_part_gx_bytes(g, p.gx) : 0;
}

// ---------------------------------------------------------------------------------- loads
// Operands requested ahead of their use: volatile, so that they stay where they are written.  KEEP: the
// lines are shared with other warps of the CTA (grad_w); the grad_x kernel streams its operands past an L1
// that the accumulators leave little of.
template <typename T, bool KEEP>
__device__ __forceinline__ void ahead_g4(const T* p, float* gv) {
    if constexpr (sizeof(T) == 4) {
        if constexpr (KEEP) asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(gv[0]), "=f"(gv[1]), "=f"(gv[2]), "=f"(gv[3]) : "l"(p));
        else asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(gv[0]), "=f"(gv[1]), "=f"(gv[2]), "=f"(gv[3]) : "l"(p));
    } else {
        unsigned a, b;
        if constexpr (KEEP) asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
        else asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
        gv[0] = __uint_as_float(a); gv[1] = __uint_as_float(b);      // (unpacked when used: unpack_g4)
    }
}
template <typename T> __device__ __forceinline__ void unpack_g4(const float* raw, float* gv) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j) gv[j] = raw[j];
    } else {
        const unsigned a = __float_as_uint(raw[0]), b = __float_as_uint(raw[1]);
        gv[0] = __uint_as_float(a << 16); gv[1] = __uint_as_float(a & 0xffff0000u);
        gv[2] = __uint_as_float(b << 16); gv[3] = __uint_as_float(b & 0xffff0000u);
    }
}
__device__ __forceinline__ float ahead_value(const float* p) {
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ahead_value(const __nv_bfloat16* p) {
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return __bfloat162float(__ushort_as_bfloat16(v));
}
template <bool WIDE, bool KEEP>
__device__ __forceinline__ Codes4<WIDE> ahead_codes4(const uint8_t* p) {
    Codes4<WIDE> r;
    if constexpr (!WIDE) {
        if constexpr (KEEP) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(r.lo) : "l"(p));
        else asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(r.lo) : "l"(p));
    } else {
        asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(r.lo), "=r"(r.hi) : "l"(p));
    }
    return r;
}

// ---------------------------------------------------------------------------------- grad_x, grad_alpha, grad_beta
__device__ __forceinline__ float load_xf(const void* x, size_t i, int xf32, float) { return __ldg(reinterpret_cast<const float*>(x) + i); }
__device__ __forceinline__ float load_xf(const void* x, size_t i, int xf32, __nv_bfloat16) {
    if (xf32) return __bfloat162float(__float2bfloat16_rn(__ldg(reinterpret_cast<const float*>(x) + i)));
    return __bfloat162float(__ldg(reinterpret_cast<const __nv_bfloat16*>(x) + i));
}

// Sums 16 values over the warp: halving butterfly, lane 2v (and 2v + 1) ends with the total of value v.
__device__ __forceinline__ float warp_sum16(float* s, int lane) {
#pragma unroll
    for (int step = 0; step < 4; ++step) {
        const int d = 16 >> step, n = 8 >> step;
        const bool up = (lane & d) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? s[i + n] : s[i];
            const float send = up ? s[i] : s[i + n];
            s[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
    }
    return s[0] + __shfl_xor_sync(0xffffffffu, s[0], 1);
}

// Byte offset tap << SH of pixel j for the min / max branch (SH 8 or 10).  Narrow codes: the nibbles of a
// quad's four codes, one per byte; one PRMT moves a byte to bits 8..15.
template <bool WIDE, int SH> struct QuadTaps;
template <int SH> struct QuadTaps<false, SH> {
    static constexpr unsigned mask = 0x0f0f0f0fu << (SH - 8);
    unsigned lo, hi;
    __device__ __forceinline__ explicit QuadTaps(const Codes4<false>& c) : lo((c.lo << (SH - 8)) & mask), hi((c.lo >> (12 - SH)) & mask) {}
    __device__ __forceinline__ unsigned tmin(int j) const { return __byte_perm(lo, 0u, 0x4404u + (unsigned)(j << 4)); }
    __device__ __forceinline__ unsigned tmax(int j) const { return __byte_perm(hi, 0u, 0x4404u + (unsigned)(j << 4)); }
};
template <> struct QuadTaps<true, 8> {
    Codes4<true> c;
    __device__ __forceinline__ explicit QuadTaps(const Codes4<true>& c_) : c(c_) {}
    __device__ __forceinline__ unsigned tmin(int j) const { return __byte_perm(j < 2 ? c.lo : c.hi, 0u, 0x4404u + (unsigned)((2 * (j & 1)) << 4)); }
    __device__ __forceinline__ unsigned tmax(int j) const { return __byte_perm(j < 2 ? c.lo : c.hi, 0u, 0x4404u + (unsigned)((2 * (j & 1) + 1) << 4)); }
};
// Shared-memory address of the winning weight of pixel j: table (at a multiple of 256 bytes) + tap * 4.
template <bool WIDE> struct QuadWeights;
template <> struct QuadWeights<false> {
    unsigned lo, hi;
    __device__ __forceinline__ explicit QuadWeights(const Codes4<false>& c) : lo((c.lo << 2) & 0x3c3c3c3cu), hi((c.lo >> 2) & 0x3c3c3c3cu) {}
    __device__ __forceinline__ unsigned tmin(unsigned table, int j) const { return __byte_perm(lo, table, 0x7650u + (unsigned)j); }
    __device__ __forceinline__ unsigned tmax(unsigned table, int j) const { return __byte_perm(hi, table, 0x7650u + (unsigned)j); }
};
template <> struct QuadWeights<true> {
    QuadTaps<true, 8> t;
    __device__ __forceinline__ explicit QuadWeights(const Codes4<true>& c) : t(c) {}
    __device__ __forceinline__ unsigned tmin(unsigned table, int j) const { return table + (t.tmin(j) >> 6); }
    __device__ __forceinline__ unsigned tmax(unsigned table, int j) const { return table + (t.tmax(j) >> 6); }
};
__device__ __forceinline__ float load_shared(unsigned at) {
    return *reinterpret_cast<const float*>(__cvta_shared_to_generic(at));
}
__device__ __forceinline__ float& at_shared(unsigned at) { return *reinterpret_cast<float*>(__cvta_shared_to_generic(at)); }
// Address base + tap * 256 of a pixel's bin.  Narrow codes: the nibbles in the high halves of the bytes, and one dot
// product of bytes picks, scales and adds one of them (7 x 7 x 512 bf16 compound: 724 -> 707 us against a byte
// permutation and an add; the table over pairs of winners has more bits than a byte's half and keeps those).
template <bool WIDE> struct BinAddress {
    QuadTaps<WIDE, 8> t;
    __device__ __forceinline__ explicit BinAddress(const Codes4<WIDE>& c) : t(c) {}
    __device__ __forceinline__ unsigned tmin(unsigned base, int j) const { return base + t.tmin(j); }
    __device__ __forceinline__ unsigned tmax(unsigned base, int j) const { return base + t.tmax(j); }
};
template <> struct BinAddress<false> {
    unsigned lo, hi;
    __device__ __forceinline__ explicit BinAddress(const Codes4<false>& c) : lo((c.lo << 4) & 0xf0f0f0f0u), hi(c.lo & 0xf0f0f0f0u) {}
    __device__ __forceinline__ unsigned tmin(unsigned base, int j) const { return __dp4a(lo, 16u << (8 * j), base); }
    __device__ __forceinline__ unsigned tmax(unsigned base, int j) const { return __dp4a(hi, 16u << (8 * j), base); }
};

// Branch values z = x + w of a quad as the forward rounds them (one rounded add; bf16: the fp32 sum of two bf16
// values keeps more than twice their bits, so rounding it equals the bf16 add).
__device__ __forceinline__ void branch_values(const float* x, const float* w, float* z, float) {
#pragma unroll
    for (int j = 0; j < 4; ++j) z[j] = __fadd_rn(x[j], w[j]);
}
__device__ __forceinline__ void branch_values(const float* x, const float* w, float* z, __nv_bfloat16) {
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(__fadd_rn(x[j], w[j]), __fadd_rn(x[j + 1], w[j + 1]));
        z[j] = __low2float(v);
        z[j + 1] = __high2float(v);
    }
}

// BR: 0 both branches, 1 min branch only, 2 max branch only.  GX: grad_x.  AB: grad_alpha / grad_beta (BR 0).
// KW: 3 or 5 for 3 x 3 (narrow codes) and 5 x 5 windows (wide codes), else 0 (any window, and images whose
// gradients or winners exceed 32-bit counts: sum_far).
// Shared memory: accumulators [4][tap][TP] floats per TP threads, then (AB) the window inputs in the same
// layout, at the end two stages of eight output channels' coefficients and (AB) weights; TP is 256 for 3 x 3 windows (and the taps of a column lie 1024 bytes apart), 64 otherwise (256
// bytes apart): one PRMT and one add address an accumulator, and the winner's input lies at a constant
// distance from it.
// Bound by the shared-memory accesses of a quad and output channel: per branch four loads and four stores of
// accumulators, four inputs, four weights.  The weights cost the training pass of N=128 C=64 K=64 32x32 fp32
// 2.27 -> 2.41 ms against sums of g * x completed by the weights times the histograms; but those are the gradient
// of an unrounded x + w, lose what x + w cancels, and are NaN where an infinite weight never wins.
// TAIL: the last stage may have output channels past K.  They repeat the last one, and their gradients are dropped
// by selection (times a zero coefficient an infinite one would be NaN); selecting in every stage costs 3 x 3 layers
// 3 %, so they have an instance for multiples of eight channels without it.
template <typename T, int BR, bool GX, bool AB, bool WIDE, int KW, bool TAIL>
__global__ void __launch_bounds__(kSgThreads, KW == 3 ? 3 : 2)
bwd_sum_gx_kernel(Geo g, const void* __restrict__ x, const T* __restrict__ w, const T* __restrict__ w2,
                  const float* __restrict__ alpha, const float* __restrict__ beta, const T* __restrict__ gy,
                  const uint8_t* __restrict__ codes, T* __restrict__ gx, float* __restrict__ part_ab, float* __restrict__ part_gx, SumGxPlan pl) {
    constexpr bool K3 = KW == 3;
    constexpr int TP = K3 ? kSgThreads : 64, TS = TP * 4;      // columns side by side, bytes between two taps
    const int RS = KW ? KW * KW : g.RS;
    const int WR = KW ? KW : g.R, WS = KW ? KW : g.S;
    const int gbytes = RS * TS * (AB ? 8 : 4);                 // bytes of TP threads
    extern __shared__ __align__(256) char smem[];
    __shared__ float part[2][kSgThreads / 32][kSgKB * 2];      // g * branch value of a warp, by stage
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int c = blockIdx.x % g.C;
    const unsigned tile = blockIdx.x / g.C;
    const int ct = tile % pl.ncol, rt = (tile / pl.ncol) % pl.nrow;
    const int n_first = (tile / pl.ncol / pl.nrow) * pl.imgs;
    const int nimg = min(pl.imgs, g.N - n_first);
    const int oh0 = rt * pl.TR, oq0 = ct * pl.TQ;
    const int tr = min(pl.TR, g.OH - oh0), tq = min(pl.TQ, (g.OW >> 2) - oq0);   // output rows, quads per row
    const int NQ1 = tr * tq, NQ = NQ1 * nimg;
    const unsigned plane = (unsigned)g.OH * (unsigned)g.OW;
    constexpr int CW = WIDE ? 2 : 1;                           // bytes per code
    constexpr bool FAR = KW == 0;
    // addresses: a base of the CTA plus a 32-bit count of the thread, elements of grad_y and quads of codes.  FAR: the
    // output channels advance the base, the count is that of the image and pixel (several images only of maps of at
    // most 256 quads); as 64-bit sums they cost 3 x 3 layers 3 %
    const T* gbase = gy + (size_t)n_first * g.K * plane;
    const uint8_t* cbase = codes + ((size_t)n_first * g.K * g.C + c) * plane * CW;
    using Count = std::conditional_t<FAR, size_t, unsigned>;
    const Count cstep = (Count)g.C * (plane >> 2);             // quads of codes between two output channels
    {
        // a thread without a quad repeats the last one into columns nobody reads
        const bool live = tid < NQ;
        const int q = min(tid, NQ - 1);
        const int il = q / NQ1, q1 = q - il * NQ1, orow = q1 / tq;
        const int oh = oh0 + orow, ow0 = (oq0 + q1 - orow * tq) * 4;
        const unsigned pix = (unsigned)(oh * g.OW + ow0);
        unsigned goff = (unsigned)(il * g.K) * plane + pix;
        unsigned coff = (unsigned)(il * g.K) * (unsigned)cstep + (pix >> 2);
        char* Ab = smem + (size_t)(tid / TP) * gbytes + (tid % TP) * 4;

        // gradients and codes of a pair of output channels are requested together, one pair ahead: the loads
        // of a pair share a scoreboard, which a longer chain of single requests would exhaust (past the last
        // channel it is read again: the staged coefficients of such a channel are zero)
        constexpr int PF = 4;
        float raw[PF][sizeof(T)];      // (4 floats, or 4 bf16 in two registers)
        Codes4<WIDE> cq[PF];
        int more = g.K - 1;
        if constexpr (AB) {            // a repeated quad has no gradient
#pragma unroll
            for (int u = 0; u < PF; ++u)
#pragma unroll
                for (int i = 0; i < (int)sizeof(T); ++i) raw[u][i] = 0.0f;
        }
        auto request = [&](int u) {
            if (!AB || live) ahead_g4<T, false>(gbase + goff, raw[u]);
            cq[u] = ahead_codes4<WIDE, false>(cbase + (size_t)coff * (4 * CW));
            if (more > 0) {
                if constexpr (FAR) { gbase += plane; cbase += cstep * (4 * CW); }
                else { goff += plane; coff += cstep; }
            }
            --more;
        };
        request(0);
        request(1);

        if constexpr (GX)
            for (int e = 0; e < 4 * RS; ++e) *reinterpret_cast<float*>(Ab + e * TS) = 0.0f;
        if constexpr (AB) {
            // the inputs of the four windows; zero outside the image and for a repeated quad
            const size_t xc = ((size_t)(n_first + il) * g.C + c) * g.H * g.W;
            const int iwq = ow0 * g.sw - g.pw;
            char* Xb = Ab + 4 * RS * TS;
#pragma unroll
            for (int r = 0; r < WR; ++r) {
                const int ih = oh * g.sh - g.ph + r * g.dh;
                const bool rok = live && ih >= 0 && ih < g.H;
                const size_t xrow = xc + (size_t)(rok ? ih : 0) * g.W;
                auto fetch = [&](int iw) { return rok && iw >= 0 && iw < g.W ? load_xf(x, xrow + iw, g.xf32, T()) : 0.0f; };
                if (KW && g.sw == 1 && g.dw == 1) {       // neighbouring windows share their columns
                    float col[KW + 3];
#pragma unroll
                    for (int i = 0; i < KW + 3; ++i) col[i] = fetch(iwq + i);
#pragma unroll
                    for (int t = 0; t < KW; ++t)
#pragma unroll
                        for (int j = 0; j < 4; ++j) *reinterpret_cast<float*>(Xb + (j * RS + r * KW + t) * TS) = col[t + j];
                } else {
                    for (int t = 0; t < WS; ++t)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            *reinterpret_cast<float*>(Xb + (j * RS + r * WS + t) * TS) = fetch(iwq + j * g.sw + t * g.dw);
                }
            }
        }

        // The operands of the next stage are requested before this stage's are used and stored behind them (one a
        // thread; the rest of a large window's weights are copied then).
        const SumStage lay = sum_stage(g.mode, RS);
        char* stage = smem + pl.smem - lay.bytes;
        const int nw = AB ? kSgKB * RS : 0, nstage = BR != 0 ? 0 : 2 * kSgKB + nw * (AB && g.mode == TCONV_PARALLEL ? 2 : 1);
        struct Operand {
            const void* from;      // of the first stage; null: all ones
            int kk, to;            // output channel within the stage, place in it
            bool coef;
        };
        auto operand = [&](int e) {
            Operand o;
            o.coef = e < 2 * kSgKB;
            if (o.coef) {
                const float* ab = (e & 1) ? beta : alpha;
                o.kk = e >> 1;
                o.to = lay.coef + 4 * e;
                o.from = ab ? ab + (size_t)o.kk * g.C + c : nullptr;
            } else {
                e -= 2 * kSgKB;
                const bool second = e >= nw;
                if (second) e -= nw;
                o.kk = e / RS;
                o.to = (second ? lay.w2 : 0) + 4 * e;
                o.from = (second ? w2 : w) + ((size_t)o.kk * g.C + c) * RS + e % RS;
            }
            return o;
        };
        auto fetch = [&](const Operand& o, int k0) {
            if (k0 + o.kk >= g.K) return 0.0f;
            if (o.coef) return o.from ? ahead_value(static_cast<const float*>(o.from) + (size_t)k0 * g.C) : 1.0f;
            return ahead_value(static_cast<const T*>(o.from) + (size_t)k0 * g.C * RS);
        };
        auto copy = [&](int e0, int k0, char* to) {
            for (int e = e0; e < nstage; e += blockDim.x) {
                const Operand o = operand(e);
                *reinterpret_cast<float*>(to + o.to) = fetch(o, k0);
            }
        };
        if constexpr (BR == 0) {
            copy(tid, 0, stage);
            __syncthreads();
        }
        int buf = 0;
        for (int k0 = 0; k0 < g.K; k0 += kSgKB, buf ^= 1) {
            const bool more_k = k0 + kSgKB < g.K;
            float ahead = 0.0f;
            if (BR == 0 && more_k && tid < nstage) ahead = fetch(operand(tid), k0 + kSgKB);
            const char* st = stage + buf * lay.stride;
            const unsigned table = (unsigned)__cvta_generic_to_shared(st);
            float s[AB ? 16 : 1];
#pragma unroll
            for (int kk = 0; kk < kSgKB; ++kk) {
                const int u = kk % PF;
                if (kk % 2 == 0) {
                    request((u + 2) % PF);
                    request((u + 3) % PF);
                }
                float gv[4];
                unpack_g4<T>(raw[u], gv);
                if constexpr (TAIL) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) gv[j] = k0 + kk < g.K ? gv[j] : 0.0f;
                }
                const float2 cf = BR == 0 ? *reinterpret_cast<const float2*>(st + lay.coef + kk * 8) : make_float2(1.0f, 1.0f);
                const QuadTaps<WIDE, K3 ? 10 : 8> taps(cq[u]);
                const QuadWeights<WIDE> wtaps(cq[u]);
                // one branch: the four pixels' accumulators are distinct, so their loads go out together
                auto branch = [&](bool is_min, float a) {
                    char* p[4];
                    float v[4], xv[4], wv[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) p[j] = Ab + (is_min ? taps.tmin(j) : taps.tmax(j));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if constexpr (GX) v[j] = *reinterpret_cast<const float*>(p[j] + j * RS * TS);
                        if constexpr (AB) {
                            xv[j] = *reinterpret_cast<const float*>(p[j] + (4 + j) * RS * TS);
                            wv[j] = load_shared((is_min ? wtaps.tmin(table, j) : wtaps.tmax(table + lay.w2, j)) + kk * RS * 4);
                        }
                    }
                    float sum = 0.0f;
                    if constexpr (GX) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) *reinterpret_cast<float*>(p[j] + j * RS * TS) = __fmaf_rn(a, gv[j], v[j]);
                    }
                    if constexpr (AB) {
                        float z[4];
                        branch_values(xv, wv, z, T());
#pragma unroll
                        for (int j = 0; j < 4; ++j) sum = __fmaf_rn(gv[j], z[j], sum);
                    }
                    return sum;
                };
                float sa = 0.0f, sb = 0.0f;
                if constexpr (BR != 2) sa = branch(true, cf.x);
                if constexpr (BR != 1) sb = branch(false, cf.y);
                if constexpr (AB) { s[2 * kk] = sa; s[2 * kk + 1] = sb; }
            }
            if constexpr (AB) {
                const float v = warp_sum16(s, lane);
                if (!(lane & 1)) part[buf][warp][lane >> 1] = v;
            }
            if (BR == 0 && more_k) {
                char* to = stage + (buf ^ 1) * lay.stride;
                if (tid < nstage) *reinterpret_cast<float*>(to + operand(tid).to) = ahead;
                copy(tid + blockDim.x, k0 + kSgKB, to);
            }
            if constexpr (BR == 0) __syncthreads();     // this stage is used, the next one and its sums are stored
            if constexpr (AB) {
                if (tid < 2 * kSgKB && 2 * k0 + tid < 2 * g.K) {
                    float t = 0.0f;
#pragma unroll
                    for (int i = 0; i < kSgThreads / 32; ++i) t += i < nwarps ? part[buf][i][tid] : 0.0f;
                    part_ab[((size_t)tile * g.C + c) * g.K * 2 + 2 * k0 + tid] = t;
                }
            }
        }
    }
    if constexpr (GX) {
        __syncthreads();
        // gather: an input element sums, over the taps, the accumulator of the output pixel that reads it
        // through that tap (lanes along the columns, one warp per input row).  An image in one tile: all
        // its inputs, straight to grad_x; else the region the tile reaches, as floats
        const float* A = reinterpret_cast<const float*>(smem);
        const int gfl = gbytes / 4;
        const bool whole = pl.nrow * pl.ncol == 1;
        const int rows = whole ? g.H : pl.ER, cols = whole ? g.W : pl.EC;
        const int up = whole ? g.ph : 0, left = whole ? g.pw : 0;      // row / column 0 of the walk in the tile's region
        float* region = part_gx + ((size_t)tile * g.C + c) * pl.ER * pl.EC;
        auto index = [&](int q, int j, int tap) { return (q / TP) * gfl + (j * RS + tap) * TP + q % TP; };
        auto store = [&](int il, int row, int col, float v) {
            if (whole) gx[(((size_t)(n_first + il) * g.C + c) * g.H + row) * g.W + col] = from_f32<T>(v);
            else region[(size_t)row * pl.EC + col] = v;
        };
        // (strides 1 and 2 divide by a shift)
        const int lh = g.sh <= 2 ? g.sh - 1 : -1, lw = g.sw <= 2 ? g.sw - 1 : -1;
        auto quot = [](int n, int stride, int shift) { return shift >= 0 ? n >> shift : n / stride; };
        for (int col = lane; col < cols; col += 32) {
            // output column that reads this one through tap column sx, or -1
            int at[KW ? KW : 1];
            auto column = [&](int sx) {
                const int nw = col + left - sx * g.dw, ow = quot(nw, g.sw, lw);
                return nw >= 0 && ow * g.sw == nw && ow < tq * 4 ? ow : -1;
            };
            if constexpr (KW != 0) {
#pragma unroll
                for (int sx = 0; sx < KW; ++sx) {
                    at[sx] = column(sx);
                    if (K3 && at[sx] >= 0) at[sx] = (at[sx] >> 2) + (at[sx] & 3) * RS * TP;   // its accumulator's index but for row and tap
                }
            }
            for (int rr = warp; rr < nimg * rows; rr += nwarps) {
                const int il = nimg == 1 ? 0 : rr / rows, row = rr - il * rows;
                float sum = 0.0f;
#pragma unroll
                for (int r = 0; r < WR; ++r) {
                    const int nh = row + up - r * g.dh, oh = quot(nh, g.sh, lh);
                    if (nh < 0 || oh * g.sh != nh || oh >= tr) continue;
                    const int qrow = il * NQ1 + oh * tq;
#pragma unroll
                    for (int sx = 0; sx < WS; ++sx) {
                        const int ow = KW ? at[KW ? sx : 0] : column(sx);
                        if constexpr (K3) {
                            if (ow >= 0) sum += A[qrow + ow + (r * WS + sx) * TP];
                        } else if (ow >= 0) sum += A[index(qrow + (ow >> 2), ow & 3, r * WS + sx)];
                    }
                }
                store(il, row, col, sum);
            }
        }
    }
}

// grad_x of an image cut into tiles: every input element adds the regions that cover it, tile rows and
// columns ascending.  grid (N * C, eight warps' tasks each; tall maps have more than the 65535 blocks of that axis).
// A warp takes four rows of 32 columns: the tiles that reach a column (two divisions) once for the four rows, the
// sums' loads together.  N=19 C=75 118x93 bf16 (85 MB) took 122 us with one thread and four divisions per element.
template <typename T>
__global__ void __launch_bounds__(256)
bwd_sum_edges_kernel(Geo g, const float* __restrict__ part_gx, T* __restrict__ gx, SumGxPlan pl) {
    constexpr int RPT = 4;
    const unsigned chunks = ((unsigned)g.W + 31) / 32;
    const unsigned n = blockIdx.x / (unsigned)g.C, c = blockIdx.x - n * (unsigned)g.C;
    const unsigned sr = pl.TR * g.sh, sc = pl.TQ * 4 * g.sw;     // input distance between two tiles
    const unsigned ER = pl.ER, EC = pl.EC, area = ER * EC;
    for (unsigned task = blockIdx.y * 8 + (threadIdx.x >> 5);; task += gridDim.y * 8) {
        const unsigned rg = task / chunks, xi = (task - rg * chunks) * 32 + (threadIdx.x & 31), y0 = rg * RPT;
        if (y0 >= (unsigned)g.H) break;
        if (xi >= (unsigned)g.W) continue;
        const unsigned x = xi + g.pw;
        const unsigned c1 = min((unsigned)pl.ncol - 1, x / sc);
        unsigned c0 = c1;
        while (c0 > 0 && x - (c0 - 1) * sc < EC) --c0;
        const bool covered = x - c1 * sc < EC;
        const float* base = part_gx + ((size_t)n * pl.nrow * pl.ncol * g.C + c) * area;
        const size_t tile = (size_t)g.C * area;
        T* out = gx + ((size_t)blockIdx.x * g.H + y0) * g.W + xi;
        // the last tile that covers each element first, all rows together; then the others, ascending
        unsigned r0[RPT], r1[RPT], at = min((unsigned)pl.nrow - 1, (y0 + g.ph) / sr);
        float sum[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const unsigned y = y0 + i + g.ph;
            while (at + 1 < (unsigned)pl.nrow && (at + 1) * sr <= y) ++at;
            r1[i] = r0[i] = at;
            while (r0[i] > 0 && y - (r0[i] - 1) * sr < ER) --r0[i];
            sum[i] = y - at * sr < ER && covered ? __ldg(base + (r1[i] * pl.ncol + c1) * tile + (y - r1[i] * sr) * EC + (x - c1 * sc)) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const unsigned y = y0 + i + g.ph;
            if (r0[i] == r1[i] && c0 == c1) {
                if (y0 + i < (unsigned)g.H) out[(size_t)i * g.W] = from_f32<T>(sum[i]);
                continue;
            }
            for (unsigned r = r0[i]; r <= r1[i]; ++r)
                for (unsigned q = c0; q <= c1; ++q)
                    if ((r != r1[i] || q != c1) && y - r * sr < ER && x - q * sc < EC)
                        sum[i] += __ldg(base + (r * pl.ncol + q) * tile + (y - r * sr) * EC + (x - q * sc));
            if (y0 + i < (unsigned)g.H) out[(size_t)i * g.W] = from_f32<T>(sum[i]);
        }
    }
}

// ---------------------------------------------------------------------------------- grad_w (and grad_bias)
// A warp owns one (k, c) pair and one share of its (image, quad) items.  Lane-private histograms,
// [bin][64] floats for two warps (bins 256 bytes apart: one PRMT turns a bin number into an offset).
// PAIRS: with both branches the bin is the pair (argmax tap, argmin tap), RS * RS bins, so one
// read-modify-write serves both; the finishing sums over rows / columns of the table give the two
// histograms.  Else one table per branch.
// FLAT: the share is a range of the flattened (image, quad) space; else an image is whole rounds of 32 quads.
// BLOCKS (not FLAT): an image is a multiple of four rounds, whose operands lie at constant distances.
// Bound by the shared-memory path (two accesses of the table per item beside the streamed operands) and the issue
// slots, so what is left out is address arithmetic.  Against one address per round with a test for the end of the
// image, and (FLAT) a test for the end of the share in every round: N=128 C=64 K=64 32x32 fp32 compound 320 -> 268 us,
// 8 x 256 x 256 channels 128x256 bf16 7704 -> 6977 us; FLAT: 28 x 28 x 128 bf16 parallel 487 -> 430 us, 7 x 7 x 512
// bf16 compound 831 -> 707 us, 56 -> 28 fp32 parallel 271 -> 255 us.
template <typename T, int BR, bool PAIRS, bool WIDE, bool FLAT, bool BLOCKS>
__global__ void __launch_bounds__(128)
bwd_sum_gw_kernel(Geo g, const T* __restrict__ gy, const uint8_t* __restrict__ codes, float* __restrict__ part, SumGwPlan pl) {
    extern __shared__ float tabs[];
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // (uniform: addresses below)
    const long wid = (long)blockIdx.x * 4 + warp;
    const int pairs = g.K * g.C;
    if (wid >= (long)pairs * pl.splits) return;
    const int split = (int)(wid / pairs), pair = (int)(wid - (long)split * pairs);
    const int k = pair / g.C, c = pair - k * g.C;
    float* tab = tabs + (size_t)(warp >> 1) * pl.nbins * 64 + (warp & 1) * 32;
    // (32-bit shared-memory addresses: 449 -> 430 us on 28 x 28 bf16 parallel against generic pointers)
    const unsigned mine = (unsigned)__cvta_generic_to_shared(tab + lane);
    const unsigned mine_max = mine + (BR == 0 ? g.RS * 256 : 0);      // (one table per branch)
    for (int b = 0; b < pl.nbins; ++b) tab[b * 64 + lane] = 0.0f;
    constexpr int CW = WIDE ? 2 : 1;
    const int NQ = g.OH * (g.OW >> 2);
    const size_t plane = (size_t)g.OH * g.OW, gstep = (size_t)g.K * plane, cstep = gstep * g.C * CW;
    const unsigned skip = 16u - (unsigned)g.RS;
    auto add_two = [&](unsigned p0, unsigned p1, float g0, float g1) {
        // both loads first; where the two bins are one, the second store holds both gradients
        const float v0 = at_shared(p0), v1 = at_shared(p1);
        const float t0 = v0 + g0;
        const float t1 = (p0 == p1 ? t0 : v1) + g1;
        at_shared(p0) = t0;
        at_shared(p1) = t1;
    };
    auto add_quad = [&](const float* gv, const Codes4<WIDE>& code) {
        if constexpr (PAIRS) {
            // four bins, one per byte (no borrow crosses a byte: each is at least skip * high nibble)
            const unsigned top = (code.lo >> 4) & 0x0f0f0f0fu, bins = code.lo - skip * top;
            auto at = [&](int j) { return mine + __byte_perm(bins, 0u, 0x4404u + (unsigned)(j << 4)); };
            add_two(at(0), at(1), gv[0], gv[1]);
            add_two(at(2), at(3), gv[2], gv[3]);
        } else {
            const BinAddress<WIDE> bin(code);
            if constexpr (BR != 2) {
                add_two(bin.tmin(mine, 0), bin.tmin(mine, 1), gv[0], gv[1]);
                add_two(bin.tmin(mine, 2), bin.tmin(mine, 3), gv[2], gv[3]);
            }
            if constexpr (BR != 1) {
                add_two(bin.tmax(mine_max, 0), bin.tmax(mine_max, 1), gv[0], gv[1]);
                add_two(bin.tmax(mine_max, 2), bin.tmax(mine_max, 3), gv[2], gv[3]);
            }
        }
    };
    // FLAT: the operands of HB rounds are requested together, while the HB rounds before them are added (the
    // loads of such a batch share a scoreboard: 290 against 270 us on the 28 x 28 transition layer); whole
    // rounds: one at a time, PF ahead
    constexpr int HB = FLAT && !PAIRS ? 2 : 4, PF = 2 * HB;
    float raw[PF][sizeof(T)];
    Codes4<WIDE> cq[PF];
    if constexpr (FLAT) {
        const int lo = split * pl.per, hi = min(g.N * NQ, lo + pl.per);
        int it = lo + lane;
        // lanes past the end read the share's last quad again; its gradient is dropped
        const int first = min(it, hi - 1);
        int n = first / NQ, q = first - n * NQ;
        const T* gp = gy + ((size_t)n * g.K + k) * plane + 4 * q;
        const uint8_t* cp = codes + ((((size_t)n * g.K + k) * g.C + c) * plane + 4 * q) * CW;
        const int dn = 32 / NQ, dq = 32 - dn * NQ;
        const size_t gadv = dn * gstep + 4 * dq, cadv = dn * cstep + 4 * dq * CW;
        const size_t gwrap = gstep - plane, cwrap = cstep - plane * CW;
        auto request = [&](int u, bool advance) {
            ahead_g4<T, true>(gp, raw[u]);
            cq[u] = ahead_codes4<WIDE, true>(cp);
            if (advance) {
                q += dq;
                gp += gadv;
                cp += cadv;
                if (q >= NQ) { q -= NQ; gp += gwrap; cp += cwrap; }
            }
        };
        auto request_to_end = [&](int u) {
            it += 32;
            request(u, it < hi);
        };
#pragma unroll
        for (int u = 0; u < HB; ++u) request_to_end(u);
        const int rounds = (hi - lo + 31) / 32, full = (hi - lo) / 32;
        int r0 = 0;
        // while all that is requested and the round behind it are whole rounds
        for (; r0 + PF + HB < full; r0 += PF, it += 32 * PF) {
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                if (u % HB == 0) {
#pragma unroll
                    for (int v = 0; v < HB; ++v) request((u + HB + v) % PF, true);
                }
                float gv[4];
                unpack_g4<T>(raw[u], gv);
                add_quad(gv, cq[u]);
            }
        }
        for (; r0 < rounds; r0 += PF) {
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                if (u % HB == 0) {
#pragma unroll
                    for (int v = 0; v < HB; ++v) request_to_end((u + HB + v) % PF);
                }
                float gv[4];
                unpack_g4<T>(raw[u], gv);
                if (lo + (r0 + u + 1) * 32 > hi) {      // the last round, or a round past it
                    const bool in = lo + (r0 + u) * 32 + lane < hi;
#pragma unroll
                    for (int j = 0; j < 4; ++j) gv[j] = in ? gv[j] : 0.0f;
                }
                add_quad(gv, cq[u]);
            }
        }
    } else if constexpr (BLOCKS) {
        const int bpi = NQ / 128;                        // blocks of an image; shares are whole blocks
        const int lo = split * (pl.per / 4), hi = min(g.N * bpi, lo + pl.per / 4);
        const int n0 = lo / bpi;
        int left = bpi - (lo - n0 * bpi), more = hi - lo;      // blocks left in the image, in the share
        const size_t off = (size_t)((lo - n0 * bpi) * 128 + lane) * 4;
        const T* gp = gy + ((size_t)n0 * g.K + k) * plane + off;
        const uint8_t* cp = codes + ((((size_t)n0 * g.K + k) * g.C + c) * plane + off) * CW;
        const size_t gwrap = gstep - plane, cwrap = cstep - plane * CW;
        auto request = [&](int u0) {                     // (past the share its last block is read again)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                ahead_g4<T, true>(gp + v * 128, raw[u0 + v]);
                cq[u0 + v] = ahead_codes4<WIDE, true>(cp + v * 128 * CW);
            }
            if (--more > 0) {
                gp += 512;
                cp += 512 * CW;
                if (--left == 0) {
                    left = bpi;
                    gp += gwrap;
                    cp += cwrap;
                }
            }
        };
        request(0);
        for (int i = lo; i < hi; i += 2) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half && i + 1 >= hi) break;
                request(half ? 0 : 4);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float gv[4];
                    unpack_g4<T>(raw[4 * half + v], gv);
                    add_quad(gv, cq[4 * half + v]);
                }
            }
        }
    } else {
        const int rpi = NQ / 32;
        const int lo = split * pl.per, hi = min(g.N * rpi, lo + pl.per);
        const int n0 = lo / rpi;
        int rr = lo - n0 * rpi, left = hi - lo - 1;      // round of its image to request next, rounds behind it
        const T* gp = gy + ((size_t)n0 * g.K + k) * plane;
        const uint8_t* cp = codes + (((size_t)n0 * g.K + k) * g.C + c) * plane * CW;
        auto request = [&](int u) {                      // (past the share its last round is read again)
            const unsigned off = (unsigned)(rr * 32 + lane) * 4u;
            ahead_g4<T, true>(gp + off, raw[u]);
            cq[u] = ahead_codes4<WIDE, true>(cp + off * CW);
            if (left > 0 && ++rr == rpi) {
                rr = 0;
                gp += gstep;
                cp += cstep;
            }
            --left;
        };
#pragma unroll
        for (int u = 0; u < PF; ++u) request(u);
        int i = lo;
        for (; i + PF <= hi; i += PF) {
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                float gv[4];
                unpack_g4<T>(raw[u], gv);
                add_quad(gv, cq[u]);
                request(u);
            }
        }
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            if (i + u >= hi) break;
            float gv[4];
            unpack_g4<T>(raw[u], gv);
            add_quad(gv, cq[u]);
        }
    }
    __syncwarp();
    // bin totals: lane l sums the bins l, l + 32, ..., starting at its own column (no bank conflicts)
    for (int b = lane; b < pl.nbins; b += 32) {
        float s = 0.0f;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) s += tab[b * 64 + ((i + lane) & 31)];
        tab[b * 64 + lane] = s;      // (column b % 32 of its own row: read by this lane only)
    }
    __syncwarp();
    auto total = [&](int b) { return tab[b * 64 + (b & 31)]; };
    float* o = part + ((size_t)split * pairs + pair) * 2 * g.RS;
    for (int t = lane; t < g.RS; t += 32) {
        float smin = 0.0f, smax = 0.0f;
        if constexpr (PAIRS) {
            for (int i = 0; i < g.RS; ++i) { smin += total(i * g.RS + t); smax += total(t * g.RS + i); }
        } else {
            smin = total(t);
            smax = BR == 0 ? total(g.RS + t) : smin;
        }
        o[t] = smin;
        o[g.RS + t] = smax;
    }
}

// ---------------------------------------------------------------------------------- finish
// Blocks [0, nb_w): grad_w / grad_w2, 256 / ws (k, c, tap) entries per block; ws slices share the splits and are
// added in slice order.  The next nb_ab blocks: grad_alpha / grad_beta, 256 / AS (c, k) entries per block; AS slices
// share the partial rows and are added in slice order.  The rest: grad_bias, a warp per output channel (the sum of a
// pair's histogram is the sum of grad_y), its lanes added in a fixed tree.  All sums are chains of loads from L2, kept eight
// deep in flight: N=92 C=3 K=12 23x33 5x5 took 42 us where one thread per channel summed splits x taps values.  Short
// blocks, so eight on an SM: 46 registers leave five.  3 -> 36 channels 1 x 15623 N=64 (7872 rows), 400 -> 197 64x45 5x5 N=3
// (24), 512 x 512 7x7 N=64 (4 rows, one slice): five blocks, an unrolled loop and what eights leave one by one 42, 32 and 55
// us; a variable number of slices and 32 registers 81, 25 and 24; constant slices, the rest in twos, 32 registers 30, 23, 24.
template <int AS>
__global__ void __launch_bounds__(256, 8)
bwd_sum_finish_kernel(Geo g, int br, int splits, const float* __restrict__ part, int rows, const float* __restrict__ part_ab,
                      const float* __restrict__ alpha, const float* __restrict__ beta, float* __restrict__ gw, float* __restrict__ gw2,
                      float* __restrict__ galpha, float* __restrict__ gbeta, float* __restrict__ gbias, unsigned nb_w,
                      unsigned nb_ab, int ws) {
    const size_t pairs = (size_t)g.K * g.C, len = pairs * 2 * g.RS;
    __shared__ float2 red[256];
    if (blockIdx.x < nb_w) {
        const int epb = 256 / ws, el = threadIdx.x % epb, sl = threadIdx.x / epb;
        const size_t i = (size_t)blockIdx.x * epb + el;
        const bool on = i < pairs * g.RS;
        const size_t pair = on ? i / g.RS : 0;
        const int t = on ? (int)(i - pair * g.RS) : 0;
        const float* p = part + pair * 2 * g.RS + t;
        float smin = 0.0f, smax = 0.0f;
#pragma unroll 8
        for (int s = sl; s < splits; s += ws) { smin += __ldg(p + s * len); smax += __ldg(p + s * len + g.RS); }
        if (ws > 1) {
            red[threadIdx.x] = make_float2(smin, smax);
            __syncthreads();
            for (int s = 1; s < ws && sl == 0; ++s) { smin += red[s * epb + el].x; smax += red[s * epb + el].y; }
        }
        if (!on || sl != 0) return;
        if (br == 0) {
            const float a = alpha ? alpha[pair] : 1.0f, b = beta ? beta[pair] : 1.0f;
            if (g.mode == TCONV_COMPOUND) {
                if (gw) gw[i] = __fmaf_rn(a, smin, b * smax);
            } else {
                if (gw) gw[i] = a * smin;
                if (gw2) gw2[i] = b * smax;
            }
        } else if (gw) {
            gw[i] = smin;
        }
        return;
    }
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    if (blockIdx.x >= nb_w + nb_ab) {
        const size_t k = (size_t)(blockIdx.x - nb_w - nb_ab) * 8 + slice;
        if (k >= (size_t)g.K) return;
        const float* p = part + k * g.C * 2 * g.RS;
        const unsigned items = (unsigned)splits * g.RS;
        float s = 0.0f;
#pragma unroll 8
        for (unsigned i = lane; i < items; i += 32) s += __ldg(p + i / (unsigned)g.RS * len + i % (unsigned)g.RS);
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) gbias[k] = s;
        return;
    }
    constexpr int EPB = 256 / AS;
    const int el = threadIdx.x % EPB, sl = threadIdx.x / EPB;
    const size_t e = (size_t)(blockIdx.x - nb_w) * EPB + el;      // c * K + k
    const size_t c = e / g.K, k = e - c * g.K;
    float2 s = make_float2(0.0f, 0.0f);
    if (e < pairs) {
        const float2* at = reinterpret_cast<const float2*>(part_ab) + sl * pairs + e;
        s = sum_in_order<8, float2>((rows - sl + AS - 1) / AS, [&](int i) { return __ldg(at + (size_t)i * AS * pairs); });
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (sl == 0 && e < pairs) {
        for (int i = 1; i < AS; ++i) { s.x += red[i * EPB + el].x; s.y += red[i * EPB + el].y; }
        if (galpha) galpha[k * g.C + c] = s.x;
        if (gbeta) gbeta[k * g.C + c] = s.y;
    }
}

// Arguments of one backward call (host side).
struct SumBwdArgs {
    Geo g;             // widened to whole quads (OW a multiple of 4)
    int dtype;
    const void *x, *w, *w2;
    const float *alpha, *beta;
    const void* gy;    // rows of g.OW elements
    const uint8_t* codes;
    void* gx;
    float *gw, *gw2, *galpha, *gbeta, *gbias;
    float* ws;         // sum_ws_bytes()
    cudaStream_t st;
    int launches;      // out
};
int bwd_sum_launch(SumBwdArgs& a);

}  // namespace tconv
