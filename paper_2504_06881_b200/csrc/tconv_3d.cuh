// Three-dimensional tropical convolution (Section 3.2 and the Conv3d forms of Sections 3.4, 3.5).
// The paper's 3-D workloads are LeNet-sized (one to sixteen channels, 5 x 5 x 5 windows on 28^3 and
// 64^3 volumes): a window has many taps and few channels, so one thread owns one output position
// for a few output channels, the weights of a channel chunk sit in shared memory and the input is
// read through L1 (neighbouring threads read neighbouring elements).  All kernels are
// deterministic and atomic-free.
#pragma once
#include "tconv_common.cuh"

namespace tconv {

struct Geo3 {
    int N, C, D, H, W, K, T, R, S;
    int sd, sh, sw, pd, ph, pw, dd, dh, dw;
    int OD, OH, OW, taps, vol;  // vol = OD*OH*OW
    int mode, chan;
};

constexpr int kFwd3Threads = 128;

// Forward.  grid (ceil(N * vol / 128), ceil(K / KT)): one thread per (n, output position) of the
// flattened range, KT output channels each.  Shared memory: weights of `cch` input channels for
// this block's KT output channels, [cc][tap][KT] (twice in parallel mode), as T.
// WIN: track the winning taps (strict compares, taps ascending); without it the extrema are plain
// min / max.  SC: the window's innermost extent S when it is 3 or 5 (unrolled), else 0.
template <typename T, int KT, bool WIN, int SC>
__global__ void __launch_bounds__(kFwd3Threads)
fwd3d_kernel(Geo3 g, int cch, const T* __restrict__ x, const T* __restrict__ w, const T* __restrict__ w2,
             const float* __restrict__ alpha, const float* __restrict__ beta,
             const float* __restrict__ bias, T* __restrict__ y, void* __restrict__ winners) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* wmin_s = reinterpret_cast<T*>(smem_raw);
    const bool par = g.mode == TCONV_PARALLEL;
    const bool twob = two_branch(g.mode);
    T* wmax_s = par ? wmin_s + (size_t)cch * g.taps * KT : wmin_s;
    const long long flat = (long long)blockIdx.x * kFwd3Threads + threadIdx.x;
    const bool live = flat < (long long)g.N * g.vol;
    const int n = live ? (int)(flat / g.vol) : 0, pos = live ? (int)(flat % g.vol) : 0;
    const int k0 = blockIdx.y * KT;
    const int ow = pos % g.OW, oh = (pos / g.OW) % g.OH, od = pos / (g.OW * g.OH);
    const int d0 = od * g.sd - g.pd, h0 = oh * g.sh - g.ph, w0 = ow * g.sw - g.pw;
    const int S = SC ? SC : g.S;
    float acc[KT], best[KT];
    int win[KT];
#pragma unroll
    for (int j = 0; j < KT; ++j) {
        acc[j] = 0.0f;
        best[j] = (g.chan == CH_MAX) ? -INFINITY : INFINITY;
        win[j] = -1;
    }
    for (int c0 = 0; c0 < g.C; c0 += cch) {
        const int ncc = min(cch, g.C - c0);
        __syncthreads();
        for (int i = threadIdx.x; i < ncc * g.taps * KT; i += kFwd3Threads) {
            const int j = i % KT, tap = (i / KT) % g.taps, cc = i / (KT * g.taps);
            const int k = k0 + j;
            const size_t wi = ((size_t)k * g.C + c0 + cc) * g.taps + tap;
            wmin_s[i] = k < g.K ? w[wi] : zero_of<T>();
            if (par) wmax_s[i] = k < g.K ? w2[wi] : zero_of<T>();
        }
        __syncthreads();
        if (!live) continue;
        for (int cc = 0; cc < ncc; ++cc) {
            const int c = c0 + cc;
            const T* xc = x + ((size_t)n * g.C + c) * g.D * g.H * g.W;
            const T* wa = wmin_s + (size_t)cc * g.taps * KT;
            const T* wb = wmax_s + (size_t)cc * g.taps * KT;
            float mn[KT], mx[KT];
            int amn[KT], amx[KT];
#pragma unroll
            for (int j = 0; j < KT; ++j) {
                mn[j] = INFINITY; mx[j] = -INFINITY; amn[j] = 0; amx[j] = 0;
            }
            int tap = 0;
            for (int t = 0; t < g.T; ++t) {
                const int id = d0 + t * g.dd;
                const bool okd = id >= 0 && id < g.D;
                for (int r = 0; r < g.R; ++r) {
                    const int ih = h0 + r * g.dh;
                    const bool okh = okd && ih >= 0 && ih < g.H;
                    const T* xrow = xc + ((size_t)(okh ? id : 0) * g.H + (okh ? ih : 0)) * g.W;
                    if constexpr (SC != 0) {
                        T xv[SC];
#pragma unroll
                        for (int s = 0; s < SC; ++s) {
                            const int iw = w0 + s * g.dw;
                            xv[s] = (okh && iw >= 0 && iw < g.W) ? xrow[iw] : zero_of<T>();
                        }
#pragma unroll
                        for (int s = 0; s < SC; ++s) {
#pragma unroll
                            for (int j = 0; j < KT; ++j) {
                                const float tmn = tap_add(xv[s], wa[(tap + s) * KT + j]);
                                const float tmx = par ? tap_add(xv[s], wb[(tap + s) * KT + j]) : tmn;
                                if constexpr (WIN) {
                                    if (tmn < mn[j]) { mn[j] = tmn; amn[j] = tap + s; }
                                    if (tmx > mx[j]) { mx[j] = tmx; amx[j] = tap + s; }
                                } else {
                                    mn[j] = fminf(mn[j], tmn);
                                    mx[j] = fmaxf(mx[j], tmx);
                                }
                            }
                        }
                        tap += SC;
                    } else {
                        for (int s = 0; s < S; ++s, ++tap) {
                            const int iw = w0 + s * g.dw;
                            T xv = zero_of<T>();
                            if (okh && iw >= 0 && iw < g.W) xv = xrow[iw];
#pragma unroll
                            for (int j = 0; j < KT; ++j) {
                                const float tmn = tap_add(xv, wa[tap * KT + j]);
                                const float tmx = par ? tap_add(xv, wb[tap * KT + j]) : tmn;
                                if constexpr (WIN) {
                                    if (tmn < mn[j]) { mn[j] = tmn; amn[j] = tap; }
                                    if (tmx > mx[j]) { mx[j] = tmx; amx[j] = tap; }
                                } else {
                                    mn[j] = fminf(mn[j], tmn);
                                    mx[j] = fmaxf(mx[j], tmx);
                                }
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < KT; ++j) {
                const int k = k0 + j;
                if (k >= g.K) continue;
                if (twob) {
                    const float a = alpha ? alpha[(size_t)k * g.C + c] : 1.0f;
                    const float b = beta ? beta[(size_t)k * g.C + c] : 1.0f;
                    acc[j] = __fmaf_rn(a, mn[j], acc[j]);
                    acc[j] = __fmaf_rn(b, mx[j], acc[j]);
                } else {
                    const bool is_min = g.mode == TCONV_MIN_PLUS;
                    const float m = is_min ? mn[j] : mx[j];
                    const int am = is_min ? amn[j] : amx[j];
                    if (g.chan == CH_SUM) acc[j] = __fadd_rn(acc[j], m);
                    else if (g.chan == CH_MAX) { if (m > best[j]) { best[j] = m; win[j] = c * g.taps + am; } }
                    else { if (m < best[j]) { best[j] = m; win[j] = c * g.taps + am; } }
                    if (is_min) amx[j] = 0; else amn[j] = 0;
                }
                if (WIN && g.chan == CH_SUM)
                    ((uint16_t*)winners)[(((size_t)n * g.K + k) * g.C + c) * g.vol + pos] =
                        (uint16_t)(amn[j] | (amx[j] << 8));
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int j = 0; j < KT; ++j) {
        const int k = k0 + j;
        if (k >= g.K) continue;
        float out = (g.chan == CH_SUM) ? acc[j] : best[j];
        if (bias) out = __fadd_rn(out, bias[k]);
        const size_t o = ((size_t)n * g.K + k) * g.vol + pos;
        if (y) y[o] = from_f32<T>(out);
        if (WIN && g.chan != CH_SUM) ((int32_t*)winners)[o] = win[j];
    }
}

// Forward for layers with too few (position, output channel) pairs to fill the GPU (a LeNet layer on 28^3
// volumes has 1024 of them): a block owns PX positions x KT output channels and splits the taps of a group of
// input channels over `parts` threads per position, one (channel, window plane) each; after every group the
// block folds the planes of a channel and adds the channels in ascending order, one thread per (position,
// output channel), so that the results are those of fwd3d_kernel.  256 threads = PX * parts.  Shared memory:
// weights of the group [cc][tap][KT] (twice in parallel mode), then the partial extrema [part][KT][PX] (min,
// max, and with winners both taps in 16 bits).  ts: planes per channel (1 or T), cg: channels per group.
template <typename T, int KT, bool WIN, int SC>
__global__ void __launch_bounds__(256)
fwd3d_split_kernel(Geo3 g, int PX, int ts, int cg, const T* __restrict__ x, const T* __restrict__ w,
                   const T* __restrict__ w2, const float* __restrict__ alpha, const float* __restrict__ beta,
                   const float* __restrict__ bias, T* __restrict__ y, void* __restrict__ winners) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const bool par = g.mode == TCONV_PARALLEL, twob = two_branch(g.mode);
    T* wmin_s = reinterpret_cast<T*>(smem_raw);
    T* wmax_s = par ? wmin_s + (size_t)cg * g.taps * KT : wmin_s;
    const int nparts = cg * ts;
    float* pmn = reinterpret_cast<float*>(smem_raw + (((size_t)cg * g.taps * KT * (par ? 2 : 1) * sizeof(T) + 15) & ~(size_t)15));
    float* pmx = pmn + nparts * KT * PX;
    uint16_t* pcode = reinterpret_cast<uint16_t*>(pmx + nparts * KT * PX);
    const int tid = threadIdx.x, px = tid % PX, part = tid / PX;
    const int pc = part / ts, pt = part - pc * ts;             // this thread's channel of the group, window plane
    const int k0 = blockIdx.y * KT;
    const long long flat0 = (long long)blockIdx.x * PX, total = (long long)g.N * g.vol;
    const long long flat = min(flat0 + px, total - 1);
    const int n = (int)(flat / g.vol), pos = (int)(flat % g.vol);
    const int ow = pos % g.OW, oh = (pos / g.OW) % g.OH, od = pos / (g.OW * g.OH);
    const int d0 = od * g.sd - g.pd, h0 = oh * g.sh - g.ph, w0 = ow * g.sw - g.pw;
    const int S = SC ? SC : g.S, RS = g.R * g.S;
    // folding thread: (output channel, position) of the block
    const int fj = tid / PX, fk = k0 + fj;
    const bool folds = tid < KT * PX && flat0 + px < total && fk < g.K;
    float acc = g.chan == CH_SUM ? 0.0f : (g.chan == CH_MAX ? -INFINITY : INFINITY);
    int win = -1;
    for (int c0 = 0; c0 < g.C; c0 += cg) {
        const int ncc = min(cg, g.C - c0);
        // (the folding threads are done with the previous group before its partials are overwritten: second barrier)
        for (int i = tid; i < ncc * g.taps * KT; i += 256) {
            // along the taps of one (channel, output channel): contiguous weights
            const int tap = i % g.taps, j = (i / g.taps) % KT, cc = i / (KT * g.taps), k = k0 + j;
            const size_t wi = ((size_t)k * g.C + c0 + cc) * g.taps + tap;
            wmin_s[(cc * g.taps + tap) * KT + j] = k < g.K ? w[wi] : zero_of<T>();
            if (par) wmax_s[(cc * g.taps + tap) * KT + j] = k < g.K ? w2[wi] : zero_of<T>();
        }
        __syncthreads();
        if (pc < ncc) {
            float mn[KT], mx[KT];
            int amn[KT], amx[KT];
#pragma unroll
            for (int j = 0; j < KT; ++j) { mn[j] = INFINITY; mx[j] = -INFINITY; amn[j] = amx[j] = 0; }
            const T* xc = x + ((size_t)n * g.C + c0 + pc) * g.D * g.H * g.W;
            const T* wa = wmin_s + (size_t)pc * g.taps * KT;
            const T* wb = wmax_s + (size_t)pc * g.taps * KT;
            const int t_end = ts == 1 ? g.T : pt + 1;
            for (int t = pt; t < t_end; ++t) {
                const int id = d0 + t * g.dd;
                const bool okd = id >= 0 && id < g.D;
                for (int r = 0; r < g.R; ++r) {
                    const int ih = h0 + r * g.dh;
                    const bool okh = okd && ih >= 0 && ih < g.H;
                    const T* xrow = xc + ((size_t)(okh ? id : 0) * g.H + (okh ? ih : 0)) * g.W;
                    const int tap0 = t * RS + r * S;
                    auto fold = [&](T xv, int tap) {
#pragma unroll
                        for (int j = 0; j < KT; ++j) {
                            const float tmn = tap_add(xv, wa[tap * KT + j]);
                            const float tmx = par ? tap_add(xv, wb[tap * KT + j]) : tmn;
                            if constexpr (WIN) {
                                if (tmn < mn[j]) { mn[j] = tmn; amn[j] = tap; }
                                if (tmx > mx[j]) { mx[j] = tmx; amx[j] = tap; }
                            } else {
                                mn[j] = fminf(mn[j], tmn);
                                mx[j] = fmaxf(mx[j], tmx);
                            }
                        }
                    };
                    if constexpr (SC != 0) {
                        T xv[SC];
#pragma unroll
                        for (int s = 0; s < SC; ++s) {
                            const int iw = w0 + s * g.dw;
                            xv[s] = (okh && iw >= 0 && iw < g.W) ? xrow[iw] : zero_of<T>();
                        }
#pragma unroll
                        for (int s = 0; s < SC; ++s) fold(xv[s], tap0 + s);
                    } else {
                        for (int s = 0; s < S; ++s) {
                            const int iw = w0 + s * g.dw;
                            fold((okh && iw >= 0 && iw < g.W) ? xrow[iw] : zero_of<T>(), tap0 + s);
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < KT; ++j) {
                const int o = (part * KT + j) * PX + px;
                pmn[o] = mn[j];
                pmx[o] = mx[j];
                if constexpr (WIN) pcode[o] = (uint16_t)(amn[j] | (amx[j] << 8));
            }
        }
        __syncthreads();
        if (folds) {
            for (int cc = 0; cc < ncc; ++cc) {
                const int c = c0 + cc;
                float mn = INFINITY, mx = -INFINITY;
                unsigned amn = 0, amx = 0;
                for (int z = 0; z < ts; ++z) {          // planes ascending: the lowest winning tap stays
                    const int o = ((cc * ts + z) * KT + fj) * PX + px;
                    const float a = pmn[o], b = pmx[o];
                    if constexpr (WIN) {
                        const unsigned cd = pcode[o];
                        if (a < mn) { mn = a; amn = cd & 0xFFu; }
                        if (b > mx) { mx = b; amx = cd >> 8; }
                    } else {
                        mn = fminf(mn, a);
                        mx = fmaxf(mx, b);
                    }
                }
                if (twob) {
                    acc = __fmaf_rn(alpha ? alpha[(size_t)fk * g.C + c] : 1.0f, mn, acc);
                    acc = __fmaf_rn(beta ? beta[(size_t)fk * g.C + c] : 1.0f, mx, acc);
                } else {
                    const bool is_min = g.mode == TCONV_MIN_PLUS;
                    const float m = is_min ? mn : mx;
                    const int am = (int)(is_min ? amn : amx);
                    if (g.chan == CH_SUM) acc = __fadd_rn(acc, m);
                    else if (g.chan == CH_MAX ? m > acc : m < acc) { acc = m; win = c * g.taps + am; }
                    if (is_min) amx = 0; else amn = 0;
                }
                if (WIN && g.chan == CH_SUM)
                    ((uint16_t*)winners)[(((size_t)n * g.K + fk) * g.C + c) * g.vol + pos] = (uint16_t)(amn | (amx << 8));
            }
        }
    }
    if (!folds) return;
    float out = acc;
    if (bias) out = __fadd_rn(out, bias[fk]);
    const size_t o = ((size_t)n * g.K + fk) * g.vol + pos;
    if (y) y[o] = from_f32<T>(out);
    if (WIN && g.chan != CH_SUM) ((int32_t*)winners)[o] = win;
}

// Taps t of one axis through which an output reads input index i: i + pad - t * dil = stride * o with
// 0 <= o < out.  The walk visits exactly those when dil is 1 (step = stride), else it tests every tap.
struct TapRange {
    int first, end, step;
};
__device__ __forceinline__ TapRange tap_range(int i, int pad, int dil, int stride, int taps, int out) {
    TapRange r;
    if (dil != 1) { r.first = 0; r.end = taps; r.step = 1; return r; }
    const int u = i + pad, last = (out - 1) * stride;
    r.first = u > last ? u - last : u % stride;      // (last is a multiple of the stride)
    r.end = min(taps, u + 1);
    r.step = stride;
    return r;
}

// grad_x in gather form.  A block of 256 threads owns 256 / slices consecutive input elements (threadIdx.x)
// and splits the output channels over blockDim.y = 1, 2, 4 or 8 slices (k = slice, slice + slices, ...): each
// thread visits, taps ascending and its channels ascending inside a tap, the outputs whose window reads its
// element; the slices' partial sums are then added in slice order.  (Small 3-D layers have few input elements:
// the slices keep enough warps in flight to hide the dependent loads.)  Four channels' winners are requested
// together; a gradient is only read where one of them is the tap.
// One instance per code form, five blocks per SM (48 registers): N=2 C=6 K=14 25^3 5^3 took 814 us with the form
// decided in the loop at 64 registers, four blocks.
constexpr int kGx3Slices = 8;

template <typename T, bool CODES, bool TWO>
__global__ void __launch_bounds__(32 * kGx3Slices, 5)
bwd3d_gx_kernel(Geo3 g, const float* __restrict__ alpha, const float* __restrict__ beta,
                const T* __restrict__ gy, const void* __restrict__ winners, T* __restrict__ gx) {
    __shared__ float part[32 * kGx3Slices];
    const size_t total = (size_t)g.N * g.C * g.D * g.H * g.W;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int slice = threadIdx.y, slices = blockDim.y;
    const bool live = i < total;
    // TWO: two branches; else the codes of a single branch or the winner index decide
    const bool is_max = g.mode == TCONV_MAX_PLUS;
    float acc = 0.0f;
    if (live) {
        const unsigned ui = (unsigned)i;                    // (every tensor has fewer than 2^31 elements)
        const int iw = (int)(ui % (unsigned)g.W);
        const unsigned t1 = ui / (unsigned)g.W;
        const int ih = (int)(t1 % (unsigned)g.H);
        const unsigned t2 = t1 / (unsigned)g.H;
        const int id = (int)(t2 % (unsigned)g.D);
        const unsigned nc = t2 / (unsigned)g.D;
        const int c = (int)(nc % (unsigned)g.C), n = (int)(nc / (unsigned)g.C);
        const uint16_t* cbase = (const uint16_t*)winners + ((size_t)n * g.K * g.C + c) * g.vol;
        const int32_t* ibase = (const int32_t*)winners + (size_t)n * g.K * g.vol;
        const T* gbase = gy + (size_t)n * g.K * g.vol;
        const int cstep = g.C * g.vol;
        const TapRange rd = tap_range(id, g.pd, g.dd, g.sd, g.T, g.OD), rh = tap_range(ih, g.ph, g.dh, g.sh, g.R, g.OH),
                       rw = tap_range(iw, g.pw, g.dw, g.sw, g.S, g.OW);
        for (int t = rd.first; t < rd.end; t += rd.step) {
            const int nd = id + g.pd - t * g.dd, od = nd / g.sd;
            if (nd < 0 || od * g.sd != nd || od >= g.OD) continue;
            for (int r = rh.first; r < rh.end; r += rh.step) {
                const int nh = ih + g.ph - r * g.dh, oh = nh / g.sh;
                if (nh < 0 || oh * g.sh != nh || oh >= g.OH) continue;
                for (int s = rw.first; s < rw.end; s += rw.step) {
                    const int nw = iw + g.pw - s * g.dw, ow = nw / g.sw;
                    if (nw < 0 || ow * g.sw != nw || ow >= g.OW) continue;
                    const unsigned tap = (unsigned)((t * g.R + r) * g.S + s);
                    const int pos = (od * g.OH + oh) * g.OW + ow;
                    const unsigned want = (unsigned)(c * g.taps) + tap;
                    auto take = [&](int k, unsigned v) {        // v: the winner code(s) of output channel k
                        if constexpr (TWO) {
                            const bool hmin = (v & 0xFFu) == tap, hmax = (v >> 8) == tap;
                            if (!(hmin || hmax)) return;
                            const float gv = to_f32(__ldg(gbase + (k * g.vol + pos)));
                            if (hmin) acc = __fmaf_rn(alpha ? alpha[k * g.C + c] : 1.0f, gv, acc);
                            if (hmax) acc = __fmaf_rn(beta ? beta[k * g.C + c] : 1.0f, gv, acc);
                        } else {
                            const unsigned mine = !CODES ? v : is_max ? v >> 8 : v & 0xFFu;
                            if (mine == (CODES ? tap : want)) acc += to_f32(__ldg(gbase + (k * g.vol + pos)));
                        }
                    };
                    auto code = [&](int k) { return CODES ? (unsigned)__ldg(cbase + (k * cstep + pos)) : (unsigned)__ldg(ibase + (k * g.vol + pos)); };
                    int k = slice;
                    for (; k + 3 * slices < g.K; k += 4 * slices) {
                        unsigned v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] = code(k + u * slices);
#pragma unroll
                        for (int u = 0; u < 4; ++u) take(k + u * slices, v[u]);
                    }
                    for (; k < g.K; k += slices) take(k, code(k));
                }
            }
        }
    }
    part[slice * blockDim.x + threadIdx.x] = acc;
    __syncthreads();
    if (slice == 0 && live) {
        float total_acc = 0.0f;
        for (int j = 0; j < slices; ++j) total_acc += part[j * blockDim.x + threadIdx.x];
        gx[i] = from_f32<T>(total_acc);
    }
}

// All parameter gradients but their last sum.  Block (k * C + c, split) walks its share of the (n, position)
// range; every thread keeps private columns in shared memory, one per tap and branch (col[tap][tb], one more
// for items that another channel won), so that an item costs one read-modify-write per branch; grad_alpha /
// grad_beta: g times the branch value, rebuilt from the winner (x zero in the padding) as the forward rounded it.
// part_hist [split][k*C+c][2][taps], part_ab [split][k*C+c][2], part_bias [split][k].
template <typename T>
__global__ void __launch_bounds__(128)
bwd3d_params_kernel(Geo3 g, int nsplit, const T* __restrict__ x, const T* __restrict__ w, const T* __restrict__ w2,
                    const T* __restrict__ gy, const void* __restrict__ winners, float* __restrict__ part_hist,
                    float* __restrict__ part_ab, float* __restrict__ part_bias) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, tb = blockDim.x, taps = g.taps;
    const int kc = blockIdx.x, k = kc / g.C, c = kc - k * g.C, split = blockIdx.y;
    const bool twob = two_branch(g.mode), codes = g.chan == CH_SUM;
    const bool use_min = g.mode != TCONV_MAX_PLUS, use_max = g.mode != TCONV_MIN_PLUS;
    const int branches = (use_min ? 1 : 0) + (use_max ? 1 : 0);
    float* cmin = reinterpret_cast<float*>(smem_raw);
    float* cmax = cmin + (use_min ? (taps + 1) * tb : 0);
    int* tofs = reinterpret_cast<int*>(cmin + branches * (taps + 1) * tb);   // input offset of a tap from its window's corner
    int* tcrd = tofs + taps;                                                 // its (depth, row, column) distance, 10 bits each
    T* wmin = reinterpret_cast<T*>(tcrd + taps);                             // weights of the pair, either branch
    T* wmax = wmin + taps;
    float* red = reinterpret_cast<float*>(tcrd + 3 * taps);                  // [3][tb / 32]
    for (int i = tid; i < branches * (taps + 1) * tb; i += tb) cmin[i] = 0.0f;
    for (int i = tid; i < taps; i += tb) {
        const int t = i / (g.R * g.S), r = (i / g.S) % g.R, s = i % g.S;
        tofs[i] = (t * g.dd * g.H + r * g.dh) * g.W + s * g.dw;
        tcrd[i] = (t << 20) | (r << 10) | s;
        if (twob) {
            wmin[i] = w[(size_t)kc * taps + i];
            wmax[i] = (g.mode == TCONV_PARALLEL ? w2 : w)[(size_t)kc * taps + i];
        }
    }
    __syncthreads();
    // (unsigned: up to 2^31 - 1 items, and a round may end past them)
    const unsigned total = (unsigned)(g.N * g.vol), per = (total + nsplit - 1) / nsplit;
    const unsigned j0 = min(total, split * per), j1 = min(total, j0 + per);
    float sa = 0.0f, sb = 0.0f, sg = 0.0f;
    constexpr int U = 4;          // items whose loads go out together
    for (unsigned jb = j0 + tid; jb < j1; jb += U * tb) {
        unsigned raw[U];
        float gv[U];
        int n[U], pos[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned j = jb + u * tb, jj = j < j1 ? j : jb;
            n[u] = (int)(jj / (unsigned)g.vol);
            pos[u] = (int)(jj - (unsigned)n[u] * (unsigned)g.vol);
            const int row = n[u] * g.K + k;
            raw[u] = codes ? (unsigned)__ldg((const uint16_t*)winners + ((row * g.C + c) * g.vol + pos[u]))
                           : (unsigned)__ldg((const int32_t*)winners + (row * g.vol + pos[u]));
            const float v = to_f32(__ldg(gy + (row * g.vol + pos[u])));
            gv[u] = j < j1 ? v : 0.0f;
        }
        int amn[U], amx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (codes) {
                amn[u] = (int)(raw[u] & 0xFFu);
                amx[u] = (int)(raw[u] >> 8);
            } else {
                const int v = (int)raw[u] - c * taps;
                amn[u] = amx[u] = (v >= 0 && v < taps) ? v : taps;
            }
        }
        if (twob) {
            float za[U], zb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned q = (unsigned)pos[u] / (unsigned)g.OW;
                const int ow = pos[u] - (int)q * g.OW, od = (int)(q / (unsigned)g.OH), oh = (int)q - od * g.OH;
                const int d0 = od * g.sd - g.pd, h0 = oh * g.sh - g.ph, w0 = ow * g.sw - g.pw;
                const T* xc = x + (size_t)(n[u] * g.C + c) * g.D * g.H * g.W;
                const int corner = (d0 * g.H + h0) * g.W + w0;
                auto at = [&](int tap, const T* wt) {
                    const int p = tcrd[tap];
                    const int id = d0 + (p >> 20) * g.dd, ih = h0 + ((p >> 10) & 1023) * g.dh, iw = w0 + (p & 1023) * g.dw;
                    const bool ok = (unsigned)id < (unsigned)g.D && (unsigned)ih < (unsigned)g.H && (unsigned)iw < (unsigned)g.W;
                    return tap_add(ok ? __ldg(xc + corner + tofs[tap]) : zero_of<T>(), wt[tap]);
                };
                za[u] = at(amn[u], wmin);
                zb[u] = at(amx[u], wmax);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (jb + u * tb >= j1) break;
                sa = __fmaf_rn(gv[u], za[u], sa);
                sb = __fmaf_rn(gv[u], zb[u], sb);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            sg += gv[u];
            if (use_min) cmin[amn[u] * tb + tid] += gv[u];
            if (use_max) cmax[amx[u] * tb + tid] += gv[u];
        }
    }
    __syncthreads();
    float* hist = part_hist + ((size_t)split * g.K * g.C + kc) * 2 * taps;
    for (int i = tid; i < 2 * taps; i += tb) {
        const bool mx = i >= taps;
        const float* col = (mx ? cmax : cmin) + (size_t)(mx ? i - taps : i) * tb;
        float s = 0.0f;
        if (mx ? use_max : use_min)
            for (int q = 0; q < tb; ++q) s += col[(q + tid) & (tb - 1)];   // rotated start: different banks
        hist[i] = s;
    }
    float v[3] = {sa, sb, sg};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], d);
        if ((tid & 31) == 0) red[q * (tb / 32) + (tid >> 5)] = v[q];
    }
    __syncthreads();
    if (tid < 3) {
        float s = 0.0f;
        for (int q = 0; q < tb / 32; ++q) s += red[tid * (tb / 32) + q];
        if (tid < 2) part_ab[((size_t)split * g.K * g.C + kc) * 2 + tid] = s;
        else if (c == 0) part_bias[(size_t)split * g.K + k] = s;
    }
}

// One block per (k, c): sums its partials over the splits in order and applies alpha / beta.
static __global__ void __launch_bounds__(128)
bwd3d_params_finish_kernel(Geo3 g, int nsplit, const float* __restrict__ alpha, const float* __restrict__ beta,
                           const float* __restrict__ part_hist, const float* __restrict__ part_ab,
                           const float* __restrict__ part_bias, float* __restrict__ gw, float* __restrict__ gw2,
                           float* __restrict__ galpha, float* __restrict__ gbeta, float* __restrict__ gbias) {
    const int kc = blockIdx.x, k = kc / g.C, c = kc - k * g.C, tid = threadIdx.x;
    const size_t pairs = (size_t)g.K * g.C;
    const bool twob = two_branch(g.mode), par = g.mode == TCONV_PARALLEL;
    const float a = twob && alpha ? alpha[kc] : 1.0f, b = twob && beta ? beta[kc] : 1.0f;
    for (int t = tid; t < g.taps; t += 128) {
        float tmin = 0.0f, tmax = 0.0f;
        for (int s = 0; s < nsplit; ++s) {
            const float* h = part_hist + (s * pairs + kc) * 2 * g.taps;
            tmin += h[t];
            tmax += h[g.taps + t];
        }
        const size_t i = (size_t)kc * g.taps + t;
        if (!twob) {
            if (gw) gw[i] = g.mode == TCONV_MIN_PLUS ? tmin : tmax;
        } else {
            if (par) {
                if (gw) gw[i] = a * tmin;
                if (gw2) gw2[i] = b * tmax;
            } else if (gw) {
                gw[i] = __fmaf_rn(a, tmin, b * tmax);
            }
        }
    }
    if (twob && tid < 2) {
        float s = 0.0f;
        for (int sp = 0; sp < nsplit; ++sp) s += part_ab[(sp * pairs + kc) * 2 + tid];
        float* to = tid == 0 ? galpha : gbeta;
        if (to) to[kc] = s;
    }
    if (gbias && c == 0 && tid == 2) {
        float s = 0.0f;
        for (int sp = 0; sp < nsplit; ++sp) s += part_bias[(size_t)sp * g.K + k];
        gbias[k] = s;
    }
}

// Sums the partials over the splits in order and applies alpha / beta: one thread per (k, c, tap).
__global__ void __launch_bounds__(256)
bwd3d_gw_finish_kernel(Geo3 g, int nsplit, const float* __restrict__ alpha, const float* __restrict__ beta,
                       const float* __restrict__ part_min, const float* __restrict__ part_max,
                       float* __restrict__ gw, float* __restrict__ gw2) {
    const size_t count = (size_t)g.K * g.C * g.taps;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    float tmin = 0.0f, tmax = 0.0f;
    for (int sp = 0; sp < nsplit; ++sp) {
        tmin += part_min[(size_t)sp * count + i];
        tmax += part_max[(size_t)sp * count + i];
    }
    const size_t kc = i / g.taps;
    if (!two_branch(g.mode)) {
        if (gw) gw[i] = (g.mode == TCONV_MIN_PLUS) ? tmin : tmax;
        return;
    }
    const float a = alpha ? alpha[kc] : 1.0f, b = beta ? beta[kc] : 1.0f;
    if (g.mode == TCONV_COMPOUND) {
        if (gw) gw[i] = __fmaf_rn(a, tmin, b * tmax);
    } else {
        if (gw) gw[i] = a * tmin;
        if (gw2) gw2[i] = b * tmax;
    }
}

// Sums partials over the splits in order: out[i] = sum_split part[(split * count + i) * stride + off].
__global__ void __launch_bounds__(256)
bwd3d_sum_splits_kernel(int count, int nsplit, int stride, int off, const float* __restrict__ part,
                        float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    float t = 0.0f;
    for (int sp = 0; sp < nsplit; ++sp) t += part[((size_t)sp * count + i) * stride + off];
    out[i] = t;
}

}  // namespace tconv
