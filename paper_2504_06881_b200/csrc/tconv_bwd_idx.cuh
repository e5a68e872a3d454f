// Backward of the Max / Min channel combine (one int32 winner c * RS + tap per output).  No atomics; every
// accumulator has one writer at a time and a fixed order.
//
//   bwd_idx_gx_kernel   a CTA owns a band of input rows of one image (all channels, or a block of them) in
//                       shared memory and adds every output's gradient at its winner.  Two outputs can only
//                       meet at an input element if their windows overlap, so the band's output rows are taken
//                       in classes of rows whose windows are disjoint (a barrier between classes), one warp per
//                       row, and inside a row the columns in classes too (program order inside the warp); then
//                       every add is a plain read-modify-write, whatever the winning channels are.
//   bwd_idx_gw_kernel   lane = output channel (few channels: several lanes each, on other pixels): each lane keeps
//                       its own histogram over (c, tap), tab[bin][32], free of conflicts.  Also grad_bias.
//   bwd_idx_gw_finish_kernel  sums the ranges' histograms in a fixed order.
//
// Measured at N=128 C=64 K=64 32x32 3x3 fp32 (67 MB of winners and gradients, 10 us at the copy rate):
// grad_x 133 -> 80 us, bound by the latency of its chain (row classes x K / 4 steps of some 800 cycles: addresses,
// then three column classes of dependent shared-memory accesses) at the few warps per SM that the tile leaves; grad_w 93 -> 23 us, memory traffic.
// One row of 10303 samples, 53 channels: 825 -> 22 us (column tiles instead of one warp along the row).
#pragma once
#include <cstring>

#include "tconv_common.cuh"

namespace tconv {

constexpr size_t kIdxSmemMost = 200 * 1024;   // opt-in ceiling set on the kernels

struct IdxGxPlan {
    int TH, bands;          // input rows per band
    int TW, ncol;           // input columns per tile, column tiles
    int CB, nblk;           // channels per CTA, channel blocks
    int gdh, mr, gdw, mc;   // output rows (columns) i and j are of one class iff (i / gd) % m agrees
    int threads;
    unsigned grid;
    size_t smem;
};
struct IdxGwPlan {
    int CB, nblk;           // channels per table, channel blocks
    int nkg;                // groups of 32 output channels
    int lk;                 // log2 of the lanes that take different output channels (the others: more pixels)
    int shift;              // 1: planes that are not a multiple of four, rows start inside a piece of four
    int timg;               // tiles of 32 pixels per lane slice, per image
    int chunks, per;        // ranges of the flattened (image, tile) space, tiles per range
    size_t smem, part_floats;
};

// Classes of one axis: outputs i < j collide iff (j - i) * stride = dil * t for a 0 <= t < taps.  Stride 1:
// only distances that are multiples of dil, so groups of dil neighbours count as one.
inline void idx_classes(int taps, int dil, int stride, int* gd, int* m) {
    if (stride == 1) { *gd = dil; *m = taps; }
    else { *gd = 1; *m = ((taps - 1) * dil) / stride + 1; }
}
__host__ __device__ inline int idx_class_count(int n, int gd, int m, int cls) {
    const int period = gd * m, rest = n % period - cls * gd;
    return n / period * gd + (rest < 0 ? 0 : rest < gd ? rest : gd);
}

// Tile (rows, columns, channel block) and threads with the shortest estimated time, in cycles.  A CTA's rows of one
// class run on a warp each, its classes and the columns of a row one after another; a step of four output channels
// takes 460 cycles + 115 per column class, or, with more warps on an SM than that hides, their 14 + 31 issue slots
// each.  Clearing and storing the tile: 244 cycles per element of a thread, more where 16 warps share an SM.  Fitted
// to 3600 launches of 21 layers (the choice is 8 % off the best on average, 39 % at worst).  Residency counts the
// registers as well: without them N=64 C=512 K=512 12x12 fp32 ran in three rounds of two CTAs per SM instead of one
// of two (549 against 187 us).
constexpr int kIdxGxRegs = 112;          // per thread, as allocated (107 used)
inline bool plan_idx_gx(const Geo& g, IdxGxPlan* best) {
    if ((double)g.K * g.OH * g.OW > 2.0e9 || (double)g.N * g.H > 2.0e9) return false;
    int gdh, mr, gdw, mc;
    idx_classes(g.R, g.dh, g.sh, &gdh, &mr);
    idx_classes(g.S, g.dw, g.sw, &gdw, &mc);
    double best_cost = -1.0;
    const int halo_h = (g.R - 1) * g.dh, halo_w = (g.S - 1) * g.dw;
    const double step = 460.0 + 115.0 * mc, slots = 14.0 + 31.0 * mc, k4 = (g.K + 3) / 4;
    for (const int nblk : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64}) {
        if (nblk > g.C) break;
        IdxGxPlan p;
        p.gdh = gdh; p.mr = mr; p.gdw = gdw; p.mc = mc;
        p.CB = (g.C + nblk - 1) / nblk;
        p.nblk = (g.C + p.CB - 1) / p.CB;
        for (int tw0 = g.W; ; tw0 = (tw0 + 1) / 2) {
            p.ncol = (g.W + tw0 - 1) / tw0;
            p.TW = (g.W + p.ncol - 1) / p.ncol;
            const size_t row = (size_t)p.CB * p.TW * sizeof(float);
            int cols = (p.TW + halo_w - 1) / g.sw + 1;               // outputs that reach a tile's columns
            if (cols > g.OW) cols = g.OW;
            for (int b = 1; ; b = b < 4 ? b + 1 : b + b / 2) {
                if (b > g.H) b = g.H;
                p.TH = (g.H + b - 1) / b;
                p.bands = (g.H + p.TH - 1) / p.TH;
                p.smem = row * p.TH + 256 * sizeof(float);
                const double ctas = (double)g.N * p.bands * p.ncol * p.nblk;
                if (p.smem <= kIdxSmemMost && ctas <= 2.0e9) {
                    int rows = (p.TH + halo_h - 1) / g.sh + 1;
                    if (rows > g.OH) rows = g.OH;
                    int tasks = idx_class_count(rows, gdh, mr, 0);
                    if (cols <= 32) tasks = (tasks + 32 / cols - 1) / (32 / cols);
                    const int warps = tasks < 1 ? 1 : tasks > 8 ? 8 : tasks;
                    for (const int nw : {warps, 8}) {                // (eight: to clear and store the tile)
                        long per_sm = (long)(228 * 1024 / (p.smem + 1024));
                        if (per_sm > 65536 / (kIdxGxRegs * 32 * nw)) per_sm = 65536 / (kIdxGxRegs * 32 * nw);
                        const double rounds = (double)(long)((ctas + 148.0 * per_sm - 1) / (148.0 * per_sm));
                        double resident = (double)(long)((ctas + 147.0) / 148.0);
                        if (resident > per_sm) resident = per_sm;
                        const double issue = resident * warps * slots, crowd = resident * nw / 16.0;
                        const double chain = (double)mr * ((tasks + warps - 1) / warps) * ((cols + 31) / 32) * k4;
                        const double cost = rounds * (chain * (issue > step ? issue : step) +
                                                      244.0 * row / 4 * p.TH / (32 * nw) * (crowd > 1.0 ? crowd : 1.0));
                        if (best_cost < 0.0 || cost < best_cost) {
                            best_cost = cost;
                            p.threads = 32 * nw;
                            p.grid = (unsigned)ctas;
                            *best = p;
                        }
                    }
                }
                if (b == g.H) break;
            }
            if (tw0 <= 32) break;
        }
    }
    return best_cost >= 0.0;
}

// The plan of a layer, or null.  The search is some microseconds of host work, so the last few are kept per host
// thread (they depend on nothing but the geometry).
inline const IdxGxPlan* idx_gx_plan(const Geo& g) {
    constexpr int kKept = 16;
    struct Entry { Geo g; IdxGxPlan plan; bool ok; };
    static thread_local Entry kept[kKept];
    static thread_local int used = 0, next = 0;
    for (int i = 0; i < used; ++i)
        if (memcmp(&kept[i].g, &g, sizeof(Geo)) == 0) return kept[i].ok ? &kept[i].plan : nullptr;
    Entry& e = kept[next];
    e.g = g;
    e.ok = plan_idx_gx(g, &e.plan);
    next = (next + 1) % kKept;
    if (used < kKept) ++used;
    return e.ok ? &e.plan : nullptr;
}

// One stage of the pixel ring: 32 lanes' winners and gradients of 32 pixels, rows padded against bank conflicts.
constexpr int kGwPitch = 36;                        // words per lane row (16-byte reads of eight lanes: all banks)
constexpr int kGwStages = 4;
constexpr size_t kGwStageBytes = 2 * 32 * kGwPitch * 4;

inline bool plan_idx_gw(const Geo& g, IdxGwPlan* p) {
    const size_t per_c = (size_t)g.RS * 32 * sizeof(float);
    if (per_c > 150 * 1024 || (double)g.N * g.K * g.OH * g.OW > 6.0e10 || (double)g.N * g.OH * g.OW > 2.0e9) return false;
    p->CB = (int)(73 * 1024 / per_c);
    if (p->CB < 1) p->CB = 1;
    if (p->CB > g.C) p->CB = g.C;
    p->nblk = (g.C + p->CB - 1) / p->CB;
    p->CB = (g.C + p->nblk - 1) / p->nblk;
    p->nblk = (g.C + p->CB - 1) / p->CB;
    p->nkg = (g.K + 31) / 32;
    p->lk = g.K > 16 ? 5 : g.K > 8 ? 4 : g.K > 4 ? 3 : g.K > 2 ? 2 : g.K > 1 ? 1 : 0;
    p->smem = per_c * p->CB + 32 * sizeof(float) + kGwStages * kGwStageBytes;
    const long plane = (long)g.OH * g.OW;
    while (p->lk < 5 && plane <= (32L << (5 - p->lk)) / 2) ++p->lk;    // small planes: no slices without pixels
    p->shift = plane % 4 != 0;
    const long tile = 32L << (5 - p->lk);
    p->timg = (int)((plane + tile - 1) / tile);
    const long tiles = (long)g.N * p->timg;
    long per_sm = (long)(227 * 1024 / (p->smem + 1024));
    if (per_sm > 6) per_sm = 6;
    if (per_sm < 1) per_sm = 1;
    long want = 148 * per_sm / ((long)p->nkg * p->nblk);
    if (want > 512) want = 512;                      // (the finishing sum walks the ranges)
    // a range's pixels cost about 20 cycles each, clearing, writing and summing its table 8 a bin
    const long most = 3 * (long)g.N * plane / (((long)p->CB * g.RS) << (5 - p->lk)) + 1;
    if (want > most) want = most;
    if (want > tiles) want = tiles;
    if (want < 1) want = 1;
    p->per = (int)((tiles + want - 1) / want);
    p->chunks = (int)((tiles + p->per - 1) / p->per);
    p->part_floats = (size_t)p->chunks * p->nkg * ((size_t)g.C * g.RS + 1) * 32;
    return true;
}

// ---------------------------------------------------------------------------------- grad_x
template <typename T>
__global__ void __launch_bounds__(256, 2)
bwd_idx_gx_kernel(Geo g, const T* __restrict__ gy, const int32_t* __restrict__ idx, T* __restrict__ gx, IdxGxPlan pl,
                  unsigned magic_rs, unsigned magic_s) {
    extern __shared__ float tile[];          // [CB][TH][TW], then a dummy word per thread
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int cblk = blockIdx.x % pl.nblk;
    int bt = blockIdx.x / pl.nblk;
    const int iw0 = (bt % pl.ncol) * pl.TW, cols = min(pl.TW, g.W - iw0);
    bt /= pl.ncol;
    const int n = bt / pl.bands, ih0 = (bt - n * pl.bands) * pl.TH;
    const int rows = min(pl.TH, g.H - ih0);
    const int c0 = cblk * pl.CB, cbn = min(pl.CB, g.C - c0);
    const int cstride = pl.TH * pl.TW, used = pl.CB * cstride;
    for (int e = tid; e < used; e += blockDim.x) tile[e] = 0.0f;
    const int num = ih0 + g.ph - (g.R - 1) * g.dh;
    const int oh_lo = num <= 0 ? 0 : (num + g.sh - 1) / g.sh;
    const int oh_hi = min(g.OH - 1, (ih0 + rows - 1 + g.ph) / g.sh);
    const int NR = max(0, oh_hi - oh_lo + 1);
    const int numw = iw0 + g.pw - (g.S - 1) * g.dw;
    const int ow_lo = numw <= 0 ? 0 : (numw + g.sw - 1) / g.sw;
    const int NC = max(0, min(g.OW - 1, (iw0 + cols - 1 + g.pw) / g.sw) - ow_lo + 1);   // output columns that reach the tile
    const unsigned plane = (unsigned)(g.OH * g.OW);
    const int32_t* ibase = idx + (size_t)n * g.K * plane;
    const T* gbase = gy + (size_t)n * g.K * plane;
    const bool packed = NC > 0 && NC <= 32;
    const int rpw = packed ? 32 / NC : 1;                          // rows a warp takes at once
    const int lr = packed ? lane / NC : 0, lcol = packed ? lane - lr * NC : lane;
    const int dummy = used + tid;
    __syncthreads();
    for (int cls = 0; cls < pl.mr; ++cls) {
        const int cnt = idx_class_count(NR, pl.gdh, pl.mr, cls);
        for (int i0 = warp * rpw; i0 < cnt; i0 += nwarps * rpw) {
            const int i = i0 + lr;
            const bool rlive = lr < rpw && i < cnt;
            const int o = (i / pl.gdh) * (pl.gdh * pl.mr) + cls * pl.gdh + i % pl.gdh;
            const int oh = oh_lo + (rlive ? o : 0);
            const int rbase = oh * g.sh - g.ph - ih0;
            for (int col0 = 0; col0 < NC; col0 += 32) {
                const int ow = ow_lo + col0 + lcol;
                const bool live = rlive && col0 + lcol < NC;
                const int cbase = ow * g.sw - g.pw - iw0;
                const int ccls = live ? (ow / pl.gdw) % pl.mc : -1;
                unsigned off = live ? (unsigned)(oh * g.OW + ow) : 0u;
                // winners and gradients of four output channels at a time, the next twelve in flight
                constexpr int U = 4, B = 4;
                int32_t id[B][U];
                float gv[B][U];
                auto request = [&](int b, int k0) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const unsigned at = off + (unsigned)min(k0 + u, g.K - 1) * plane;
                        id[b][u] = __ldg(ibase + at);
                        gv[b][u] = to_f32(__ldg(gbase + at));
                    }
                };
                auto add = [&](int b, int k0) {
                    int at[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const unsigned v = (unsigned)id[b][u];
                        const unsigned c = magic_rs ? __umulhi(v, magic_rs) : v;       // v / RS (magic 0: RS == 1)
                        const unsigned tap = v - c * g.RS;
                        const unsigned r = (tap * magic_s) >> 16;                      // tap / S, tap < 256
                        const int tr = rbase + (int)r * g.dh, tc = cbase + (int)(tap - r * g.S) * g.dw;
                        const bool hit = k0 + u < g.K && (unsigned)tr < (unsigned)rows && (unsigned)tc < (unsigned)cols &&
                                         (unsigned)((int)c - c0) < (unsigned)cbn;
                        at[u] = hit ? ((int)c - c0) * cstride + tr * pl.TW + tc : dummy;
                    }
                    for (int cc = 0; cc < pl.mc; ++cc) {
                        if (ccls == cc) {
                            // all loads first; where two of the four meet, the later store holds both gradients
                            float v[U];
#pragma unroll
                            for (int u = 0; u < U; ++u) v[u] = tile[at[u]];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
#pragma unroll
                                for (int w = 0; w < u; ++w) v[u] = at[w] == at[u] ? v[w] : v[u];
                                v[u] += gv[b][u];
                            }
#pragma unroll
                            for (int u = 0; u < U; ++u) tile[at[u]] = v[u];
                        }
                        __syncwarp();
                    }
                };
#pragma unroll
                for (int b = 0; b < B - 1; ++b) request(b, b * U);
                for (int k0 = 0; k0 < g.K; k0 += B * U) {
#pragma unroll
                    for (int b = 0; b < B; ++b) {
                        if (k0 + b * U >= g.K) break;
                        request((b + B - 1) % B, k0 + (b + B - 1) * U);
                        add(b, k0 + b * U);
                    }
                }
            }
        }
        __syncthreads();
    }
    // rows of all channels, one warp each, lanes along the columns (whole rows of a channel in one go)
    const bool wide = cols == g.W;
    const int len = wide ? rows * cols : cols, per_c = wide ? 1 : rows;
    for (int t = warp; t < cbn * per_c; t += nwarps) {
        const int c = t / per_c, r = t - c * per_c;
        T* o = gx + ((size_t)n * g.C + c0 + c) * g.H * g.W + (size_t)(ih0 + r) * g.W + iw0;
        const float* from = tile + c * cstride + r * pl.TW;
        for (int e = lane; e < len; e += 32) o[e] = from_f32<T>(from[e]);
    }
}

// ---------------------------------------------------------------------------------- grad_w, grad_bias
// bytes of a piece of 16 (8), then zeros
__device__ __forceinline__ void gw_copy16(unsigned dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void gw_copy8(unsigned dst, const void* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// Elements s .. s + 3 of eight.
__device__ __forceinline__ uint4 gw_shift(const uint4& a, const uint4& b, int s) {
    const bool one = s & 1, two = s & 2;
    const unsigned t0 = one ? a.y : a.x, t1 = one ? a.z : a.y, t2 = one ? a.w : a.z, t3 = one ? b.x : a.w, t4 = one ? b.y : b.x,
                   t5 = one ? b.z : b.y;
    return make_uint4(two ? t2 : t0, two ? t3 : t1, two ? t4 : t2, two ? t5 : t3);
}

// SHIFT: planes that are not a multiple of four.  A row of 32 pixels may start inside a piece of four; its nine pieces
// are copied whole and four pixels selected out of two pieces when they are read.  Copied pixel by pixel such planes
// took four times the copies (N=64 C=512 K=512 15x15 bf16: 818 us).
template <typename T, bool SHIFT>
__global__ void __launch_bounds__(32)
bwd_idx_gw_kernel(Geo g, const T* __restrict__ gy, const int32_t* __restrict__ idx, float* __restrict__ part,
                  float* __restrict__ part_b, IdxGwPlan pl) {
    extern __shared__ __align__(16) float smem_gw[];
    // ring [kGwStages][winners, gradients][32][kGwPitch], then the table [CB * RS + 1][32]
    float* tab = smem_gw + kGwStages * (kGwStageBytes / 4);
    const int lane = threadIdx.x;
    const int cblk = blockIdx.x % pl.nblk, kg = blockIdx.x / pl.nblk, chunk = blockIdx.y;
    const int c0 = cblk * pl.CB, nb = min(pl.CB, g.C - c0) * g.RS, b0 = c0 * g.RS;
    const int plane = g.OH * g.OW;
    const int total = g.N * pl.timg;
    const int i0 = chunk * pl.per, i1 = min(total, i0 + pl.per);
    const int tile_px = 32 << (5 - pl.lk), kmask = (1 << pl.lk) - 1;
    constexpr bool HALF = sizeof(T) == 2;
    const int n0 = i0 / pl.timg, t0 = i0 - n0 * pl.timg;
    int n = n0, t = t0, next = i0;
    // Pixels past the plane's end and output channels past K arrive as zeros: nothing added.
    auto request = [&](int stage) {
        if (next < i1) {
            float* st = smem_gw + stage * (kGwStageBytes / 4);
            const unsigned si = (unsigned)__cvta_generic_to_shared(st), sg = si + 32 * kGwPitch * 4;
            // piece j (four pixels) of a row: `left` pixels of the row and those before it in its first piece remain
            auto copy = [&](int row, int j) {
                const int k = kg * 32 + (row & kmask), p0 = t * tile_px + (row >> pl.lk) * 32, cnt = min(32, plane - p0);
                const bool on = k < g.K && cnt > 0;
                size_t at = on ? ((size_t)n * g.K + k) * plane + p0 : 0;
                const int before = SHIFT ? (int)(at & 3) : 0;
                const int left = on ? min(4, max(0, cnt + before - 4 * j)) : 0;
                at = left ? at - before + 4 * j : 0;
                gw_copy16(si + (row * kGwPitch + 4 * j) * 4, idx + at, left * 4);
                if constexpr (HALF) gw_copy8(sg + row * (kGwPitch * 2) + j * 8, gy + at, left * 2);
                else gw_copy16(sg + (row * kGwPitch + 4 * j) * 4, gy + at, left * 4);
            };
#pragma unroll
            for (int u = 0; u < 8; ++u) copy(u * 4 + (lane >> 3), lane & 7);       // eight lanes, 32 pixels of one row
            if constexpr (SHIFT) copy(lane, 8);
            if (++t == pl.timg) { t = 0; ++n; }
        }
        ++next;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float sum = 0.0f;
    auto add = [&](const int4& q, const float4& f) {
        const int id[4] = {q.x, q.y, q.z, q.w};
        const float gv[4] = {f.x, f.y, f.z, f.w};
        int at[4];
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)                               // (another block's channel: the spare row)
            at[u] = (int)min((unsigned)(id[u] - b0), (unsigned)nb) * 32 + lane;
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = tab[at[u]];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int w = 0; w < u; ++w) v[u] = at[w] == at[u] ? v[w] : v[u];
            v[u] += gv[u];
            sum += gv[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) tab[at[u]] = v[u];
    };
#pragma unroll
    for (int s = 0; s < kGwStages - 1; ++s) request(s);
    float4* tab4 = reinterpret_cast<float4*>(tab);
#pragma unroll 4
    for (int e = lane; e < (pl.CB * g.RS + 1) * 8; e += 32) tab4[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int stage = 0;
    const unsigned kmine = kg * 32 + (lane & kmask);
    unsigned nu = n0;                                             // image of the tile in use
    int tu = t0;
    for (int i = i0; i < i1; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGwStages - 2) : "memory");
        __syncwarp();
        request((stage + kGwStages - 1) % kGwStages);
        const float* st = smem_gw + stage * (kGwStageBytes / 4);
        const int before = SHIFT ? (int)(((nu * g.K + kmine) * (unsigned)plane) & 3u) : 0;
        if (++tu == pl.timg) { tu = 0; ++nu; }
        const uint4* ri = reinterpret_cast<const uint4*>(st + lane * kGwPitch);
        auto grads = [&](int j) {                                 // (bf16: four in two words)
            if constexpr (HALF) {
                const uint2 f = reinterpret_cast<const uint2*>(st + 32 * kGwPitch + lane * (kGwPitch / 2))[j];
                return make_uint4(f.x, f.y, 0u, 0u);
            } else {
                return reinterpret_cast<const uint4*>(st + 32 * kGwPitch + lane * kGwPitch)[j];
            }
        };
        uint4 q = ri[0], f = grads(0);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int j1 = SHIFT ? j + 1 : (j + 1) & 7;
            const uint4 q1 = ri[j1], f1 = grads(j1);
            uint4 w = q, v = f;
            if constexpr (SHIFT) {
                w = gw_shift(q, q1, before);
                if constexpr (HALF) {
                    const bool two = before & 2;
                    const unsigned h = (before & 1) * 16, a = two ? f.y : f.x, b = two ? f1.x : f.y, c = two ? f1.y : f1.x;
                    v.x = __funnelshift_r(a, b, h);
                    v.y = __funnelshift_r(b, c, h);
                } else {
                    v = gw_shift(f, f1, before);
                }
            }
            if constexpr (HALF) v = make_uint4(v.x << 16, v.x & 0xffff0000u, v.y << 16, v.y & 0xffff0000u);
            add(make_int4(w.x, w.y, w.z, w.w),
                make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)));
            q = q1;
            f = f1;
        }
        stage = (stage + 1) % kGwStages;
        __syncwarp();
    }
    const size_t CRS = (size_t)g.C * g.RS;
    float4* o = reinterpret_cast<float4*>(part + (((size_t)chunk * pl.nkg + kg) * CRS + b0) * 32);
#pragma unroll 4
    for (int e = lane; e < nb * 8; e += 32) o[e] = tab4[e];
    if (cblk == 0) part_b[((size_t)chunk * pl.nkg + kg) * 32 + lane] = sum;
}

// gw[k][bin] = sum over the ranges of part[range][k / 32][bin][k % 32]: a block takes four bins of 32 output
// channels, up to eight slices of the ranges each (blockDim.z), added in slice order; the block past the last bin
// sums grad_bias.  Two ranges of 512 x 512 channels with eight slices, six of them idle: 79 us.
static __global__ void __launch_bounds__(1024)
bwd_idx_gw_finish_kernel(Geo g, IdxGwPlan pl, const float* __restrict__ part, const float* __restrict__ part_b,
                         float* __restrict__ gw, float* __restrict__ gbias) {
    __shared__ float red[8][4][33];
    const int kk = threadIdx.x, bin4 = threadIdx.y, slice = threadIdx.z, slices = blockDim.z, kg = blockIdx.y;
    const size_t CRS = (size_t)g.C * g.RS, bin = (size_t)blockIdx.x * 4 + bin4;
    const bool bias = blockIdx.x == gridDim.x - 1;
    float s = 0.0f;
    if (bias ? bin4 == 0 : bin < CRS) {
        const float* p = bias ? part_b + (size_t)kg * 32 + kk : part + ((size_t)kg * CRS + bin) * 32 + kk;
        const size_t step = (bias ? (size_t)pl.nkg : (size_t)pl.nkg * CRS) * 32;
#pragma unroll 8
        for (int ch = slice; ch < pl.chunks; ch += slices) s += __ldg(p + ch * step);
    }
    red[slice][bin4][kk] = s;
    __syncthreads();
    if (slice != 0) return;
    // four adjacent bins of an output channel to adjacent threads
    const int t = bin4 * 32 + kk, k2 = t >> 2, b2 = t & 3, k = kg * 32 + k2;
    float v = 0.0f;
    for (int i = 0; i < slices; ++i) v += red[i][b2][k2];
    if (k >= g.K) return;
    for (int l = k2 + (1 << pl.lk); l < 32; l += 1 << pl.lk) {     // the channel's other lanes
        for (int i = 0; i < slices; ++i) v += red[i][b2][l];
    }
    if (bias) {
        if (b2 == 0 && gbias) gbias[k] = v;
    } else if (gw && (size_t)blockIdx.x * 4 + b2 < CRS) {
        gw[(size_t)k * CRS + (size_t)blockIdx.x * 4 + b2] = v;
    }
}

}  // namespace tconv
