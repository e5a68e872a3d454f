// Register-only throughput probes of the add + max/min instruction mixes the
// tropical kernels can be built from.  Each thread keeps a TK x TP block of
// running extrema and folds taps x[j] + w[i] into them, exactly the inner loop of
// the forward pass minus its memory traffic.  The x operands must change from one
// iteration to the next (an empty asm barrier is not enough: the assembler, which
// never sees it, would hoist the loop-invariant tap sums out of the loop and the
// probe would measure min/max alone).  Two ways, both built (template flag FEED),
// and the caller takes the better rate: advancing adds (TP + 1 extra adds per
// TK * TP * 2 taps, left uncorrected), or feedback: TP + 1 of the tap sums an
// iteration forms anyway become the next iteration's x operands, so that every
// instruction of the loop body is a tap sum or a min / max.
#pragma once
#include <type_traits>

#include "tconv_common.cuh"
#include "tconv_winners.cuh"

namespace tconv {

#define TCONV_OPAQUE_F(v) asm volatile("" : "+f"(v))
#define TCONV_OPAQUE_R(v) asm volatile("" : "+r"(v))

enum {
    PROBE_F32_ADD_MAX2 = 0,      // max-plus / min-plus: add, 2-input max
    PROBE_F32_ADD_MAX3,          // two adds feed one 3-input max
    PROBE_F32_ADD2_MAX3,         // packed add of two channels, 3-input max over two taps
    PROBE_F32_ADD_MINMAX2,       // compound: add, min, max
    PROBE_F32_ADD_MINMAX3,       // compound: two adds feed a 3-input min and a 3-input max
    PROBE_F32_ADD2_MINMAX3,      // compound with packed adds
    PROBE_F32_2ADD_MINMAX2,      // parallel: two adds, min, max
    PROBE_F32_2ADD_MINMAX3,      // parallel with 3-input min / max
    PROBE_F32_2ADD2_MINMAX3,     // parallel with packed adds and 3-input min / max
    PROBE_BF16X2_ADD_MAX,        // bf16 pairs: add, max
    PROBE_BF16X2_ADD_MINMAX,     // bf16 pairs, compound
    PROBE_BF16X2_2ADD_MINMAX,    // bf16 pairs, parallel
    PROBE_F32_ADD_ONLY,          // adds alone (sum-reduced), the FP32 pipe by itself
    PROBE_F32_MAX2_ONLY,         // 2-input max alone
    PROBE_F32_MAX3_ONLY,         // 3-input max alone
    PROBE_F32_WIN_SINGLE,        // Sum form with winners, one branch: sums, extremum, first equal row and tap
    PROBE_F32_WIN_COMPOUND,      // the same for compound (shared sums, two branches)
    PROBE_F32_WIN_PARALLEL,      // the same for parallel (two sets of sums)
    PROBE_BF16X2_FMA_MAX,        // bf16 pairs, every tap sum as fma(x, 1, w) (same rounding, the other pipe)
    PROBE_BF16X2_FMA_MINMAX,
    PROBE_BF16X2_2FMA_MINMAX,
    PROBE_BF16X2_MIX_MAX,        // bf16 pairs, tap sums alternate between add and fma(x, 1, w)
    PROBE_BF16X2_MIX_MINMAX,
    PROBE_BF16X2_2MIX_MINMAX,
    PROBE_COUNT
};

static const char* const kProbeNames[PROBE_COUNT] = {
    "f32_add_max2",       "f32_add_max3",      "f32_add2_max3",   "f32_add_minmax2",
    "f32_add_minmax3",    "f32_add2_minmax3",  "f32_2add_minmax2", "f32_2add_minmax3",
    "f32_2add2_minmax3",  "bf16x2_add_max",    "bf16x2_add_minmax", "bf16x2_2add_minmax",
    "f32_add_only",       "f32_max2_only",     "f32_max3_only",   "f32_win_single",
    "f32_win_compound",   "f32_win_parallel",  "bf16x2_fma_max",  "bf16x2_fma_minmax",
    "bf16x2_2fma_minmax", "bf16x2_mix_max",    "bf16x2_mix_minmax", "bf16x2_2mix_minmax"};

__host__ __device__ constexpr bool probe_is_bf16(int v) {
    return (v >= PROBE_BF16X2_ADD_MAX && v <= PROBE_BF16X2_2ADD_MINMAX) ||
           (v >= PROBE_BF16X2_FMA_MAX && v <= PROBE_BF16X2_2MIX_MINMAX);
}

// Taps folded per thread per loop iteration, by variant (must match the kernel).
__host__ inline int probe_taps_per_iter(int v) {
    if (probe_is_bf16(v)) return 4 * 8 * 2 * 2;               // 4 channel pairs x 8 pixels x 2 lanes x 2 taps
    switch (v) {
        case PROBE_F32_WIN_SINGLE:
        case PROBE_F32_WIN_COMPOUND:
        case PROBE_F32_WIN_PARALLEL: return 4 * 4 * 9;        // 4 channels x 4 pixels x a 3x3 window
        default: return 8 * 4 * 2;                            // 8 channels x 4 pixels x 2 taps
    }
}

template <int V, bool FEED>
__global__ void __launch_bounds__(256) alu_probe_kernel(int iters, float seed, float* sink) {
    constexpr int TK = 8, TP = 4;
    if constexpr (probe_is_bf16(V)) {
        // packed bf16 pairs: a register holds two tap sums.  Three ways to form a tap sum with one
        // bf16 rounding: add.bf16x2, fma.bf16x2(x, 1, w) (the multiply by one is exact, so the
        // result is the same; it issues to the fused-multiply-add pipe), or the two alternating;
        // min / max are nested in pairs so that the assembler may fuse them into 3-input forms.
        constexpr int KP = 4, PX = 8;
        constexpr int KIND = (V >= PROBE_BF16X2_MIX_MAX) ? 2 : (V >= PROBE_BF16X2_FMA_MAX) ? 1 : 0;   // 0 add, 1 fma, 2 mix
        constexpr int BASE = KIND == 2 ? PROBE_BF16X2_MIX_MAX : KIND == 1 ? PROBE_BF16X2_FMA_MAX : PROBE_BF16X2_ADD_MAX;
        constexpr int SHAPE = V - BASE;                                // 0 max, 1 min + max, 2 parallel
        __nv_bfloat162 x[PX + 1], wa[KP], wb[KP], va[KP], vb[KP];
        __nv_bfloat162 mn[KP][PX], mx[KP][PX];
        const __nv_bfloat162 dx2 = __float2bfloat162_rn(seed * 0.0078125f);
        __nv_bfloat162 one2 = __float2bfloat162_rn(1.0f);
        TCONV_OPAQUE_R(*reinterpret_cast<unsigned*>(&one2));
        for (int j = 0; j <= PX; ++j) x[j] = __float2bfloat162_rn(seed * (float)(j + threadIdx.x));
        for (int i = 0; i < KP; ++i) {
            wa[i] = __float2bfloat162_rn(seed * (float)(i + 3));
            wb[i] = __float2bfloat162_rn(seed * (float)(i + 5));
            va[i] = __float2bfloat162_rn(seed * (float)(i + 7));
            vb[i] = __float2bfloat162_rn(seed * (float)(i + 9));
            for (int j = 0; j < PX; ++j) { mn[i][j] = x[j]; mx[i][j] = x[j]; }
        }
        auto tap = [&](const __nv_bfloat162& xv, const __nv_bfloat162& wv, bool second) {
            if (KIND == 1 || (KIND == 2 && second)) return __hfma2(xv, one2, wv);
            return __hadd2(xv, wv);
        };
        for (int it = 0; it < iters; ++it) {
            __nv_bfloat162 xn[PX + 1];                                  // next iteration's operands
            if constexpr (!FEED) {
#pragma unroll
                for (int j = 0; j <= PX; ++j) xn[j] = __hadd2(x[j], dx2);
            }
#pragma unroll
            for (int i = 0; i < KP; ++i) {
                TCONV_OPAQUE_R(*reinterpret_cast<unsigned*>(&wa[i]));
                TCONV_OPAQUE_R(*reinterpret_cast<unsigned*>(&wb[i]));
                TCONV_OPAQUE_R(*reinterpret_cast<unsigned*>(&va[i]));
                TCONV_OPAQUE_R(*reinterpret_cast<unsigned*>(&vb[i]));
            }
#pragma unroll
            for (int i = 0; i < KP; ++i)
#pragma unroll
                for (int j = 0; j < PX; ++j) {
                    const __nv_bfloat162 t0 = tap(x[j], wa[i], false);
                    const __nv_bfloat162 t1 = tap(x[j + 1], wb[i], true);
                    if constexpr (FEED) {
                        if (i == 0) { xn[j] = t0; if (j == PX - 1) xn[PX] = t1; }
                    }
                    if constexpr (SHAPE == 0) {
                        mx[i][j] = __hmax2(__hmax2(mx[i][j], t0), t1);
                    } else if constexpr (SHAPE == 1) {
                        mx[i][j] = __hmax2(__hmax2(mx[i][j], t0), t1);
                        mn[i][j] = __hmin2(__hmin2(mn[i][j], t0), t1);
                    } else {
                        const __nv_bfloat162 u0 = tap(x[j], va[i], true);
                        const __nv_bfloat162 u1 = tap(x[j + 1], vb[i], false);
                        mx[i][j] = __hmax2(__hmax2(mx[i][j], u0), u1);
                        mn[i][j] = __hmin2(__hmin2(mn[i][j], t0), t1);
                    }
                }
#pragma unroll
            for (int j = 0; j <= PX; ++j) x[j] = xn[j];
        }
        __nv_bfloat162 r = mx[0][0];
        for (int i = 0; i < KP; ++i)
            for (int j = 0; j < PX; ++j) r = __hadd2(r, __hadd2(mx[i][j], mn[i][j]));
        if (__low2float(r) == 12345.678f) sink[0] = __high2float(r);
    } else if constexpr (V == PROBE_F32_WIN_SINGLE || V == PROBE_F32_WIN_COMPOUND || V == PROBE_F32_WIN_PARALLEL) {
        // The winner-emitting Sum-form inner loop: per pair of output channels and pixel, nine packed tap sums, their
        // extrema by rows, the channel combine, the winning taps (add_winner) and the code bytes; the inputs in
        // registers, a pass's weights from shared memory as the kernel reads them (another set every other iteration).
        // Parallel: a pass per branch, as the kernel does.  Compound: one pass with both branches, as the kernel does,
        // or (FEED) a pass per branch too, the sums formed anew from a second copy of the weights: the better of the two
        // is what the mix can do (measured 5.68 and 6.04 Ttap/s, parallel 6.04).
        constexpr bool TWOB = (V != PROBE_F32_WIN_SINGLE), PARB = (V == PROBE_F32_WIN_PARALLEL);
        __shared__ __align__(16) float ws[2][2][2][9][2];            // iteration, branch, channel pair, tap, channel
        for (int e = threadIdx.x; e < 2 * 2 * 2 * 9 * 2; e += blockDim.x) {
            const int id = V == PROBE_F32_WIN_COMPOUND ? e / 72 * 36 + e % 36 : e;       // (compound: both branches alike)
            (&ws[0][0][0][0][0])[e] = seed * (float)(id * 37 % 101 + 3);
        }
        __syncthreads();
        float x[12], acc[4][4], al[4], be[4];
        unsigned codes = 0u;
        const float dx = seed * 1.0e-3f;
        for (int j = 0; j < 12; ++j) x[j] = seed * (float)(j + threadIdx.x);
        for (int k = 0; k < 4; ++k) {
            al[k] = seed * (float)(k + 1); be[k] = seed * (float)(k + 2);
            for (int j = 0; j < 4; ++j) acc[k][j] = 0.0f;
        }
#pragma unroll 1
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int j = 0; j < 12; ++j) x[j] = __fadd_rn(x[j], dx);     // operands change every iteration
#pragma unroll
            for (int kp = 0; kp < 2; ++kp) {
                float cnt[2][2] = {{8388608.0f, 8388608.0f}, {8388608.0f, 8388608.0f}};
                auto pass = [&](auto min_branch, auto max_branch, int branch) {
                    constexpr bool DO_MIN = decltype(min_branch)::value, DO_MAX = decltype(max_branch)::value;
                    float wa[9][2];
#pragma unroll
                    for (int t = 0; t < 9; ++t) {
                        const float2 v = *reinterpret_cast<const float2*>(ws[it & 1][branch][kp][t]);
                        wa[t][0] = v.x; wa[t][1] = v.y;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float t[9][2], lo[2] = {0.0f, 0.0f}, hi[2] = {0.0f, 0.0f}, rmin[2][3], rmax[2][3];
#pragma unroll
                        for (int i = 0; i < 9; ++i) add2(x[j + i], wa[i][0], wa[i][1], t[i][0], t[i][1]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const auto th = [&](int i) { return t[i][h]; };
                            if constexpr (DO_MIN) lo[h] = fold_rows<3, 3>(th, true, rmin[h]);
                            if constexpr (DO_MAX) hi[h] = fold_rows<3, 3>(th, false, rmax[h]);
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float& a = acc[2 * kp + h][j];
                            if constexpr (TWOB) {
                                if constexpr (DO_MIN) a = __fmaf_rn(al[2 * kp + h], lo[h], a);
                                if constexpr (DO_MAX) a = __fmaf_rn(be[2 * kp + h], hi[h], a);
                            } else {
                                a = __fadd_rn(a, hi[h]);
                            }
                        }
                        const float unit = j % 2 ? 256.0f : 1.0f;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const auto th = [&](int i) { return t[i][h]; };
                            if constexpr (DO_MIN) add_winner<3, 3>(th, rmin[h], lo[h], unit, cnt[h][j / 2]);
                            if constexpr (DO_MAX) add_winner<3, 3>(th, rmax[h], hi[h], 16.0f * unit, cnt[h][j / 2]);
                        }
                    }
                };
                if constexpr (!TWOB) {
                    pass(std::false_type(), std::true_type(), 0);
                } else if constexpr (PARB || FEED) {
                    pass(std::true_type(), std::false_type(), 0);
                    pass(std::false_type(), std::true_type(), 1);
                } else {
                    pass(std::true_type(), std::true_type(), 0);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) codes ^= __byte_perm(__float_as_uint(cnt[h][0]), __float_as_uint(cnt[h][1]), 0x5410);
            }
        }
        float r = __uint_as_float(codes);
        for (int k = 0; k < 4; ++k)
            for (int j = 0; j < 4; ++j) r += acc[k][j];
        if (r == 12345.678f) sink[0] = r;
    } else {
        float x[TP + 1], w0[TK], w1[TK], v0[TK], v1[TK];
        float mn[TK][TP], mx[TK][TP];
        const float dx = seed * 1.0e-3f;
        for (int j = 0; j <= TP; ++j) x[j] = seed * (float)(j + threadIdx.x);
        for (int i = 0; i < TK; ++i) {
            w0[i] = seed * (float)(i + 3);
            w1[i] = seed * (float)(i + 5);
            v0[i] = seed * (float)(i + 7);
            v1[i] = seed * (float)(i + 9);
            for (int j = 0; j < TP; ++j) { mn[i][j] = x[j]; mx[i][j] = x[j]; }
        }
        for (int it = 0; it < iters; ++it) {
            constexpr bool no_adds = (V == PROBE_F32_MAX2_ONLY || V == PROBE_F32_MAX3_ONLY);
            float xn[TP + 1];                                            // next iteration's operands
            if constexpr (no_adds || !FEED) {
#pragma unroll
                for (int j = 0; j <= TP; ++j) xn[j] = __fadd_rn(x[j], dx);
            }
#pragma unroll
            for (int i = 0; i < TK; ++i) {
                TCONV_OPAQUE_F(w0[i]); TCONV_OPAQUE_F(w1[i]);
                TCONV_OPAQUE_F(v0[i]); TCONV_OPAQUE_F(v1[i]);
            }
            constexpr bool packed = (V == PROBE_F32_ADD2_MAX3 || V == PROBE_F32_ADD2_MINMAX3 ||
                                     V == PROBE_F32_2ADD2_MINMAX3);
            constexpr bool par = (V == PROBE_F32_2ADD_MINMAX2 || V == PROBE_F32_2ADD_MINMAX3 ||
                                  V == PROBE_F32_2ADD2_MINMAX3);
#pragma unroll
            for (int i = 0; i < TK; i += 2)
#pragma unroll
                for (int j = 0; j < TP; ++j) {
                    // two taps (window positions j, j+1) for the channel pair (i, i+1)
                    float ta0, tb0, ta1, tb1;      // min-branch sums: tap 0 / 1, channel i / i+1
                    float ua0, ub0, ua1, ub1;      // max-branch sums (parallel only)
                    if constexpr (V == PROBE_F32_MAX2_ONLY || V == PROBE_F32_MAX3_ONLY) {
                        ta0 = x[j]; tb0 = w0[i]; ta1 = x[j + 1]; tb1 = w1[i + 1];
                    } else if constexpr (packed) {
                        add2(x[j], w0[i], w0[i + 1], ta0, tb0);
                        add2(x[j + 1], w1[i], w1[i + 1], ta1, tb1);
                    } else {
                        ta0 = __fadd_rn(x[j], w0[i]); tb0 = __fadd_rn(x[j], w0[i + 1]);
                        ta1 = __fadd_rn(x[j + 1], w1[i]); tb1 = __fadd_rn(x[j + 1], w1[i + 1]);
                    }
                    if constexpr (par) {
                        if constexpr (packed) {
                            add2(x[j], v0[i], v0[i + 1], ua0, ub0);
                            add2(x[j + 1], v1[i], v1[i + 1], ua1, ub1);
                        } else {
                            ua0 = __fadd_rn(x[j], v0[i]); ub0 = __fadd_rn(x[j], v0[i + 1]);
                            ua1 = __fadd_rn(x[j + 1], v1[i]); ub1 = __fadd_rn(x[j + 1], v1[i + 1]);
                        }
                    } else {
                        ua0 = ta0; ub0 = tb0; ua1 = ta1; ub1 = tb1;
                    }
                    if constexpr (!no_adds && FEED) {
                        if (i == 0) { xn[j] = ta0; if (j == TP - 1) xn[TP] = ta1; }
                    }
                    if constexpr (V == PROBE_F32_ADD_ONLY) {
                        mx[i][j] += ta0 + ta1;          // 4 adds per 2 taps: an upper bound
                        mx[i + 1][j] += tb0 + tb1;      // on what the FP32 pipe sustains
                    } else if constexpr (V == PROBE_F32_ADD_MAX2 || V == PROBE_F32_MAX2_ONLY) {
                        mx[i][j] = fmaxf(fmaxf(mx[i][j], ta0), ta1);
                        mx[i + 1][j] = fmaxf(fmaxf(mx[i + 1][j], tb0), tb1);
                    } else if constexpr (V == PROBE_F32_ADD_MAX3 || V == PROBE_F32_ADD2_MAX3 ||
                                         V == PROBE_F32_MAX3_ONLY) {
                        mx[i][j] = ext3(mx[i][j], ta0, ta1, false);
                        mx[i + 1][j] = ext3(mx[i + 1][j], tb0, tb1, false);
                    } else if constexpr (V == PROBE_F32_ADD_MINMAX2 || V == PROBE_F32_2ADD_MINMAX2) {
                        mx[i][j] = fmaxf(fmaxf(mx[i][j], ua0), ua1);
                        mx[i + 1][j] = fmaxf(fmaxf(mx[i + 1][j], ub0), ub1);
                        mn[i][j] = fminf(fminf(mn[i][j], ta0), ta1);
                        mn[i + 1][j] = fminf(fminf(mn[i + 1][j], tb0), tb1);
                    } else {
                        mx[i][j] = ext3(mx[i][j], ua0, ua1, false);
                        mx[i + 1][j] = ext3(mx[i + 1][j], ub0, ub1, false);
                        mn[i][j] = ext3(mn[i][j], ta0, ta1, true);
                        mn[i + 1][j] = ext3(mn[i + 1][j], tb0, tb1, true);
                    }
                }
#pragma unroll
            for (int j = 0; j <= TP; ++j) x[j] = xn[j];
        }
        float r = 0.0f;
        for (int i = 0; i < TK; ++i)
            for (int j = 0; j < TP; ++j) r += mx[i][j] + mn[i][j];
        if (r == 12345.678f) sink[0] = r;
    }
}

}  // namespace tconv
