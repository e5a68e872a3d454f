// Launches of the Sum-form backward kernels (tconv_bwd_sum.cuh).
#include <algorithm>

#include "tconv_bwd_sum.cuh"

namespace tconv {
namespace {

template <typename T, int BR, bool GX, bool AB, bool WIDE, int KW, bool TAIL>
int launch_gx(SumBwdArgs& a, const SumGxPlan& pl, float* part_ab, float* part_gx) {
    auto kern = bwd_sum_gx_kernel<T, BR, GX, AB, WIDE, KW, TAIL>;
    if (allow_smem(kern, kSgSmemAttr) != cudaSuccess) return TCONV_ERR_CUDA;
    kern<<<pl.ctas * (unsigned)a.g.C, pl.threads, pl.smem, a.st>>>(
        a.g, a.x, (const T*)a.w, (const T*)a.w2, a.alpha, a.beta, (const T*)a.gy, a.codes, (T*)a.gx, part_ab, part_gx, pl);
    ++a.launches;
    return TCONV_OK;
}
// 3 x 3 and 5 x 5 windows have instances of their own (constant address offsets, unrolled windows).
template <typename T, int BR, bool GX, bool AB>
int launch_gx_window(SumBwdArgs& a, const SumGxPlan& pl, float* part_ab, float* part_gx) {
    const Geo& g = a.g;
    const bool far = sum_far(g);
    if (g.wide) return g.R == 5 && g.S == 5 && !far ? launch_gx<T, BR, GX, AB, true, 5, true>(a, pl, part_ab, part_gx)
                                                    : launch_gx<T, BR, GX, AB, true, 0, true>(a, pl, part_ab, part_gx);
    if (g.R != 3 || g.S != 3 || far) return launch_gx<T, BR, GX, AB, false, 0, true>(a, pl, part_ab, part_gx);
    return g.K % kSgKB ? launch_gx<T, BR, GX, AB, false, 3, true>(a, pl, part_ab, part_gx)
                       : launch_gx<T, BR, GX, AB, false, 3, false>(a, pl, part_ab, part_gx);
}

template <typename T, int BR, bool PAIRS, bool WIDE>
int launch_gw(SumBwdArgs& a, const SumGwPlan& pl, float* part) {
    // fp32, one branch, wide codes: the loop over whole blocks takes 72 registers, seven CTAs an SM where the plan counts on
    // eight, the loop over whole rounds 60.  Where that second round of CTAs is the price and shares are long, whole rounds:
    // 24 -> 6 channels 5x5 128x256 N=25 (1116 CTAs of 208 rounds) 81 against 64 us, 64 -> 72 32x32 N=64 (1152 of 512) 186
    // against 149, 24 -> 24 32x64 N=32 (1152 of 64) 27.7 against 25.5; else blocks: 13 -> 29 16x96 N=50 (1131 of 52) 19.3
    // against 21.4, 64 -> 64 64x64 N=4 (8192 of 16) 50 against 52.  Blocks within 64 registers spill: 72, 169 and 27.5 us.
    const bool second = sizeof(T) == 4 && WIDE && BR != 0 && pl.grid > 148 * 7 && pl.grid <= 148 * 8 && pl.per >= 64;
    auto kern = pl.flat ? bwd_sum_gw_kernel<T, BR, PAIRS, WIDE, true, false>
                : pl.blocks && !second ? bwd_sum_gw_kernel<T, BR, PAIRS, WIDE, false, true> : bwd_sum_gw_kernel<T, BR, PAIRS, WIDE, false, false>;
    if (allow_smem(kern, kBwdSmemAttr) != cudaSuccess) return TCONV_ERR_CUDA;
    kern<<<pl.grid, 128, pl.smem, a.st>>>(a.g, (const T*)a.gy, a.codes, part, pl);
    ++a.launches;
    return TCONV_OK;
}
template <typename T, int BR>
int launch_gw_window(SumBwdArgs& a, const SumGwPlan& pl, float* part) {
    if (a.g.wide) return launch_gw<T, BR, false, true>(a, pl, part);
    if (BR == 0 && pl.pairs) return launch_gw<T, BR, BR == 0, false>(a, pl, part);
    return launch_gw<T, BR, false, false>(a, pl, part);
}

template <typename T>
int launch_all(SumBwdArgs& a) {
    const Geo& g = a.g;
    const SumPlans& plans = sum_plans(g, (int)sizeof(T));
    if (!plans.ok) return TCONV_ERR_UNSUPPORTED;
    const SumGxPlan& xp = plans.gx;
    const SumGwPlan& gp = plans.gw;
    const bool two = two_branch(g.mode);
    const int br = two ? 0 : (g.mode == TCONV_MIN_PLUS ? 1 : 2);
    const bool ab = two && (a.galpha || a.gbeta), params = a.gw || a.gw2 || a.gbias || ab;
    float* part = a.ws;
    float* part_ab = a.ws + sum_part_gw_bytes(g, gp) / sizeof(float);
    float* part_gx = part_ab + sum_part_ab_bytes(g, xp) / sizeof(float);
    int rc = TCONV_OK;
    if (ab) rc = a.gx ? launch_gx_window<T, 0, true, true>(a, xp, part_ab, part_gx) : launch_gx_window<T, 0, false, true>(a, xp, part_ab, part_gx);
    else if (a.gx) rc = br == 0 ? launch_gx_window<T, 0, true, false>(a, xp, part_ab, part_gx)
                        : br == 1 ? launch_gx_window<T, 1, true, false>(a, xp, part_ab, part_gx) : launch_gx_window<T, 2, true, false>(a, xp, part_ab, part_gx);
    if (rc == TCONV_OK && a.gx && xp.nrow * xp.ncol > 1) {
        const unsigned tasks = (unsigned)((g.H + 3) / 4) * (unsigned)((g.W + 31) / 32);
        bwd_sum_edges_kernel<T><<<dim3((unsigned)(g.N * g.C), std::min((tasks + 7) / 8, 65535u)), 256, 0, a.st>>>(g, part_gx, (T*)a.gx, xp);
        ++a.launches;
    }
    if (rc != TCONV_OK || !params) return rc;
    rc = br == 0 ? launch_gw_window<T, 0>(a, gp, part) : br == 1 ? launch_gw_window<T, 1>(a, gp, part) : launch_gw_window<T, 2>(a, gp, part);
    if (rc != TCONV_OK) return rc;
    const size_t pairs = (size_t)g.K * g.C;
    // slices of the splits: a power of two, about eight splits each
    int ws = 1;
    while (ws < 32 && ws * 8 < gp.splits) ws *= 2;
    // sixteen slices of the rows of grad_alpha / grad_beta; one where a slice would hold one row at most and the entries
    // fill the SMs (512 x 512 channels 7 x 7, four rows: 55 -> 24 us; the order of the sums is the same)
    const int as = xp.ctas <= 16 && pairs >= 148 * 256 ? 1 : 16;
    const unsigned nb_w = a.gw || a.gw2 ? (unsigned)((pairs * g.RS * ws + 255) / 256) : 0u, nb_ab = ab ? (unsigned)((pairs * as + 255) / 256) : 0u;
    const unsigned nb_bias = a.gbias ? (unsigned)((g.K + 7) / 8) : 0u;
    auto finish = as == 1 ? bwd_sum_finish_kernel<1> : bwd_sum_finish_kernel<16>;
    finish<<<nb_w + nb_ab + nb_bias, 256, 0, a.st>>>(g, br, gp.splits, part, (int)xp.ctas, part_ab, a.alpha, a.beta, a.gw, a.gw2,
                                                     a.galpha, a.gbeta, a.gbias, nb_w, nb_ab, ws);
    ++a.launches;
    return TCONV_OK;
}

}  // namespace

int bwd_sum_launch(SumBwdArgs& a) {
    return a.dtype == TCONV_F32 ? launch_all<float>(a) : launch_all<__nv_bfloat16>(a);
}

}  // namespace tconv
