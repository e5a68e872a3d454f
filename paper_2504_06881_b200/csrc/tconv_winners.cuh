// Extrema of fp32 tap sums and their winning taps, on registers.
#pragma once

namespace tconv {

__device__ __forceinline__ float ext3(float a, float b, float c, bool is_min) {
    float d;
    if (is_min) asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    else asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float ext2(float a, float b, bool is_min) {
    return is_min ? fminf(a, b) : fmaxf(a, b);
}
// {lo, hi} = {x + wlo, x + whi}: one packed fp32 add for two output channels.
__device__ __forceinline__ void add2(float x, float wlo, float whi, float& lo, float& hi) {
    unsigned long long xx, ww, tt;
    asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ww) : "f"(wlo), "f"(whi));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(tt) : "l"(xx), "l"(ww));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(tt));
}
// Extremum of N values (N odd) with 3-input min / max: a fresh chain opens with three values, every later step folds two more.
template <int N>
__device__ __forceinline__ float fold_values(const float* v, bool is_min) {
    static_assert(N % 2 == 1, "windows of 1, 3 or 5");
    float m = v[0];
#pragma unroll
    for (int i = 1; i < N; i += 2) m = ext3(m, v[i], v[i + 1], is_min);
    return m;
}
// Extremum of the R x S tap sums t(.), row by row; row[r] keeps the rows' own.
template <int R, int S, typename Taps>
__device__ __forceinline__ float fold_rows(Taps t, bool is_min, float* row) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float v[S];
#pragma unroll
        for (int i = 0; i < S; ++i) v[i] = t(r * S + i);
        row[r] = fold_values<S>(v, is_min);
    }
    return fold_values<R>(row, is_min);
}
// Adds unit times the lowest tap whose sum equals the extremum m to code: the first row whose extremum is m, by
// selection that row's taps but the last, and the first of them that is m.  The row and column counts go to code as
// predicated adds (FMA pipe: the compares and selects keep the half-rate pipe busy).  Comparisons only, so any
// finite or infinite sums do; a NaN (a tap in neutral padding) equals nothing.
template <int R, int S, typename Taps>
__device__ __forceinline__ void add_winner(Taps t, const float* row, float m, float unit, float& code) {
    static_assert((R == 1 && S == 3) || (R == 3 && S == 3) || (R == 5 && S == 5), "windows of the tiled kernels");
    if constexpr (R == 1) {
        asm("{\n\t.reg .pred q0, q1;\n\t"
            "setp.neu.f32 q0, %1, %3;\n\t"
            "setp.neu.and.f32 q1, %2, %3, q0;\n\t"
            "@q0 add.rn.f32 %0, %0, %4;\n\t"
            "@q1 add.rn.f32 %0, %0, %4;\n\t}"
            : "+f"(code) : "f"(t(0)), "f"(t(1)), "f"(m), "f"(unit));
    } else if constexpr (R == 3) {
        asm("{\n\t.reg .pred p0, p1, q0, q1;\n\t.reg .f32 u0, u1;\n\t"
            "setp.neu.f32 p0, %1, %3;\n\t"
            "setp.neu.and.f32 p1, %2, %3, p0;\n\t"
            "selp.f32 u0, %6, %4, p0;\n\t"
            "selp.f32 u1, %7, %5, p0;\n\t"
            "selp.f32 u0, %8, u0, p1;\n\t"
            "selp.f32 u1, %9, u1, p1;\n\t"
            "setp.neu.f32 q0, u0, %3;\n\t"
            "setp.neu.and.f32 q1, u1, %3, q0;\n\t"
            "@p0 add.rn.f32 %0, %0, %11;\n\t"
            "@p1 add.rn.f32 %0, %0, %11;\n\t"
            "@q0 add.rn.f32 %0, %0, %10;\n\t"
            "@q1 add.rn.f32 %0, %0, %10;\n\t}"
            : "+f"(code)
            : "f"(row[0]), "f"(row[1]), "f"(m), "f"(t(0)), "f"(t(1)), "f"(t(3)), "f"(t(4)), "f"(t(6)), "f"(t(7)),
              "f"(unit), "f"(3.0f * unit));
    } else {
        asm("{\n\t.reg .pred p0, p1, p2, p3;\n\t.reg .f32 u0, u1, u2, u3, five;\n\t"
            "mul.rn.f32 five, %6, 0f40A00000;\n\t"
            "setp.neu.f32 p0, %1, %5;\n\t"
            "setp.neu.and.f32 p1, %2, %5, p0;\n\t"
            "setp.neu.and.f32 p2, %3, %5, p1;\n\t"
            "setp.neu.and.f32 p3, %4, %5, p2;\n\t"
            "selp.f32 u0, %11, %7, p0;\n\tselp.f32 u1, %12, %8, p0;\n\tselp.f32 u2, %13, %9, p0;\n\tselp.f32 u3, %14, %10, p0;\n\t"
            "selp.f32 u0, %15, u0, p1;\n\tselp.f32 u1, %16, u1, p1;\n\tselp.f32 u2, %17, u2, p1;\n\tselp.f32 u3, %18, u3, p1;\n\t"
            "selp.f32 u0, %19, u0, p2;\n\tselp.f32 u1, %20, u1, p2;\n\tselp.f32 u2, %21, u2, p2;\n\tselp.f32 u3, %22, u3, p2;\n\t"
            "selp.f32 u0, %23, u0, p3;\n\tselp.f32 u1, %24, u1, p3;\n\tselp.f32 u2, %25, u2, p3;\n\tselp.f32 u3, %26, u3, p3;\n\t"
            "@p0 add.rn.f32 %0, %0, five;\n\t@p1 add.rn.f32 %0, %0, five;\n\t@p2 add.rn.f32 %0, %0, five;\n\t@p3 add.rn.f32 %0, %0, five;\n\t"
            "setp.neu.f32 p0, u0, %5;\n\t"
            "setp.neu.and.f32 p1, u1, %5, p0;\n\t"
            "setp.neu.and.f32 p2, u2, %5, p1;\n\t"
            "setp.neu.and.f32 p3, u3, %5, p2;\n\t"
            "@p0 add.rn.f32 %0, %0, %6;\n\t@p1 add.rn.f32 %0, %0, %6;\n\t@p2 add.rn.f32 %0, %0, %6;\n\t@p3 add.rn.f32 %0, %0, %6;\n\t}"
            : "+f"(code)
            : "f"(row[0]), "f"(row[1]), "f"(row[2]), "f"(row[3]), "f"(m), "f"(unit),
              "f"(t(0)), "f"(t(1)), "f"(t(2)), "f"(t(3)), "f"(t(5)), "f"(t(6)), "f"(t(7)), "f"(t(8)),
              "f"(t(10)), "f"(t(11)), "f"(t(12)), "f"(t(13)), "f"(t(15)), "f"(t(16)), "f"(t(17)), "f"(t(18)),
              "f"(t(20)), "f"(t(21)), "f"(t(22)), "f"(t(23)));
    }
}

}  // namespace tconv
