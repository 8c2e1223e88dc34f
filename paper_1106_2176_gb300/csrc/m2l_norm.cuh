// Powers of two that bring the operands of the tensor-core M2L into the range
// of FP16 (all exact): the factor of a coefficient and the scale
// of a level's rows.
#pragma once

#include <cstdint>

namespace fmm {

constexpr int m2l_degree(int k)  // of packed coefficient k (degree n at offset n^2: (n, 0), then Re and Im of (n, m))
{
    int n = 0;
    while ((n + 1) * (n + 1) <= k) n++;
    return n;
}

// round(log2 sqrt((n+m)! (n-m)!)): the factorials of the solid harmonics,
// |R_n^m| <= r^n / sqrt((n+m)! (n-m)!)
constexpr int m2l_fact_exp(int k)
{
    const int n = m2l_degree(k), m = (k - n * n + 1) / 2;
    double x = 1.0;
    for (int i = 2; i <= n + m; i++) x *= i;
    for (int i = 2; i <= n - m; i++) x *= i;
    int e = 0;
    while (x >= 2.0) {
        x /= 4.0;
        e++;
    }
    return e;
}

// log2 of the factor a of a coefficient of M~: the factorials, and 2^-n
constexpr int m2l_norm_exp(int k) { return m2l_fact_exp(k) - m2l_degree(k); }

constexpr int M2L_NORM_N = 128;  // p <= 11: 121 coefficients

struct M2LNorm {
    float a[M2L_NORM_N];
};

constexpr M2LNorm m2l_norm_make()
{
    M2LNorm t{};
    for (int k = 0; k < M2L_NORM_N; k++) {
        float f = 1.f;
        for (int e = m2l_norm_exp(k); e > 0; e--) f *= 2.f;
        for (int e = m2l_norm_exp(k); e < 0; e++) f *= 0.5f;
        t.a[k] = f;
    }
    return t;
}

static __constant__ M2LNorm c_m2l_norm = m2l_norm_make();

__device__ __forceinline__ float m2l_norm(int k) { return c_m2l_norm.a[k]; }

// |x| as bits, in the order of the floats; 0 for infinities and NaN, which do
// not set a level's scale
__device__ __forceinline__ unsigned m2l_mag(float x)
{
    const unsigned b = __float_as_uint(x) & 0x7fffffffu;
    return b < 0x7f800000u ? b : 0u;
}

// the exponent e of a level's scale 2^e: its largest coefficient then lies in
// [2^14, 2^15) (none: 0)
__device__ __forceinline__ int m2l_exponent(unsigned mag)
{
    const int e = (int)(mag >> 23);
    return e == 0 ? 0 : 14 - (e - 127);
}

// 2^e, -126 <= e <= 127
__device__ __forceinline__ float m2l_pow2(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }

// the row maximum of one cell (by one warp, after its row is written) to *cmax
// and into its level's: a plain read first, so that almost no cell needs the atomic
__device__ __forceinline__ void m2l_row_max(const float *Mc, int PP, int lane, unsigned *cmax, unsigned *lmax)
{
    unsigned best = 0;
    for (int k = lane; k < PP; k += 32) best = max(best, m2l_mag(__ldcg(Mc + k) * m2l_norm(k)));
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane != 0) return;
    *cmax = best;
    if (best > *(volatile unsigned *)lmax) atomicMax(lmax, best);
}

// Workspace of one evaluation, zero before it: the level maxima (word l), which
// levels are wide (bit l), and the tiles' counters.
constexpr int M2LW_WIDE = 24, M2LW_CNT = 32;

// FP16 rounds a row scaled with its level to 2^-40 of the level's largest
// coefficient: a cell within 2^-16 of it keeps 2^-24 of its own largest
// coefficient, FP32's rounding, a lower one fewer bits.
constexpr int M2L_SPAN = 16;

// Whether the lost bits may show at a target cell c of level l: an expansion whose
// largest coefficient is a is a potential of about a / w one cell width w away, so
// the potential at c is about the largest a / w of c and its ancestors (the root's:
// the whole system as seen from afar) or more, and FP32 leaves 2^-24 of that open
// anyway. Exposed: 2^-16 of the level's largest a / w and less. (N = 10^6 Plummer:
// 43 of 60,000 cells lie 2^-16 and more below their level's largest; none is exposed.)
__device__ inline bool m2l_exposed(int c, int l, unsigned lmax, const unsigned *cmax, const int *parent)
{
    const int need = (int)(lmax >> 23) - M2L_SPAN + l;
    if ((int)(cmax[c] >> 23) + l > need || (int)(cmax[0] >> 23) > need) return false;
    for (int a = parent[c], la = l - 1; a > 0; a = parent[a], la--)
        if ((int)(cmax[a] >> 23) + la > need) return false;
    return true;
}

// marks cell c's level l in the workspace (and *any) if it is exposed
__device__ inline void m2l_mark(int c, int l, const unsigned *cmax, const int *parent, unsigned *ws, unsigned *any)
{
    const unsigned lm = ws[l];
    if ((int)(lm >> 23) - (int)(cmax[c] >> 23) < M2L_SPAN || ((*(volatile unsigned *)(ws + M2LW_WIDE) >> l) & 1u)) return;
    if (!m2l_exposed(c, l, lm, cmax, parent)) return;
    atomicOr(ws + M2LW_WIDE, 1u << l);
    if (any) atomicOr(any, 1u);
}

}  // namespace fmm
