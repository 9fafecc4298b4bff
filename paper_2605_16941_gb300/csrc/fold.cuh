// fold.cuh -- the running softmax state of one scored row and the fold of 32 logits into it, shared by the two
// score kernels (score.cu, score_vmajor.cu).
#pragma once

#include <cstdint>

#include "ptx.cuh"

namespace wino {

constexpr float kLog2e = 1.4426950408889634f;

// Running softmax state of one row (one thread).
struct RowState {
    float m, s0, s1, s2, s3, tlog;
    float u0, u1, u2, u3;  // entropy variant: sum of exp(l - m) (l - m) log2(e)
    int32_t am;
};

// The fold of 32 logits is the score kernels' epilogue; its instruction count sets their time at small d.  Two
// exponents' FMAs and two sums' additions go in one packed instruction (same rounding as scalar ones), the maximum is a
// tree of three-operand maxima, and the argmax, needed whenever the maximum moves (most chunks of a short sweep), is
// searched only in the first group of 8 that holds it (44 instructions instead of 67: d = 256, V = 64000, N = 2048 76.0
// -> 74.0 us per step; with scalar FMAs, additions and maxima 89.5).
//
// Fold 32 consecutive logits x (columns v .. v + 31; those at or past cvalid are not logits) into the row
// state: online max with rescaling, four partial sums of 2^((l - m) log2 e), argmax (an earlier column
// keeps it on ties), and the target's logit when it lies among them.
template <bool kEntropy>
__device__ __forceinline__ void fold32(RowState &r, float (&x)[32], int v, int cvalid, int tgt)
{
    if (cvalid < 32) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j >= cvalid)
                x[j] = -INFINITY;  // past V (TMA zero fill) or past the tile (another tile's columns)
    }
    float c4[4];  // the maxima of 8 columns each
#pragma unroll
    for (int g = 0; g < 4; ++g)
        c4[g] = fmaxf(ptx::max3(x[8 * g], x[8 * g + 1], x[8 * g + 2]),
                      ptx::max3(ptx::max3(x[8 * g + 3], x[8 * g + 4], x[8 * g + 5]), x[8 * g + 6], x[8 * g + 7]));
    const float cm = fmaxf(ptx::max3(c4[0], c4[1], c4[2]), c4[3]);
    if (cm > r.m) {  // strict: an earlier column keeps the argmax on ties
        // the first group of 8 that holds the maximum, then the first of its columns
        const bool g0 = c4[0] == cm, g1 = c4[1] == cm, g2 = c4[2] == cm;
        int j0 = 7;
#pragma unroll
        for (int j = 6; j >= 0; --j) {
            const float y = g0 ? x[j] : (g1 ? x[8 + j] : (g2 ? x[16 + j] : x[24 + j]));
            if (y == cm)
                j0 = j;
        }
        r.am = v + j0 + (g0 ? 0 : (g1 ? 8 : (g2 ? 16 : 24)));
        const float scale = ptx::ex2((r.m - cm) * kLog2e);
        if (kEntropy && r.m != -INFINITY) {  // u' = scale * (u + (m - cm) log2(e) * s)
            const float dl = (r.m - cm) * kLog2e;
            r.u0 = scale * fmaf(dl, r.s0, r.u0);
            r.u1 = scale * fmaf(dl, r.s1, r.u1);
            r.u2 = scale * fmaf(dl, r.s2, r.u2);
            r.u3 = scale * fmaf(dl, r.s3, r.u3);
        }
        r.s0 *= scale;
        r.s1 *= scale;
        r.s2 *= scale;
        r.s3 *= scale;
        r.m = cm;
    }
    const float mb2 = r.m * kLog2e;
    const float2 l2e = make_float2(kLog2e, kLog2e), nmb2 = make_float2(-mb2, -mb2);
    float2 s01 = make_float2(r.s0, r.s1), s23 = make_float2(r.s2, r.s3);
    float2 u01 = make_float2(r.u0, r.u1), u23 = make_float2(r.u2, r.u3);
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        float2 t01 = ptx::fma2(make_float2(x[j + 0], x[j + 1]), l2e, nmb2);
        float2 t23 = ptx::fma2(make_float2(x[j + 2], x[j + 3]), l2e, nmb2);
        if (kEntropy) {  // t = (l - m) log2(e), kept finite (masked columns are -inf; 2^-200 is 0 in fp32 anyway)
            t01 = make_float2(fmaxf(t01.x, -200.f), fmaxf(t01.y, -200.f));
            t23 = make_float2(fmaxf(t23.x, -200.f), fmaxf(t23.y, -200.f));
        }
        const float2 e01 = make_float2(ptx::ex2(t01.x), ptx::ex2(t01.y));
        const float2 e23 = make_float2(ptx::ex2(t23.x), ptx::ex2(t23.y));
        s01 = ptx::add2(s01, e01);
        s23 = ptx::add2(s23, e23);
        if (kEntropy) {
            u01 = ptx::fma2(e01, t01, u01);
            u23 = ptx::fma2(e23, t23, u23);
        }
    }
    r.s0 = s01.x;
    r.s1 = s01.y;
    r.s2 = s23.x;
    r.s3 = s23.y;
    if (kEntropy) {
        r.u0 = u01.x;
        r.u1 = u01.y;
        r.u2 = u23.x;
        r.u3 = u23.y;
    }
    const int tj = tgt - v;
    if ((unsigned)tj < 32u) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            r.tlog = (j == tj) ? x[j] : r.tlog;
    }
}

// Fold the softmax state (m2, s2, i2) into (m, s, i): the larger max wins, the smaller index on equal maxima.
__device__ __forceinline__ void combine(float &m, float &s, int32_t &i, float m2, float s2, int32_t i2)
{
    const float M = fmaxf(m, m2);
    const float a = (m == -INFINITY) ? 0.f : s * ptx::ex2((m - M) * kLog2e);
    const float b = (m2 == -INFINITY) ? 0.f : s2 * ptx::ex2((m2 - M) * kLog2e);
    if (m2 > m || (m2 == m && i2 < i))
        i = i2;
    m = M;
    s = a + b;
}

// As combine, also folding u = sum exp(l - m) (l - m) log2(e) (rescaled to the new max like s).
__device__ __forceinline__ void combine_u(float &m, float &s, float &u, int32_t &i, float m2, float s2, float u2,
                                          int32_t i2)
{
    const float M = fmaxf(m, m2);
    float a = 0.f, b = 0.f, ua = 0.f, ub = 0.f;
    if (m != -INFINITY) {
        const float al = ptx::ex2((m - M) * kLog2e);
        a = s * al;
        ua = al * fmaf((m - M) * kLog2e, s, u);
    }
    if (m2 != -INFINITY) {
        const float bl = ptx::ex2((m2 - M) * kLog2e);
        b = s2 * bl;
        ub = bl * fmaf((m2 - M) * kLog2e, s2, u2);
    }
    if (m2 > m || (m2 == m && i2 < i))
        i = i2;
    m = M;
    s = a + b;
    u = ua + ub;
}

}  // namespace wino
