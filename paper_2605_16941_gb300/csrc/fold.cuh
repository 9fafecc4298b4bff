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
    float cm = x[0];
#pragma unroll
    for (int j = 1; j < 32; ++j)
        cm = fmaxf(cm, x[j]);
    if (cm > r.m) {  // strict: an earlier column keeps the argmax on ties
        int j0 = 31;
#pragma unroll
        for (int j = 31; j >= 0; --j)
            if (x[j] == cm)
                j0 = j;
        r.am = v + j0;
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
    if (!kEntropy) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            r.s0 += ptx::ex2(fmaf(x[j + 0], kLog2e, -mb2));
            r.s1 += ptx::ex2(fmaf(x[j + 1], kLog2e, -mb2));
            r.s2 += ptx::ex2(fmaf(x[j + 2], kLog2e, -mb2));
            r.s3 += ptx::ex2(fmaf(x[j + 3], kLog2e, -mb2));
        }
    } else {
        // t = (l - m) log2(e), kept finite (masked columns are -inf; 2^-200 is 0 in fp32 anyway)
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const float t0 = fmaxf(fmaf(x[j + 0], kLog2e, -mb2), -200.f);
            const float t1 = fmaxf(fmaf(x[j + 1], kLog2e, -mb2), -200.f);
            const float t2 = fmaxf(fmaf(x[j + 2], kLog2e, -mb2), -200.f);
            const float t3 = fmaxf(fmaf(x[j + 3], kLog2e, -mb2), -200.f);
            const float e0 = ptx::ex2(t0), e1 = ptx::ex2(t1), e2 = ptx::ex2(t2), e3 = ptx::ex2(t3);
            r.s0 += e0;
            r.s1 += e1;
            r.s2 += e2;
            r.s3 += e3;
            r.u0 = fmaf(e0, t0, r.u0);
            r.u1 = fmaf(e1, t1, r.u1);
            r.u2 = fmaf(e2, t2, r.u2);
            r.u3 = fmaf(e3, t3, r.u3);
        }
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
