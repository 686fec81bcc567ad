// Device code of the structured Pauli contraction shared by its projection kernel
// (project_pauli.cu, where the method is described) and the kernel that runs many steps of a small
// problem (fused_small.cu).
#pragma once

#include "qst_internal.cuh"
#include "f32x2.cuh"

namespace qst {

struct PauliArgs {
    const float *A;          // [rows][d_pad] packed rho
    const float4 *wq;        // [18][6^(Q-2)] (w, w, a, a) of output pair 2 j, 2 j + 1 of block p at [j][p]
    const float2 *wc;        // [18][6^(Q-2)] their counts
    const int32_t *perm;     // [36][6^(Q-2)] output k of block p -> setting-major projector index, at [k][p] (Q = 1: [6])
    const float *ptot;       // [3^Q] shots P_k of setting k
    double *out;             // [rows] the deviance sum (one column group)
    float *p_out;            // [rows][KD] (P_OUT only): p = q / t
    const double *trace;     // [rows] exact trace of the stored rho (P_OUT only)
    int64_t rows;
    int d_pad, KD;
    int poisson;             // 1: each setting adds -mu_k (S_k / t - 1) (Poisson; S_k / t - 1 is a few ulps
                             // here, the Pauli settings being complete) instead of -P_k log(S_k / t)
};

// The six children of one split at an entry: s = A + C, x = B + B^dag, y = i(B - B^dag) there.
__device__ __forceinline__ void six(float s, float x, float y, float a, float c, float o[6]) {
    o[0] = 0.5f * (s + x);
    o[1] = 0.5f * (s - x);
    o[2] = 0.5f * (s + y);
    o[3] = 0.5f * (s - y);
    o[4] = a;
    o[5] = c;
}

// The last split of one 2 x 2 block [[e00, Re b], [Im b*, e11]] and the deviance terms of its
// six outputs, pairs j0 .. j0 + 2 of this thread's weights: (S +- 2 Re b), (S +- 2 Im b*) are
// 2 q of X+- and Y+- (the 1/2 sits in their weights), (e00, e11) are q of Z+-.
template <bool P_OUT>
__device__ __forceinline__ void last_split(float e00, float e01, float e10, float e11, const PauliArgs &a, int j0,
                                           int stride, int blk, float2 &dev, float2 &comp, int &xmin,
                                           float (&sh)[3], float (&sl)[3], float *p_row, int o0, float inv_t) {
    float4 wq[3];   // the three pairs' weights, requested before the arithmetic that needs them
    float2 wc[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        wq[j] = a.wq[(j0 + j) * stride + blk];
        wc[j] = a.wc[(j0 + j) * stride + blk];
    }
    const float S = e00 + e11;
    const float2 q2[3] = {fma2(splat2(e01), make_float2(2.0f, -2.0f), splat2(S)),
                          fma2(splat2(e10), make_float2(2.0f, -2.0f), splat2(S)), make_float2(e00, e11)};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float4 w = wq[j];
        const float2 cnt = wc[j];
        const float2 x = fma2(q2[j], make_float2(w.x, w.y), make_float2(w.z, w.w));
        xmin = min(xmin, min(__float_as_int(x.x), __float_as_int(x.y)));
        kahan_fma2(dev, comp, cnt, log_poly2(x));   // compensated: far from the posterior the terms are O(c)
        // the setting sum of this pair's q (2 q for X, Y): high parts on the grid, exactly
        const float2 C = splat2(j < 2 ? 24.0f : 12.0f);
        const float2 hq = sub2(add2(q2[j], C), C), lq = sub2(q2[j], hq);
        sh[j] += hq.x + hq.y;
        sl[j] += lq.x + lq.y;
        if constexpr (P_OUT) {
            if (p_row) {
                const float h = j < 2 ? 0.5f : 1.0f;
                p_row[a.perm[(o0 + 2 * j) * stride + blk]] = h * q2[j].x * inv_t;
                p_row[a.perm[(o0 + 2 * j + 1) * stride + blk]] = h * q2[j].y * inv_t;
            }
        }
    }
}

}  // namespace qst
