// Device code of the proposal and Algorithm 1 shared by the per-step proposal kernels (propose.cu)
// and the kernel that runs many steps of a small problem (fused_small.cu): the shared-memory layout
// of a chain, Box-Muller, column moves, exact sums and the refinement of U.
#pragma once

#include "qst_internal.cuh"
#include "f32x2.cuh"

namespace qst {

constexpr int kProposeThreads = 128;
// the refinement of U (PASSES = 3): at most this many first-order passes, another one while the
// chain's largest |Y| entry exceeds kRefineTol (the residual of a pass is about |Y|^2)
constexpr int kRefinePasses = 3;
constexpr float kRefineTol = 0x1p-13f;

// The refinement keeps Q's and H's columns unpadded at D = 16 (16 floats each, so that five CTAs
// fit on an SM), where the 16 lanes of a chain reaching block b of their own columns would hit
// 8 of the 32 banks.  So block b (4 floats) of Q's column c is stored at b ^ ((c >> 1) & 3), and
// of H's column c at b ^ ((c >> 1) & 3) ^ 2: a chain's lanes then cover all 32 banks, and the Q
// and H columns of one index, which the refinement's products read side by side, never share
// banks.  Within a block the order is kept, so every value and every result is unchanged.
// (QC == D only for that layout; every other one is padded and unswizzled.)
template <int D, int QC>
__device__ __forceinline__ int qsw(int c) { return (QC == D && D == 16) ? ((c >> 1) & 3) : 0; }
template <int D, int QC>
__device__ __forceinline__ int hsw(int c) { return (QC == D && D == 16) ? (((c >> 1) & 3) ^ 2) : 0; }

// Shared memory per chain (floats), laid out so every access is free of bank conflicts:
//   area A: the real and imaginary planes of H's columns as they are orthogonalised (column
//           stride D + 4, so that 128-bit accesses of eight consecutive lanes' columns hit
//           different banks) -> W row-major (complex, rows padded to D + 2) once U is no
//           longer needed;
//   area B: F, dense complex column-major (only i <= j + 1 is written and read) -> packed
//           rho (row stride D + 1).
// The per-chain stride is an odd multiple of 16 floats, so the two chains of a warp that
// read the same offset in their own areas use opposite halves of the banks.
//   area R (PASSES = 3 only): the upper triangle of R from the Gram-Schmidt sweep, packed
//           (column c, row k <= c at c (c + 1) / 2 + k, complex), which the refinement's
//           triangular solve reads; area B then holds H's original columns during the
//           refinement's products.  At D = 16 the Q planes are unpadded there (area A stays at
//           W's 576 floats), which keeps five CTAs on an SM.

template <int D, int PASSES = 2, int THREADS = kProposeThreads>
struct Shape {
    static constexpr int d = D * D;
    static constexpr int chains_per_block = THREADS / D;
    static constexpr int row_stride = D + 2;                    // float2 per row of W (padded)
    static constexpr int qcol = (PASSES == 3 && D == 16) ? D : D + 4;   // floats per column of a Q plane
    static constexpr int pk_stride = D + 1;                     // floats per row of the staged rho
    static constexpr int area_a = (2 * D * qcol > 2 * D * row_stride) ? 2 * D * qcol : 2 * D * row_stride;
    static constexpr int area_b = (2 * D * D > D * pk_stride) ? 2 * D * D : D * pk_stride;
    static constexpr int area_r = (PASSES == 3) ? D * (D + 1) : 0;
    static constexpr int raw = area_a + area_b + area_r;
    static constexpr int smem_floats = (raw + 31) / 32 * 32 + 16;
};

// Box-Muller with the fast hardware log, reciprocal square root and sine/cosine: the angle is
// reduced to 2 pi (v - 1/2) in (-pi, pi), where the intrinsics are accurate to ~2^-21
// absolute, and cos/sin(2 pi v) = -cos/-sin(2 pi (v - 1/2)).  v - 1/2 is exact.  The radius
// sqrt(t), t = -2 ln u >= 2^-23, is t rsqrt(t) (a few ulps).  The normals agree with the FP64
// Box-Muller of the same uniforms to about 1e-6 relative.
__device__ __forceinline__ void gaussian_pair_fast(uint32_t wu, uint32_t wv, float &z0, float &z1) {
    const float u = Philox::uniform(wu);
    const float v = Philox::uniform(wv);
    const float t = -2.0f * __logf(u);
    const float radius = t * rsqrtf(t);
    float s, c;
    __sincosf(6.283185307179586f * (v - 0.5f), &s, &c);
    z0 = -radius * c;
    z1 = -radius * s;
}

// a D-float column into / from registers, 128-bit at a time where D allows
template <int D>
__device__ __forceinline__ void load_column(const float *src, float (&v)[D], int s = 0) {
    if constexpr (D >= 4) {
#pragma unroll
        for (int i = 0; i < D; i += 4) {
            const float4 t = *reinterpret_cast<const float4 *>(src + 4 * ((i / 4) ^ s));
            v[i] = t.x;
            v[i + 1] = t.y;
            v[i + 2] = t.z;
            v[i + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < D; ++i) v[i] = src[i];
    }
}
template <int D>
__device__ __forceinline__ void store_column(float *dst, const float (&v)[D]) {
    if constexpr (D >= 4) {
#pragma unroll
        for (int i = 0; i < D; i += 4)
            *reinterpret_cast<float4 *>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < D; ++i) dst[i] = v[i];
    }
}

// a D-float column as D/2 pairs of consecutive entries (for the packed f32x2 arithmetic).  `s`:
// the column's 4-float blocks are stored in the order b ^ s (the swizzle of the unpadded
// 16-float columns of the refinement, kSwizzle below; 0 elsewhere)
template <int D>
__device__ __forceinline__ void load_column2(const float *src, float2 (&v)[D / 2], int s = 0) {
    if constexpr (D >= 4) {
#pragma unroll
        for (int p = 0; p < D / 2; p += 2) {
            const float4 t = *reinterpret_cast<const float4 *>(src + 4 * ((p / 2) ^ s));
            v[p] = make_float2(t.x, t.y);
            v[p + 1] = make_float2(t.z, t.w);
        }
    } else {
        v[0] = *reinterpret_cast<const float2 *>(src);
    }
}
template <int D>
__device__ __forceinline__ void store_column2(float *dst, const float2 (&v)[D / 2], int s = 0) {
    if constexpr (D >= 4) {
#pragma unroll
        for (int p = 0; p < D / 2; p += 2)
            *reinterpret_cast<float4 *>(dst + 4 * ((p / 2) ^ s)) = make_float4(v[p].x, v[p].y, v[p + 1].x, v[p + 1].y);
    } else {
        *reinterpret_cast<float2 *>(dst) = v[0];
    }
}

__device__ __forceinline__ float hsum(float2 v) { return v.x + v.y; }

// x rounded to TF32 (11 significant bits, nearest, ties away from zero), in an FP32 container
// whose low 13 mantissa bits are zero; x - tf32_rna(x) is exact in FP32
__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

template <int D>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
    for (int off = D / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Exact sum over the D lanes of a chain as an unevaluated pair hi + lo (TwoSum at every level).
template <int D>
__device__ __forceinline__ void group_sum_exact(float v, float &hi, float &lo) {
    float err = 0.0f;
#pragma unroll
    for (int off = D / 2; off > 0; off >>= 1) {
        const float pv = __shfl_xor_sync(0xffffffffu, v, off);
        const float pe = __shfl_xor_sync(0xffffffffu, err, off);
        // both partners form the same sum: order the operands by lane so they round alike
        const bool low = (threadIdx.x & off) == 0;
        const float x = low ? v : pv, y = low ? pv : v;
        const float sum = x + y;
        const float bb = sum - x;
        const float e = (x - (sum - bb)) + (y - bb);
        err = (low ? err + pe : pe + err) + e;
        v = sum;
    }
    hi = v;
    lo = err;
}

// q^dag p for the lane's own column q = (qr, qi) (pairs of rows, in registers) and a column p
// in shared memory (real and imaginary planes), without rounding error in the products and
// the sum: each product is accumulated into s1, which carries the offset `offset` = 1.5 2^(e+1)
// and so holds its running sum rounded to multiples of 2^(e-22) exactly (every partial sum of
// one accumulator must stay below 2^e); the FMA's rounding error x y - (s1' - s1) is formed
// exactly by a second FMA and summed in s2, where it is at most 2^(e-23).  The result is
// returned as (re, im), minus `sub` on the real part (subtracted while the sum is still
// exact); its error is about 2^(e-45) per product.
template <int D>
__device__ __forceinline__ float2 sum_products_exact(const float2 (&qr)[D / 2], const float2 (&qi)[D / 2],
                                                     const float *pre, const float *pim, float offset, float sub,
                                                     int s = 0) {
    // four accumulators: qr pr + qi pi (real part), qr pi and qi pr (imaginary part, subtracted
    // at the end); each a grid sum s1 and an error sum s2
    float2 a1 = make_float2(offset, offset), b1 = a1, c1 = a1;
    float2 a2 = make_float2(0.f, 0.f), b2 = a2, c2 = a2;
    auto step = [](float2 &s1, float2 &s2, float2 x, float2 y) {
        const float2 n = __ffma2_rn(x, y, s1);
        s2 = __fadd2_rn(s2, __ffma2_rn(x, y, sub2(s1, n)));   // + (x y - (n - s1)): the rounding error
        s1 = n;
    };
    // the column p is read two row pairs (one 128-bit load per plane) at a time
#pragma unroll
    for (int p0 = 0; p0 < D / 2; p0 += (D >= 4 ? 2 : 1)) {
        float2 pr[2], pi[2];
        if constexpr (D >= 4) {
            const float4 r4 = *reinterpret_cast<const float4 *>(pre + 4 * ((p0 / 2) ^ s));   // (block swizzle s)
            const float4 i4 = *reinterpret_cast<const float4 *>(pim + 4 * ((p0 / 2) ^ s));
            pr[0] = make_float2(r4.x, r4.y);
            pr[1] = make_float2(r4.z, r4.w);
            pi[0] = make_float2(i4.x, i4.y);
            pi[1] = make_float2(i4.z, i4.w);
        } else {
            pr[0] = *reinterpret_cast<const float2 *>(pre);
            pi[0] = *reinterpret_cast<const float2 *>(pim);
        }
#pragma unroll
        for (int u = 0; u < (D >= 4 ? 2 : 1); ++u) {
            const int p = p0 + u;
            step(a1, a2, qr[p], pr[u]);   // Re: qr pr + qi pi
            step(a1, a2, qi[p], pi[u]);
            step(b1, b2, qr[p], pi[u]);   // Im: qr pi - qi pr
            step(c1, c2, qi[p], pr[u]);
        }
    }
    // the grid parts minus their offsets are exact, and so are their sums and differences
    const float re_grid = ((a1.x - offset) + (a1.y - offset)) - sub;
    const float im_grid = ((b1.x - offset) + (b1.y - offset)) - ((c1.x - offset) + (c1.y - offset));
    return make_float2(re_grid + (a2.x + a2.y), im_grid + ((b2.x + b2.y) - (c2.x + c2.y)));
}

// The rest of a refinement pass at D >= 32 (the solve, Y's upper part and diagonal, U = Q1 -
// Q1 Y^dag), with rolled loops and Y's row j kept in place in area B: unrolled over registers, as
// refine_pass does for D <= 16, the pass is several thousand straight-line instructions at D = 32
// and the warps stall on instruction fetch.  The arithmetic of each entry is refine_pass's.  Lane j
// writes only row j of area B: its lower part (read by the other lanes for their upper parts only
// after the barrier below), then its diagonal and upper part, which no other lane reads.
template <int D, int QC>
__device__ __noinline__ float refine_tail_rolled(float *qre, float *qim, float *hre, float *him, const float2 *rpk,
                                                 int j, float2 mjj, bool apply) {
    auto cidx = [](int r, int cc) { return cc * D + (r ^ cc); };
    // forward substitution on row j: entries c < j only (the row has no unknowns beyond)
#pragma unroll 1
    for (int c0 = 0; c0 < j; ++c0) {
        const float inv_r = rpk[c0 * (c0 + 1) / 2 + c0].y;
        const int o0 = cidx(j, c0);
        const float ar = hre[o0] * inv_r, ai = him[o0] * inv_r;
        hre[o0] = ar;
        him[o0] = ai;
#pragma unroll 2
        for (int c = c0 + 1; c < j; ++c) {
            const float2 r = rpk[c * (c + 1) / 2 + c0];   // R[c0][c]
            const int o = cidx(j, c);
            hre[o] -= ar * r.x - ai * r.y;
            him[o] -= ar * r.y + ai * r.x;
        }
    }
    // diagonal: Re Y_jj = (N_jj - 1) / 2; Im Y_jj makes R_jj real
    float ydi = mjj.y;
    float ymax = 0.0f;
#pragma unroll 1
    for (int k = 0; k < j; ++k) {
        const float2 r = rpk[j * (j + 1) / 2 + k];   // R[k][j]
        const float yr = hre[cidx(j, k)], yi = him[cidx(j, k)];
        ydi -= yr * r.y + yi * r.x;
        ymax = fmaxf(ymax, fmaxf(fabsf(yr), fabsf(yi)));
    }
    const float2 ydiag = make_float2(0.5f * hre[cidx(j, j)], ydi * rpk[j * (j + 1) / 2 + j].y);
    __syncwarp();   // every lane's lower row is in place
    // upper part: Y[j][c] = N_jc - conj(Y[c][j]), c > j, over N_jc; every lane walks the same c
    // (its entries (j, c) and (c, j) then lie in distinct banks across the lanes)
#pragma unroll 2
    for (int c = 1; c < D; ++c) {
        if (c > j) {
            const float yr = hre[cidx(j, c)] - hre[cidx(c, j)], yi = him[cidx(j, c)] + him[cidx(c, j)];
            hre[cidx(j, c)] = yr;
            him[cidx(j, c)] = yi;
            ymax = fmaxf(ymax, fmaxf(fabsf(yr), fabsf(yi)));
        }
    }
    hre[cidx(j, j)] = ydiag.x;
    him[cidx(j, j)] = ydiag.y;
    ymax = fmaxf(ymax, fmaxf(fabsf(ydiag.x), fabsf(ydiag.y)));
#pragma unroll
    for (int off = D / 2; off >= 1; off /= 2) ymax = fmaxf(ymax, __shfl_xor_sync(0xffffffffu, ymax, off, D));
    // U = Q1 - Q1 Y^dag: column j is q_j - sum_k q_k conj(Y[j][k]), in two halves of rows as in
    // refine_pass
    constexpr int HP = D / 4;   // row pairs per half
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        float2 cr[HP], ci[HP];
#pragma unroll
        for (int p = 0; p < HP; ++p) cr[p] = ci[p] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int k = 0; k < D; ++k) {
            const float ykr = hre[cidx(j, k)], yki = him[cidx(j, k)];
            const float2 yx = make_float2(ykr, ykr), yy = make_float2(yki, yki), myy = make_float2(-yki, -yki);
#pragma unroll
            for (int p = 0; p < HP; p += 2) {   // (vr + i vi)(y.x - i y.y), a 4-float block of rows at a time
                const int o = k * QC + 2 * (half * HP + p);
                const float4 r4 = *reinterpret_cast<const float4 *>(qre + o);
                const float4 i4 = *reinterpret_cast<const float4 *>(qim + o);
                const float2 vr[2] = {make_float2(r4.x, r4.y), make_float2(r4.z, r4.w)};
                const float2 vi[2] = {make_float2(i4.x, i4.y), make_float2(i4.z, i4.w)};
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    cr[p + u] = __ffma2_rn(vr[u], yx, __ffma2_rn(vi[u], yy, cr[p + u]));
                    ci[p + u] = __ffma2_rn(vi[u], yx, __ffma2_rn(vr[u], myy, ci[p + u]));
                }
            }
        }
        __syncwarp();   // every lane has read this half of every q_k
        if (apply) {
#pragma unroll
            for (int p = 0; p < HP; p += 2) {
                const int o = j * QC + 2 * (half * HP + p);
                float4 *ur = reinterpret_cast<float4 *>(qre + o);
                float4 *ui = reinterpret_cast<float4 *>(qim + o);
                const float4 u0 = *ur, u1 = *ui;
                const float2 a0 = sub2(make_float2(u0.x, u0.y), cr[p]), a1 = sub2(make_float2(u0.z, u0.w), cr[p + 1]);
                const float2 b0 = sub2(make_float2(u1.x, u1.y), ci[p]), b1 = sub2(make_float2(u1.z, u1.w), ci[p + 1]);
                *ur = make_float4(a0.x, a0.y, a1.x, a1.y);
                *ui = make_float4(b0.x, b0.y, b1.x, b1.y);
            }
        }
        __syncwarp();
    }
    return ymax;
}

// The rest of a pass for D <= 16, over registers: the triangular solve on row j of C (area B), Y's
// upper part and diagonal, U = Q1 - Q1 Y^dag.  `apply`: write this lane's column of the refined U.
// GRP = 2: two groups of D lanes share a chain, and each updates one half of U's rows.  SHARED: more
// than one lane holds row j, so the solved entries replace M's only after all of them have read those.
template <int D, int QC, bool SHARED, int GRP = 1>
__device__ __forceinline__ float refine_tail(float *qre, float *qim, float *hre, float *him, const float2 *rpk, int j,
                                             float2 mjj, bool apply, int grp = 0) {
    auto cidx = [](int r, int cc) { return cc * D + (r ^ cc); };
    // Y, row j, in registers: y[c] = Y[j][c].  Forward substitution, right-looking: after
    // Y[j][c0] = (M_jc0 - ...) / R_c0c0 every later entry of the row takes its share
    // -Y[j][c0] R[c0][c] at once, so each R entry is read once for all lanes; entries at
    // c >= j stay zero (the lane's row has no such unknowns) until the upper part below.
    float2 y[D];
#pragma unroll
    for (int c = 0; c < D; ++c)
        y[c] = (c < j) ? make_float2(hre[cidx(j, c)], him[cidx(j, c)]) : make_float2(0.f, 0.f);
#pragma unroll
    for (int c0 = 0; c0 < D - 1; ++c0) {
        const float inv_r = rpk[c0 * (c0 + 1) / 2 + c0].y;
        y[c0] = make_float2(y[c0].x * inv_r, y[c0].y * inv_r);
#pragma unroll
        for (int c = c0 + 1; c < D - 1; ++c) {
            const float2 r = rpk[c * (c + 1) / 2 + c0];   // R[c0][c]
            y[c].x -= y[c0].x * r.x - y[c0].y * r.y;
            y[c].y -= y[c0].x * r.y + y[c0].y * r.x;
        }
    }
    // diagonal: Re Y_jj = (N_jj - 1) / 2; Im Y_jj makes R_jj real
    float ydi = mjj.y;
#pragma unroll
    for (int k = 0; k < D - 1; ++k) {
        const float2 r = rpk[j * (j + 1) / 2 + (k < j ? k : 0)];   // R[k][j] (k < j)
        if (k < j) ydi -= y[k].x * r.y + y[k].y * r.x;
    }
    const float2 ydiag = make_float2(0.5f * hre[cidx(j, j)], ydi * rpk[j * (j + 1) / 2 + j].y);
    // upper part: Y[j][c] = N_jc - conj(Y[c][j]), c > j, through area B
    if constexpr (SHARED) __syncwarp();   // the lanes that share this row have read it
#pragma unroll
    for (int c = 0; c < D - 1; ++c)
        if (c < j) {
            hre[cidx(j, c)] = y[c].x;
            him[cidx(j, c)] = y[c].y;
        }
    __syncwarp();   // every lane's lower row is in place
#pragma unroll
    for (int c = 1; c < D; ++c)
        if (c > j) y[c] = make_float2(hre[cidx(j, c)] - hre[cidx(c, j)], him[cidx(j, c)] + him[cidx(c, j)]);
#pragma unroll
    for (int c = 0; c < D; ++c)
        if (c == j) y[c] = ydiag;
    // the chain's largest |Y| entry decides whether another pass follows
    float ymax = 0.0f;
#pragma unroll
    for (int c = 0; c < D; ++c) ymax = fmaxf(ymax, fmaxf(fabsf(y[c].x), fabsf(y[c].y)));
#pragma unroll
    for (int off = D / 2; off >= 1; off /= 2) ymax = fmaxf(ymax, __shfl_xor_sync(0xffffffffu, ymax, off, D));
    // U = Q1 - Q1 Y^dag: column j is q_j - sum_k q_k conj(Y[j][k]); the correction is summed
    // on its own (it is small) and subtracted once.  Rows go in two halves: a half is
    // overwritten only after every lane has read that half of every column.
    constexpr int HP = (D >= 4) ? D / 4 : 1;   // row pairs per half
    static_assert(GRP == 1 || D >= 4, "halves");
#pragma unroll
    for (int h = 0; h < (D >= 4 && GRP == 1 ? 2 : 1); ++h) {
        const int half = GRP == 1 ? h : grp;
        float2 cr[HP], ci[HP];
#pragma unroll
        for (int p = 0; p < HP; ++p) cr[p] = ci[p] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const float2 yx = make_float2(y[k].x, y[k].x), yy = make_float2(y[k].y, y[k].y);
            const float2 myy = make_float2(-y[k].y, -y[k].y);   // conj(y) = (y.x, -y.y)
            if constexpr (HP % 2 == 0) {   // column k's rows read a 4-float block (two pairs) at a time
#pragma unroll
                for (int p = 0; p < HP; p += 2) {   // (vr + i vi)(y.x - i y.y)
                    const int row = 2 * (half * HP + p);
                    const int o = k * QC + 4 * ((row >> 2) ^ qsw<D, QC>(k));
                    const float4 r4 = *reinterpret_cast<const float4 *>(qre + o);
                    const float4 i4 = *reinterpret_cast<const float4 *>(qim + o);
                    const float2 vr[2] = {make_float2(r4.x, r4.y), make_float2(r4.z, r4.w)};
                    const float2 vi[2] = {make_float2(i4.x, i4.y), make_float2(i4.z, i4.w)};
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        cr[p + u] = __ffma2_rn(vr[u], yx, __ffma2_rn(vi[u], yy, cr[p + u]));
                        ci[p + u] = __ffma2_rn(vi[u], yx, __ffma2_rn(vr[u], myy, ci[p + u]));
                    }
                }
            } else {
#pragma unroll
                for (int p = 0; p < HP; ++p) {   // (vr + i vi)(y.x - i y.y)
                    const int row = 2 * (half * HP + p);
                    const int o = k * QC + 4 * ((row >> 2) ^ qsw<D, QC>(k)) + (row & 3);
                    const float2 vr = *reinterpret_cast<const float2 *>(qre + o);
                    const float2 vi = *reinterpret_cast<const float2 *>(qim + o);
                    cr[p] = __ffma2_rn(vr, yx, __ffma2_rn(vi, yy, cr[p]));
                    ci[p] = __ffma2_rn(vi, yx, __ffma2_rn(vr, myy, ci[p]));
                }
            }
        }
        __syncwarp();   // every lane has read this half of every q_k
        if (apply) {
            if constexpr (HP % 2 == 0) {   // two row pairs, one 4-float block, at a time
#pragma unroll
                for (int p = 0; p < HP; p += 2) {
                    const int row = 2 * (half * HP + p);
                    float4 *ur = reinterpret_cast<float4 *>(qre + j * QC + 4 * ((row >> 2) ^ qsw<D, QC>(j)));
                    float4 *ui = reinterpret_cast<float4 *>(qim + j * QC + 4 * ((row >> 2) ^ qsw<D, QC>(j)));
                    const float4 u0 = *ur, u1 = *ui;
                    const float2 a0 = sub2(make_float2(u0.x, u0.y), cr[p]), a1 = sub2(make_float2(u0.z, u0.w), cr[p + 1]);
                    const float2 b0 = sub2(make_float2(u1.x, u1.y), ci[p]), b1 = sub2(make_float2(u1.z, u1.w), ci[p + 1]);
                    *ur = make_float4(a0.x, a0.y, a1.x, a1.y);
                    *ui = make_float4(b0.x, b0.y, b1.x, b1.y);
                }
            } else {
#pragma unroll
                for (int p = 0; p < HP; ++p) {
                    const int row = 2 * (half * HP + p);
                    float2 *ur = reinterpret_cast<float2 *>(qre + j * QC + row);
                    float2 *ui = reinterpret_cast<float2 *>(qim + j * QC + row);
                    *ur = sub2(*ur, cr[p]);
                    *ui = sub2(*ui, ci[p]);
                }
            }
        }
        __syncwarp();
    }
    return ymax;
}

// One first-order pass of the refinement of U (step 2b of the D <= 16 kernel below, where the
// method is described).  `again`: a pass after the first, which reads H's column j back from y'
// into area B (it held C) and U's column j as this lane's vector; `apply`: write the refined U
// (a further pass runs for the whole warp when any of its chains needs it, and the others
// discard theirs, so a chain's bits never depend on its neighbours).  SHARED as in refine_tail.
// Returns the chain's largest |Y| entry.
template <int D, int QC, bool SHARED = false>
__device__ __forceinline__ float refine_pass(float2 (&hr)[D / 2], float2 (&hi)[D / 2], float *qre, float *qim,
                                             float *hre, float *him, const float2 *rpk, const float *gsrc, int j,
                                             bool again, bool apply) {
    constexpr int d = D * D;
    auto cidx = [](int r, int cc) { return cc * D + (r ^ cc); };
    if (again) {   // H's column j into area B again (it held C), U's column j as the vector
#pragma unroll
        for (int i = 0; i < D; i += (D >= 4 ? 4 : 1)) {
            if constexpr (D >= 4) {
                const int o = j * D + 4 * ((i / 4) ^ hsw<D, QC>(j));
                *reinterpret_cast<float4 *>(hre + o) = *reinterpret_cast<const float4 *>(gsrc + 2 * d + j * D + i);
                *reinterpret_cast<float4 *>(him + o) = *reinterpret_cast<const float4 *>(gsrc + 3 * d + j * D + i);
            } else {
                hre[j * D + i] = gsrc[2 * d + j * D + i];
                him[j * D + i] = gsrc[3 * d + j * D + i];
            }
        }
        load_column2<D>(qre + j * QC, hr, qsw<D, QC>(j));
        load_column2<D>(qim + j * QC, hi, qsw<D, QC>(j));
        __syncwarp();
    }
#pragma unroll 1
    for (int cc = 0; cc < D; ++cc) {
        const bool lower = cc < j;   // M_jc = q_j^dag h_c; at c = j (and above) N_jc = q_j^dag q_c
        const float *pre = lower ? hre + cc * D : qre + cc * QC;
        const float *pim = lower ? him + cc * D : qim + cc * QC;
        // every partial sum of M stays below 2^6 (|h| < 64), of N below 2^1
        const float2 res = sum_products_exact<D>(hr, hi, pre, pim, lower ? 192.0f : 6.0f, cc == j ? 1.0f : 0.0f,
                                                 lower ? hsw<D, QC>(cc) : qsw<D, QC>(cc));
        __syncwarp();   // every lane is done with column c of H
        hre[cidx(j, cc)] = res.x;
        him[cidx(j, cc)] = res.y;
    }
    // M_jj, the one entry of the row not formed above: its column of H now holds C, so h_j is
    // read again from the proposal's own y' (or the evaluated row; for an inactive lane the
    // first chain's row, in bounds, whose result is not used)
    const float2 mjj = sum_products_exact<D>(hr, hi, gsrc + 2 * d + j * D, gsrc + 3 * d + j * D, 192.0f, 0.0f);
    __syncwarp();
    static_assert(!SHARED || D <= 16, "the rolled tail solves in place: one lane per row");
    if constexpr (D >= 32)
        return refine_tail_rolled<D, QC>(qre, qim, hre, him, rpk, j, mjj, apply);
    else
        return refine_tail<D, QC, SHARED>(qre, qim, hre, him, rpk, j, mjj, apply);
}

// refine_pass's first pass where two groups of D lanes share a chain: the groups take the entries of
// row j of C in turn (two of H's columns are freed per step), and half of U's rows each.
template <int D, int QC>
__device__ __forceinline__ float refine_pass_split(const float2 (&hr)[D / 2], const float2 (&hi)[D / 2], float *qre,
                                                   float *qim, float *hre, float *him, const float2 *rpk,
                                                   const float *gsrc, int j, int grp) {
    constexpr int d = D * D;
#pragma unroll 1
    for (int c2 = 0; c2 < D; c2 += 2) {
        const int cc = c2 + grp;
        const bool lower = cc < j;
        const float2 res = sum_products_exact<D>(hr, hi, lower ? hre + cc * D : qre + cc * QC,
                                                 lower ? him + cc * D : qim + cc * QC, lower ? 192.0f : 6.0f,
                                                 cc == j ? 1.0f : 0.0f, lower ? hsw<D, QC>(cc) : qsw<D, QC>(cc));
        __syncwarp();   // every lane is done with columns c2 and c2 + 1 of H
        hre[cc * D + (j ^ cc)] = res.x;
        him[cc * D + (j ^ cc)] = res.y;
    }
    const float2 mjj = sum_products_exact<D>(hr, hi, gsrc + 2 * d + j * D, gsrc + 3 * d + j * D, 192.0f, 0.0f);
    __syncwarp();
    return refine_tail<D, QC, true, 2>(qre, qim, hre, him, rpk, j, mjj, true, grp);
}

// The passes after the first, for the few chains whose first pass left |Y| above kRefineTol: out
// of line, so that the common path keeps its registers.  `own`: this lane writes its column of U (where
// several lanes repeat a chain's columns (SHARED), one of them does).
template <int D, int QC, bool SHARED>
__device__ __noinline__ void refine_more(float *qre, float *qim, float *hre, float *him, const float2 *rpk,
                                         const float *gsrc, int j, float ymax, bool own) {
    float2 hr[D / 2], hi[D / 2];
#pragma unroll 1
    for (int pass = 1; pass < kRefinePasses && __any_sync(0xffffffffu, ymax > kRefineTol); ++pass) {
        const bool need = ymax > kRefineTol;
        const float next = refine_pass<D, QC, SHARED>(hr, hi, qre, qim, hre, him, rpk, gsrc, j, true, need && own);
        ymax = need ? next : ymax;
    }
}

}  // namespace qst
