// Proposal and density-matrix assembly (the proposal of Algorithm 2, Algorithm 1).
//
// One chain is handled by D consecutive lanes; lane j owns column j of the D x D
// blocks G and H (the latent layout is column-major, so a column is D contiguous
// floats of each of the four parts).  Per chain:
//   1. eta from Philox (tag 1, step j) and y' = sqrt(1 - beta^2) y + beta eta, one
//      Philox block (four entries) at a time, a chain's lanes on consecutive blocks; y' goes to the
//      chain's other y buffer (the accept kernel flips to it); lane j takes H's column j through
//      shared memory and keeps it in registers.  G's columns are read back from y' in step 3.
//      (With every lane on its own column's blocks an access touched 32 pieces of 16 bytes in as
//      many sectors or lines; consecutive blocks took the kernel from 536 to 524 us at 65536
//      four-qubit chains, from 292 to 258 us at 8192 five-qubit ones and from 348 to 332 us at
//      1024 six-qubit ones.)
//   2. QR of H (Algorithm 1).  Modified Gram-Schmidt: at step k lane k publishes its
//      (unnormalised) column v_k, and every lane j > k loads it, forms |v_k|^2 and v_k^dag h_j
//      itself and removes the projection -- no lane works alone on a normalisation.  The
//      columns are normalised at the end.  MGS yields the unitary factor whose R has a
//      positive real diagonal, i.e. U = Q Lambda of Algorithm 1.  Its FP32 columns are
//      orthogonal only to O(cond(H) 2^-24); with PASSES = 2 they are re-orthogonalised once:
//      Q1 = Q2 R2 with R2 = chol(Q1^dag Q1) = I + F + O(E^2), E = Q1^dag Q1 - I,
//      F = strict upper part of E plus half its (real) diagonal, so Q2 = Q1 (I - F) is the
//      same QR factor of H to O(E^2) (E < 1e-4 after one pass for cond(H) < 1e4, so E^2
//      is below FP32 rounding).  Unlike a second Gram-Schmidt sweep this is two balanced
//      products: lane a forms entries (a, a + t) of E, then row a of Q1 (I - F).
//   3. W = (U + I) G, lane j computing column j;
//   4. rho = W W^dag / Tr: lane a computes entries (a, a+t mod D) for t = 0..D/2
//      (the Hermitian half, balanced over lanes), packed as vec_h and scaled by the FP32
//      reciprocal of the trace.  The rounding of that scaling is not left in the
//      probabilities: the exact sum t of the *stored* FP32 diagonal (1 up to a few ulps,
//      formed by a TwoSum reduction) is written too, and the likelihood uses
//      p = (vec_h . P) / t, i.e. subtracts N log t in FP64.  Then sum_l p_kl = 1 holds to
//      the contraction's rounding, with no coherent shift of every probability (which
//      would cost N * 2^-24 in log L);
//   5. the packed row is stored as FP32 and, for the tensor-core contraction, as the
//      exact three-term bf16 split hi + mid + lo.
#include "propose_dev.cuh"

namespace qst {
namespace {

constexpr int kThreads = kProposeThreads;
struct ProposeArgs {
    const float *x_eval;        // MODE_EVAL: [rows][nx] latent vectors
    float *y;                   // [2][R][nx]
    const uint8_t *cur;         // [R]
    const float2 *coef;         // [R] (sqrt(1 - beta^2), beta) as floats
    float *rho_out;             // [rows][d_pad] packed rho (FP32-normalised)
    __nv_bfloat16 *split_out;   // [rows][3][d_pad] bf16 hi/mid/lo, or null
    float *split_tf;            // [rows][tf_splits][d_pad] TF32 hi[, lo], or null
    int tf_splits;              // 1 or 2
    double *trace_out;          // [rows] exact trace of the stored rho (1 up to rounding)
    float *rho_norm_out;        // MODE_EVAL, optional: [rows][d] copy of the packed rho
    int64_t rows;
    int64_t R;
    int64_t chain_offset;
    uint64_t seed;
    uint32_t step;
    StepState *step_dev;         // MODE_STEP: when not null the step is the one after this counter's, opened here
    int mode;
    int d_pad;
    Philox::RoundKeys rk;        // the generator's round keys for `seed`
};

// THREADS: the CTA size (chains per CTA = THREADS / D); 128 by default, 64 or 32 when the
// autotuner finds that a small problem covers more SMs that way.  The register budget per
// thread is the same for every size: that of five 128-thread CTAs per SM (96 registers), at eight
// lanes per chain of seven (72, nothing spilled but 4 bytes with 32 threads: 65536 three-qubit chains
// 94 -> 89 us, 16384 29.1 -> 28.1).
template <int D>
constexpr int propose_ctas() {
    return D == 8 ? 7 : 5;
}

// GRP = 2: two groups of D lanes share a chain.  They take the latent blocks, the refinement's dot
// products and its update of U, W (at four qubits) and rho's entries in turn, and repeat the sweep
// and the triangular solve, whose steps depend on one another: the shorter step while there are too
// few chains to fill the chip (propose_split).
template <int D, int PASSES, int THREADS = kThreads, int GRP = 1>
__global__ void __launch_bounds__(THREADS, (GRP == 1 ? propose_ctas<D>() : 5) * kThreads / THREADS) propose_kernel(ProposeArgs a) {
    using S = Shape<D, PASSES, THREADS>;
    constexpr int d = S::d;
    constexpr int nx = 4 * d;
    constexpr int RS = S::row_stride;
    constexpr int QC = S::qcol;
    constexpr int PK = S::pk_stride;
    extern __shared__ __align__(16) float smem[];

    constexpr int LPC = D * GRP;         // lanes per chain
    const int j = threadIdx.x % D;       // owned column (and, in steps 2b and 4, owned row)
    const int l = threadIdx.x % LPC, grp = GRP == 1 ? 0 : l / D;
    const int g = threadIdx.x / LPC;     // chain slot in the block
    const int64_t c = (int64_t)blockIdx.x * (THREADS / LPC) + g;
    const bool active = c < a.rows;
    const uint32_t step = (a.step_dev && a.mode == MODE_STEP) ? a.step_dev->step + 1u : a.step;
    if (a.step_dev && a.mode == MODE_STEP && blockIdx.x == 0 && threadIdx.x == 0) open_step(a.step_dev);
    float *sm = smem + g * S::smem_floats;
    float *qre = sm, *qim = sm + D * QC;                 // Q planes (column stride QC)
    float2 *wsm = reinterpret_cast<float2 *>(sm);        // W row-major (row stride RS), replaces Q
    float *fre = sm + S::area_a, *fim = fre + D * D;     // F column-major (stride D), re / im planes
    float *packed = sm + S::area_a;                      // staged rho (row stride PK), replaces F
    float *hre = sm + S::area_a, *him = hre + D * D;     // PASSES = 3: H's columns (stride D), in area B
    float2 *rpk = reinterpret_cast<float2 *>(sm + S::area_a + S::area_b);   // PASSES = 3: packed R

    // ---- 1. latent proposal --------------------------------------------------------------
    float coef_y = 1.0f, coef_eta = 0.0f;
    int cur = 0;
    if (active && a.mode == MODE_STEP) {
        cur = a.cur[c];
        const float2 cf = a.coef[c];
        coef_y = cf.x;
        coef_eta = cf.y;
    } else if (a.mode == MODE_INIT) {
        coef_y = 0.0f;
        coef_eta = 1.0f;
    }
    const int64_t cc = active ? c : 0;
    const uint32_t chain_id = (uint32_t)(a.chain_offset + cc);
    const uint32_t tag = (a.mode == MODE_INIT) ? TAG_INIT : TAG_PROPOSAL;
    const float *ysrc = a.y + ((int64_t)cur * a.R + cc) * nx;
    float *ydst = a.y + ((int64_t)(1 - cur) * a.R + cc) * nx;
    // where G's column j is read back in step 3: this chain's y' writes, or the input row
    const float *gsrc = (a.mode == MODE_EVAL) ? a.x_eval + cc * nx : ydst;
    float2 hr[D / 2], hi[D / 2];   // H's column j, entries (2p, 2p + 1) in pair p
    if constexpr (D >= 4) {
        // A part is d/4 Philox blocks of four entries.  Lane l takes blocks l, l + LPC, ..: a chain's
        // lanes then read and write consecutive 16-byte pieces of y, and H's blocks reach the lanes that own
        // their columns through shared memory (area B where the refinement keeps H's columns
        // anyway, the Q planes otherwise).
        // At D = 4 a block is its lane's column and needs neither (through shared memory the kernel took 30.6
        // instead of 28.7 us for 65536 chains).
        constexpr int BPC = D / 4;   // blocks per column
        auto stage = [&](float *plane_h, float *plane_q, int blk, float4 v, float2 (&own)[D / 2]) {
            const int col = blk / BPC, r = blk % BPC;
            if constexpr (D == 4) {
                own[0] = make_float2(v.x, v.y);
                own[1] = make_float2(v.z, v.w);
            } else if constexpr (PASSES == 3) {
                *reinterpret_cast<float4 *>(plane_h + col * D + 4 * (r ^ hsw<D, QC>(col))) = v;
            } else {
                *reinterpret_cast<float4 *>(plane_q + col * QC + 4 * (r ^ qsw<D, QC>(col))) = v;
            }
        };
#pragma unroll 1
        for (int part = 0; part < 4; ++part) {
            const int e0 = part * d + 4 * l;    // element index of this lane's first block
            float4 y0[D / 4 / GRP];
#pragma unroll
            for (int q = 0; q < D / 4 / GRP; ++q) {
                y0[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (active && a.mode == MODE_STEP) y0[q] = *reinterpret_cast<const float4 *>(ysrc + e0 + 4 * LPC * q);
                if (active && a.mode == MODE_EVAL) y0[q] = *reinterpret_cast<const float4 *>(a.x_eval + cc * nx + e0 + 4 * LPC * q);
            }
#pragma unroll
            for (int q = 0; q < D / 4 / GRP; ++q) {
                float4 yn = y0[q];
                if (a.mode != MODE_EVAL) {
                    const uint4 w = Philox::block(make_uint4((uint32_t)(e0 / 4 + LPC * q), step, chain_id, tag), a.rk);
                    float z0, z1, z2, z3;
                    gaussian_pair_fast(w.x, w.y, z0, z1);
                    gaussian_pair_fast(w.z, w.w, z2, z3);
                    yn.x = __fmaf_rn(coef_y, y0[q].x, coef_eta * z0);
                    yn.y = __fmaf_rn(coef_y, y0[q].y, coef_eta * z1);
                    yn.z = __fmaf_rn(coef_y, y0[q].z, coef_eta * z2);
                    yn.w = __fmaf_rn(coef_y, y0[q].w, coef_eta * z3);
                    if (active) *reinterpret_cast<float4 *>(ydst + e0 + 4 * LPC * q) = yn;
                }
                if (part == 2) stage(hre, qre, l + LPC * q, yn, hr);
                if (part == 3) stage(him, qim, l + LPC * q, yn, hi);
            }
        }
        if constexpr (D > 4) {
            __syncwarp();
            if constexpr (PASSES == 3) {
                load_column2<D>(hre + j * D, hr, hsw<D, QC>(j));
                load_column2<D>(him + j * D, hi, hsw<D, QC>(j));
            } else {
                load_column2<D>(qre + j * QC, hr, qsw<D, QC>(j));
                load_column2<D>(qim + j * QC, hi, qsw<D, QC>(j));
                __syncwarp();   // (the sweep publishes its columns there)
            }
        }
    } else {
        // D == 2: each part is one Philox block shared by the two lanes; lane j takes pair j
#pragma unroll
        for (int part = 0; part < 4; ++part) {
            const int e = part * d + j * D;
            float y0v = 0.0f, y1v = 0.0f;
            if (a.mode == MODE_EVAL) {
                if (active) {
                    y0v = a.x_eval[cc * nx + e];
                    y1v = a.x_eval[cc * nx + e + 1];
                }
            } else {
                const uint4 w = Philox::block(make_uint4((uint32_t)part, step, chain_id, tag), a.rk);
                float z0, z1;
                gaussian_pair_fast(j == 0 ? w.x : w.z, j == 0 ? w.y : w.w, z0, z1);
                float o0 = 0.0f, o1 = 0.0f;
                if (a.mode == MODE_STEP && active) {
                    o0 = ysrc[e];
                    o1 = ysrc[e + 1];
                }
                y0v = __fmaf_rn(coef_y, o0, coef_eta * z0);
                y1v = __fmaf_rn(coef_y, o1, coef_eta * z1);
                if (active) {
                    ydst[e] = y0v;
                    ydst[e + 1] = y1v;
                }
            }
            if (part == 2) {
                hr[0] = make_float2(y0v, y1v);
            } else if (part == 3) {
                hi[0] = make_float2(y0v, y1v);
            }
        }
    }

    if constexpr (PASSES == 3 && D <= 4) {   // H's original columns, for the refinement after the sweep (above for D > 4)
        store_column2<D>(hre + j * D, hr, hsw<D, QC>(j));
        store_column2<D>(him + j * D, hi, hsw<D, QC>(j));
    }

    // ---- 2a. modified Gram-Schmidt on the columns of H (Algorithm 1) ---------------------------
    // Every lane loads the published column v_k and forms r = v_k^dag h with its own column h
    // (packed f32x2 products over pairs of rows).  Lane k's column is v_k itself, so its r is
    // |v_k|^2, which the other lanes take by shuffle.  Lanes j > k project; lane k keeps
    // 1/|v_k|; a lane j < k holds its final v_j, so its r is conj(v_j^dag v_k) and gives the
    // Gram entry E_jk = q_j^dag q_k of the normalised columns for the re-orthogonalisation --
    // the entries become available exactly as lanes fall idle, so the Gram matrix costs no
    // separate pass.
    // PASSES = 0 (the Hilbert-Schmidt prior) skips steps 2 and the U term of step 3: W = G
    if constexpr (PASSES > 0) {
    float inv_own = 0.0f;   // 1 / |v_j| of this lane's final column
#pragma unroll 1
    for (int k = 0; k < D; ++k) {
        if (j == k) {   // column k is final: publish it
            store_column2<D>(qre + k * QC, hr, qsw<D, QC>(k));
            store_column2<D>(qim + k * QC, hi, qsw<D, QC>(k));
        }
        __syncwarp();
        float2 vr[D / 2], vi[D / 2];
        load_column2<D>(qre + k * QC, vr, qsw<D, QC>(k));
        load_column2<D>(qim + k * QC, vi, qsw<D, QC>(k));
        // r = v^dag h = sum (vr hr + vi hi) + i sum (vr hi - vi hr)
        float2 a0 = make_float2(0.f, 0.f), a1 = a0, b0 = a0, b1 = a0;
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            a0 = __ffma2_rn(vr[p], hr[p], a0);
            a1 = __ffma2_rn(vi[p], hi[p], a1);
            b0 = __ffma2_rn(vr[p], hi[p], b0);
            b1 = __ffma2_rn(vi[p], hr[p], b1);
        }
        const float rr = hsum(a0) + hsum(a1);
        const float ri = hsum(b0) - hsum(b1);
        const float nk = __shfl_sync(0xffffffffu, rr, k, D);   // |v_k|^2 from lane k
        // one hardware reciprocal square root, uniform over the lanes: its few-ulp error in the
        // projection coefficient or the norm is of the size of the FP32 rounding the sweep
        // already leaves, and the re-orthogonalisation removes both to first order
        const float rs = rsqrtf(nk);
        // h -= (r / |v|^2) v on lanes j > k; the coefficient is zero elsewhere, which leaves h
        // unchanged, so the warp runs one branch-free path
        const float coef = (j > k) ? rs * rs : 0.0f;
        const float sr = rr * coef, si = ri * coef;
        const float2 msr = make_float2(-sr, -sr), psi = make_float2(si, si), msi = make_float2(-si, -si);
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            hr[p] = __ffma2_rn(msr, vr[p], __ffma2_rn(psi, vi[p], hr[p]));
            hi[p] = __ffma2_rn(msr, vi[p], __ffma2_rn(msi, vr[p], hi[p]));
        }
        inv_own = (j == k) ? rs : inv_own;
        if constexpr (PASSES == 2) {
            if (j < k) {
                const float sc = inv_own * rs;             // E_jk = conj(r) / (|v_j| |v_k|), j < k
                fre[k * D + j] = rr * sc;
                fim[k * D + j] = -ri * sc;
            }
        }
        if constexpr (PASSES == 3) {
            // the triangular factor the refinement solves with (FP32 suffices there): R_kj =
            // v_k^dag h_j / |v_k| above the diagonal; the diagonal slot holds (|v_k|, 1 / |v_k|)
            if (j > k) rpk[j * (j + 1) / 2 + k] = make_float2(rr * rs, ri * rs);
            if (j == k) rpk[k * (k + 1) / 2 + k] = make_float2(nk * rs, rs);
        }
    }
    {   // normalise the own column and publish it
        const float2 sc = make_float2(inv_own, inv_own);
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            hr[p] = __fmul2_rn(hr[p], sc);
            hi[p] = __fmul2_rn(hi[p], sc);
        }
        __syncwarp();
        store_column2<D>(qre + j * QC, hr, qsw<D, QC>(j));
        store_column2<D>(qim + j * QC, hi, qsw<D, QC>(j));
        __syncwarp();
    }
    }   // PASSES > 0

    if constexpr (PASSES == 3) {
        // ---- 2b. refinement of Q1 to the QR factor of H beyond FP32 ----------------------------
        // An FP32 Gram-Schmidt factor Q1 is the exact factor of a matrix within 2^-24 of H, so it
        // misses U by about cond(H) 2^-24 -- and near the posterior U + I is nearly singular, so
        // that error reaches rho.  With Q1 = U V, V = I + X small: N = Q1^dag Q1 = I + X + X^dag
        // (first order) and M = Q1^dag H = V^dag R, whose strictly lower part is that of X^dag R.
        // So X^dag (called Y below) has: strictly lower part from the triangular system
        // lower(Y R) = lower(M), upper part N - conj(lower part)^T, real diagonal (N_jj - 1) / 2,
        // imaginary diagonal from the real diagonal of R; and U = Q1 V^-1 = Q1 (I - Y^dag) to
        // first order.  The step leaves about |Y|^2 (|Y| ~ cond(H) 2^-24): below FP32 rounding
        // while every |Y| entry is below 2^-14 (cond(H) up to ~10^3).  A chain above that repeats
        // the step from the refined U, its H and the same R; each pass squares the residual, and
        // three passes cover cond(H) up to ~10^6.  (The posterior's chains reach cond(H) ~10^5:
        // one chain in 1024 of a four-qubit problem with 81,000 shots after 2000 steps, which a
        // single pass left 6e-3 from the oracle's log L.)
        // The lower part of M and N - I are tiny differences of O(1) products, so they are formed
        // without rounding error: lane j forms row j (c < j: M_jc = q_j^dag h_c; c > j: N_jc =
        // q_j^dag q_c) with error-free products (sum_products_exact), its own q_j in (hr, hi) and
        // the other vector read from shared memory -- the lanes take different vectors at the
        // same step only through their addresses, so every lane does useful work at every step.
        // Lanes c > j then solve row j of the lower system as M_jc arrives (R from the sweep).
        // C[j][c] (row j = lane j) is kept in area B: step c frees H's column c, whose 2 D floats
        // take the D lanes' results of that step -- element (r, c) at c D + (r ^ c) of the real
        // (hre) and imaginary (him) planes, so that the lanes' writes of a step, a lane's reads
        // of its row and the reads of a column all hit distinct banks.
        float ymax;
        if constexpr (GRP == 2)
            ymax = refine_pass_split<D, QC>(hr, hi, qre, qim, hre, him, rpk, gsrc, j, grp);
        else
            ymax = refine_pass<D, QC>(hr, hi, qre, qim, hre, him, rpk, gsrc, j, false, true);
        if (__any_sync(0xffffffffu, ymax > kRefineTol))
            refine_more<D, QC, (GRP > 1)>(qre, qim, hre, him, rpk, gsrc, j, ymax, grp == 0);
    }

    if constexpr (PASSES == 2) {
        // ---- 2b. re-orthogonalisation Q2 = Q1 (I - F), F = strict upper part of E (formed in
        // the sweep above) plus half the diagonal E_jj = |q_j|^2 - 1 of the stored columns ------
        {
            float2 n = make_float2(0.f, 0.f);
#pragma unroll
            for (int p = 0; p < D / 2; ++p) n = __ffma2_rn(hr[p], hr[p], __ffma2_rn(hi[p], hi[p], n));
            fre[j * D + j] = 0.5f * (hsum(n) - 1.0f);
            fim[j * D + j] = 0.0f;
            if (j + 1 < D) {   // F[j+1][j] = 0: read in the pair (j, j+1) of column j
                fre[j * D + j + 1] = 0.0f;
                fim[j * D + j + 1] = 0.0f;
            }
        }
        __syncwarp();
        // row a of Q2: x_m - sum_{i <= m} x_i F[i][m], x = row a of Q1 (lane a = j), as pairs
        // (x_2p, x_2p+1); a pair that reaches past m meets F[m+1][m] = 0
        {
            float2 xr[D / 2], xi[D / 2];
#pragma unroll
            for (int p = 0; p < D / 2; ++p) {
                xr[p] = make_float2(qre[(2 * p) * QC + j], qre[(2 * p + 1) * QC + j]);
                xi[p] = make_float2(qim[(2 * p) * QC + j], qim[(2 * p + 1) * QC + j]);
            }
#pragma unroll
            for (int m = D - 1; m >= 0; --m) {   // descending: x_m is still Q1's when row m is formed
                float2 ca = make_float2(0.f, 0.f), cb = ca, cc2 = ca, cd = ca;
#pragma unroll
                for (int p = 0; 2 * p <= m; ++p) {
                    float2 fx, fy;   // F[2p][m], F[2p+1][m]
                    if constexpr (D >= 4) {
                        if ((p & 1) == 0) {
                            const float4 f4x = *reinterpret_cast<const float4 *>(fre + m * D + 2 * p);
                            const float4 f4y = *reinterpret_cast<const float4 *>(fim + m * D + 2 * p);
                            fx = make_float2(f4x.x, f4x.y);
                            fy = make_float2(f4y.x, f4y.y);
                        } else {
                            fx = *reinterpret_cast<const float2 *>(fre + m * D + 2 * p);
                            fy = *reinterpret_cast<const float2 *>(fim + m * D + 2 * p);
                        }
                    } else {
                        fx = *reinterpret_cast<const float2 *>(fre + m * D + 2 * p);
                        fy = *reinterpret_cast<const float2 *>(fim + m * D + 2 * p);
                    }
                    ca = __ffma2_rn(xr[p], fx, ca);    // sum xr fx
                    cb = __ffma2_rn(xi[p], fy, cb);    // sum xi fy
                    cc2 = __ffma2_rn(xr[p], fy, cc2);  // sum xr fy
                    cd = __ffma2_rn(xi[p], fx, cd);    // sum xi fx
                }
                const float dr = hsum(ca) - hsum(cb), di = hsum(cc2) + hsum(cd);
                if (m & 1) {
                    xr[m / 2].y -= dr;
                    xi[m / 2].y -= di;
                } else {
                    xr[m / 2].x -= dr;
                    xi[m / 2].x -= di;
                }
            }
#pragma unroll
            for (int p = 0; p < D / 2; ++p) {
                qre[(2 * p) * QC + j] = xr[p].x;
                qre[(2 * p + 1) * QC + j] = xr[p].y;
                qim[(2 * p) * QC + j] = xi[p].x;
                qim[(2 * p + 1) * QC + j] = xi[p].y;
            }
        }
        __syncwarp();
    }

    if constexpr (D == 16) {
        // ---- 3. W = (U + I) G in 4x4 register blocks: lane (bi, bj) forms W[4bi.., 4bj..] -----
        // G is staged row-major as separate real and imaginary planes in area B (free between
        // the re-orthogonalisation and the packed rho), so that columns (4bj, 4bj+1) and
        // (4bj+2, 4bj+3) of a row are f32x2 pairs and U's entries enter broadcast: eight
        // packed FMAs per row of U instead of sixteen scalar ones.
        float *gsr = sm + S::area_a, *gsi = gsr + D * D;
        {
            if constexpr (GRP == 2) {   // a plane per group
                float v[D];
#pragma unroll
                for (int i = 0; i < D; ++i) v[i] = 0.0f;
                if (active) load_column<D>(gsrc + grp * d + j * D, v);
                float *plane = grp ? gsi : gsr;
#pragma unroll
                for (int i = 0; i < D; ++i) plane[i * D + j] = v[i];
            } else {
                float gr[D], gi[D];
                if (active) {
                    load_column<D>(gsrc + j * D, gr);
                    load_column<D>(gsrc + d + j * D, gi);
                } else {
#pragma unroll
                    for (int i = 0; i < D; ++i) gr[i] = gi[i] = 0.0f;
                }
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    gsr[i * D + j] = gr[i];
                    gsi[i * D + j] = gi[i];
                }
            }
        }
        __syncwarp();
        const int bi = j >> 2, bj = j & 3;
        // W[4bi + r][4bj + 2h .. 4bj + 2h + 1], two rows at a time: the products of Re U (and G
        // itself, the identity's term) in one pair of chains (wr, wi), those of Im U in another
        // (xr, xi), added at the end -- each chain half as long, with the rounding of the two
        // sums kept apart until the one final add (the assembly's log L error grows with the
        // length of the chains that form W).  The first two rows wait in registers until
        // every lane is done with U, whose storage W takes.
        constexpr int NB = 2 / GRP;   // pairs of rows per lane
        float2 wr[2 * NB][2], wi[2 * NB][2];
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
            const int hb = GRP == 1 ? nb : grp;
            float2 ar[2][2], ai[2][2], xr[2][2], xi[2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int row = 4 * bi + 2 * hb + r;
                const float4 g4r = *reinterpret_cast<const float4 *>(gsr + row * D + 4 * bj);
                const float4 g4i = *reinterpret_cast<const float4 *>(gsi + row * D + 4 * bj);
                ar[r][0] = make_float2(g4r.x, g4r.y);
                ar[r][1] = make_float2(g4r.z, g4r.w);
                ai[r][0] = make_float2(g4i.x, g4i.y);
                ai[r][1] = make_float2(g4i.z, g4i.w);
                xr[r][0] = xr[r][1] = xi[r][0] = xi[r][1] = make_float2(0.f, 0.f);
            }
#pragma unroll 4
            for (int k = 0; k < (PASSES > 0 ? D : 0); ++k) {
                const float2 ur2 = *reinterpret_cast<const float2 *>(qre + k * QC + 4 * (bi ^ qsw<D, QC>(k)) + 2 * hb);
                const float2 ui2 = *reinterpret_cast<const float2 *>(qim + k * QC + 4 * (bi ^ qsw<D, QC>(k)) + 2 * hb);
                const float4 g4r = *reinterpret_cast<const float4 *>(gsr + k * D + 4 * bj);
                const float4 g4i = *reinterpret_cast<const float4 *>(gsi + k * D + 4 * bj);
                const float2 gr2[2] = {make_float2(g4r.x, g4r.y), make_float2(g4r.z, g4r.w)};
                const float2 gi2[2] = {make_float2(g4i.x, g4i.y), make_float2(g4i.z, g4i.w)};
                const float ur[2] = {ur2.x, ur2.y}, ui[2] = {ui2.x, ui2.y};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float2 pu = make_float2(ur[r], ur[r]), pi = make_float2(ui[r], ui[r]);
                    const float2 mi = make_float2(-ui[r], -ui[r]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        ar[r][h] = __ffma2_rn(pu, gr2[h], ar[r][h]);
                        xr[r][h] = __ffma2_rn(mi, gi2[h], xr[r][h]);
                        ai[r][h] = __ffma2_rn(pu, gi2[h], ai[r][h]);
                        xi[r][h] = __ffma2_rn(pi, gr2[h], xi[r][h]);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    wr[2 * nb + r][h] = __fadd2_rn(ar[r][h], xr[r][h]);
                    wi[2 * nb + r][h] = __fadd2_rn(ai[r][h], xi[r][h]);
                }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 2 * NB; ++r) {   // W row-major with padded rows (replaces Q)
            float2 *row = wsm + (4 * bi + (GRP == 1 ? 0 : 2 * grp) + r) * RS + 4 * bj;
            *reinterpret_cast<float4 *>(row) = make_float4(wr[r][0].x, wi[r][0].x, wr[r][0].y, wi[r][0].y);
            *reinterpret_cast<float4 *>(row + 2) = make_float4(wr[r][1].x, wi[r][1].x, wr[r][1].y, wi[r][1].y);
        }
        __syncwarp();
    } else {
    // ---- 3. W = (U + I) G, column j: W[:,j] = G[:,j] + sum_k U[:,k] G[k,j] ------------------
        float gr[D], gi[D], wr[D], wi[D];
        if (active) {
            load_column<D>(gsrc + j * D, gr);
            load_column<D>(gsrc + d + j * D, gi);
        } else {
    #pragma unroll
            for (int i = 0; i < D; ++i) {
                gr[i] = 0.0f;
                gi[i] = 0.0f;
            }
        }
    #pragma unroll
        for (int i = 0; i < D; ++i) {
            wr[i] = gr[i];
            wi[i] = gi[i];
        }
    #pragma unroll
        for (int k = 0; k < (PASSES > 0 ? D : 0); ++k) {
            float ur[D], ui[D];
            load_column<D>(qre + k * QC, ur, qsw<D, QC>(k));
            load_column<D>(qim + k * QC, ui, qsw<D, QC>(k));
    #pragma unroll
            for (int i = 0; i < D; ++i) {
                wr[i] = __fmaf_rn(ur[i], gr[k], __fmaf_rn(-ui[i], gi[k], wr[i]));
                wi[i] = __fmaf_rn(ur[i], gi[k], __fmaf_rn(ui[i], gr[k], wi[i]));
            }
        }
        __syncwarp();
        // W row-major with padded rows: W[i][j] at wsm[i * RS + j] (replaces Q)
    #pragma unroll
        for (int i = 0; i < D; ++i) wsm[i * RS + j] = make_float2(wr[i], wi[i]);
        __syncwarp();
    
    }

    // ---- 4. rho = W W^dag / Tr: lane a owns entries (a, a + t mod D), t = 0..D/2 ------------
    // (W W^dag)_ab = sum_m W[a,m] conj(W[b,m]): with the row of b read as complex pairs
    // (Re, Im) W[b,m], Re is the sum of both halves of (Re, Im) W[a,m] * (Re, Im) W[b,m] and Im
    // that of (Im, -Re) W[a,m] * (Re, Im) W[b,m]
    const int arow = j;
    float2 wa[D], wc[D];   // (Re, Im) W[a,m] and (Im, -Re) W[a,m]
#pragma unroll
    for (int m = 0; m < D; m += 2) {
        const float4 v = *reinterpret_cast<const float4 *>(wsm + arow * RS + m);
        wa[m] = make_float2(v.x, v.y);
        wa[m + 1] = make_float2(v.z, v.w);
        wc[m] = make_float2(v.y, -v.x);
        wc[m + 1] = make_float2(v.w, -v.z);
    }
    float diag;
    {
        float2 d0 = make_float2(0.f, 0.f), d1 = d0;
#pragma unroll
        for (int m = 0; m < D; m += 2) {
            d0 = __ffma2_rn(wa[m], wa[m], d0);
            d1 = __ffma2_rn(wa[m + 1], wa[m + 1], d1);
        }
        diag = hsum(d0) + hsum(d1);
    }
    const float inv_tr = 1.0f / group_sum<D>(diag);
    const float diag_n = diag * inv_tr;
    float tr_hi, tr_lo;
    group_sum_exact<D>(diag_n, tr_hi, tr_lo);   // exact trace of the stored diagonal
    packed[arow * PK + arow] = diag_n;
    // For t = D/2 lanes a and a + D/2 both form the entry pair {a, a + D/2}; the two results are
    // bitwise equal (the same products, accumulated in the same order, negated where the
    // conjugate is taken), so both stores may stand.
#pragma unroll 1
    for (int t = 1 + grp; t <= D / 2; t += GRP) {
        const int b = (arow + t) & (D - 1);
        float2 re0 = make_float2(0.f, 0.f), im0 = re0, re1 = re0, im1 = re0;
#pragma unroll
        for (int m = 0; m < D; m += 2) {
            const float4 wb = *reinterpret_cast<const float4 *>(wsm + b * RS + m);
            const float2 b0 = make_float2(wb.x, wb.y), b1 = make_float2(wb.z, wb.w);
            re0 = __ffma2_rn(wa[m], b0, re0);
            im0 = __ffma2_rn(wc[m], b0, im0);
            re1 = __ffma2_rn(wa[m + 1], b1, re1);
            im1 = __ffma2_rn(wc[m + 1], b1, im1);
        }
        const float re = (hsum(re0) + hsum(re1)) * inv_tr;
        const float im = (hsum(im0) + hsum(im1)) * inv_tr;
        const bool upper = arow < b;
        packed[arow * PK + b] = upper ? re : im;
        packed[b * PK + arow] = upper ? -im : re;
    }
    if (active && l == 0) a.trace_out[c] = (double)tr_hi + (double)tr_lo;
    __syncwarp();

    // ---- 5. store packed rho (FP32) and its exact bf16 split ----------------------------------
    if (active) {
        float *dst = a.rho_out + c * a.d_pad;
        for (int e = 4 * l; e < d; e += 4 * LPC) {
            // entries e .. e+3 of the row-major packed rho, staged with row stride PK
            auto staged = [&](int ee) { return packed[(ee / D) * PK + (ee % D)]; };
            const float4 v = make_float4(staged(e), staged(e + 1), staged(e + 2), staged(e + 3));
            *reinterpret_cast<float4 *>(dst + e) = v;
            if (a.rho_norm_out) *reinterpret_cast<float4 *>(a.rho_norm_out + c * d + e) = v;
            if (a.split_out) {
                const float vv[4] = {v.x, v.y, v.z, v.w};
                __nv_bfloat16 hs[4], ms[4], ls[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    hs[u] = __float2bfloat16_rn(vv[u]);
                    const float r1 = vv[u] - __bfloat162float(hs[u]);
                    ms[u] = __float2bfloat16_rn(r1);
                    const float r2 = r1 - __bfloat162float(ms[u]);
                    ls[u] = __float2bfloat16_rn(r2);
                }
                __nv_bfloat16 *sp = a.split_out + c * 3 * (int64_t)a.d_pad + e;
                *reinterpret_cast<uint2 *>(sp) = *reinterpret_cast<const uint2 *>(hs);
                *reinterpret_cast<uint2 *>(sp + a.d_pad) = *reinterpret_cast<const uint2 *>(ms);
                *reinterpret_cast<uint2 *>(sp + 2 * a.d_pad) = *reinterpret_cast<const uint2 *>(ls);
            }
            if (a.split_tf) {   // TF32 hi = v rounded to 11 significant bits, lo = TF32(v - hi)
                const float4 hi = make_float4(tf32_rna(v.x), tf32_rna(v.y), tf32_rna(v.z), tf32_rna(v.w));
                float *sp = a.split_tf + c * (int64_t)a.tf_splits * a.d_pad + e;
                *reinterpret_cast<float4 *>(sp) = hi;
                if (a.tf_splits == 2)
                    *reinterpret_cast<float4 *>(sp + a.d_pad) = make_float4(
                        tf32_rna(v.x - hi.x), tf32_rna(v.y - hi.y), tf32_rna(v.z - hi.z), tf32_rna(v.w - hi.w));
            }
        }
    }
}

// W = G + U G for one lane's block of 4 rows x 8 columns: rows 4 bi .. 4 bi + 3, columns 4 bj .. and
// HALF + 4 bj ...  U column-major at stride qc (entry i of a column at at(i)), G row-major [D][D];
// W's real and imaginary planes replace U's, row-major at stride qc (entry i of a row at at(i)),
// after `sync` has seen every lane done with U.  An entry is sum_k U_ik G_kj in k's order (the two
// products of a part one FMA after the other), then G_ij added.
template <int D, int HALF, bool HAS_U, class At, class Sync>
__device__ __forceinline__ void w_blocks(float *qre, float *qim, const float *gsr, const float *gsi, int bi, int bj, int qc,
                                         At at, Sync sync) {
    float2 wr[4][4], wi[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int h = 0; h < 4; ++h) wr[r][h] = wi[r][h] = make_float2(0.f, 0.f);
    auto row_pairs = [&](const float *g, int row, float2 (&v)[4]) {
        const float4 x = *reinterpret_cast<const float4 *>(g + row * D + 4 * bj);
        const float4 y = *reinterpret_cast<const float4 *>(g + row * D + HALF + 4 * bj);
        v[0] = make_float2(x.x, x.y);
        v[1] = make_float2(x.z, x.w);
        v[2] = make_float2(y.x, y.y);
        v[3] = make_float2(y.z, y.w);
    };
    if constexpr (HAS_U) {
#pragma unroll 2
        for (int k = 0; k < D; ++k) {
            const float4 ur4 = *reinterpret_cast<const float4 *>(qre + k * qc + at(4 * bi));
            const float4 ui4 = *reinterpret_cast<const float4 *>(qim + k * qc + at(4 * bi));
            float2 gr2[4], gi2[4];
            row_pairs(gsr, k, gr2);
            row_pairs(gsi, k, gi2);
            const float ur[4] = {ur4.x, ur4.y, ur4.z, ur4.w}, ui[4] = {ui4.x, ui4.y, ui4.z, ui4.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float2 pu = make_float2(ur[r], ur[r]), pi = make_float2(ui[r], ui[r]);
                const float2 mi = make_float2(-ui[r], -ui[r]);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    wr[r][h] = __ffma2_rn(pu, gr2[h], __ffma2_rn(mi, gi2[h], wr[r][h]));
                    wi[r][h] = __ffma2_rn(pu, gi2[h], __ffma2_rn(pi, gr2[h], wi[r][h]));
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float2 g[4];
        row_pairs(gsr, 4 * bi + r, g);
#pragma unroll
        for (int h = 0; h < 4; ++h) wr[r][h] = __fadd2_rn(wr[r][h], g[h]);
        row_pairs(gsi, 4 * bi + r, g);
#pragma unroll
        for (int h = 0; h < 4; ++h) wi[r][h] = __fadd2_rn(wi[r][h], g[h]);
    }
    sync();   // U is read by every lane before W replaces it
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float *re = qre + (4 * bi + r) * qc, *im = qim + (4 * bi + r) * qc;
        *reinterpret_cast<float4 *>(re + at(4 * bj)) = make_float4(wr[r][0].x, wr[r][0].y, wr[r][1].x, wr[r][1].y);
        *reinterpret_cast<float4 *>(re + at(HALF + 4 * bj)) = make_float4(wr[r][2].x, wr[r][2].y, wr[r][3].x, wr[r][3].y);
        *reinterpret_cast<float4 *>(im + at(4 * bj)) = make_float4(wi[r][0].x, wi[r][0].y, wi[r][1].x, wi[r][1].y);
        *reinterpret_cast<float4 *>(im + at(HALF + 4 * bj)) = make_float4(wi[r][2].x, wi[r][2].y, wi[r][3].x, wi[r][3].y);
    }
}

// ---- five qubits (D = 32): one warp per chain ----------------------------------------------
// The same algorithm with the same lane ownership (lane j: column j, then row j), but at D = 32 a
// lane cannot also hold the operand it is multiplied with, so that operand is streamed from
// shared memory four complex entries (two 128-bit loads) at a time.  With PASSES = 3 the
// refinement of U runs as in the D <= 16 kernel (refine_pass); its copy of H and the packed R take
// 4.2 KB more per chain, so that form runs two chains per CTA (THREADS = 64): five CTAs, ten
// warps, on an SM.
template <int PASSES = 2, int THREADS = kThreads>
struct WideShape {
    static constexpr int D = 32;
    static constexpr int d = D * D;
    static constexpr int chains_per_block = THREADS / D;
    static constexpr int qcol = D + 4;                      // floats per column of a Q plane
    static constexpr int pk_stride = D + 1;
    static constexpr int area_a = 2 * D * qcol;             // Q planes, then W as two planes of stride qcol
    static constexpr int area_b = 2 * D * D;                // F planes (PASSES = 3: H's columns), then the staged rho
    static constexpr int area_r = (PASSES == 3) ? D * (D + 1) : 0;   // PASSES = 3: packed R
    static constexpr int smem_floats = (area_a + area_b + area_r + 31) / 32 * 32 + 16;
};
using Wide = WideShape<>;
static_assert(Wide::area_b >= Wide::D * Wide::pk_stride, "areas");

template <int PASSES, int THREADS = kThreads>
__global__ void __launch_bounds__(THREADS, 3 * kThreads / THREADS) propose_kernel_d32(ProposeArgs a) {
    using S = WideShape<PASSES, THREADS>;
    constexpr int D = S::D, d = S::d, nx = 4 * d, QC = S::qcol, PK = S::pk_stride;
    extern __shared__ __align__(16) float smem[];
    const int j = threadIdx.x % D;
    const int g = threadIdx.x / D;
    const int64_t c = (int64_t)blockIdx.x * S::chains_per_block + g;
    const bool active = c < a.rows;
    const uint32_t step = (a.step_dev && a.mode == MODE_STEP) ? a.step_dev->step + 1u : a.step;
    if (a.step_dev && a.mode == MODE_STEP && blockIdx.x == 0 && threadIdx.x == 0) open_step(a.step_dev);
    float *sm = smem + g * S::smem_floats;
    float *qre = sm, *qim = sm + D * QC;                 // Q planes (column stride QC)
    float *wre = sm, *wim = sm + D * QC;                 // W planes (row stride QC), replace Q
    float *fre = sm + S::area_a, *fim = fre + D * D;     // F column-major (stride D), re / im planes
    float *packed = sm + S::area_a;                      // staged rho (row stride PK), replaces F
    float *hre = sm + S::area_a, *him = hre + D * D;     // PASSES = 3: H's columns (stride D), in area B
    float2 *rpk = reinterpret_cast<float2 *>(sm + S::area_a + S::area_b);   // PASSES = 3: packed R

    // ---- 1. latent proposal (as in the D <= 16 kernel: lane j takes blocks j, j + 32, .. of each part,
    // H's blocks go through the Q planes to the lanes that own their columns) ---------------------
    float coef_y = 1.0f, coef_eta = 0.0f;
    int cur = 0;
    if (active && a.mode == MODE_STEP) {
        cur = a.cur[c];
        const float2 cf = a.coef[c];
        coef_y = cf.x;
        coef_eta = cf.y;
    } else if (a.mode == MODE_INIT) {
        coef_y = 0.0f;
        coef_eta = 1.0f;
    }
    const int64_t cc = active ? c : 0;
    const uint32_t chain_id = (uint32_t)(a.chain_offset + cc);
    const uint32_t tag = (a.mode == MODE_INIT) ? TAG_INIT : TAG_PROPOSAL;
    const float *ysrc = a.y + ((int64_t)cur * a.R + cc) * nx;
    float *ydst = a.y + ((int64_t)(1 - cur) * a.R + cc) * nx;
    const float *gsrc = (a.mode == MODE_EVAL) ? a.x_eval + cc * nx : ydst;
    float2 hr[D / 2], hi[D / 2];   // H's column j, entries (2p, 2p + 1) in pair p
#pragma unroll 1
    for (int part = 0; part < 4; ++part) {
        const int e0 = part * d + 4 * j;
        float4 y0[D / 4];
#pragma unroll
        for (int q = 0; q < D / 4; ++q) {
            y0[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (active && a.mode == MODE_STEP) y0[q] = *reinterpret_cast<const float4 *>(ysrc + e0 + 4 * D * q);
            if (active && a.mode == MODE_EVAL) y0[q] = *reinterpret_cast<const float4 *>(a.x_eval + cc * nx + e0 + 4 * D * q);
        }
#pragma unroll
        for (int q = 0; q < D / 4; ++q) {
            float4 yn = y0[q];
            if (a.mode != MODE_EVAL) {
                const uint4 w = Philox::block(make_uint4((uint32_t)(e0 / 4 + D * q), step, chain_id, tag), a.rk);
                float z0, z1, z2, z3;
                gaussian_pair_fast(w.x, w.y, z0, z1);
                gaussian_pair_fast(w.z, w.w, z2, z3);
                yn.x = __fmaf_rn(coef_y, y0[q].x, coef_eta * z0);
                yn.y = __fmaf_rn(coef_y, y0[q].y, coef_eta * z1);
                yn.z = __fmaf_rn(coef_y, y0[q].z, coef_eta * z2);
                yn.w = __fmaf_rn(coef_y, y0[q].w, coef_eta * z3);
                if (active) *reinterpret_cast<float4 *>(ydst + e0 + 4 * D * q) = yn;
            }
            const int blk = j + D * q, at = blk / (D / 4) * QC + 4 * (blk % (D / 4));
            if (part == 2) *reinterpret_cast<float4 *>(qre + at) = yn;
            if (part == 3) *reinterpret_cast<float4 *>(qim + at) = yn;
        }
    }
    __syncwarp();
    load_column2<D>(qre + j * QC, hr);
    load_column2<D>(qim + j * QC, hi);
    __syncwarp();   // (the sweep publishes its columns there)
    if constexpr (PASSES == 3) {   // H's original columns, for the refinement after the sweep
        store_column2<D>(hre + j * D, hr);
        store_column2<D>(him + j * D, hi);
    }

    // ---- 2a. modified Gram-Schmidt, the published column streamed in chunks --------------------
    // As in the D <= 16 kernel: every lane forms r = v_k^dag h (lane k's is |v_k|^2, shuffled to
    // the others), one uniform rsqrt, a branch-free projection (zero coefficient on lanes
    // j <= k), and the lanes j < k form the Gram entries of the re-orthogonalisation.
    float inv_own = 0.0f;
#pragma unroll 1
    for (int k = 0; k < (PASSES > 0 ? D : 0); ++k) {   // (PASSES = 0, the Hilbert-Schmidt prior: no QR)
        if (j == k) {
            store_column2<D>(qre + k * QC, hr);
            store_column2<D>(qim + k * QC, hi);
        }
        __syncwarp();
        float2 vr[D / 2], vi[D / 2];   // held for the projection too: the broadcast loads are what bounds the sweep
        load_column2<D>(qre + k * QC, vr);
        load_column2<D>(qim + k * QC, vi);
        float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0, a3 = a0, b0 = a0, b1 = a0, b2 = a0, b3 = a0;
#pragma unroll
        for (int p = 0; p < D / 2; p += 2) {
            a0 = __ffma2_rn(vr[p], hr[p], a0);
            a1 = __ffma2_rn(vi[p], hi[p], a1);
            b0 = __ffma2_rn(vr[p], hi[p], b0);
            b1 = __ffma2_rn(vi[p], hr[p], b1);
            a2 = __ffma2_rn(vr[p + 1], hr[p + 1], a2);
            a3 = __ffma2_rn(vi[p + 1], hi[p + 1], a3);
            b2 = __ffma2_rn(vr[p + 1], hi[p + 1], b2);
            b3 = __ffma2_rn(vi[p + 1], hr[p + 1], b3);
        }
        const float rr = (hsum(a0) + hsum(a1)) + (hsum(a2) + hsum(a3));
        const float ri = (hsum(b0) - hsum(b1)) + (hsum(b2) - hsum(b3));
        const float nk = __shfl_sync(0xffffffffu, rr, k);   // |v_k|^2 from lane k
        const float rs = rsqrtf(nk);
        const float coef = (j > k) ? rs * rs : 0.0f;
        const float sr = rr * coef, si = ri * coef;
        const float2 msr = make_float2(-sr, -sr), psi = make_float2(si, si), msi = make_float2(-si, -si);
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            hr[p] = __ffma2_rn(msr, vr[p], __ffma2_rn(psi, vi[p], hr[p]));
            hi[p] = __ffma2_rn(msr, vi[p], __ffma2_rn(msi, vr[p], hi[p]));
        }
        inv_own = (j == k) ? rs : inv_own;
        if constexpr (PASSES == 2) {
            if (j < k) {
                const float sc = inv_own * rs;   // E_jk = conj(r) / (|v_j| |v_k|), j < k
                fre[k * D + j] = rr * sc;
                fim[k * D + j] = -ri * sc;
            }
        }
        if constexpr (PASSES == 3) {   // R for the refinement's solve, as in the D <= 16 kernel
            if (j > k) rpk[j * (j + 1) / 2 + k] = make_float2(rr * rs, ri * rs);
            if (j == k) rpk[k * (k + 1) / 2 + k] = make_float2(nk * rs, rs);
        }
    }
    if constexpr (PASSES > 0) {   // normalise the own column and publish it
        const float2 sc = make_float2(inv_own, inv_own);
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            hr[p] = __fmul2_rn(hr[p], sc);
            hi[p] = __fmul2_rn(hi[p], sc);
        }
        __syncwarp();
        store_column2<D>(qre + j * QC, hr);
        store_column2<D>(qim + j * QC, hi);
        __syncwarp();
    }

    if constexpr (PASSES == 3) {
        // ---- 2b. refinement of Q1 to the QR factor of H beyond FP32 (the D <= 16 kernel's step 2b:
        // error-free M and N rows per lane, the triangular solve, U = Q1 - Q1 Y^dag, repeated while
        // the chain's largest |Y| entry exceeds kRefineTol) ----------------------------------------
        const float ymax = refine_pass<D, QC>(hr, hi, qre, qim, hre, him, rpk, gsrc, j, false, true);
        if (__any_sync(0xffffffffu, ymax > kRefineTol)) refine_more<D, QC, false>(qre, qim, hre, him, rpk, gsrc, j, ymax, true);
    }

    if constexpr (PASSES == 2) {
        // ---- 2b. Q2 = Q1 (I - F): F's diagonal, then row a of Q1 (I - F) (as in D <= 16) ----------
        {
            float2 n = make_float2(0.f, 0.f);
#pragma unroll
            for (int p = 0; p < D / 2; ++p) n = __ffma2_rn(hr[p], hr[p], __ffma2_rn(hi[p], hi[p], n));
            fre[j * D + j] = 0.5f * (hsum(n) - 1.0f);
            fim[j * D + j] = 0.0f;
            if (j + 1 < D) {
                fre[j * D + j + 1] = 0.0f;
                fim[j * D + j + 1] = 0.0f;
            }
        }
        __syncwarp();
        {
            float2 xr[D / 2], xi[D / 2];
#pragma unroll
            for (int p = 0; p < D / 2; ++p) {
                xr[p] = make_float2(qre[(2 * p) * QC + j], qre[(2 * p + 1) * QC + j]);
                xi[p] = make_float2(qim[(2 * p) * QC + j], qim[(2 * p + 1) * QC + j]);
            }
#pragma unroll
            for (int m = D - 1; m >= 0; --m) {
                float2 ca = make_float2(0.f, 0.f), cb = ca, cc2 = ca, cd = ca;
#pragma unroll
                for (int p = 0; 2 * p <= m; ++p) {
                    float2 fx, fy;   // F[2p][m], F[2p+1][m]
                    if ((p & 1) == 0) {
                        const float4 f4x = *reinterpret_cast<const float4 *>(fre + m * D + 2 * p);
                        const float4 f4y = *reinterpret_cast<const float4 *>(fim + m * D + 2 * p);
                        fx = make_float2(f4x.x, f4x.y);
                        fy = make_float2(f4y.x, f4y.y);
                    } else {
                        fx = *reinterpret_cast<const float2 *>(fre + m * D + 2 * p);
                        fy = *reinterpret_cast<const float2 *>(fim + m * D + 2 * p);
                    }
                    ca = __ffma2_rn(xr[p], fx, ca);
                    cb = __ffma2_rn(xi[p], fy, cb);
                    cc2 = __ffma2_rn(xr[p], fy, cc2);
                    cd = __ffma2_rn(xi[p], fx, cd);
                }
                const float dr = hsum(ca) - hsum(cb), di = hsum(cc2) + hsum(cd);
                if (m & 1) {
                    xr[m / 2].y -= dr;
                    xi[m / 2].y -= di;
                } else {
                    xr[m / 2].x -= dr;
                    xi[m / 2].x -= di;
                }
            }
#pragma unroll
            for (int p = 0; p < D / 2; ++p) {
                qre[(2 * p) * QC + j] = xr[p].x;
                qre[(2 * p + 1) * QC + j] = xr[p].y;
                qim[(2 * p) * QC + j] = xi[p].x;
                qim[(2 * p + 1) * QC + j] = xi[p].y;
            }
        }
        __syncwarp();
    }

    // ---- 3. W = G + U G in blocks of 4 rows x 8 columns per lane (rows 4 bi .., columns 4 bj .. and
    // 16 + 4 bj ..), each entry the sum over k in order and then G's entry: a k costs six 128-bit
    // loads, of which a warp reads 128 bytes each at most, where column j per lane took sixteen
    // broadcast ones.  G is staged row-major as real and imaginary planes in area B.
    {
        float *gsr = sm + S::area_a, *gsi = gsr + D * D;
#pragma unroll
        for (int q = 0; q < D / 4; ++q) {
            float4 g4r = make_float4(0.f, 0.f, 0.f, 0.f), g4i = g4r;
            if (active) {
                g4r = *reinterpret_cast<const float4 *>(gsrc + j * D + 4 * q);
                g4i = *reinterpret_cast<const float4 *>(gsrc + d + j * D + 4 * q);
            }
            gsr[(4 * q) * D + j] = g4r.x;
            gsr[(4 * q + 1) * D + j] = g4r.y;
            gsr[(4 * q + 2) * D + j] = g4r.z;
            gsr[(4 * q + 3) * D + j] = g4r.w;
            gsi[(4 * q) * D + j] = g4i.x;
            gsi[(4 * q + 1) * D + j] = g4i.y;
            gsi[(4 * q + 2) * D + j] = g4i.z;
            gsi[(4 * q + 3) * D + j] = g4i.w;
        }
        __syncwarp();
        w_blocks<D, 16, (PASSES > 0)>(qre, qim, gsr, gsi, j >> 2, j & 3, QC, [](int i) { return i; },
                                            [] { __syncwarp(); });
        __syncwarp();
    }

    // ---- 4. rho = W W^dag / Tr, lane a: entries (a, a + t mod D), row b streamed --------------
    // Re (W W^dag)_ab = sum Re W_am Re W_bm + Im W_am Im W_bm and Im = sum Im W_am Re W_bm -
    // Re W_am Im W_bm, on pairs of columns m.  For t = D/2 lanes a and a + D/2 both form the pair
    // {a, a + D/2}; the results are bitwise equal (the same products in the same order), so both
    // stores may stand.
    const int arow = j;
    float2 war[D / 2], wai[D / 2];
#pragma unroll
    for (int p = 0; p < D / 2; p += 2) {
        const float4 r4 = *reinterpret_cast<const float4 *>(wre + arow * QC + 2 * p);
        const float4 i4 = *reinterpret_cast<const float4 *>(wim + arow * QC + 2 * p);
        war[p] = make_float2(r4.x, r4.y);
        war[p + 1] = make_float2(r4.z, r4.w);
        wai[p] = make_float2(i4.x, i4.y);
        wai[p + 1] = make_float2(i4.z, i4.w);
    }
    float diag;
    {
        float2 d0 = make_float2(0.f, 0.f), d1 = d0;
#pragma unroll
        for (int p = 0; p < D / 2; ++p) {
            d0 = __ffma2_rn(war[p], war[p], d0);
            d1 = __ffma2_rn(wai[p], wai[p], d1);
        }
        diag = hsum(d0) + hsum(d1);
    }
    const float inv_tr = 1.0f / group_sum<D>(diag);
    const float diag_n = diag * inv_tr;
    float tr_hi, tr_lo;
    group_sum_exact<D>(diag_n, tr_hi, tr_lo);
    __syncwarp();   // every lane holds its W row before F's area becomes the staged rho
    packed[arow * PK + arow] = diag_n;
#pragma unroll 1
    for (int t = 1; t <= D / 2; ++t) {
        const int b = (arow + t) & (D - 1);
        float2 re = make_float2(0.f, 0.f), ima = re, imb = re;
#pragma unroll
        for (int p = 0; p < D / 2; p += 2) {
            const float4 r4 = *reinterpret_cast<const float4 *>(wre + b * QC + 2 * p);
            const float4 i4 = *reinterpret_cast<const float4 *>(wim + b * QC + 2 * p);
            const float2 br0 = make_float2(r4.x, r4.y), br1 = make_float2(r4.z, r4.w);
            const float2 bi0 = make_float2(i4.x, i4.y), bi1 = make_float2(i4.z, i4.w);
            re = __ffma2_rn(wai[p], bi0, __ffma2_rn(war[p], br0, re));
            ima = __ffma2_rn(wai[p], br0, ima);
            imb = __ffma2_rn(war[p], bi0, imb);
            re = __ffma2_rn(wai[p + 1], bi1, __ffma2_rn(war[p + 1], br1, re));
            ima = __ffma2_rn(wai[p + 1], br1, ima);
            imb = __ffma2_rn(war[p + 1], bi1, imb);
        }
        const float rv = hsum(re) * inv_tr;
        const float iv = (hsum(ima) - hsum(imb)) * inv_tr;
        const bool upper = arow < b;
        packed[arow * PK + b] = upper ? rv : iv;
        packed[b * PK + arow] = upper ? -iv : rv;
    }
    if (active && j == 0) a.trace_out[c] = (double)tr_hi + (double)tr_lo;
    __syncwarp();

    // ---- 5. store packed rho (FP32) and its exact bf16 split ----------------------------------
    if (active) {
        float *dst = a.rho_out + c * a.d_pad;
        for (int e = 4 * j; e < d; e += 4 * D) {
            auto staged = [&](int ee) { return packed[(ee / D) * PK + (ee % D)]; };
            const float4 v = make_float4(staged(e), staged(e + 1), staged(e + 2), staged(e + 3));
            *reinterpret_cast<float4 *>(dst + e) = v;
            if (a.rho_norm_out) *reinterpret_cast<float4 *>(a.rho_norm_out + c * d + e) = v;
            if (a.split_out) {
                const float vv[4] = {v.x, v.y, v.z, v.w};
                __nv_bfloat16 hs[4], ms[4], ls[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    hs[u] = __float2bfloat16_rn(vv[u]);
                    const float r1 = vv[u] - __bfloat162float(hs[u]);
                    ms[u] = __float2bfloat16_rn(r1);
                    const float r2 = r1 - __bfloat162float(ms[u]);
                    ls[u] = __float2bfloat16_rn(r2);
                }
                __nv_bfloat16 *sp = a.split_out + c * 3 * (int64_t)a.d_pad + e;
                *reinterpret_cast<uint2 *>(sp) = *reinterpret_cast<const uint2 *>(hs);
                *reinterpret_cast<uint2 *>(sp + a.d_pad) = *reinterpret_cast<const uint2 *>(ms);
                *reinterpret_cast<uint2 *>(sp + 2 * a.d_pad) = *reinterpret_cast<const uint2 *>(ls);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// D = 64 (six qubits): one 128-thread CTA per chain, two threads per column (thread 2 j + h holds
// rows 32 h .. 32 h + 31 of column j).  The same steps as the kernels above, with CTA barriers
// where those use warp ones: the latent proposal and H's column half in registers; modified
// Gram-Schmidt with each column normalised by its owner pair and published to shared memory
// (the others project it out; pairs whose column is final form the Gram entries); the
// first-order re-orthogonalisation Q1 (I - F) (R21) by rows; W = (U + I) G by column halves;
// the Hermitian half of W W^dag by rows, the two threads of a row splitting its columns.
// ---------------------------------------------------------------------------------------
struct Wide64 {
    static constexpr int D = 64;
    static constexpr int d = D * D;
    static constexpr int threads = 128;
    // floats per column of a Q plane (per row of W): entry i sits at i + 4 (i / 32), so the two
    // halves a thread pair works on fall in different 16-byte bank groups and the eight float4
    // accesses of a quarter warp in distinct ones (72 = 18 groups of 4 floats per column)
    static constexpr int qcol = D + 8;
    static constexpr int pk_stride = D + 1;
    static constexpr int area_a = 2 * D * qcol;         // Q planes, then W as two planes of row stride qcol
    // F's planes are row-major; 68 floats a row keep the sweep's stores (one row per column pair) to two
    // rows per bank and the rows 16-byte aligned
    static constexpr int frow = D + 4;
    static constexpr int area_b = 2 * D * frow;         // F planes, then G's planes, then the staged rho
    static constexpr int smem_floats = area_a + area_b + 2 * D + 32;
};
static_assert(Wide64::area_b >= Wide64::D * Wide64::pk_stride, "areas");

template <int PASSES>
__global__ void __launch_bounds__(Wide64::threads, 3) propose_kernel_d64(ProposeArgs a) {
    using S = Wide64;
    constexpr int D = S::D, d = S::d, nx = 4 * d, QC = S::qcol, PK = S::pk_stride, H2 = D / 2;
    extern __shared__ __align__(16) float smem[];
    float *qre = smem, *qim = smem + D * QC;             // Q planes (column stride QC)
    float *wre = smem, *wim = smem + D * QC;             // W planes (row stride QC), replace Q
    float *fre = smem + S::area_a, *fim = fre + D * S::frow;   // F row-major (F[p][m] at p frow + m)
    float *packed = smem + S::area_a;                    // staged rho (row stride PK), replaces F
    float *rowv = smem + S::area_a + S::area_b;          // [D] per-row values (diagonal of W W^dag)
    const int t = threadIdx.x;
    const int j = t >> 1, hh = t & 1, r0 = H2 * hh;      // column (or row) j, half hh
    const int r0s = r0 + 4 * hh;                         // where half hh starts within a column (row)
    const unsigned pair_mask = 3u << ((t & 31) & ~1);
    const int64_t c = blockIdx.x;                        // one chain per CTA; the grid is exactly rows
    const uint32_t step = (a.step_dev && a.mode == MODE_STEP) ? a.step_dev->step + 1u : a.step;
    if (a.step_dev && a.mode == MODE_STEP && blockIdx.x == 0 && threadIdx.x == 0) open_step(a.step_dev);

    // ---- 1. latent proposal: this thread's 32 entries of column j of each part -----------------
    float coef_y = 1.0f, coef_eta = 0.0f;
    int cur = 0;
    if (a.mode == MODE_STEP) {
        cur = a.cur[c];
        const float2 cf = a.coef[c];
        coef_y = cf.x;
        coef_eta = cf.y;
    } else if (a.mode == MODE_INIT) {
        coef_y = 0.0f;
        coef_eta = 1.0f;
    }
    const uint32_t chain_id = (uint32_t)(a.chain_offset + c);
    const uint32_t tag = (a.mode == MODE_INIT) ? TAG_INIT : TAG_PROPOSAL;
    const float *ysrc = a.y + ((int64_t)cur * a.R + c) * nx;
    float *ydst = a.y + ((int64_t)(1 - cur) * a.R + c) * nx;
    const float *gsrc = (a.mode == MODE_EVAL) ? a.x_eval + c * nx : ydst;
    float2 hr[H2 / 2], hi[H2 / 2];   // rows r0 + 2p, r0 + 2p + 1 of H's column j in pair p
#pragma unroll 1
    for (int part = 0; part < 4; ++part) {
        // thread t takes blocks t, t + 128, ..; H's reach the threads that own them through the Q planes
        const int e0 = part * d + 4 * t;
        float4 y0[H2 / 4];
#pragma unroll
        for (int q = 0; q < H2 / 4; ++q) {
            y0[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (a.mode == MODE_STEP) y0[q] = *reinterpret_cast<const float4 *>(ysrc + e0 + 4 * S::threads * q);
            if (a.mode == MODE_EVAL) y0[q] = *reinterpret_cast<const float4 *>(a.x_eval + c * nx + e0 + 4 * S::threads * q);
        }
#pragma unroll
        for (int q = 0; q < H2 / 4; ++q) {
            float4 yn = y0[q];
            if (a.mode != MODE_EVAL) {
                const uint4 w = Philox::block(make_uint4((uint32_t)(e0 / 4 + S::threads * q), step, chain_id, tag), a.rk);
                float z0, z1, z2, z3;
                gaussian_pair_fast(w.x, w.y, z0, z1);
                gaussian_pair_fast(w.z, w.w, z2, z3);
                yn.x = __fmaf_rn(coef_y, y0[q].x, coef_eta * z0);
                yn.y = __fmaf_rn(coef_y, y0[q].y, coef_eta * z1);
                yn.z = __fmaf_rn(coef_y, y0[q].z, coef_eta * z2);
                yn.w = __fmaf_rn(coef_y, y0[q].w, coef_eta * z3);
                *reinterpret_cast<float4 *>(ydst + e0 + 4 * S::threads * q) = yn;
            }
            const int blk = t + S::threads * q, r = blk % (D / 4);
            const int at = blk / (D / 4) * QC + 4 * r + 4 * (r / (D / 8));
            if (part == 2) *reinterpret_cast<float4 *>(qre + at) = yn;
            if (part == 3) *reinterpret_cast<float4 *>(qim + at) = yn;
        }
    }
    if constexpr (PASSES == 2) {   // F's entries below the diagonal count as zero
        for (int e = 4 * t; e < 2 * D * S::frow; e += 4 * S::threads)
            *reinterpret_cast<float4 *>(fre + e) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();   // y' (read back as G) is written, H staged
    load_column2<H2>(qre + j * QC + r0s, hr);
    load_column2<H2>(qim + j * QC + r0s, hi);
    __syncthreads();   // (the sweep publishes its columns there)

    // ---- 2a. modified Gram-Schmidt: q_k = v_k / |v_k| published by its pair, projected out ------
#pragma unroll 1
    for (int k = 0; k < (PASSES > 0 ? D : 0); ++k) {   // (PASSES = 0, the Hilbert-Schmidt prior: no QR)
        if (j == k) {
            float2 n2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int p = 0; p < H2 / 2; ++p) n2 = __ffma2_rn(hr[p], hr[p], __ffma2_rn(hi[p], hi[p], n2));
            float n = hsum(n2);
            n += __shfl_xor_sync(pair_mask, n, 1);
            const float2 rs = make_float2(rsqrtf(n), rsqrtf(n));
#pragma unroll
            for (int p = 0; p < H2 / 2; ++p) {
                hr[p] = __fmul2_rn(hr[p], rs);
                hi[p] = __fmul2_rn(hi[p], rs);
            }
            store_column2<H2>(qre + k * QC + r0s, hr);
            store_column2<H2>(qim + k * QC + r0s, hi);
        }
        __syncthreads();
        // r = q_k^dag h over this half, then both halves
        float2 vr[H2 / 2], vi[H2 / 2];   // held for the projection too
        load_column2<H2>(qre + k * QC + r0s, vr);
        load_column2<H2>(qim + k * QC + r0s, vi);
        float2 a0 = make_float2(0.f, 0.f), a1 = a0, b0 = a0, b1 = a0;
#pragma unroll
        for (int p = 0; p < H2 / 2; p += 2) {
            a0 = __ffma2_rn(vr[p], hr[p], __ffma2_rn(vr[p + 1], hr[p + 1], a0));
            a1 = __ffma2_rn(vi[p], hi[p], __ffma2_rn(vi[p + 1], hi[p + 1], a1));
            b0 = __ffma2_rn(vr[p], hi[p], __ffma2_rn(vr[p + 1], hi[p + 1], b0));
            b1 = __ffma2_rn(vi[p], hr[p], __ffma2_rn(vi[p + 1], hr[p + 1], b1));
        }
        float rr = hsum(a0) + hsum(a1), ri = hsum(b0) - hsum(b1);
        rr += __shfl_xor_sync(0xffffffffu, rr, 1);
        ri += __shfl_xor_sync(0xffffffffu, ri, 1);
        if (j > k) {   // h -= r q_k
            const float2 msr = make_float2(-rr, -rr), psi = make_float2(ri, ri), msi = make_float2(-ri, -ri);
#pragma unroll
            for (int p = 0; p < H2 / 2; ++p) {
                hr[p] = __ffma2_rn(msr, vr[p], __ffma2_rn(psi, vi[p], hr[p]));
                hi[p] = __ffma2_rn(msr, vi[p], __ffma2_rn(msi, vr[p], hi[p]));
            }
        } else if (PASSES == 2 && j < k && hh == 0) {   // E_jk = q_j^dag q_k = conj(q_k^dag q_j)
            fre[j * S::frow + k] = rr;
            fim[j * S::frow + k] = -ri;
        }
    }

    if constexpr (PASSES == 2) {
        {   // F's diagonal: (|q_j|^2 - 1) / 2
            float2 n2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int p = 0; p < H2 / 2; ++p) n2 = __ffma2_rn(hr[p], hr[p], __ffma2_rn(hi[p], hi[p], n2));
            float n = hsum(n2);
            n += __shfl_xor_sync(0xffffffffu, n, 1);
            if (hh == 0) {
                fre[j * S::frow + j] = 0.5f * (n - 1.0f);
                fim[j * S::frow + j] = 0.0f;
            }
        }
        __syncthreads();
        // ---- 2b. Q2 = Q1 (I - F) in blocks of 4 rows x 4 columns per thread: columns 32 .. 63 first (they
        // need every column of Q1), then 0 .. 31 (which need those only).  An entry is Q1_am - sum over
        // p of Q1_ap F_pm in p's order; the terms p > m of a block are zeros of F.  Warp w takes columns
        // 8 w .. 8 w + 7 of the low half and the mirrored ones of the high half, so the warps' sums are
        // equally long (72 terms).  (A row per thread pair, one column after the other, took four scalar
        // loads for two packed FMAs: 332 us for 1024 chains, 263 this way.)
        const int bi = t & 15, bj = t >> 4;
        const int x0 = 4 * bi + 4 * (bi >> 3);   // where rows 4 bi .. sit within a column
        float2 q2r[4][2], q2i[4][2];             // Q2 of the block, pairs of columns
        auto block = [&](int m0, int terms) {    // columns m0 .. m0 + 3
            float2 rr[4][2], ii[4][2], ri[4][2], ir[4][2];   // sums of xr fr, xi fi, xr fi, xi fr
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) rr[r][h2] = ii[r][h2] = ri[r][h2] = ir[r][h2] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int p = 0; p < terms; ++p) {
                const float4 xr4 = *reinterpret_cast<const float4 *>(qre + p * QC + x0);
                const float4 xi4 = *reinterpret_cast<const float4 *>(qim + p * QC + x0);
                const float4 fr4 = *reinterpret_cast<const float4 *>(fre + p * S::frow + m0);
                const float4 fi4 = *reinterpret_cast<const float4 *>(fim + p * S::frow + m0);
                const float xr[4] = {xr4.x, xr4.y, xr4.z, xr4.w}, xi[4] = {xi4.x, xi4.y, xi4.z, xi4.w};
                const float2 fr[2] = {make_float2(fr4.x, fr4.y), make_float2(fr4.z, fr4.w)};
                const float2 fi[2] = {make_float2(fi4.x, fi4.y), make_float2(fi4.z, fi4.w)};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 pr = make_float2(xr[r], xr[r]), pi = make_float2(xi[r], xi[r]);
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) {
                        rr[r][h2] = __ffma2_rn(pr, fr[h2], rr[r][h2]);
                        ii[r][h2] = __ffma2_rn(pi, fi[h2], ii[r][h2]);
                        ri[r][h2] = __ffma2_rn(pr, fi[h2], ri[r][h2]);
                        ir[r][h2] = __ffma2_rn(pi, fr[h2], ir[r][h2]);
                    }
                }
            }
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4) {
                const float4 xr4 = *reinterpret_cast<const float4 *>(qre + (m0 + c4) * QC + x0);
                const float4 xi4 = *reinterpret_cast<const float4 *>(qim + (m0 + c4) * QC + x0);
                const float xr[4] = {xr4.x, xr4.y, xr4.z, xr4.w}, xi[4] = {xi4.x, xi4.y, xi4.z, xi4.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (c4 & 1) {
                        q2r[r][c4 / 2].y = xr[r] - (rr[r][c4 / 2].y - ii[r][c4 / 2].y);
                        q2i[r][c4 / 2].y = xi[r] - (ri[r][c4 / 2].y + ir[r][c4 / 2].y);
                    } else {
                        q2r[r][c4 / 2].x = xr[r] - (rr[r][c4 / 2].x - ii[r][c4 / 2].x);
                        q2i[r][c4 / 2].x = xi[r] - (ri[r][c4 / 2].x + ir[r][c4 / 2].x);
                    }
                }
            }
        };
        auto put = [&](int m0) {
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                float *c0 = qre + (m0 + 2 * h2) * QC + x0, *c1 = qim + (m0 + 2 * h2) * QC + x0;
                *reinterpret_cast<float4 *>(c0) = make_float4(q2r[0][h2].x, q2r[1][h2].x, q2r[2][h2].x, q2r[3][h2].x);
                *reinterpret_cast<float4 *>(c0 + QC) = make_float4(q2r[0][h2].y, q2r[1][h2].y, q2r[2][h2].y, q2r[3][h2].y);
                *reinterpret_cast<float4 *>(c1) = make_float4(q2i[0][h2].x, q2i[1][h2].x, q2i[2][h2].x, q2i[3][h2].x);
                *reinterpret_cast<float4 *>(c1 + QC) = make_float4(q2i[0][h2].y, q2i[1][h2].y, q2i[2][h2].y, q2i[3][h2].y);
            }
        };
        const int w8 = 8 * (t >> 5);
        block(H2 + 4 * (7 - bj), H2 + 32 - w8);
        __syncthreads();   // every thread has read the high columns
        put(H2 + 4 * (7 - bj));
        block(4 * bj, w8 + 8);
        __syncthreads();
        put(4 * bj);
        __syncthreads();
    } else {
        __syncthreads();
    }

    // ---- 3. W = G + U G in blocks of 4 rows x 8 columns per thread (w_blocks), G staged row-major in
    // area B (F is no longer needed) ------------------------------------------------------------------
    {
        float *gsr = smem + S::area_a, *gsi = gsr + D * D;
#pragma unroll
        for (int q = 0; q < H2 / 4; ++q) {
            const float4 g4r = *reinterpret_cast<const float4 *>(gsrc + j * D + r0 + 4 * q);
            const float4 g4i = *reinterpret_cast<const float4 *>(gsrc + d + j * D + r0 + 4 * q);
            const float gr[4] = {g4r.x, g4r.y, g4r.z, g4r.w}, gi[4] = {g4i.x, g4i.y, g4i.z, g4i.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                gsr[(r0 + 4 * q + u) * D + j] = gr[u];
                gsi[(r0 + 4 * q + u) * D + j] = gi[u];
            }
        }
        __syncthreads();
        w_blocks<D, H2, (PASSES > 0)>(qre, qim, gsr, gsi, t >> 3, t & 7, QC, [](int i) { return i + 4 * (i >> 5); },
                                      [] { __syncthreads(); });
        __syncthreads();
    }

    // ---- 4. rho = W W^dag / Tr: row a = j, this thread's half of the columns m ------------------
    const int arow = j;
    float2 war[H2 / 2], wai[H2 / 2];
#pragma unroll
    for (int p = 0; p < H2 / 2; p += 2) {
        const float4 r4 = *reinterpret_cast<const float4 *>(wre + arow * QC + r0s + 2 * p);
        const float4 i4 = *reinterpret_cast<const float4 *>(wim + arow * QC + r0s + 2 * p);
        war[p] = make_float2(r4.x, r4.y);
        war[p + 1] = make_float2(r4.z, r4.w);
        wai[p] = make_float2(i4.x, i4.y);
        wai[p + 1] = make_float2(i4.z, i4.w);
    }
    {
        float2 d0 = make_float2(0.f, 0.f), d1 = d0;
#pragma unroll
        for (int p = 0; p < H2 / 2; ++p) {
            d0 = __ffma2_rn(war[p], war[p], d0);
            d1 = __ffma2_rn(wai[p], wai[p], d1);
        }
        float diag = hsum(d0) + hsum(d1);
        diag += __shfl_xor_sync(0xffffffffu, diag, 1);
        if (hh == 0) rowv[arow] = diag;
    }
    __syncthreads();
    float tr = 0.0f;   // Tr W W^dag in row order (every thread alike)
    for (int r = 0; r < D; ++r) tr += rowv[r];
    const float inv_tr = 1.0f / tr;
    if (hh == 0) packed[arow * PK + arow] = rowv[arow] * inv_tr;
#pragma unroll 1
    for (int s = 1; s <= D / 2; ++s) {
        const int b = (arow + s) & (D - 1);
        float2 re = make_float2(0.f, 0.f), ima = re, imb = re;
#pragma unroll
        for (int p = 0; p < H2 / 2; p += 2) {
            const float4 r4 = *reinterpret_cast<const float4 *>(wre + b * QC + r0s + 2 * p);
            const float4 i4 = *reinterpret_cast<const float4 *>(wim + b * QC + r0s + 2 * p);
            const float2 br0 = make_float2(r4.x, r4.y), br1 = make_float2(r4.z, r4.w);
            const float2 bi0 = make_float2(i4.x, i4.y), bi1 = make_float2(i4.z, i4.w);
            re = __ffma2_rn(wai[p], bi0, __ffma2_rn(war[p], br0, re));
            ima = __ffma2_rn(wai[p], br0, ima);
            imb = __ffma2_rn(war[p], bi0, imb);
            re = __ffma2_rn(wai[p + 1], bi1, __ffma2_rn(war[p + 1], br1, re));
            ima = __ffma2_rn(wai[p + 1], br1, ima);
            imb = __ffma2_rn(war[p + 1], bi1, imb);
        }
        // both halves, in the same order for both threads of the pair
        float rs = hsum(re), is = hsum(ima) - hsum(imb);
        const float rs_o = __shfl_xor_sync(0xffffffffu, rs, 1), is_o = __shfl_xor_sync(0xffffffffu, is, 1);
        const float rv = (hh == 0 ? rs + rs_o : rs_o + rs) * inv_tr;
        const float iv = (hh == 0 ? is + is_o : is_o + is) * inv_tr;
        if (hh == 0) {
            const bool upper = arow < b;
            packed[arow * PK + b] = upper ? rv : iv;
            packed[b * PK + arow] = upper ? -iv : rv;
        }
    }
    if (t == 0) {   // the exact trace of the stored (normalised) diagonal, in row order
        float th = 0.0f, tl = 0.0f;
        for (int r = 0; r < D; ++r) {
            const float x = rowv[r] * inv_tr;
            const float sum = th + x, bp = sum - th;
            tl += (th - (sum - bp)) + (x - bp);
            th = sum;
        }
        a.trace_out[c] = (double)th + (double)tl;
    }
    __syncthreads();

    // ---- 5. store packed rho (FP32) -----------------------------------------------------------
    float *dst = a.rho_out + c * a.d_pad;
    for (int e = 4 * t; e < d; e += 4 * S::threads) {
        auto staged = [&](int ee) { return packed[(ee / D) * PK + (ee % D)]; };
        const float4 v = make_float4(staged(e), staged(e + 1), staged(e + 2), staged(e + 3));
        *reinterpret_cast<float4 *>(dst + e) = v;
        if (a.rho_norm_out) *reinterpret_cast<float4 *>(a.rho_norm_out + c * d + e) = v;
    }
}

template <int PASSES>
cudaError_t launch_propose_d64(const ProposeArgs &a, cudaStream_t s) {
    using S = Wide64;
    const size_t smem = sizeof(float) * S::smem_floats;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(propose_kernel_d64<PASSES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(propose_kernel_d64<PASSES>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    if (a.rows <= 0) return cudaSuccess;
    propose_kernel_d64<PASSES><<<(unsigned)a.rows, S::threads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int PASSES>
cudaError_t launch_propose_d32(const ProposeArgs &a, cudaStream_t s) {
    constexpr int THREADS = (PASSES == 3) ? 64 : kThreads;   // two chains per CTA with the refinement
    using S = WideShape<PASSES, THREADS>;
    const size_t smem = sizeof(float) * S::smem_floats * S::chains_per_block;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(propose_kernel_d32<PASSES, THREADS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(propose_kernel_d32<PASSES, THREADS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const int64_t blocks = (a.rows + S::chains_per_block - 1) / S::chains_per_block;
    if (blocks == 0) return cudaSuccess;
    propose_kernel_d32<PASSES, THREADS><<<(unsigned)blocks, THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

template <int D, int PASSES, int THREADS, int GRP = 1>
cudaError_t launch_propose_small(const ProposeArgs &a, int64_t rows, cudaStream_t s) {
    using S = Shape<D, PASSES, THREADS>;
    constexpr int chains = THREADS / (D * GRP);
    const size_t smem = sizeof(float) * S::smem_floats * chains;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(propose_kernel<D, PASSES, THREADS, GRP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(propose_kernel<D, PASSES, THREADS, GRP>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const int64_t blocks = (rows + chains - 1) / chains;
    if (blocks == 0) return cudaSuccess;
    propose_kernel<D, PASSES, THREADS, GRP><<<(unsigned)blocks, THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

template <int D, int PASSES>
cudaError_t launch_propose_pd(const ProblemView &p, int mode, uint32_t step, StepState *step_dev,
                              const float *x_eval, int64_t rows, bool want_split, float *rho_norm_out, cudaStream_t s) {
    ProposeArgs a;
    a.x_eval = x_eval;
    a.y = p.y;
    a.cur = p.cur;
    a.coef = p.coef;
    a.rho_out = p.rho_prop;
    a.split_out = (want_split && p.tc_kind == TC_BF16X3) ? static_cast<__nv_bfloat16 *>(p.rho_split) : nullptr;
    a.split_tf = (want_split && (p.tc_kind == TC_TF32 || p.tc_kind == TC_TF32X2)) ? static_cast<float *>(p.rho_split)
                                                                                   : nullptr;
    a.tf_splits = tc_splits(p.tc_kind);
    a.trace_out = p.trace_prop;
    a.rho_norm_out = (mode == MODE_EVAL) ? rho_norm_out : nullptr;
    a.rows = rows;
    a.R = p.R;
    a.chain_offset = p.chain_offset;
    a.seed = p.seed;
    a.rk = Philox::round_keys(p.seed);
    a.step = step;
    a.step_dev = step_dev;
    a.mode = mode;
    a.d_pad = p.d_pad;
    // the six-qubit kernel has no refinement: it takes the FP32 re-orthogonalisation
    constexpr int WIDE_PASSES = PASSES == 3 ? 2 : PASSES;
    if constexpr (D == 64) {
        if (a.split_out || a.split_tf) return cudaErrorNotSupported;   // no tensor-core form at D = 64
        return launch_propose_d64<WIDE_PASSES>(a, s);
    } else if constexpr (D == 32) {
        if (a.split_tf) return cudaErrorNotSupported;   // the TF32 forms stop at D = 16
        return launch_propose_d32<PASSES>(a, s);
    } else {
        // the CTA sizes the autotuner may pick are built for the default QR (3) and the
        // Hilbert-Schmidt prior (0); other settings run 128-thread CTAs
        if constexpr (PASSES == 3 && D >= 8) {
            if (propose_split(p, rows, mode != MODE_EVAL)) return launch_propose_small<D, PASSES, 64, 2>(a, rows, s);
        }
        if constexpr (PASSES == 0 || PASSES == 3) {
            if (p.propose_threads == 32) return launch_propose_small<D, PASSES, 32>(a, rows, s);
            if (p.propose_threads == 64) return launch_propose_small<D, PASSES, 64>(a, rows, s);
        }
        return launch_propose_small<D, PASSES, kThreads>(a, rows, s);
    }
}

template <int D>
cudaError_t launch_propose_d(const ProblemView &p, int mode, uint32_t step, StepState *step_dev, const float *x_eval,
                             int64_t rows, bool want_split, float *rho_norm_out, cudaStream_t s) {
    if (p.qr_passes == 0) return launch_propose_pd<D, 0>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
    if (p.qr_passes == 1) return launch_propose_pd<D, 1>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
    if (p.qr_passes == 2) return launch_propose_pd<D, 2>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
    return launch_propose_pd<D, 3>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
}

}  // namespace

// Two groups of lanes per chain (64-thread CTAs) at three and four qubits with the default QR and no
// CTA size asked for, up to two warps per scheduler at four qubits and one at three.  us at one / two
// groups: four qubits 64 chains 23.9 / 17.9, 1001 25.1 / 23.7, 2000 31.6 / 34.8; three qubits 64 chains
// 11.8 / 10.5, 1000 12.5 / 9.8, 2000 11.9 / 12.7.  In a step the handle's other problems of that size run at
// the same time and count as well, since the extra instructions then cost more than they shorten (277
// four-qubit chains beside 2087: 54 us per step with one group, 58 with two).
bool propose_split(const ProblemView &p, int64_t rows, bool step) {
    if (p.qr_passes != 3 || p.propose_fixed) return false;
    return (p.D == 16 || p.D == 8) && rows + (step ? p.beside : 0) <= 1216;
}

cudaError_t launch_propose(const ProblemView &p, int mode, uint32_t step, StepState *step_dev, const float *x_eval,
                           int64_t n_eval, bool want_split, float *rho_norm_out, uint32_t *status, cudaStream_t s) {
    (void)status;
    const int64_t rows = (mode == MODE_EVAL) ? n_eval : p.R;
    switch (p.D) {
        case 2: return launch_propose_d<2>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        case 4: return launch_propose_d<4>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        case 8: return launch_propose_d<8>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        case 16: return launch_propose_d<16>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        case 32: return launch_propose_d<32>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        case 64: return launch_propose_d<64>(p, mode, step, step_dev, x_eval, rows, want_split, rho_norm_out, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace qst
