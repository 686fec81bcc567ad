// Many steps of a one- or two-qubit problem in one launch (Algorithm 2 with Algorithm 1 inside).
//
// At D = 2 and 4 a chain's step is a few hundred arithmetic operations; as separate proposal,
// projection and accept kernels a step costs four dependent launches (14.7 us per step for 64
// one-qubit chains, 19.3 us for 4096 two-qubit chains) of which the arithmetic is a fraction.
// Chains never interact, so here the lanes of a chain run whole steps on their own: the latent
// state, rho and the chain's scalars stay in registers, the small matrices in a few hundred bytes
// of shared memory, and nothing but warp barriers orders a step.  A CTA is one warp, so that few
// chains spread over many SMs: 1.8 us per step for 64 one-qubit chains, 4.9 us for 4096 two-qubit
// chains.  Values are formed by the same operations in the same order as in the per-step kernels,
// with one exception: of log t, |t - 1| a few ulps, the second and third order (below 1e-14) are
// formed in FP32 here and in FP64 in the accept kernel.  They differ by 1e-22, times the counts far
// below log L's last bit: over 20 million proposals of one and two qubits no bit of log L differs
// (tests/test_gpu_many_log_l.py), so the chains are the same bits.  In FP64 here as well a step takes
// a fifth longer (64 one-qubit chains 1.8 -> 2.2 us, 4096 two-qubit chains 4.9 -> 5.3).
//
// What bounds a step here is one warp's chain of dependent instructions, and in it the FP64
// instructions (a sub-partition takes 64 cycles for each, conversions from FP32 included), so
// conversions are done on the integer pipe (f2d), t's parts stay in FP32 and only the sums that
// form log L are FP64.  Lanes per chain (LPC): with 4 D lanes the generator's blocks, the
// refinement's dot products and the settings go side by side, one per lane, where D lanes take
// four in turn; the steps that need only D lanes (the sweep, W, rho) are repeated by the other
// lanes.  That is the shorter step, but more instructions per chain, so it is used until the
// chip is full (the line is in launch_steps).
//
// Pooling (Eq. BME2) is the one step with an order across chains: the per-step accept kernel adds
// a CTA's 128 chains in FP32 in a fixed order and then into its FP64 slot.  So a launch writes the
// kept states of its chains to a history buffer and fused_pool_kernel adds them afterwards in that
// order, all kept steps of a launch in parallel.
#include <algorithm>

#include "pauli_dev.cuh"
#include "propose_dev.cuh"

namespace qst {
namespace {

constexpr int kWarp = 32;
constexpr int kMinCtas = 16;   // per SM: 128 registers (168 leave room for 12 warps, and 4096 chains then took a second wave)
constexpr int kSettingSlots = 4;   // settings per D lanes: up to 4 D of them (a power of two per chain)

struct FusedArgs {
    ProblemView p;
    SamplerParams sp;
    const StepState *base;   // the problem's step counter, as it was before this call
    uint32_t off;            // steps of earlier launches of this call
    int nsteps;
    int thin;
    int64_t burn_in;
    float *hist;             // [kept step of this launch][R][d]
    Philox::RoundKeys rk;
};

// kept steps among 1..j: the multiples of `thin` beyond `burn_in`
__device__ __forceinline__ int64_t kept_up_to(int64_t j, int thin, int64_t burn_in) {
    return j <= burn_in ? 0 : j / thin - burn_in / thin;
}

// (double)x by integer operations.  A denormal counts as zero: what is converted here are sums of terms of
// 1e-7 and more and their rounding errors, the smallest of them above 1e-20
__device__ __forceinline__ double f2d(float x) {
    const uint32_t b = __float_as_uint(x), e = b & 0x7f800000u;
    const uint32_t rebias = e == 0x7f800000u ? 0x70000000u : 0x38000000u;   // exponent 255 -> 2047, else + 896
    uint32_t hi = ((b & 0x7fffffffu) >> 3) + rebias, lo = b << 29;
    if (e == 0u) hi = lo = 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)lo);
}

template <int D, int PASSES, int LPC>
struct FusedShape {
    using S = Shape<D, PASSES, kWarp>;
    static constexpr int d = D * D, nx = 4 * d;
    // a chain's floats: the proposal's areas, then y'.  The stride is 4 mod 32, so that the eight (or
    // sixteen) chains of a warp reading the same offset fall in different bank groups
    static constexpr int raw = S::area_a + S::area_b + S::area_r + nx;
    static constexpr int stride = (raw + 27) / 32 * 32 + 4;
    static_assert(stride >= raw, "chain stride");
};

// One setting of the FP32 form (project_fp32_small_kernel's arithmetic): its FP64 contribution.
template <int D, bool POISSON>
__device__ __forceinline__ double setting_fp32(const float (&ar)[D * D], const float *ps, const float *cnt,
                                               const float *invf, float pk, int KD, int k, float t_hi, float t_lo) {
    constexpr int d = D * D;
    float q[D];
#pragma unroll
    for (int l = 0; l < D; ++l) q[l] = 0.0f;
#pragma unroll
    for (int i = 0; i < d; ++i) {   // one FMA chain per outcome, the setting's D outcomes side by side
        float pv[D];
        if constexpr (D == 4) {
            const float4 v = *reinterpret_cast<const float4 *>(ps + i * KD + k * D);
            pv[0] = v.x;
            pv[1] = v.y;
            pv[2] = v.z;
            pv[3] = v.w;
        } else {
            const float2 v = *reinterpret_cast<const float2 *>(ps + i * KD + k * D);
            pv[0] = v.x;
            pv[1] = v.y;
        }
#pragma unroll
        for (int l = 0; l < D; ++l) q[l] = __fmaf_rn(ar[i], pv[l], q[l]);
    }
    float sum = 0.0f, comp = 0.0f, small = 0.0f, sh = 0.0f, sl = 0.0f;
#pragma unroll
    for (int l = 0; l < D; ++l) {
        const int col = k * D + l;
        const float cv = cnt[col];
        if (cv > 0.0f) {   // Kahan: sum - comp
            const float y = __fmaf_rn(cv, deviance_log(q[l] * invf[col]), -comp);
            const float tt = sum + y;
            comp = (tt - sum) - y;
            sum = tt;
        }
        const float hq = (q[l] + 12.0f) - 12.0f;   // S_k as an exact pair
        sh += hq;
        sl += q[l] - hq;
    }
    if constexpr (POISSON) {   // -mu_k (S_k / t - 1)
        float ph, pl;
        poisson_setting(pk, sh, sl, t_hi, t_lo, ph, pl);
        const float y = -ph - comp;
        const float tt = sum + y;
        comp = (tt - sum) - y;
        sum = tt;
        small -= pl;
    } else {   // -P_k log(S_k / t)
        const float rel = ((sh - t_hi) + (sl - t_lo)) / t_hi;
        const float l1p = fabsf(rel) < 0x1p-10f ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                                : log1pf(rel);
        small -= pk * l1p;
    }
    return (f2d(sum) - f2d(comp)) + f2d(small);
}

// The structured Pauli form at one and two qubits (project_pauli_kernel's arithmetic with one
// thread per chain): m, the packed rho.
template <int D, bool POISSON>
__device__ __forceinline__ double pauli_small(const float (&m)[D * D], const PauliArgs &pa, float t_hi, float t_lo) {
    float2 dev = splat2(0.0f), comp = splat2(0.0f);
    int xmin = 0x7fffffff;
    const float inv_thi = 1.0f / t_hi;
    auto renorm = [&](float sh, float sl, float unit, int k) {
        const float rel = ((unit * sh - t_hi) + (unit * sl - t_lo)) * inv_thi;
        if constexpr (POISSON) return -__ldg(pa.ptot + k) * rel;
        const float l1p = fabsf(rel) < 0x1p-10f ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                                : log1pf(rel);
        return -__ldg(pa.ptot + k) * l1p;
    };
    float extra = 0.0f;
    float sh[3], sl[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) sh[j] = sl[j] = 0.0f;
    if constexpr (D == 2) {
        last_split<false>(m[0], m[1], m[2], m[3], pa, 0, 1, 0, dev, comp, xmin, sh, sl, nullptr, 0, 0.0f);
#pragma unroll
        for (int j = 0; j < 3; ++j) extra += renorm(sh[j], sl[j], j < 2 ? 0.5f : 1.0f, j);
    } else {
        float e00[6], e01[6], e10[6], e11[6];
        six(m[0] + m[10], 2.0f * m[2], 2.0f * m[8], m[0], m[10], e00);
        six(m[1] + m[11], m[3] + m[6], m[9] + m[12], m[1], m[11], e01);
        six(m[4] + m[14], m[12] - m[9], m[6] - m[3], m[4], m[14], e10);
        six(m[5] + m[15], 2.0f * m[7], 2.0f * m[13], m[5], m[15], e11);
#pragma unroll
        for (int c1 = 0; c1 < 6; ++c1) {
            last_split<false>(e00[c1], e01[c1], e10[c1], e11[c1], pa, 3 * c1, 1, 0, dev, comp, xmin, sh, sl, nullptr, 0,
                              0.0f);
            if (c1 & 1) {
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    extra += renorm(sh[j], sl[j], j < 2 ? 0.5f : 1.0f, 3 * (c1 >> 1) + j);
                    sh[j] = sl[j] = 0.0f;
                }
            }
        }
    }
    float acc_hi, acc_lo;
    two_sum(dev.x, dev.y, acc_hi, acc_lo);
    acc_lo += extra - (comp.x + comp.y);
    if (xmin < 0x00800000) acc_hi = -INFINITY;
    return f2d(acc_hi) + f2d(acc_lo);
}

template <int D, int PASSES, int LPC, bool PAULI, bool POISSON>
__global__ void __launch_bounds__(kWarp, kMinCtas) fused_small_kernel(const __grid_constant__ FusedArgs a) {
    using F = FusedShape<D, PASSES, LPC>;
    using S = typename F::S;
    constexpr int d = F::d, nx = F::nx, RS = S::row_stride, QC = S::qcol, PK = S::pk_stride;
    constexpr int GRP = LPC / D;          // groups of D lanes per chain
    constexpr int NP = 4 / GRP;           // parts of the latent state (and settings' slots) per lane
    static_assert(GRP == 1 || GRP == 2 || GRP == 4, "lanes per chain");
    static_assert(PASSES == 0 || PASSES == 3, "the default QR and the Hilbert-Schmidt prior");
    extern __shared__ __align__(16) float smem[];
    const ProblemView &p = a.p;
    const int l = threadIdx.x % LPC, g = threadIdx.x / LPC;   // lane of the chain, chain of the warp
    const int j = l % D;                  // owned column (and row); lanes l, l + D, .. share it
    const int grp = l / D, p0 = grp * NP; // its group, and the first part of the latent state it holds
    const bool own = l < D;               // of the lanes that share a column, the one that writes
    constexpr int chains = kWarp / LPC;   // of this CTA
    const int64_t c = (int64_t)blockIdx.x * chains + g;
    const bool active = c < p.R;
    // an idle group repeats the last chain, which is of this warp, and writes nothing (another warp's chain
    // could be written back while it is read)
    const int64_t cc = active ? c : p.R - 1;
    float *sm = smem + g * F::stride;
    float *qre = sm, *qim = sm + D * QC;
    float2 *wsm = reinterpret_cast<float2 *>(sm);
    float *packed = sm + S::area_a;
    float *hre = sm + S::area_a, *him = hre + D * D;
    float2 *rpk = reinterpret_cast<float2 *>(sm + S::area_a + S::area_b);
    float *ysm = sm + S::area_a + S::area_b + S::area_r;
    // the FP32 form's projectors [d][KD], counts and weights, once per launch
    float *ps = smem + chains * F::stride, *cnt_s = ps + d * p.KD, *invf_s = cnt_s + p.KD;
    const int K = p.KD / D;
    if constexpr (!PAULI) {
        for (int e = threadIdx.x; e < d * p.KD; e += kWarp) ps[e] = p.P32[(int64_t)(e / p.KD) * p.KD_pad + (e % p.KD)];
        for (int e = threadIdx.x; e < p.KD; e += kWarp) {
            cnt_s[e] = p.cnt[e];
            invf_s[e] = p.invf[e];
        }
        __syncwarp();
    }
    PauliArgs pa{};
    if constexpr (PAULI) {
        pa.wq = p.pauli_wq;
        pa.wc = p.pauli_wc;
        pa.ptot = p.ptot;
    }

    // the chain's state
    const uint32_t step0 = a.base->step + a.off;   // steps taken before this launch
    const int64_t kept0 = kept_up_to(step0, a.thin, a.burn_in);
    int64_t kept_idx = a.base->kept_count + kept0 - kept_up_to(a.base->step, a.thin, a.burn_in);   // of the next kept step
    uint32_t until_kept = (uint32_t)a.thin - step0 % (uint32_t)a.thin;          // steps to the next multiple of T
    uint32_t until_adapt = a.sp.adapt_interval > 0 ? (uint32_t)a.sp.adapt_interval - step0 % (uint32_t)a.sp.adapt_interval : 0u;
    const uint32_t chain_id = (uint32_t)(p.chain_offset + cc);
    float2 coef = p.coef[cc];
    double logl_cur = p.logl_cur[cc], beta = p.beta[cc];
    int32_t win = p.acc_win[cc];
    int64_t acc_total = p.acc_total[cc];
    float *yst = p.y + ((int64_t)p.cur[cc] * p.R + cc) * nx;
    float y[NP][D], rc[D];   // column j of this lane's parts of the latent state; row j of the packed rho
#pragma unroll
    for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int i = 0; i < D; ++i) y[q][i] = yst[(p0 + q) * d + j * D + i];
#pragma unroll
    for (int i = 0; i < D; ++i) rc[i] = p.rho_cur[cc * p.d_pad + j * D + i];
    float *hist = a.hist + cc * d + j * D;
    float log_alphas = 0.0f;   // log alpha of LPC steps, one per lane

#pragma unroll 1
    for (int s = 0; s < a.nsteps; ++s) {
        const uint32_t step = step0 + 1u + (uint32_t)s;
        if (s % LPC == 0) {   // the accept draws of the next LPC steps
            const uint4 w = Philox::block(make_uint4(0u, step + (uint32_t)l, chain_id, TAG_ALPHA), a.rk);
            log_alphas = logf(((float)(w.x >> 9) + 0.5f) * 0x1p-23f);
        }
        const float log_alpha = __shfl_sync(0xffffffffu, log_alphas, s % LPC, LPC);
        // ---- latent proposal (propose_kernel, step 1) ----
        float yn[NP][D];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int part = p0 + q;
            if constexpr (D == 4) {
                const uint4 w = Philox::block(make_uint4((uint32_t)(part * 4 + j), step, chain_id, TAG_PROPOSAL), a.rk);
                float z0, z1, z2, z3;
                gaussian_pair_fast(w.x, w.y, z0, z1);
                gaussian_pair_fast(w.z, w.w, z2, z3);
                yn[q][0] = __fmaf_rn(coef.x, y[q][0], coef.y * z0);
                yn[q][1] = __fmaf_rn(coef.x, y[q][1], coef.y * z1);
                yn[q][2] = __fmaf_rn(coef.x, y[q][2], coef.y * z2);
                yn[q][3] = __fmaf_rn(coef.x, y[q][3], coef.y * z3);
                *reinterpret_cast<float4 *>(ysm + part * d + j * D) = make_float4(yn[q][0], yn[q][1], yn[q][2], yn[q][3]);
            } else {
                const uint4 w = Philox::block(make_uint4((uint32_t)part, step, chain_id, TAG_PROPOSAL), a.rk);
                float z0, z1;
                gaussian_pair_fast(j == 0 ? w.x : w.z, j == 0 ? w.y : w.w, z0, z1);
                yn[q][0] = __fmaf_rn(coef.x, y[q][0], coef.y * z0);
                yn[q][1] = __fmaf_rn(coef.x, y[q][1], coef.y * z1);
                *reinterpret_cast<float2 *>(ysm + part * d + j * D) = make_float2(yn[q][0], yn[q][1]);
            }
        }
        float gr[D], gi[D];            // G's column j
        float2 hr[D / 2], hi[D / 2];   // H's column j
        if constexpr (GRP > 1) {
            __syncwarp();   // the chain's other lanes' parts
            load_column<D>(ysm + j * D, gr);
            load_column<D>(ysm + d + j * D, gi);
            load_column2<D>(ysm + 2 * d + j * D, hr);
            load_column2<D>(ysm + 3 * d + j * D, hi);
        } else {
#pragma unroll
            for (int i = 0; i < D; ++i) {
                gr[i] = yn[0][i];
                gi[i] = yn[NP > 1 ? 1 : 0][i];
            }
#pragma unroll
            for (int q = 0; q < D / 2; ++q) {
                hr[q] = make_float2(yn[NP > 2 ? 2 : 0][2 * q], yn[NP > 2 ? 2 : 0][2 * q + 1]);
                hi[q] = make_float2(yn[NP > 3 ? 3 : 0][2 * q], yn[NP > 3 ? 3 : 0][2 * q + 1]);
            }
        }
        // ---- QR of H and the refinement of U (steps 2a, 2b) ----
        if constexpr (PASSES == 3) {
            store_column2<D>(hre + j * D, hr);
            store_column2<D>(him + j * D, hi);
            float inv_own = 0.0f;
#pragma unroll
            for (int k = 0; k < D; ++k) {
                if (j == k) {
                    store_column2<D>(qre + k * QC, hr);
                    store_column2<D>(qim + k * QC, hi);
                }
                __syncwarp();
                float2 vr[D / 2], vi[D / 2];
                load_column2<D>(qre + k * QC, vr);
                load_column2<D>(qim + k * QC, vi);
                float2 a0 = make_float2(0.f, 0.f), a1 = a0, b0 = a0, b1 = a0;
#pragma unroll
                for (int q = 0; q < D / 2; ++q) {
                    a0 = __ffma2_rn(vr[q], hr[q], a0);
                    a1 = __ffma2_rn(vi[q], hi[q], a1);
                    b0 = __ffma2_rn(vr[q], hi[q], b0);
                    b1 = __ffma2_rn(vi[q], hr[q], b1);
                }
                const float rr = hsum(a0) + hsum(a1);
                const float ri = hsum(b0) - hsum(b1);
                const float nk = __shfl_sync(0xffffffffu, rr, k, D);
                const float rs = rsqrtf(nk);
                const float cf = (j > k) ? rs * rs : 0.0f;
                const float sr = rr * cf, si = ri * cf;
                const float2 msr = make_float2(-sr, -sr), psi = make_float2(si, si), msi = make_float2(-si, -si);
#pragma unroll
                for (int q = 0; q < D / 2; ++q) {
                    hr[q] = __ffma2_rn(msr, vr[q], __ffma2_rn(psi, vi[q], hr[q]));
                    hi[q] = __ffma2_rn(msr, vi[q], __ffma2_rn(msi, vr[q], hi[q]));
                }
                inv_own = (j == k) ? rs : inv_own;
                if (j > k) rpk[j * (j + 1) / 2 + k] = make_float2(rr * rs, ri * rs);
                if (j == k) rpk[k * (k + 1) / 2 + k] = make_float2(nk * rs, rs);
            }
            const float2 sc = make_float2(inv_own, inv_own);
#pragma unroll
            for (int q = 0; q < D / 2; ++q) {
                hr[q] = __fmul2_rn(hr[q], sc);
                hi[q] = __fmul2_rn(hi[q], sc);
            }
            __syncwarp();
            store_column2<D>(qre + j * QC, hr);
            store_column2<D>(qim + j * QC, hi);
            __syncwarp();
            float ymax;
            if constexpr (GRP > 1) {
                // refine_pass with row j's entries of C shared out over the groups: columns cc = grp, grp + GRP, ..
                // (mod D), all of them formed before any replaces H
                constexpr int NC = D > GRP ? D / GRP : 1;
                float2 res[NC];
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const int cc1 = (grp + i * GRP) % D;
                    const bool lower = cc1 < j;
                    res[i] = sum_products_exact<D>(hr, hi, lower ? hre + cc1 * D : qre + cc1 * QC,
                                                   lower ? him + cc1 * D : qim + cc1 * QC, lower ? 192.0f : 6.0f,
                                                   cc1 == j ? 1.0f : 0.0f);
                }
                const float2 mjj = sum_products_exact<D>(hr, hi, hre + j * D, him + j * D, 192.0f, 0.0f);
                __syncwarp();   // every lane is done with H's columns
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const int cc1 = (grp + i * GRP) % D;
                    hre[cc1 * D + (j ^ cc1)] = res[i].x;
                    him[cc1 * D + (j ^ cc1)] = res[i].y;
                }
                __syncwarp();
                ymax = refine_tail<D, QC, true>(qre, qim, hre, him, rpk, j, mjj, own);
            } else {
                ymax = refine_pass<D, QC>(hr, hi, qre, qim, hre, him, rpk, ysm, j, false, true);
            }
            if (__any_sync(0xffffffffu, ymax > kRefineTol))
                refine_more<D, QC, (GRP > 1)>(qre, qim, hre, him, rpk, ysm, j, ymax, own);
        }
        // ---- W = (U + I) G and rho = W W^dag / Tr (steps 3, 4) ----
        float wr[D], wi[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            wr[i] = gr[i];
            wi[i] = gi[i];
        }
#pragma unroll
        for (int k = 0; k < (PASSES > 0 ? D : 0); ++k) {
            float ur[D], ui[D];
            load_column<D>(qre + k * QC, ur);
            load_column<D>(qim + k * QC, ui);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                wr[i] = __fmaf_rn(ur[i], gr[k], __fmaf_rn(-ui[i], gi[k], wr[i]));
                wi[i] = __fmaf_rn(ur[i], gi[k], __fmaf_rn(ui[i], gr[k], wi[i]));
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < D; ++i) wsm[i * RS + j] = make_float2(wr[i], wi[i]);
        __syncwarp();
        float2 wa[D], wc[D];
#pragma unroll
        for (int m = 0; m < D; m += 2) {
            const float4 v = *reinterpret_cast<const float4 *>(wsm + j * RS + m);
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
        group_sum_exact<D>(diag_n, tr_hi, tr_lo);
        packed[j * PK + j] = diag_n;
#pragma unroll
        for (int t = 1; t <= D / 2; ++t) {
            const int b = (j + t) & (D - 1);
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
            const bool upper = j < b;
            packed[j * PK + b] = upper ? re : im;
            packed[b * PK + j] = upper ? -im : re;
        }
        // t = t_hi + t_lo, t_hi the FP32 nearest (the per-step kernels' split of the FP64 trace)
        const float t_hi = tr_hi + tr_lo, t_lo = tr_lo - (t_hi - tr_hi);
        __syncwarp();

        // ---- log L (the projection kernels) ----
        float ar[d];
#pragma unroll
        for (int i = 0; i < d; ++i) ar[i] = packed[(i / D) * PK + i % D];
        double v = 0.0;
        if constexpr (PAULI) {
            v = pauli_small<D, POISSON>(ar, pa, t_hi, t_lo);
        } else {
            // lane l takes settings l, l + LPC, ..; their sum is the binary tree of the per-step kernel's
            // shuffles (its absent settings contribute zero)
            double part[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                part[i] = 0.0;
                const int k = l + LPC * i;
                if (LPC * i < K) {   // (uniform)
                    const int kk = k < K ? k : K - 1;
                    const double one = setting_fp32<D, POISSON>(ar, ps, cnt_s, invf_s, __ldg(p.ptot + kk), p.KD, kk, t_hi, t_lo);
                    part[i] = k < K ? one : 0.0;
#pragma unroll
                    for (int off = 1; off < LPC; off <<= 1)
                        if (off < K) part[i] += __shfl_xor_sync(0xffffffffu, part[i], off);   // (uniform)
                }
            }
            v = part[0];
            if (NP > 1 && LPC < K) v += part[NP > 1 ? 1 : 0];
            if (NP > 2 && 2 * LPC < K) v += part[NP > 2 ? 2 : 0] + part[NP > 3 ? 3 : 0];
            // fewer settings than lanes: the tree's sum is in its own lanes only, and all of the chain's need it
            if (K < LPC) v = __shfl_sync(0xffffffffu, v, 0, LPC);   // (uniform)
        }

        // ---- accept, adaptation (accept_kernel, phase 1) ----
        const float itr = 1.0f / t_hi;
        const float dlf = (t_hi - 1.0f) + t_lo;
        double log_t;   // log1p(t - 1): t - 1 exactly in FP64, the second and third order (1e-14) in FP32
        if (fabsf(dlf) < 0x1p-10f)
            log_t = (f2d(t_hi - 1.0f) + f2d(t_lo)) - f2d(dlf * dlf * (0.5f - dlf * (1.0f / 3.0f)));
        else
            log_t = log((double)tr_hi + (double)tr_lo);
        const double logl_prop = p.C0 - p.Ntot * log_t + v;
        const bool acc = f2d(log_alpha) < logl_prop - logl_cur;
        if (acc) {
            logl_cur = logl_prop;
            win += 1;
            acc_total += 1;
        }
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int i = 0; i < D; ++i) y[q][i] = acc ? yn[q][i] : y[q][i];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const float nv = packed[j * PK + i] * itr;
            rc[i] = acc ? nv : rc[i];
        }
        if (p.trace_steps > 0 && step <= (uint32_t)p.trace_steps && active && l == 0) {
            const int64_t t = (int64_t)(step - 1) * p.R + c;
            p.trace_acc[t] = acc ? 1 : 0;
            p.trace_logl[t] = logl_prop;
        }
        if (a.sp.adapt_interval > 0 && --until_adapt == 0u) {
            until_adapt = (uint32_t)a.sp.adapt_interval;
            const double rate = (double)win / (double)a.sp.adapt_interval;
            if (rate > a.sp.acc_hi) beta = a.sp.adapt_factor * beta;
            if (rate < a.sp.acc_lo) beta = beta / a.sp.adapt_factor;
            if (beta > a.sp.beta_max) beta = a.sp.beta_max;
            coef = make_float2((float)sqrt(1.0 - beta * beta), (float)beta);
            win = 0;
        }
        // ---- kept states: history for the pooling, trajectories ----
        if (--until_kept == 0u) {
            until_kept = (uint32_t)a.thin;
            if ((int64_t)step > a.burn_in) {
                if (active && own) {
#pragma unroll
                    for (int i = 0; i < D; ++i) hist[i] = rc[i];
                    if (c < p.n_diag && kept_idx < p.traj_cap) {
                        float *tj = p.traj + ((int64_t)c * p.traj_cap + kept_idx) * d + j * D;
#pragma unroll
                        for (int i = 0; i < D; ++i) tj[i] = rc[i];
                    }
                }
                hist += p.R * d;
                kept_idx += 1;
            }
        }
        __syncwarp();   // the areas are written again in the next step
    }

    if (!active) return;
#pragma unroll
    for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int i = 0; i < D; ++i) yst[(p0 + q) * d + j * D + i] = y[q][i];
    if (own)
#pragma unroll
        for (int i = 0; i < D; ++i) p.rho_cur[c * p.d_pad + j * D + i] = rc[i];
    if (l == 0) {
        p.logl_cur[c] = logl_cur;
        p.beta[c] = beta;
        p.coef[c] = coef;
        p.acc_win[c] = win;
        p.acc_total[c] = acc_total;
    }
}

// Adds the kept states of a launch to the pool slots as accept_kernel does, step by step: slot b's
// 128 chains in FP32 -- P = 1024 / d partial sums over chains q, q + P, ..., added in the order of q
// -- and each step's sum in FP64.  One CTA per slot; a thread forms one entry's sum of one step
// (the loads of a warp cover the d entries of consecutive steps' rows), then d threads add them up.
constexpr int kPoolThreads = 256;
template <int D>
__global__ void __launch_bounds__(kPoolThreads) fused_pool_kernel(ProblemView p, const StepState *base, uint32_t off,
                                                                  int nsteps, int thin, int64_t burn_in,
                                                                  const float *hist) {
    constexpr int d = D * D, P = 1024 / d, lanes = kPoolThreads / d;
    __shared__ float sums[lanes][d];
    const int64_t j0 = (int64_t)base->step + off;
    const int n = (int)(kept_up_to(j0 + nsteps, thin, burn_in) - kept_up_to(j0, thin, burn_in));
    const int e = threadIdx.x % d, tl = threadIdx.x / d;
    const int64_t c0 = (int64_t)blockIdx.x * p.accept_cpc;
    const int nc = (int)min((int64_t)p.accept_cpc, p.R - c0);
    double *slot = p.pool + (int64_t)blockIdx.x * d;
    double acc = threadIdx.x < d ? slot[e] : 0.0;
    for (int t0 = 0; t0 < n; t0 += lanes) {
        if (t0 + tl < n) {
            const float *h = hist + ((int64_t)(t0 + tl) * p.R + c0) * d + e;
            float tot = 0.0f;
            const int nq = min(P, nc);
#pragma unroll 16
            for (int q = 0; q < nq; ++q) {
                float sum = 0.0f;
                if constexpr (P >= 128) {
                    sum += h[(int64_t)q * d];
                } else {
                    sum += h[(int64_t)q * d];
                    if (q + P < nc) sum += h[(int64_t)(q + P) * d];
                }
                tot = q == 0 ? sum : tot + sum;
            }
            sums[tl][e] = tot;
        }
        __syncthreads();
        if (threadIdx.x < d) {
            const int m = min(lanes, n - t0);
            for (int t = 0; t < m; ++t) acc += (double)sums[t][e];
        }
        __syncthreads();
    }
    if (threadIdx.x < d && n > 0) slot[e] = acc;
}

constexpr int kAdvanceThreads = 128;
__global__ void __launch_bounds__(kAdvanceThreads) advance_steps_kernel(StepState *st, int count, uint32_t n) {
    for (int i = threadIdx.x; i < count; i += kAdvanceThreads) {
        StepState &q = st[i];
        if (!q.multi) continue;
        const int64_t j0 = q.step, j1 = j0 + n;
        q.step = (uint32_t)j1;
        q.kept_count += kept_up_to(j1, (int)q.thin, q.burn_in) - kept_up_to(j0, (int)q.thin, q.burn_in);
    }
}

__global__ void fork_kernel() {}

template <int D, int PASSES, int LPC, bool PAULI, bool POISSON>
cudaError_t launch_steps_w(const FusedArgs &a, cudaStream_t s) {
    using F = FusedShape<D, PASSES, LPC>;
    constexpr int chains = kWarp / LPC;
    const size_t smem = sizeof(float) * (chains * F::stride + (PAULI ? 0 : (F::d + 2) * a.p.KD));
    const int64_t blocks = (a.p.R + chains - 1) / chains;
    fused_small_kernel<D, PASSES, LPC, PAULI, POISSON><<<(unsigned)blocks, kWarp, smem, s>>>(a);
    return cudaGetLastError();
}
template <int D, int PASSES, bool PAULI, bool POISSON>
cudaError_t launch_steps(const FusedArgs &a, cudaStream_t s) {
    // Lanes per chain by the number of chains: 4 D while a step is one warp's latency, 2 D, then D
    // once the extra instructions cost more than they shorten.  us per step at 4 D / 2 D / D lanes:
    //   one qubit, FP32    1024: 1.9 / 2.0 / 2.8   4096: 2.1 / 2.0 / 2.8   16384: 4.6 / 3.0 / 3.3   32768: 8.2 / 5.4 / 4.6
    //   one qubit, Pauli   1024: 1.7 / 1.8 / 2.0   4096: 1.9 / 1.8 / 2.0   12288: 3.6 / 2.5 / 2.5
    //   two qubits, FP32   1024: 3.2 / 4.4 / 5.8   4096: 4.8 / 4.9 / 6.0    6144: 7.6 / 5.7 / 6.4    8192: 8.5 / 6.9 / 6.6
    //   two qubits, Pauli  1024: 4.0 / 4.5 / 5.1   4096: 6.8 / 4.8 / 5.2    6144: 10  / 6.1 / 5.6
    constexpr int64_t kMost4 = D == 2 ? 2560 : PAULI ? 2048 : 4096;
    constexpr int64_t kMost2 = D == 2 ? (PAULI ? 8192 : 20480) : PAULI ? 5120 : 7168;
    if (a.p.R <= kMost4) return launch_steps_w<D, PASSES, 4 * D, PAULI, POISSON>(a, s);
    if (a.p.R <= kMost2) return launch_steps_w<D, PASSES, 2 * D, PAULI, POISSON>(a, s);
    return launch_steps_w<D, PASSES, D, PAULI, POISSON>(a, s);
}

template <int D>
cudaError_t launch_steps_d(const FusedArgs &a, cudaStream_t s) {
    const bool po = a.p.poisson != 0;
    if (a.p.qr_passes == 0) {
        if (a.p.pauli) return po ? launch_steps<D, 0, true, true>(a, s) : launch_steps<D, 0, true, false>(a, s);
        return po ? launch_steps<D, 0, false, true>(a, s) : launch_steps<D, 0, false, false>(a, s);
    }
    if (a.p.pauli) return po ? launch_steps<D, 3, true, true>(a, s) : launch_steps<D, 3, true, false>(a, s);
    return po ? launch_steps<D, 3, false, true>(a, s) : launch_steps<D, 3, false, false>(a, s);
}

}  // namespace

// The rule: one and two qubits, in the structured Pauli form or in the FP32 form of one column
// group and at most 4 D settings (every lane then has at most four), with the default QR or the
// Hilbert-Schmidt prior, up to kFusedMaxState floats of rho over the chains (the history of a
// launch holds that many per kept step).  At that limit, 65536 two-qubit chains, a step still takes
// 38 us here against 58 us in per-step kernels in the FP32 form, and 32 us against 33 us in the Pauli
// form, where the chip is full either way; 262144 one-qubit chains take 36 against 87 us.
constexpr int64_t kFusedMaxState = 1 << 20;
bool fused_possible(const ProblemView &p, bool may_be_pauli) {
    if (p.D > 4 || p.R * p.d > kFusedMaxState) return false;
    if (p.qr_passes != 0 && p.qr_passes != 3) return false;
    if (p.pauli || may_be_pauli) return true;
    return p.tc_kind == TC_NONE && p.KD / p.D <= kSettingSlots * p.D && p.KD <= 128;
}
bool fused_supported(const ProblemView &p) { return fused_possible(p, false) && (p.pauli || p.ngroups == 1); }

// Kept steps one launch may cover: a history of at most 16 MB, and 512 of them.
int fused_kept_steps(const ProblemView &p) {
    const int64_t row = p.R * p.d * (int64_t)sizeof(float);
    return (int)std::min<int64_t>(512, (16ll << 20) / row);
}

cudaError_t launch_fused_steps(const ProblemView &p, const SamplerParams &sp, const StepState *base, uint32_t off,
                               int nsteps, int thin, int64_t burn_in, float *hist, cudaStream_t s) {
    FusedArgs a;
    a.p = p;
    a.sp = sp;
    a.base = base;
    a.off = off;
    a.nsteps = nsteps;
    a.thin = thin;
    a.burn_in = burn_in;
    a.hist = hist;
    a.rk = Philox::round_keys(p.seed);
    return p.D == 2 ? launch_steps_d<2>(a, s) : launch_steps_d<4>(a, s);
}

cudaError_t launch_fused_pool(const ProblemView &p, const StepState *base, uint32_t off, int nsteps, int thin,
                              int64_t burn_in, const float *hist, cudaStream_t s) {
    if (p.D == 2)
        fused_pool_kernel<2><<<p.n_slots, kPoolThreads, 0, s>>>(p, base, off, nsteps, thin, burn_in, hist);
    else
        fused_pool_kernel<4><<<p.n_slots, kPoolThreads, 0, s>>>(p, base, off, nsteps, thin, burn_in, hist);
    return cudaGetLastError();
}

cudaError_t launch_fork(cudaStream_t s) {
    fork_kernel<<<1, 1, 0, s>>>();
    return cudaGetLastError();
}

cudaError_t launch_advance_steps(StepState *st, int count, uint32_t n, cudaStream_t s) {
    advance_steps_kernel<<<1, kAdvanceThreads, 0, s>>>(st, count, n);
    return cudaGetLastError();
}

}  // namespace qst
