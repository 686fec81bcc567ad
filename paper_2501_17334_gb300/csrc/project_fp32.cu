// Plain FP32 form of the projector contraction and log-likelihood (Sec. II,
// p_kl = Tr Lambda_kl rho; Eq. likelihood).
//
// p = A . P with A = packed vec_h(rho) rows [rows][d_pad] and P the packed projector
// matrix [d_pad][KD_pad].  A CTA owns 128 chains and sweeps a group of 128-column
// tiles; each thread keeps an 8 x 8 register tile.  The K sum runs in chunks of 32 terms:
// after each chunk the tile is added into a second-level sum (a thread-private array in
// shared memory) and restarted, so no FP32 chain is longer than 32 terms -- a 256-term chain
// rounds at the scale of its running sum 256 times, which at four qubits is most of the FP32
// form's log L error.  The epilogue evaluates the
// likelihood in deviance form, every setting k renormalised by its own sum S_k = sum_l q_kl,
//     log L = C0 - N log t + sum_k [ sum_{c_kl > 0} c_kl log(q_kl invf_kl) - P_k log(S_k / t) ],
// invf_kl = P_k / c_kl (q = vec_h(rho) . P, t the exact trace of the stored rho), which equals
// sum c log p exactly in real arithmetic (C0 = -sum c log invf; S_k = t for a complete POVM)
// and cancels the rounding the FP32 sums of a setting share.  S_k is summed exactly as a
// hi + lo pair over the four threads that hold the setting's 16 columns; each thread sums its
// deviance terms with a compensated (Kahan) sum carried as a pair into the FP64 combine of the
// 16 threads sharing a chain, and one FP64 partial per (column group, chain) is written.  The
// constant and trace terms are added by the accept kernel.
#include <algorithm>
#include <atomic>

#include "qst_internal.cuh"
#include "f32x2.cuh"

namespace qst {
namespace {

constexpr int BM = 128, BN = 128, BK = 16, kThreads = 256;
constexpr int kChunkSteps = 2;   // K steps of BK per chunk of the sum (32 terms)
// dynamic shared memory: the A and B stages, the column weights and the second-level sums
constexpr size_t kSmemBytes = sizeof(float) * (2 * BK * BM + 2 * BK * BN + 2 * BN + 64 * kThreads);

struct ProjectArgs {
    const float *A;      // [rows][d_pad]
    const float *P;      // [d_pad][KD_pad]
    const float *cnt;    // [KD_pad]
    const float *invf;   // [KD_pad]
    const float *ptot;   // [KD_pad / D] shots P_k of each setting
    double *out;         // [ngroups][rows]
    float *p_out;        // [rows][KD] or null: p = q / t
    const double *trace; // [rows] t, the exact trace of the stored rho (used only for p_out)
    int64_t rows;
    int d_pad, KD, KD_pad;
    int D;               // outcomes per setting (a setting's columns are consecutive)
    int tiles_per_group;
    int poisson;         // 1: each setting adds -mu_k (S_k / t - 1) (Poisson) instead of -P_k log(S_k / t)
};

// POISSON: the Poisson likelihood's setting term (a compile-time choice, so that the multinomial
// instantiation carries none of its code)
template <bool POISSON>
__global__ void __launch_bounds__(kThreads) project_fp32_kernel(ProjectArgs a) {
    extern __shared__ __align__(16) float dyn[];
    float (*As)[BK][BM] = reinterpret_cast<float (*)[BK][BM]>(dyn);
    float (*Bs)[BK][BN] = reinterpret_cast<float (*)[BK][BN]>(dyn + 2 * BK * BM);
    float *cnt_s = dyn + 2 * BK * BM + 2 * BK * BN, *invf_s = cnt_s + BN;
    float *tot = invf_s + BN;   // [64][kThreads]: element e of this thread's tile at e * kThreads + tid

    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int n_tiles_total = a.KD_pad / BN;
    const int t_begin = blockIdx.y * a.tiles_per_group;
    const int t_end = min(t_begin + a.tiles_per_group, n_tiles_total);

    // per row: the compensated deviance sum (sum - comp) and the small renormalisation terms
    float rowsum[8], rowcomp[8], rowsmall[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) rowsum[i] = rowcomp[i] = rowsmall[i] = 0.0f;
    float trace_hi[8], trace_lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = (i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4);
        const int64_t row = m0 + r;
        const double t = (row < a.rows) ? a.trace[row] : 1.0;
        trace_hi[i] = (float)t;
        trace_lo[i] = (float)(t - (double)trace_hi[i]);
    }

    const int k_steps = a.d_pad / BK;
    for (int nt = t_begin; nt < t_end; ++nt) {
        const int n0 = nt * BN;
        float acc[8][8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) acc[i][jj] = 0.0f;

        // register staging for the next K slice
        float4 ra[2], rb[2];
        auto load_global = [&](int k0) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int idx = tid + u * kThreads;   // 0..511
                const int r = idx / 4, q = idx % 4;
                const int64_t row = m0 + r;
                ra[u] = (row < a.rows) ? *reinterpret_cast<const float4 *>(a.A + row * a.d_pad + k0 + 4 * q)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                const int kk = idx / 32, cq = idx % 32;
                rb[u] = *reinterpret_cast<const float4 *>(a.P + (int64_t)(k0 + kk) * a.KD_pad + n0 + 4 * cq);
            }
        };
        auto store_shared = [&](int buf) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int idx = tid + u * kThreads;
                const int r = idx / 4, q = idx % 4;
                As[buf][4 * q + 0][r] = ra[u].x;
                As[buf][4 * q + 1][r] = ra[u].y;
                As[buf][4 * q + 2][r] = ra[u].z;
                As[buf][4 * q + 3][r] = ra[u].w;
                const int kk = idx / 32, cq = idx % 32;
                *reinterpret_cast<float4 *>(&Bs[buf][kk][4 * cq]) = rb[u];
            }
        };

        if (tid < BN) {
            cnt_s[tid] = a.cnt[n0 + tid];
            invf_s[tid] = a.invf[n0 + tid];
        }
        load_global(0);
        store_shared(0);
        __syncthreads();
        for (int ks = 0; ks < k_steps; ++ks) {
            const int buf = ks & 1;
            if (ks + 1 < k_steps) load_global((ks + 1) * BK);
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) {
                const float4 a0 = *reinterpret_cast<const float4 *>(&As[buf][kk][ty * 4]);
                const float4 a1 = *reinterpret_cast<const float4 *>(&As[buf][kk][64 + ty * 4]);
                const float4 b0 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][tx * 4]);
                const float4 b1 = *reinterpret_cast<const float4 *>(&Bs[buf][kk][64 + tx * 4]);
                const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int jj = 0; jj < 8; ++jj) acc[i][jj] = __fmaf_rn(av[i], bv[jj], acc[i][jj]);
            }
            if (ks + 1 < k_steps) {
                store_shared(buf ^ 1);
            }
            // end of a 32-term chunk (not the last one): fold the tile into the second-level sum
            if (ks % kChunkSteps == kChunkSteps - 1 && ks + 1 < k_steps) {
                const bool first = ks == kChunkSteps - 1;
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int jj = 0; jj < 8; ++jj) {
                        float *t = tot + (i * 8 + jj) * kThreads + tid;
                        *t = first ? acc[i][jj] : *t + acc[i][jj];
                        acc[i][jj] = 0.0f;
                    }
            }
            __syncthreads();
        }
        if (k_steps > kChunkSteps) {   // the last chunk joins the earlier ones
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) acc[i][jj] = tot[(i * 8 + jj) * kThreads + tid] + acc[i][jj];
        }

        // epilogue: deviance terms of this tile, and the renormalisation of its settings.  The
        // four columns jj = 4h .. 4h + 3 of this thread belong to one setting, whose other twelve
        // columns are held by the threads tx ^ 1, tx ^ 2, tx ^ 3 (16 columns per setting, D = 16;
        // for D < 16 a group of four columns holds whole settings, for D = 32 two groups of
        // threads form one setting)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = (i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4);
            const int64_t row = m0 + r;
            const float inv_tr = (a.p_out && row < a.rows) ? (float)(1.0 / a.trace[row]) : 0.0f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float sh = 0.0f, sl = 0.0f;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int jj = 4 * h + u;
                    const int col = (jj < 4) ? tx * 4 + jj : 64 + tx * 4 + (jj - 4);
                    const float pv = acc[i][jj];
                    const float cv = cnt_s[col];
                    if (cv > 0.0f) {   // Kahan: rowsum - rowcomp
                        const float y = __fmaf_rn(cv, deviance_log(pv * invf_s[col]), -rowcomp[i]);
                        const float tt = rowsum[i] + y;
                        rowcomp[i] = (tt - rowsum[i]) - y;
                        rowsum[i] = tt;
                    }
                    // S_k as an exact pair: every q in (-4, 4) split at 2^-20 (the hi parts add exactly)
                    const float hq = (pv + 12.0f) - 12.0f;
                    sh += hq;
                    sl += pv - hq;
                    if (a.p_out && row < a.rows && n0 + col < a.KD) a.p_out[row * a.KD + n0 + col] = pv * inv_tr;
                }
                // the setting's sum over the threads holding its columns (exact for the hi parts)
                const int col0 = (h == 0) ? tx * 4 : 64 + tx * 4;
                // threads per setting: D / 4 (1 .. 16, consecutive tx); at D = 2 a thread's four
                // columns hold two settings and the renormalisation is left out (the plain
                // deviance form alone is exact too)
                const int per = a.D / 4;
#pragma unroll
                for (int off = 1; off < 16; off <<= 1) {
                    if (off < per) {
                        sh += __shfl_xor_sync(0xffffffffu, sh, off);
                        sl += __shfl_xor_sync(0xffffffffu, sl, off);
                    }
                }
                if constexpr (POISSON) {
                    // Poisson: -mu_k (S_k / t - 1) per setting, its large part into the compensated
                    // sum; at D = 2 a thread's four columns are two whole settings
                    auto add_poisson = [&](float mu, float s_hi, float s_lo) {
                        float ph, pl;
                        poisson_setting(mu, s_hi, s_lo, trace_hi[i], trace_lo[i], ph, pl);
                        const float y = -ph - rowcomp[i];
                        const float tt = rowsum[i] + y;
                        rowcomp[i] = (tt - rowsum[i]) - y;
                        rowsum[i] = tt;
                        rowsmall[i] -= pl;
                    };
                    if (per >= 1) {
                        if ((tx & (per - 1)) == 0 && n0 + col0 < a.KD) add_poisson(a.ptot[(n0 + col0) / a.D], sh, sl);
                    } else {
#pragma unroll
                        for (int s2 = 0; s2 < 2; ++s2) {
                            if (n0 + col0 + 2 * s2 >= a.KD) continue;
                            float s_hi = 0.0f, s_lo = 0.0f;
#pragma unroll
                            for (int u = 2 * s2; u < 2 * s2 + 2; ++u) {
                                const float pv = acc[i][4 * h + u];
                                const float hq = (pv + 12.0f) - 12.0f;
                                s_hi += hq;
                                s_lo += pv - hq;
                            }
                            add_poisson(a.ptot[(n0 + col0 + 2 * s2) / 2], s_hi, s_lo);
                        }
                    }
                } else if (per >= 1 && (tx & (per - 1)) == 0 && n0 + col0 < a.KD) {   // (multinomial)
                    // one thread per setting adds -P_k log(S_k / t)
                    const float pk = a.ptot[(n0 + col0) / a.D];
                    const float rel = ((sh - trace_hi[i]) + (sl - trace_lo[i])) / trace_hi[i];
                    const float l1p = fabsf(rel) < 0x1p-10f
                                          ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                          : log1pf(rel);
                    rowsmall[i] -= pk * l1p;
                }
            }
        }
        __syncthreads();   // cnt_s / invf_s reuse
    }

    // combine the 16 threads (tx) that share each row, in FP64
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        double v = ((double)rowsum[i] - (double)rowcomp[i]) + (double)rowsmall[i];
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        const int r = (i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4);
        const int64_t row = m0 + r;
        if (tx == 0 && row < a.rows) a.out[(int64_t)blockIdx.y * a.rows + row] = v;
    }
}

// ---- small problems (D <= 4, at most 32 settings, KD <= 128): one thread per (chain, setting) --
// The tiled kernel above is several thousand unrolled instructions; for a one- or two-qubit
// problem its few warps run them once per step from a cold instruction cache (about 40 us per
// launch for 64 one-qubit or 4096 two-qubit chains, most of it stalled on instruction fetch).  Here a thread
// forms its setting's D values q_kl = sum_i A_ri P_i,(kD+l) as one FMA chain over i (d <= 16
// terms), their deviance terms (compensated, as above), the setting's exact sum S_k and its
// renormalisation term, and the KP threads of a chain (KP >= K, a power of two, so that a chain's
// threads share a warp) add their partials in FP64 by shuffles: one partial per chain, the
// single column group this size has.  P (d x KD floats) is staged in shared memory.
template <int D, bool POISSON>
__global__ void __launch_bounds__(256) project_fp32_small_kernel(ProjectArgs a, int K, int KP) {
    constexpr int d = D * D;
    extern __shared__ __align__(16) float ps[];
    const int KD = a.KD;
    for (int e = threadIdx.x; e < d * KD; e += blockDim.x) ps[e] = a.P[(int64_t)(e / KD) * a.KD_pad + (e % KD)];
    __syncthreads();
    const int k = threadIdx.x % KP;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x / KP) + threadIdx.x / KP;
    double v = 0.0;
    if (row < a.rows && k < K) {
        float ar[d];
#pragma unroll
        for (int i = 0; i < d; i += 4) {
            const float4 t4 = *reinterpret_cast<const float4 *>(a.A + row * a.d_pad + i);
            ar[i] = t4.x;
            ar[i + 1] = t4.y;
            ar[i + 2] = t4.z;
            ar[i + 3] = t4.w;
        }
        const double t = a.trace[row];
        const float t_hi = (float)t, t_lo = (float)(t - (double)t_hi);
        const float inv_tr = a.p_out ? (float)(1.0 / t) : 0.0f;
        float sum = 0.0f, comp = 0.0f, small = 0.0f, sh = 0.0f, sl = 0.0f;
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const int col = k * D + l;
            float q = 0.0f;
#pragma unroll
            for (int i = 0; i < d; ++i) q = __fmaf_rn(ar[i], ps[i * KD + col], q);
            const float cv = a.cnt[col];
            if (cv > 0.0f) {   // Kahan: sum - comp
                const float y = __fmaf_rn(cv, deviance_log(q * a.invf[col]), -comp);
                const float tt = sum + y;
                comp = (tt - sum) - y;
                sum = tt;
            }
            const float hq = (q + 12.0f) - 12.0f;   // S_k as an exact pair, as above
            sh += hq;
            sl += q - hq;
            if (a.p_out) a.p_out[row * KD + col] = q * inv_tr;
        }
        if constexpr (POISSON) {   // -mu_k (S_k / t - 1)
            float ph, pl;
            poisson_setting(a.ptot[k], sh, sl, t_hi, t_lo, ph, pl);
            const float y = -ph - comp;
            const float tt = sum + y;
            comp = (tt - sum) - y;
            sum = tt;
            small -= pl;
        } else {   // -P_k log(S_k / t)
            const float rel = ((sh - t_hi) + (sl - t_lo)) / t_hi;
            const float l1p = fabsf(rel) < 0x1p-10f ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                                    : log1pf(rel);
            small -= a.ptot[k] * l1p;
        }
        v = ((double)sum - (double)comp) + (double)small;
    }
    for (int off = 1; off < KP; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (k == 0 && row < a.rows) a.out[row] = v;
}

// ---- three and four qubits: the rows of P that a setting does not use are left out -------------
// A Pauli setting's D elements share their nonzero rows: of the 256 packed rows of a four-qubit
// setting 136, 72, 40, 24 or 16 are used (with 0 .. 4 Z factors; 70 on average), of the 64 rows at
// three qubits 23.  So each setting gets a list of the rows where any of its elements is nonzero,
// with their P entries (fp32_lists_kernel; a general POVM's lists are simply full), and the K sum
// runs over the list, in the rows' order and in the same 32-row chunks as the tiled kernel above:
// the terms left out are exact zeros, so every q has the tiled kernel's bits.
//
// A CTA keeps the packed rho of M = 32 C chains in shared memory, transposed ([row][chain], 128 KB
// at D = 16, four-chain groups xor-swizzled by the row so that both the transposing stores and the
// 128-bit loads spread over the banks), and its warps take settings: lane i has chains 4 i .. 4 i + 3
// (and 128 + 4 i .. at D = 8) and all D outcomes of the setting, 64 accumulators in f32x2 pairs, so
// that a row costs one 128-bit load of rho and D/4 broadcast loads of P for 32 packed FMAs (C = 4).  The
// lists stream through a small per-warp ring (cp.async).  The settings of all tiles, ordered by the
// length of their lists, are laid end to end by cost (rows plus kSpEpilogue for the logarithms) and
// cut into equal pieces, one per CTA, so that all SMs are busy whatever the number of chains; a tile
// that several CTAs share has one partial sum per CTA.
// 10007 four-qubit chains with p written take 103 us, 65536 without 465 us, against 330 and 1740 us by
// the tiled kernel (an FMA-bound time would be 32 and 210 us: with 255 registers two warps share a
// scheduler, and a row's 128-bit loads keep the shared-memory pipe half busy).
constexpr int kSpStages = 3;
constexpr int kSpEpilogue = 24;       // a setting's logarithms, in rows of the K sum
constexpr int kSpMaxSettings = 1024;  // the lengths of all lists sit in shared memory
constexpr int kSpBatch = 32;          // listed rows per stage of the ring

template <int D, int C>   // C: chains per lane
struct SparseShape {
    static constexpr int d = D * D, M = 32 * C;               // chains per tile
    static constexpr int warps = C == 4 ? 8 : 16, threads = 32 * warps;
    // a stage: P rows, their row codes, then the setting's weights: (invf, invf, add, add) and counts per
    // column pair, shots
    static constexpr int wts = kSpBatch * (D + 1);
    static constexpr int stage_floats = (wts + 3 * D + 1 + 3) / 4 * 4;
    // fixed part; the cost prefix [K + 1] (int), the lengths [K] and the order [K] (u16) follow
    static constexpr int floats = d * M + warps * kSpStages * stage_floats;
    static_assert(2 * M <= kSpStages * stage_floats, "the final sums reuse the ring");
};

struct SparseArgs {
    const float *A;            // [rows][d_pad]
    const float *val;          // [K][d][D] P entries of the listed rows
    const uint32_t *code;      // [K][d] row codes: 512 row + 16 ((row / 4) mod 32), + 1 on a 32-row chunk's last
    const uint16_t *len;       // [K] rows listed
    const float4 *colw;        // [KD / 2] (invf, invf, add, add) per column pair
    const float *cnt, *ptot;
    double *out;               // [ngroups][rows]
    float *p_out;              // [rows][KD]
    const double *trace;
    int64_t rows;
    int d_pad, K, KD;
    int ngroups;
    int wide_p;                // p_out's rows are 32-byte aligned: 256-bit stores
};

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// packed pairs kept as 64-bit values, so that one splat of a chain's value serves all its products
__device__ __forceinline__ uint64_t splat_u64(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float2 unpack_u64(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma_u64(uint64_t &acc, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void add_u64(uint64_t &sum, uint64_t v) {
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(sum) : "l"(v));
}
__device__ __forceinline__ void st_global_8(float *dst, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// sum + rest += c v: the product's part on the grid of `sum` (whose exponent no add changes), and the rest of
// it, which the second FMA forms exactly
__device__ __forceinline__ void add_product(float2 &sum, float2 &rest, float2 c, float2 v) {
    const float2 n = fma2(c, v, sum);
    rest = add2(rest, fma2(c, v, sub2(sum, n)));
    sum = n;
}
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

template <int D, int C, bool POISSON, bool P_OUT>
__global__ void __launch_bounds__(SparseShape<D, C>::threads, 1) project_fp32_sparse_kernel(SparseArgs a) {
    using S = SparseShape<D, C>;
    constexpr int d = S::d, M = S::M, kSpWarps = S::warps, kSpThreads = S::threads;
    // A unit of work: one setting, at D = 8 settings k and k + 8 of a 128-column tile of P (16 settings).
    // There the deviance terms are added as the tiled kernel adds them -- one running Kahan sum per
    // four outcomes (packed here: outcomes u and u + 4), through the unit's two settings -- since
    // with few settings the order of that sum is the largest difference left between the two kernels
    // (1e-9 of log L).
    constexpr bool PAIR = D == 8;
    const int units = PAIR ? a.K / 16 * 8 + min(8, a.K % 16) : a.K;
    auto first_of = [&](int u) { return PAIR ? u / 8 * 16 + u % 8 : u; };
    auto has_second = [&](int k) { return PAIR && k % 16 < 8 && k + 8 < a.K; };
    extern __shared__ __align__(1024) float sp_sm[];
    float *As = sp_sm;                                  // [row][M], swizzled
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    float *ring = As + d * M + warp * kSpStages * S::stage_floats;
    int *pre = reinterpret_cast<int *>(sp_sm + S::floats);               // [units + 1] cost of the units before
    uint16_t *len_s = reinterpret_cast<uint16_t *>(pre + a.K + 1), *order = len_s + a.K;   // units, longest first
    for (int i = tid; i < a.K; i += kSpThreads) len_s[i] = a.len[i];
    __syncthreads();
    auto cost = [&](int u) {
        const int k = first_of(u);
        return (int)len_s[k] + kSpEpilogue + (has_second(k) ? (int)len_s[k + 8] + kSpEpilogue : 0);
    };
    for (int u = tid; u < units; u += kSpThreads) {
        const int n = cost(u);
        int rank = 0;
        for (int o = 0; o < units; ++o) {
            const int m = cost(o);
            rank += (m > n || (m == n && o < u)) ? 1 : 0;
        }
        order[rank] = (uint16_t)u;
    }
    __syncthreads();
    if (warp == 0) {   // exclusive prefix sums of the costs in that order
        int base = 0;
        for (int r = 0; r < units; r += 32) {
            int v = r + lane < units ? cost(order[r + lane]) : 0;
            const int own = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += up;
            }
            if (r + lane < units) pre[r + lane] = base + v - own;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) pre[units] = base;
    }
    __syncthreads();
    // this CTA's piece [x0, x1) of the tiles' costs, W each; a unit belongs where its cost starts
    const int64_t tiles = (a.rows + M - 1) / M, W = pre[units];
    const int64_t piece = (tiles * W + gridDim.x - 1) / gridDim.x;
    const int64_t x0 = blockIdx.x * piece, x1 = min(x0 + piece, tiles * W);
    auto first_from = [&](int64_t x) {   // first position of the order whose cost starts at x or later
        int lo = 0, hi = units;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (pre[mid] < x) lo = mid + 1;
            else hi = mid;
        }
        return lo;
    };
    const uint32_t ring_base = (uint32_t)__cvta_generic_to_shared(ring);

    for (int64_t tile = x0 / W; tile * W < x1; ++tile) {
        // this tile's units: positions [r0, r1) of the order
        const int r0 = first_from(x0 - tile * W), r1 = first_from(x1 - tile * W);
        const int64_t m0 = tile * M;
        __syncthreads();   // the previous tile's rows and final sums are done with (and the order is in place)
        // rho, transposed: a warp reads 128 rows' entries of one chain at a time
#pragma unroll 8
        for (int i = tid; i < (r0 < r1 ? M * (d / 4) : 0); i += kSpThreads) {
            const int c = i / (d / 4), q = i - c * (d / 4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (m0 + c < a.rows) v = *reinterpret_cast<const float4 *>(a.A + (m0 + c) * a.d_pad + 4 * q);
            // chain c at C ((c / C) ^ (row / 4 mod 32)) + c mod C of rows 4 q .. 4 q + 3
            float *dst = As + 4 * q * M + (C * ((c / C) ^ (q & 31)) + c % C);
            dst[0] = v.x;
            dst[M] = v.y;
            dst[2 * M] = v.z;
            dst[3 * M] = v.w;
        }
        __syncthreads();

        float t_hi[C], t_lo[C];      // exact trace of this lane's chains
        float tot_hi[C], tot_lo[C];  // their sums over this warp's settings
        float inv_t[C], inv_p[C];    // 1 / t
        bool dead[C];                // a counted outcome with q <= 0
        float2 run[C], run_c[C];     // D = 8: the running deviance sums of a unit
        float run_small[C];
        auto chain = [&](int i) { return C * lane + i; };
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int64_t row = m0 + chain(i);
            const double t = row < a.rows ? a.trace[row] : 1.0;
            t_hi[i] = (float)t;
            t_lo[i] = (float)(t - (double)t_hi[i]);
            inv_t[i] = 1.0f / t_hi[i];
            inv_p[i] = P_OUT ? (float)(1.0 / t) : 0.0f;
            tot_hi[i] = tot_lo[i] = 0.0f;
            dead[i] = false;
        }

        // this warp's units: positions warp, 2 W - 1 - warp, 2 W + warp, .. of the range (a snake, so
        // that long and short lists even out), their lists in batches of kSpBatch rows
        const int count = r1 - r0;
        auto unit_at = [&](int n) {   // first setting of this warp's n-th unit, or -1
            const int pos = n * kSpWarps + ((n & 1) ? kSpWarps - 1 - warp : warp);
            return pos < count ? first_of(order[r0 + pos]) : -1;
        };
        auto after = [&](int k, int &n) { return has_second(k) ? k + 8 : unit_at(++n); };   // the setting after k
        int pf_n = 0, pf_k = unit_at(0), pf_at = 0;   // next batch to request: setting and position
        auto fetch = [&](int stage) {
            if (pf_k >= 0) {
                const int n = min(kSpBatch, len_s[pf_k] - pf_at);
                const float *src = a.val + ((int64_t)pf_k * d + pf_at) * D;
                const uint32_t dst = ring_base + 4u * (uint32_t)(stage * S::stage_floats);
#pragma unroll
                for (int u = 0; u < kSpBatch * D / 128; ++u) {
                    const int i = lane + 32 * u;
                    if (i < n * (D / 4)) cp_async16(dst + 16u * i, src + 4 * i);
                }
                if (lane < n) cp_async4(dst + 4u * (kSpBatch * D + lane), a.code + (int64_t)pf_k * d + pf_at + lane);
                pf_at += kSpBatch;
                if (pf_at >= len_s[pf_k]) {   // the setting's last batch: its weights come along
                    if (lane < D / 2)
                        cp_async16(dst + 4u * (S::wts + 4 * lane), a.colw + pf_k * (D / 2) + lane);
                    else if (lane < 3 * D / 4)
                        cp_async16(dst + 4u * (S::wts + 4 * lane), a.cnt + pf_k * D + 4 * (lane - D / 2));
                    else if (lane == 31)
                        cp_async4(dst + 4u * (S::wts + 3 * D), a.ptot + pf_k);
                    pf_at = 0;
                    pf_k = after(pf_k, pf_n);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        int k = pf_k, at = 0, num = 0;   // the batch in hand
#pragma unroll
        for (int st = 0; st < kSpStages - 1; ++st) fetch(st);
        int stage = 0, fill = kSpStages - 1;
        uint64_t sum[C][D / 2], acc[C][D / 2];   // the setting's q so far, and the chunk's part (packed pairs)
#pragma unroll
        for (int i = 0; i < C; ++i)
#pragma unroll
            for (int l = 0; l < D / 2; ++l) {
                sum[i][l] = 0ull;
                acc[i][l] = 0ull;
            }
        while (k >= 0) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kSpStages - 2) : "memory");
            __syncwarp();   // every lane's copies of this stage have landed, and the stage two back is free
            fetch(fill);
            fill = fill + 1 == kSpStages ? 0 : fill + 1;
            const float *vals = ring + stage * S::stage_floats;
            const uint32_t *codes = reinterpret_cast<const uint32_t *>(vals + kSpBatch * D);
            stage = stage + 1 == kSpStages ? 0 : stage + 1;
            const int n = min(kSpBatch, len_s[k] - at);
            auto multiply = [&](int e) {
                // the code is the byte offset of the row and its swizzle for C = 4
                const char *at_a = reinterpret_cast<const char *>(As) + (((codes[e] / (4 / C)) ^ (4u * C * lane)) & ~(4u * C - 1u));
                uint64_t av[C];
                if constexpr (C == 4) {
                    const float4 a4 = *reinterpret_cast<const float4 *>(at_a);
                    av[0] = splat_u64(a4.x);
                    av[C - 3] = splat_u64(a4.y);
                    av[C - 2] = splat_u64(a4.z);
                    av[C - 1] = splat_u64(a4.w);
                } else {
                    av[0] = splat_u64(*reinterpret_cast<const float *>(at_a));
                }
                ulonglong2 p4[D / 4];
#pragma unroll
                for (int l = 0; l < D / 4; ++l) p4[l] = *reinterpret_cast<const ulonglong2 *>(vals + e * D + 4 * l);
#pragma unroll
                for (int i = 0; i < C; ++i)
#pragma unroll
                    for (int l = 0; l < D / 4; ++l) {
                        fma_u64(acc[i][2 * l], av[i], p4[l].x);
                        fma_u64(acc[i][2 * l + 1], av[i], p4[l].y);
                    }
            };
            // runs of rows of one 32-row chunk of P; a chunk's end joins its sum to the earlier ones
            unsigned ends = __ballot_sync(0xffffffffu, lane < n && (codes[lane] & 1u));
            int e = 0;
            while (e < n) {
                const int stop = ends ? __ffs(ends) : n;   // (a chunk may go on in the next batch)
#pragma unroll 4
                for (; e < stop; ++e) multiply(e);
                if (ends == 0u) break;
                ends &= ends - 1u;
#pragma unroll
                for (int i = 0; i < C; ++i)
#pragma unroll
                    for (int l = 0; l < D / 2; ++l) {
                        add_u64(sum[i][l], acc[i][l]);
                        acc[i][l] = 0ull;
                    }
            }
            at += n;
            if (at < len_s[k]) continue;

            // ---- the setting's q are complete: its deviance terms and renormalisation ----
            const float *wts = vals + S::wts;
            const float pk = wts[3 * D];
            if constexpr (PAIR) {
                if (k % 16 < 8) {   // the unit begins
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        run[i] = run_c[i] = splat2(0.0f);
                        run_small[i] = 0.0f;
                    }
                }
                float2 sh[C], sl[C];
                int xmin[C];
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    sh[i] = sl[i] = splat2(0.0f);
                    xmin[i] = 0x7fffffff;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    // outcomes u and u + 4: weights (invf, invf, add, add) of pairs u / 2 and u / 2 + 2, element u % 2
                    const float2 w = make_float2(wts[4 * (u / 2) + u % 2], wts[4 * (u / 2 + 2) + u % 2]);
                    const float2 add = make_float2(wts[4 * (u / 2) + 2 + u % 2], wts[4 * (u / 2 + 2) + 2 + u % 2]);
                    const float2 cn = make_float2(wts[2 * D + u], wts[2 * D + u + 4]);
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        const float2 s0 = unpack_u64(sum[i][u / 2]), s1 = unpack_u64(sum[i][u / 2 + 2]);
                        const float2 q = u % 2 ? make_float2(s0.y, s1.y) : make_float2(s0.x, s1.x);
                        const float2 h = sub2(add2(q, splat2(12.0f)), splat2(12.0f));   // S_k as an exact pair
                        sh[i] = add2(sh[i], h);
                        sl[i] = add2(sl[i], sub2(q, h));
                        const float2 x = fma2(q, w, add);
                        xmin[i] = min(xmin[i], min(__float_as_int(x.x), __float_as_int(x.y)));
                        float2 s = run[i], c = run_c[i];
                        kahan_fma2(s, c, cn, log_poly2(x));
                        if (cn.x > 0.0f) {   // (an outcome without counts leaves the sum as it is)
                            run[i].x = s.x;
                            run_c[i].x = c.x;
                        }
                        if (cn.y > 0.0f) {
                            run[i].y = s.y;
                            run_c[i].y = c.y;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    const float s_hi = sh[i].x + sh[i].y, s_lo = sl[i].x + sl[i].y;
                    if constexpr (POISSON) {   // the large part joins the first four outcomes' sum
                        float ph, pl;
                        poisson_setting(pk, s_hi, s_lo, t_hi[i], t_lo[i], ph, pl);
                        const float y = -ph - run_c[i].x;
                        const float tt = run[i].x + y;
                        run_c[i].x = (tt - run[i].x) - y;
                        run[i].x = tt;
                        run_small[i] -= pl;
                    } else {
                        const float rel = ((s_hi - t_hi[i]) + (s_lo - t_lo[i])) * inv_t[i];
                        const float l1p = fabsf(rel) < 0x1p-10f
                                              ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                              : log1pf(rel);
                        run_small[i] -= pk * l1p;
                    }
                    dead[i] |= xmin[i] < 0x00800000;
                    if (!has_second(k)) add_setting(tot_hi[i], tot_lo[i], run[i], run_c[i], -run_small[i]);
                }
            } else if (pk > 0.0f) {
                // The setting's sum starts at 1.5 2^k, with 2^(k-1) above any sum of its terms (counts below
                // 2^(e+1) in all, |log| < 2^7, k = e + 9), so it stays on one grid and add_product loses
                // nothing.  (A Kahan sum from zero took as many instructions, rounded every product and lost part
                // of an add's error whenever a term was larger than the sum so far.  rms error of log L on
                // the stored rho, relative, over 60000 four-qubit Pauli states: the tiled kernel's sums
                // 8.40e-10, Kahan sums from zero 8.44e-10, these 7.33e-10.
                // Where the compiler schedules them worst, 65536 chains without p, they cost 453 -> 465 us.)
                float total = pk;
                if constexpr (POISSON) {   // the counts may exceed mu
                    total = 0.0f;
#pragma unroll
                    for (int l = 0; l < D; ++l) total += wts[2 * D + l];
                }
                const float base = __int_as_float((__float_as_int(total) & 0x7f800000) + (9 << 23) + 0x400000);
                float2 sh[C], sl[C], dev[C], rest[C];
                int xmin[C];
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    sh[i] = sl[i] = rest[i] = splat2(0.0f);
                    dev[i] = splat2(base);
                    xmin[i] = 0x7fffffff;
                }
#pragma unroll
                for (int l = 0; l < D / 2; ++l) {
                    const float4 w = *reinterpret_cast<const float4 *>(wts + 4 * l);
                    const float2 cn = *reinterpret_cast<const float2 *>(wts + 2 * D + 2 * l);
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        const float2 q = unpack_u64(sum[i][l]);
                        const float2 h = sub2(add2(q, splat2(12.0f)), splat2(12.0f));   // S_k as an exact pair
                        sh[i] = add2(sh[i], h);
                        sl[i] = add2(sl[i], sub2(q, h));
                        const float2 x = fma2(q, make_float2(w.x, w.y), make_float2(w.z, w.w));
                        xmin[i] = min(xmin[i], min(__float_as_int(x.x), __float_as_int(x.y)));
                        add_product(dev[i], rest[i], cn, log_poly2(x));
                    }
                }
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    dev[i] = sub2(dev[i], splat2(base));   // (exact)
                    const float s_hi = sh[i].x + sh[i].y, s_lo = sl[i].x + sl[i].y;
                    if constexpr (POISSON) {
                        float ph, pl;
                        poisson_setting(pk, s_hi, s_lo, t_hi[i], t_lo[i], ph, pl);
                        add_setting_pair(tot_hi[i], tot_lo[i], dev[i], neg2(rest[i]), ph, pl);
                    } else {
                        const float rel = ((s_hi - t_hi[i]) + (s_lo - t_lo[i])) * inv_t[i];
                        const float l1p = fabsf(rel) < 0x1p-10f
                                              ? rel * __fmaf_rn(rel, __fmaf_rn(rel, 0.33333334f, -0.5f), 1.0f)
                                              : log1pf(rel);
                        add_setting(tot_hi[i], tot_lo[i], dev[i], neg2(rest[i]), pk * l1p);
                    }
                    dead[i] |= xmin[i] < 0x00800000;
                }
            }
            if constexpr (P_OUT) {
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    const int64_t row = m0 + chain(i);
                    if (row >= a.rows) continue;
                    float *dst = a.p_out + row * a.KD + k * D;
#pragma unroll
                    for (int l = 0; l < D; l += 8) {
                        float v[8];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 q = unpack_u64(sum[i][l / 2 + u]);
                            v[2 * u] = q.x * inv_p[i];
                            v[2 * u + 1] = q.y * inv_p[i];
                        }
                        if (a.wide_p) {
                            st_global_8(dst + l, v);
                        } else {
#pragma unroll
                            for (int u = 0; u < 8; ++u) dst[l + u] = v[u];
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < C; ++i)
#pragma unroll
                for (int l = 0; l < D / 2; ++l) sum[i][l] = 0ull;
            at = 0;
            k = after(k, num);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // every warp is done with its ring: the final sums take its place
        float *fin = As + d * M;   // [2][warp][M]
#pragma unroll
        for (int i = 0; i < C; ++i) {
            fin[warp * M + chain(i)] = dead[i] ? -INFINITY : tot_hi[i];
            fin[(kSpWarps + warp) * M + chain(i)] = tot_lo[i];
        }
        __syncthreads();
        if (tid < M && m0 + tid < a.rows) {
            float hi = 0.0f, lo = 0.0f;
            bool ninf = false;
#pragma unroll
            for (int w = 0; w < kSpWarps; ++w) {
                const float h = fin[w * M + tid];
                ninf |= h == -INFINITY;
                float e;
                two_sum(hi, h, hi, e);
                lo += e + fin[(kSpWarps + w) * M + tid];
            }
            // partial of the g-th CTA of this tile; the last one clears the partials no CTA has
            const int64_t g = (int64_t)blockIdx.x - tile * W / piece;
            a.out[g * a.rows + m0 + tid] = ninf ? -INFINITY : (double)hi + (double)lo;
            if (x1 >= (tile + 1) * W)
                for (int64_t z = g + 1; z < a.ngroups; ++z) a.out[z * a.rows + m0 + tid] = 0.0;
        }
    }
}

// The lists of setting blockIdx.x: a warp per 32-row chunk reads the setting's D columns of P ([d][ld]).
template <int D>
__global__ void __launch_bounds__(D * D) fp32_lists_kernel(const float *P, int ld, float *val, uint32_t *code, uint16_t *len) {
    constexpr int d = D * D;
    __shared__ int count[d / 32];
    const int k = blockIdx.x, lane = threadIdx.x % 32, ch = threadIdx.x / 32, row = threadIdx.x;
    float *v = val + (int64_t)k * d * D;
    uint32_t *c = code + (int64_t)k * d;
    const float *src = P + (int64_t)row * ld + k * D;
    float x[D];
    bool any = false;
#pragma unroll
    for (int l = 0; l < D; ++l) x[l] = src[l];
#pragma unroll
    for (int l = 0; l < D; ++l) any |= !(x[l] == 0.0f);
    const unsigned on = __ballot_sync(0xffffffffu, any);
    if (lane == 0) count[ch] = __popc(on);
    __syncthreads();
    int before = 0, n = 0;
#pragma unroll
    for (int o = 0; o < d / 32; ++o) {
        before += o < ch ? count[o] : 0;
        n += count[o];
    }
    if (any) {
        const int at = before + __popc(on & ((1u << lane) - 1u));
#pragma unroll
        for (int l = 0; l < D; ++l) v[at * D + l] = x[l];
        c[at] = 512u * (uint32_t)row + 16u * ((row >> 2) & 31) + (lane == 31 - __clz(on) ? 1u : 0u);
    }
    if (n == 0 && row < D) v[row] = 0.0f;   // no element of the setting is nonzero: one row of zeros, so
    if (row == 0) {                         // that its q = 0 are formed
        if (n == 0) c[0] = 1u;
        len[k] = (uint16_t)(n == 0 ? 1 : n);
    }
}

}  // namespace

// The sparse kernel covers three and four qubits (at five a tile of rho does not fit shared memory).
bool fp32_lists(const ProblemView &p) { return (p.D == 8 || p.D == 16) && p.KD / p.D <= kSpMaxSettings; }
size_t fp32_list_values(const ProblemView &p) { return fp32_lists(p) ? (size_t)p.d * p.KD : 0; }
size_t fp32_list_codes(const ProblemView &p) { return fp32_lists(p) ? (size_t)p.d * (p.KD / p.D) : 0; }
size_t fp32_list_lengths(const ProblemView &p) { return fp32_lists(p) ? (size_t)(p.KD / p.D) : 0; }

cudaError_t launch_fp32_lists(const ProblemView &p, const float *P, int ld, float *val, uint32_t *code, uint16_t *len,
                              cudaStream_t s) {
    const unsigned K = (unsigned)(p.KD / p.D);
    if (p.D == 16)
        fp32_lists_kernel<16><<<K, 256, 0, s>>>(P, ld, val, code, len);
    else
        fp32_lists_kernel<8><<<K, 64, 0, s>>>(P, ld, val, code, len);
    return cudaGetLastError();
}

namespace {
constexpr int kSms = 152;
int sparse_units(const ProblemView &p) {   // of a tile: settings, at D = 8 pairs of them
    const int K = p.KD / p.D;
    return p.D == 8 ? K / 16 * 8 + std::min(8, K % 16) : K;
}
// rows of P over all settings' lists, each with kSpEpilogue for its logarithms (a Pauli problem's number
// where the lists are not known on the host)
int64_t sparse_cost(const ProblemView &p) {
    const int64_t K = p.KD / p.D;
    return (p.sp_rows > 0 ? p.sp_rows : (p.D == 16 ? 70 : 23) * K) + kSpEpilogue * K;
}
// Chains per lane: four (the row's P entries serve 128 chains), or one (shorter settings, more of them)
// while there is little work per warp.  us at four / one chains per lane with p written, Pauli settings:
// four qubits 1 row 27 / 17, 1000 rows 43 / 31, 4096 rows 68 / 59, 6000 rows 77 / 80, 10007 rows 103 / 119;
// three qubits 1000 rows 20 / 14, 6000 rows 24 / 23, 10007 rows 25 / 29.  So the line at four qubits lies
// at 40 tiles of 128 chains, or as many listed rows where the lists are longer (81 bases without zeros: 2000
// rows 72 / 84, 3000 rows 90 / 109).  A few settings take four as well while every CTA then has one, but
// two or more with one (a setting without zeros, 16384 rows: 33 / 63; 16 of them, 1000 rows: 33 / 35).
int sparse_c(const ProblemView &p, int64_t rows) {
    const int64_t K = p.KD / p.D, tiles = (rows + 127) / 128;
    if (p.D == 8) return tiles * K >= 1600 ? 4 : 1;
    if (tiles * sparse_cost(p) >= 300000) return 4;
    return K <= 16 && tiles * K <= kSms && (rows + 31) / 32 * K > 2 * kSms ? 4 : 1;
}
// CTAs of the sparse kernel: one per SM (fewer only where there are fewer settings); a tile's piece of
// the costs then meets at most ceil(CTAs / tiles) + 1 of them
int64_t sparse_tiles(const ProblemView &p, int64_t rows) {
    const int M = 32 * sparse_c(p, rows);
    return (rows + M - 1) / M;
}
int64_t sparse_ctas(const ProblemView &p, int64_t rows) {
    return std::min<int64_t>(kSms, sparse_tiles(p, rows) * sparse_units(p));
}
int sparse_groups(int64_t tiles, int64_t ctas) { return (int)((ctas + tiles - 1) / tiles) + 1; }
}  // namespace

// Whether the list kernel is the faster one at this many rows.  The tiled kernel takes a wave of tiles of
// 128 rows x 128 columns after the other; the list kernel an even share of the listed rows for every SM, but at
// least a setting's list per warp, twice where a CTA's share spans two tiles, and the ordering of
// many settings.  Lists without zeros save nothing, so around whole waves of tiles the tiled kernel wins.  us by
// these estimates and measured, tiled / list: four qubits, 81 bases 1000 rows 56 / 58 (57 / 58), 1500 rows
// 56 / 70 (56 / 66), 2000 rows 100 / 73 (99 / 68); 1000 bases 64 rows 56 / 101 (56 / 97), 1000 rows 318 / 282
// (353 / 305); Pauli settings 1500 rows 56 / 29 (57 / 35); three qubits, 300 bases 1000 rows 33 / 35 (33 / 35), 1400
// rows 51 / 38 (51 / 39).
bool fp32_list_form(const ProblemView &p, int64_t rows) {
    if (!fp32_lists(p)) return false;
    if (p.sp_rows == 0) return true;   // the lists' lengths are not known on the host
    const int64_t tiles = (rows + 127) / 128, K = p.KD / p.D, units = sparse_units(p), total = sparse_cost(p);
    const double waves = (double)((tiles * (p.KD_pad / BN) + kSms - 1) / kSms);
    const double cost = (double)total / kSms;   // per tile and SM
    const double one = (p.sp_most + kSpEpilogue) * (units < K ? 2.0 : 1.0);
    // the CTAs' even shares end inside tiles, unless they happen to divide them
    auto spans = [&](int64_t t) { return t > 1 && t * units > kSms && (kSms % t != 0 || t * total % kSms != 0); };
    double list;
    if (p.D == 8) {
        list = 9.0 + 0.05 * (tiles * cost / 8 + one * (spans(tiles) ? 1.58 : 1.0)) + 0.0244 * units * ((units + 255) / 256);
    } else if (sparse_c(p, rows) == 4) {
        list = 6.0 + 0.085 * (tiles * cost / 8 + one * (spans(tiles) ? 1.67 : 1.0)) + 0.02 * K * ((K + 255) / 256);
    } else {
        const int64_t t32 = (rows + 31) / 32;
        const double more = !spans(t32) ? 1.0 : t32 >= 2 * kSms ? 0.35 : 1.35;
        list = 3.0 + 0.079 * (t32 * cost / 16 * std::max(1.0, 12.0 / K) + one * more) + 0.025 * K * ((K + 511) / 512);
    }
    return list <= (p.D == 8 ? 14.0 + 18.7 * waves : 13.0 + 43.5 * waves);
}

int fp32_list_groups(const ProblemView &p, int64_t rows) {
    return sparse_groups(sparse_tiles(p, rows), sparse_ctas(p, rows));
}

int fp32_ngroups(const ProblemView &p, int64_t rows) {
    if (fp32_list_form(p, rows)) return fp32_list_groups(p, rows);
    // enough CTAs to fill the machine: split the columns when there are few row tiles
    const int64_t mt = (rows + BM - 1) / BM;
    const int nt = p.KD_pad / BN;
    int g = 1;
    while (g < nt && mt * g < 2 * 152) g *= 2;
    return g > nt ? nt : g;
}

namespace {
template <int D, int C, bool POISSON, bool P_OUT>
cudaError_t launch_sparse(const SparseArgs &a, unsigned blocks, cudaStream_t s) {
    using S = SparseShape<D, C>;
    const size_t smem = sizeof(float) * (S::floats + a.K + 1) + 2 * sizeof(uint16_t) * (size_t)a.K;
    constexpr size_t most = sizeof(float) * (S::floats + kSpMaxSettings + 1) + 2 * sizeof(uint16_t) * (size_t)kSpMaxSettings;
    static_assert(most <= 227 * 1024, "shared memory");
    static std::atomic<unsigned long long> attr_set{0};   // opted into once per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !((attr_set.load() >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(project_fp32_sparse_kernel<D, C, POISSON, P_OUT>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set.fetch_or(1ull << dev);
    }
    project_fp32_sparse_kernel<D, C, POISSON, P_OUT><<<blocks, S::threads, smem, s>>>(a);
    return cudaGetLastError();
}
template <int D, int C>
cudaError_t launch_sparse_dc(const SparseArgs &a, bool poisson, unsigned blocks, cudaStream_t s) {
    if (a.p_out) return poisson ? launch_sparse<D, C, true, true>(a, blocks, s) : launch_sparse<D, C, false, true>(a, blocks, s);
    return poisson ? launch_sparse<D, C, true, false>(a, blocks, s) : launch_sparse<D, C, false, false>(a, blocks, s);
}
template <int D>
cudaError_t launch_sparse_d(const SparseArgs &a, bool poisson, int c, unsigned blocks, cudaStream_t s) {
    return c == 4 ? launch_sparse_dc<D, 4>(a, poisson, blocks, s) : launch_sparse_dc<D, 1>(a, poisson, blocks, s);
}
}  // namespace

namespace {
template <bool POISSON>
cudaError_t launch_fp32(const ProjectArgs &a, dim3 grid, cudaStream_t s) {
    // more than 48 KB of dynamic shared memory: opted into once per device
    static unsigned long long attr_set = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && !((attr_set >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(project_fp32_kernel<POISSON>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set |= 1ull << dev;
    }
    project_fp32_kernel<POISSON><<<grid, kThreads, kSmemBytes, s>>>(a);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_project_fp32(const ProblemView &p, const float *A, int64_t rows, double *out_part, float *p_out,
                                cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    if (p.KD_pad % BN != 0 || p.d_pad % BK != 0) return cudaErrorInvalidValue;
    ProjectArgs a;
    a.A = A;
    a.P = p.P32;
    a.cnt = p.cnt;
    a.invf = p.invf;
    a.ptot = p.ptot;
    a.D = p.D;
    a.out = out_part;
    a.p_out = p_out;
    a.trace = p.trace_prop;
    a.rows = rows;
    a.d_pad = p.d_pad;
    a.KD = p.KD;
    a.KD_pad = p.KD_pad;
    a.poisson = p.poisson;
    const int K = p.KD / p.D;
    if (p.D <= 4 && p.KD <= 128 && K <= 32 && p.ngroups == 1) {   // one column group: the small kernel
        int KP = 1;
        while (KP < K) KP <<= 1;
        const unsigned blocks = (unsigned)((rows + (256 / KP) - 1) / (256 / KP));
        const size_t smem = sizeof(float) * (size_t)p.D * p.D * p.KD;
        if (p.D == 2) {
            if (a.poisson) project_fp32_small_kernel<2, true><<<blocks, 256, smem, s>>>(a, K, KP);
            else project_fp32_small_kernel<2, false><<<blocks, 256, smem, s>>>(a, K, KP);
        } else {
            if (a.poisson) project_fp32_small_kernel<4, true><<<blocks, 256, smem, s>>>(a, K, KP);
            else project_fp32_small_kernel<4, false><<<blocks, 256, smem, s>>>(a, K, KP);
        }
        return cudaGetLastError();
    }
    if (p.sp_val && fp32_list_form(p, rows)) {
        SparseArgs b;
        b.A = A;
        b.val = p.sp_val;
        b.code = p.sp_code;
        b.len = p.sp_len;
        b.colw = p.colw;
        b.cnt = p.cnt;
        b.ptot = p.ptot;
        b.out = out_part;
        b.p_out = p_out;
        b.trace = p.trace_prop;
        b.rows = rows;
        b.d_pad = p.d_pad;
        b.K = K;
        b.KD = p.KD;
        b.wide_p = reinterpret_cast<uintptr_t>(p_out) % 32 == 0;   // (KD is a multiple of 8)
        b.ngroups = p.ngroups;
        // the view's groups bound the CTAs that may share a tile
        const int64_t tiles = sparse_tiles(p, rows);
        int64_t ctas = sparse_ctas(p, rows);
        if (sparse_groups(tiles, ctas) > p.ngroups) ctas = std::max<int64_t>(1, (p.ngroups - 1) * tiles);
        const int c = sparse_c(p, rows);
        return p.D == 16 ? launch_sparse_d<16>(b, p.poisson != 0, c, (unsigned)ctas, s)
                         : launch_sparse_d<8>(b, p.poisson != 0, c, (unsigned)ctas, s);
    }
    const int nt = p.KD_pad / BN;
    const int groups = p.ngroups;
    a.tiles_per_group = (nt + groups - 1) / groups;
    dim3 grid((unsigned)((rows + BM - 1) / BM), (unsigned)groups);
    return a.poisson ? launch_fp32<true>(a, grid, s) : launch_fp32<false>(a, grid, s);
}

}  // namespace qst
