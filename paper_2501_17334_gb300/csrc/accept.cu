// Accept / reject, step-size adaptation, thinning and pooling (Algorithm 2,
// Eq. BME2), the diagnostics reductions (Eq. ACFrho, Eq. IACT) and small test hooks.
#include "qst_internal.cuh"
#include "f32x2.cuh"

#include <atomic>

namespace qst {
namespace {

constexpr int kChainsPerCta = 128;   // the most chains one accept CTA takes (ProblemView::accept_cpc)
constexpr int kThreads = 256;

struct AcceptArgs {
    ProblemView p;
    SamplerParams sp;
    int mode;          // MODE_INIT or MODE_STEP
    uint32_t step;     // j
    int kept;          // j is a kept step (j % T == 0 and j > burn_in)
    int64_t kept_idx;  // index of this kept state (0-based) in the trajectories
    StepState *step_dev; // when not null: step, kept and kept_idx are the open step's, which this closes
};

// One CTA owns chains [C b, C b + C) and pool slot b, C = p.accept_cpc <= 128.
__global__ void __launch_bounds__(kThreads) accept_kernel(AcceptArgs a) {
    const ProblemView &p = a.p;
    if (a.step_dev) {   // (a is this thread's copy of the parameters)
        a.step = a.step_dev->j;
        a.kept = a.step_dev->kept;
        a.kept_idx = a.step_dev->kept_idx;
        if (blockIdx.x == 0 && threadIdx.x == 0) {   // (no CTA of this launch reads these two)
            a.step_dev->step = a.step;
            a.step_dev->kept_count = a.kept_idx + a.kept;
        }
    }
    __shared__ uint8_t flag[kChainsPerCta];
    __shared__ float inv_tr[kChainsPerCta];
    const int tid = threadIdx.x;
    const int64_t c0 = (int64_t)blockIdx.x * p.accept_cpc;
    const int nc = (int)min((int64_t)p.accept_cpc, p.R - c0);

    // ---- phase 1: one thread per chain -------------------------------------------------
    if (tid < kChainsPerCta) {
        uint8_t acc = 0;
        float itr = 0.0f;
        if (tid < nc) {
            const int64_t c = c0 + tid;
            // log L(y') = C0 + sum_{c>0} c log(q invf) - N log t: q = vec_h(rho) . P for the
            // stored FP32 rho, t its exact trace, p = q / t
            const double tr = p.trace_prop[c];
            itr = 1.0f / (float)tr;
            // log t: t is the exact trace of an already normalised rho, so |t - 1| is a few ulps;
            // three terms of log1p(t - 1) then leave less than (t - 1)^4 / 4, far below FP64
            // rounding (FP64 log would cost ~30 of the scarce FP64 FMAs; it is kept for
            // |t - 1| >= 2^-10)
            const double dl = tr - 1.0;
            double logl_prop = p.C0 - p.Ntot * (fabs(dl) < 0x1p-10 ? dl * (1.0 - dl * (0.5 - dl * (1.0 / 3.0))) : log(tr));
            for (int g = 0; g < p.ngroups; ++g) logl_prop += p.logl_part[(int64_t)g * p.R + c];
            if (a.mode == MODE_INIT) {
                acc = 1;
                p.logl_cur[c] = logl_prop;
                p.cur[c] = 1;   // the initial proposal always lands in slot 1
            } else {
                // accept test: alpha ~ U(0,1), accept iff log alpha < log L(y') - log L(y)
                const uint32_t chain_id = (uint32_t)(p.chain_offset + c);
                const uint4 w = Philox::block(make_uint4(0u, a.step, chain_id, TAG_ALPHA),
                                              (uint32_t)(p.seed & 0xffffffffu), (uint32_t)(p.seed >> 32));
                const float alpha = ((float)(w.x >> 9) + 0.5f) * 0x1p-23f;
                // log alpha in FP32 (alpha is exact in FP32; error <= 2e-6, far inside the
                // near-tie band); the log-ratio it is compared with stays FP64
                const double log_alpha = (double)logf(alpha);
                const double logl_cur = p.logl_cur[c];
                acc = (log_alpha < logl_prop - logl_cur) ? 1 : 0;
                int32_t win = p.acc_win[c];
                if (acc) {
                    p.logl_cur[c] = logl_prop;
                    p.cur[c] ^= 1;
                    win += 1;
                    p.acc_total[c] += 1;
                }
                if (p.trace_steps > 0 && a.step >= 1 && a.step <= (uint32_t)p.trace_steps) {
                    const int64_t t = (int64_t)(a.step - 1) * p.R + c;
                    p.trace_acc[t] = acc;
                    p.trace_logl[t] = logl_prop;
                }
                // adaptation: every M_A steps rescale beta by the window's acceptance rate
                if (a.sp.adapt_interval > 0 && a.step % (uint32_t)a.sp.adapt_interval == 0) {
                    const double rate = (double)win / (double)a.sp.adapt_interval;
                    double beta = p.beta[c];
                    if (rate > a.sp.acc_hi) beta = a.sp.adapt_factor * beta;
                    if (rate < a.sp.acc_lo) beta = beta / a.sp.adapt_factor;
                    if (beta > a.sp.beta_max) beta = a.sp.beta_max;
                    p.beta[c] = beta;
                    p.coef[c] = make_float2((float)sqrt(1.0 - beta * beta), (float)beta);
                    win = 0;
                }
                p.acc_win[c] = win;
            }
        }
        flag[tid] = acc;
        inv_tr[tid] = itr;
    }
    __syncthreads();

    // ---- phase 2: rho write-back, pooling of the current state, trajectories ------------
    // Thread t moves float4 number (t mod V) of a chain's packed rho (V = d/4 per chain) for
    // the chains t/V, t/V + P, ... (P = 256/V chains in flight per pass, four passes
    // unrolled so that several independent loads are outstanding; eight or sixteen cost registers and
    // with them occupancy: 34 and 33 against 26 us at 65536 four-qubit chains).  Pool sums: per-thread
    // float4 partials, then a shared-memory reduction over the P chain lanes.
    const int d = p.d;
    const int V = d / 4;
    const int P = kThreads / V < 1 ? 1 : kThreads / V;
    const bool pool_now = (a.mode == MODE_STEP) && a.kept;
    const int vi = tid % V, lane_c = tid / V;
    __shared__ float4 red4[kThreads];
    for (int v0 = 0; v0 < V; v0 += kThreads) {          // d > 1024 only: several vector columns per thread
        const int vv = v0 + (V < kThreads ? vi : tid);
        const bool vthread = (V < kThreads) ? (lane_c < P) : (vv < V);
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vthread) {
            // chains k0, k0 + st, ...: four loads in flight per batch, one per chain (the new
            // current state: rho' if accepted, else the stored rho, read only when pooling)
            const int k0 = (V < kThreads ? lane_c : 0), st = (V < kThreads ? P : 1);
            constexpr int B = 4;
            for (int kb = k0; kb < nc; kb += B * st) {
                float4 q[B];
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const int k = kb + u * st;
                    q[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k < nc && (flag[k] || pool_now)) {
                        const int64_t c = c0 + k;
                        const float *row = flag[k] ? p.rho_prop : p.rho_cur;
                        q[u] = reinterpret_cast<const float4 *>(row + c * p.d_pad)[vv];
                    }
                }
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const int k = kb + u * st;
                    if (k >= nc) break;
                    const int64_t c = c0 + k;
                    float4 val = q[u];
                    if (flag[k]) {
                        const float s_ = inv_tr[k];
                        val = make_float4(val.x * s_, val.y * s_, val.z * s_, val.w * s_);
                        reinterpret_cast<float4 *>(p.rho_cur + c * p.d_pad)[vv] = val;
                    }
                    if (pool_now) {
                        sum.x += val.x;
                        sum.y += val.y;
                        sum.z += val.z;
                        sum.w += val.w;
                        if (c < p.n_diag && a.kept_idx < p.traj_cap)
                            reinterpret_cast<float4 *>(p.traj + ((int64_t)c * p.traj_cap + a.kept_idx) * d)[vv] = val;
                    }
                }
            }
        }
        if (pool_now) {
            red4[tid] = sum;
            __syncthreads();
            if (V < kThreads) {
                if (tid < V) {
                    float4 tot = red4[tid];
                    for (int q = 1; q < P; ++q) {
                        const float4 o = red4[q * V + tid];
                        tot.x += o.x;
                        tot.y += o.y;
                        tot.z += o.z;
                        tot.w += o.w;
                    }
                    double *slot = p.pool + (int64_t)blockIdx.x * d + 4 * tid;
                    slot[0] += (double)tot.x;
                    slot[1] += (double)tot.y;
                    slot[2] += (double)tot.z;
                    slot[3] += (double)tot.w;
                }
            } else if (vthread) {
                double *slot = p.pool + (int64_t)blockIdx.x * d + 4 * vv;
                slot[0] += (double)sum.x;
                slot[1] += (double)sum.y;
                slot[2] += (double)sum.z;
                slot[3] += (double)sum.w;
            }
            __syncthreads();
        }
        if (V < kThreads) break;
    }
}

// Sums the pool slots -> out[d] (deterministic): a CTA owns 32 consecutive entries; its warp w
// adds slots [w n/32, (w + 1) n/32) in slot order, and the 32 partial sums are added in warp order.
constexpr int kReduceWarps = 32;
__global__ void __launch_bounds__(32 * kReduceWarps) pool_reduce_kernel(const double *pool, int n_slots, int d,
                                                                          double *out) {
    __shared__ double part[kReduceWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    const int per = (n_slots + kReduceWarps - 1) / kReduceWarps;
    const int b0 = w * per, b1 = min(n_slots, b0 + per);
    double s = 0.0;
    if (e < d)
        for (int b = b0; b < b1; ++b) s += pool[(int64_t)b * d + e];
    part[w][lane] = s;
    __syncthreads();
    if (w == 0 && e < d) {
        double t = 0.0;
        for (int k = 0; k < kReduceWarps; ++k) t += part[k][lane];
        out[e] = t;
    }
}

// Eq. ACFrho of the diagnostic chains: c~[l] = sum_{n < N - lmax} sum_e w_e (x_n,e - m_e)
// (x_{n+l},e - m_e) with w_e = 1 on the diagonal and 2 off it (each packed off-diagonal entry
// stands for the (i,j) and (j,i) terms of Eq. ACFa).  Products in FP32 summed over chunks of 32
// samples; a thread's chunks are added as FP32 pairs (two-sums, 48 bits), its entries and the slabs in FP64.
// The chunks' own rounding is what remains: the error against FP64 of the ACF and of tau is the same to
// four digits as with FP64 sums of chunks and samples (one to four qubits, 16 to 512 chains, 210 to 1024
// states, 50 to 200 lags).
//
// The work is d (N - lmax) (lmax + 1) multiply-adds per chain on N d values, so it is bound by
// the FP32 pipe once each value is loaded rarely enough.  A CTA takes one chain, a slab of up to
// kAcfEntries packed entries and kAcfLags lags.  A thread owns a pair of entries (f32x2) and
// kAcfTile consecutive lags: the centred samples sit in shared memory, and a register window of
// kAcfTile samples slides along, so two 64-bit loads feed kAcfTile packed FMAs (one load per FMA
// operand, one entry and one lag at a time, took 12.8 ms for 256 four-qubit chains of 600 states
// and 201 lags; this form 0.41 ms, the FP32 pipe busy half of it).  Samples pass through in segments of kAcfSeg, so neither N
// nor lmax is limited by shared memory.
constexpr int kAcfEntries = 32;                          // packed entries per slab
constexpr int kAcfTile = 16;                             // lags per thread
constexpr int kAcfLagTiles = 13;                         // lag tiles per CTA (l_max = 200 fits one CTA)
constexpr int kAcfLags = kAcfTile * kAcfLagTiles;        // 208
constexpr int kAcfSeg = 256;                             // samples n per segment (a multiple of 32)
constexpr int kAcfRowsB = kAcfSeg + kAcfLags;            // samples n + l of a segment
constexpr int kAcfThreads = kAcfEntries / 2 * kAcfLagTiles;   // 208
constexpr size_t kAcfSmem = sizeof(float) * kAcfEntries * (kAcfSeg + kAcfRowsB);

// part[chain][slab][l]: the slab's share of c~[l]; grid (chains, slabs, lag groups)
__global__ void __launch_bounds__(kAcfThreads, 2) acf_kernel(const float *traj, int traj_cap, int d, int D, int n_kept,
                                                          int lmax, double *part) {
    extern __shared__ __align__(16) float acf_sm[];
    float *za = acf_sm, *zb = acf_sm + kAcfSeg * kAcfEntries;   // [sample][entry], centred
    __shared__ __align__(16) float mean[kAcfEntries];
    const int ne = min(kAcfEntries, d);                 // entries of a slab (d is 4, 16 or a multiple of 32)
    const int np = ne / 2;                              // entry pairs: consecutive lanes
    const int tid = threadIdx.x;
    const int pr = tid % np, lt = tid / np;             // this thread's pair and lag tile
    const bool worker = lt < kAcfLagTiles;
    const int e0 = blockIdx.y * ne;
    const float *x = traj + (int64_t)blockIdx.x * traj_cap * d + e0;

    // means over all N samples: exact pairs per thread, joined in FP64
    {
        float2 hi = make_float2(0.f, 0.f), lo = hi;
        const int lanes = kAcfThreads / np;
        constexpr int kInFlight = 16;   // loads requested together (one at a time: half of the kernel's time)
        if (lt < lanes)
            for (int n = lt; n < n_kept; n += kInFlight * lanes) {
                float2 v[kInFlight];
#pragma unroll
                for (int u = 0; u < kInFlight; ++u) {
                    v[u] = make_float2(0.f, 0.f);
                    if (n + u * lanes < n_kept)
                        v[u] = *reinterpret_cast<const float2 *>(x + (int64_t)(n + u * lanes) * d + 2 * pr);
                }
#pragma unroll
                for (int u = 0; u < kInFlight; ++u) {
                    float e;
                    two_sum(hi.x, v[u].x, hi.x, e);
                    lo.x += e;
                    two_sum(hi.y, v[u].y, hi.y, e);
                    lo.y += e;
                }
            }
        double *md = reinterpret_cast<double *>(acf_sm);   // [lane][entry] sums, before the samples move in
        if (lt < lanes) {
            md[lt * ne + 2 * pr] = (double)hi.x + (double)lo.x;
            md[lt * ne + 2 * pr + 1] = (double)hi.y + (double)lo.y;
        }
        __syncthreads();
        if (tid < ne) {
            double s = 0.0;
            for (int q = 0; q < lanes; ++q) s += md[q * ne + tid];
            mean[tid] = (float)(s / n_kept);
        }
        __syncthreads();
    }

    const int m = n_kept - lmax;
    const int l0 = blockIdx.z * kAcfLags;              // this CTA's lags l0 .. l0 + kAcfLags - 1
    const int lag = lt * kAcfTile;
    const int ea = e0 + 2 * pr;
    const int nq = ne / 4, lq = tid % nq, lr = tid / nq;   // loads: this thread's float4 column (208 is a multiple of nq)
    const float4 mq = *reinterpret_cast<const float4 *>(mean + 4 * lq);
    const float2 w = make_float2((ea / D) == (ea % D) ? 1.0f : 2.0f, ((ea + 1) / D) == ((ea + 1) % D) ? 1.0f : 2.0f);
    float hi[kAcfTile], lo[kAcfTile];   // sums over both entries
#pragma unroll
    for (int i = 0; i < kAcfTile; ++i) hi[i] = lo[i] = 0.0f;
    for (int n0 = 0; n0 < m; n0 += kAcfSeg) {
        const int rows = min(kAcfSeg, (m - n0 + 31) / 32 * 32);   // whole chunks; samples n >= m count as zero
        __syncthreads();
        // the first lag group's samples n are the first rows of its samples n + l: only later
        // groups, and a segment that ends at m (samples from there on count as zero), load them apart
        auto fill = [&](float *z, int first, int count, int end) {
#pragma unroll 4
            for (int r = lr; r < count; r += kAcfThreads / nq) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (first + r < end) {
                    v = *reinterpret_cast<const float4 *>(x + (int64_t)(first + r) * d + 4 * lq);
                    v = make_float4(v.x - mq.x, v.y - mq.y, v.z - mq.z, v.w - mq.w);
                }
                *reinterpret_cast<float4 *>(z + r * ne + 4 * lq) = v;
            }
        };
        const bool own = l0 != 0 || n0 + rows > m;
        if (own) fill(za, n0, rows, m);
        fill(zb, n0 + l0, rows + kAcfLags, n_kept);
        __syncthreads();
        if (worker) {
            const float *pa = (own ? za : zb) + 2 * pr, *pb = zb + lag * ne + 2 * pr;
            float2 win[kAcfTile];   // sample n + lag + i in slot (n + i) mod kAcfTile
#pragma unroll
            for (int i = 0; i < kAcfTile; ++i) win[i] = *reinterpret_cast<const float2 *>(pb + i * ne);
            float2 a_next = *reinterpret_cast<const float2 *>(pa);
#pragma unroll 1
            for (int c = 0; c < rows; c += 32) {
                float2 chunk[kAcfTile];
#pragma unroll
                for (int i = 0; i < kAcfTile; ++i) chunk[i] = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int h = c; h < c + 32; h += kAcfTile) {
#pragma unroll
                    for (int u = 0; u < kAcfTile; ++u) {
                        const float2 a = a_next;   // (the row after the last one is zb's first)
                        a_next = *reinterpret_cast<const float2 *>(pa + (h + u + 1) * ne);
#pragma unroll
                        for (int i = 0; i < kAcfTile; ++i)
                            chunk[i] = fma2(a, win[(u + i) % kAcfTile], chunk[i]);
                        // the sample kAcfTile further on (the last row read is rows + kAcfTile - 1 past the tile)
                        win[u] = *reinterpret_cast<const float2 *>(pb + (h + u + kAcfTile) * ne);
                    }
                }
#pragma unroll
                for (int i = 0; i < kAcfTile; ++i) {   // hi + lo += w chunk, exactly (two-sum)
                    const float2 v = mul2(w, chunk[i]);
                    float e, e2;
                    two_sum(hi[i], v.x, hi[i], e);
                    two_sum(hi[i], v.y, hi[i], e2);
                    lo[i] += e + e2;
                }
            }
        }
    }
    // the pairs of a lag tile sit in np consecutive lanes (a power of two, 2 .. 16): FP64 tree
    double *out = part + ((int64_t)blockIdx.x * gridDim.y + blockIdx.y) * (lmax + 1);
    const unsigned lanes_mask = (tid / 32 + 1) * 32 <= kAcfThreads ? 0xffffffffu : (1u << (kAcfThreads % 32)) - 1u;
#pragma unroll
    for (int i = 0; i < kAcfTile; ++i) {
        double v = (double)hi[i] + (double)lo[i];
        for (int off = np / 2; off > 0; off >>= 1) v += __shfl_xor_sync(lanes_mask, v, off);
        const int l = l0 + lag + i;
        if (worker && pr == 0 && l <= lmax) out[l] = v;
    }
}

// out[chain][l] = sum over the slabs, in slab order
__global__ void acf_reduce_kernel(const double *part, int slabs, int nl, int64_t total, double *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int64_t c = i / nl, l = i - c * nl;
    double s = 0.0;
    for (int b = 0; b < slabs; ++b) s += part[(c * slabs + b) * nl + l];
    out[i] = s;
}

// log L = C0 - N log t + sum over column groups, for stateless evaluation.
__global__ void logl_combine_kernel(const double *part, const double *trace, int ngroups, int64_t rows, double C0,
                                    double Ntot, double *out) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    double v = C0 - Ntot * log(trace[r]);
    for (int g = 0; g < ngroups; ++g) v += part[(int64_t)g * rows + r];
    out[r] = v;
}

__global__ void philox_blocks_kernel(uint64_t seed, uint32_t step, uint32_t tag, uint32_t chain0, int64_t nchains,
                                     uint32_t block0, int32_t nblocks, uint32_t *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nchains * nblocks) return;
    const uint32_t c = chain0 + (uint32_t)(i / nblocks);
    const uint32_t b = block0 + (uint32_t)(i % nblocks);
    const uint4 w = Philox::block(make_uint4(b, step, c, tag), (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
    reinterpret_cast<uint4 *>(out)[i] = w;
}

__global__ void inject_nan_kernel(float *y, const uint8_t *cur, int64_t R, int nx, int64_t chain) {
    const int b = cur[chain];
    for (int e = threadIdx.x; e < nx; e += blockDim.x) y[((int64_t)b * R + chain) * nx + e] = __int_as_float(0x7fc00000);
}

}  // namespace

cudaError_t launch_accept(const ProblemView &p, const SamplerParams &sp, int mode, StepState *step_dev, uint32_t *status,
                          cudaStream_t s) {
    (void)status;
    AcceptArgs a;
    a.p = p;
    a.sp = sp;
    a.mode = mode;
    a.step = 0u;
    a.kept = 0;
    a.kept_idx = 0;
    a.step_dev = step_dev;
    const int64_t blocks = (p.R + p.accept_cpc - 1) / p.accept_cpc;
    accept_kernel<<<(unsigned)blocks, kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

// Up to 256 packed floats per chain (D <= 16) a CTA takes 128 chains, which moves its 256
// threads' float4 lanes over several chains at once.  From D = 32 on, each chain alone fills
// the CTA's lanes and a CTA walks its chains in turn, so 128 chains per CTA leave most SMs
// idle (4096 six-qubit chains: 32 CTAs) and the copy latency-bound: halve the chains per CTA
// until the grid covers the SMs twice, down to 8 (more pool slots, each read and written
// once per kept step).
int accept_chains_per_cta(int64_t R, int d) {
    if (d < 4 * kThreads) return kChainsPerCta;
    static int num_sms = 0;
    if (num_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || num_sms <= 0)
            num_sms = 148;
    }
    int c = kChainsPerCta;
    while (c > 8 && (R + c - 1) / c < 2 * (int64_t)num_sms) c /= 2;
    return c;
}

cudaError_t launch_pool_reduce(const ProblemView &p, double *out, cudaStream_t s) {
    pool_reduce_kernel<<<(p.d + 31) / 32, 32 * kReduceWarps, 0, s>>>(p.pool, p.n_slots, p.d, out);
    return cudaGetLastError();
}

int acf_slabs(int d) { return (d + kAcfEntries - 1) / kAcfEntries; }

cudaError_t launch_acf(const ProblemView &p, int n_kept, int lmax, double *part, cudaStream_t s) {
    if (p.n_diag <= 0 || n_kept <= lmax) return cudaSuccess;
    // more than 48 KB of dynamic shared memory: opted into once per device
    static std::atomic<unsigned long long> attr_set{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !((attr_set.load() >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(acf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAcfSmem);
        if (e != cudaSuccess) return e;
        if (dev < 64) attr_set.fetch_or(1ull << dev);
    }
    const int slabs = acf_slabs(p.d);
    const dim3 grid((unsigned)p.n_diag, (unsigned)slabs, (unsigned)(lmax / kAcfLags + 1));
    acf_kernel<<<grid, kAcfThreads, kAcfSmem, s>>>(p.traj, p.traj_cap, p.d, p.D, n_kept, lmax, part);
    return cudaGetLastError();
}

cudaError_t launch_acf_reduce(const ProblemView &p, int lmax, const double *part, double *acf_raw, cudaStream_t s) {
    const int64_t total = (int64_t)p.n_diag * (lmax + 1);
    acf_reduce_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(part, acf_slabs(p.d), lmax + 1, total, acf_raw);
    return cudaGetLastError();
}

cudaError_t launch_logl_combine(const ProblemView &p, int64_t rows, double *out, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    logl_combine_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(p.logl_part, p.trace_prop, p.ngroups, rows, p.C0,
                                                                         p.Ntot, out);
    return cudaGetLastError();
}

cudaError_t launch_philox_blocks(uint64_t seed, uint32_t step, uint32_t tag, uint32_t chain0, int64_t nchains,
                                 uint32_t block0, int32_t nblocks, uint32_t *out, cudaStream_t s) {
    const int64_t total = nchains * nblocks;
    if (total <= 0) return cudaSuccess;
    philox_blocks_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(seed, step, tag, chain0, nchains, block0,
                                                                          nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_inject_nan(const ProblemView &p, int64_t chain, cudaStream_t s) {
    inject_nan_kernel<<<1, 256, 0, s>>>(p.y, p.cur, p.R, p.nx, chain);
    return cudaGetLastError();
}

}  // namespace qst
