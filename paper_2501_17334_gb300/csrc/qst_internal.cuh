// Internal definitions of the GB300 sampler: device-side problem view, kernel
// argument blocks, the counter-based generator and launch declarations.
#pragma once

#include "log_poly.h"
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace qst {

// Device status bits (read back by synchronising calls).
enum : uint32_t {
    STATUS_TIMEOUT = 1u << 0,     // a bounded mbarrier wait gave up
    STATUS_BOUNDS = 1u << 1,      // a kernel's own bounds check failed
    STATUS_BAD_LAUNCH = 1u << 2,  // a kernel was launched with an unsupported shape
};

// Stream tags of the counter layout (block, step j, global chain id, tag).
enum : uint32_t { TAG_INIT = 0, TAG_PROPOSAL = 1, TAG_ALPHA = 2 };

enum ProposeMode : int { MODE_INIT = 0, MODE_STEP = 1, MODE_EVAL = 2 };

// ---------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32->64
// multiplications whose high halves are xored into the other two words with the
// round key, the key bumped by the Weyl constants after every round.
// ---------------------------------------------------------------------------------------
struct Philox {
    static constexpr uint32_t kMulA = 0xD2511F53u;
    static constexpr uint32_t kMulB = 0xCD9E8D57u;
    static constexpr uint32_t kWeylA = 0x9E3779B9u;
    static constexpr uint32_t kWeylB = 0xBB67AE85u;

    __device__ __forceinline__ static uint4 block(uint4 ctr, uint32_t key_lo, uint32_t key_hi) {
#pragma unroll
        for (int round = 0; round < 10; ++round) {
            const uint32_t pa_hi = __umulhi(kMulA, ctr.x);
            const uint32_t pa_lo = kMulA * ctr.x;
            const uint32_t pb_hi = __umulhi(kMulB, ctr.z);
            const uint32_t pb_lo = kMulB * ctr.z;
            ctr = make_uint4(pb_hi ^ ctr.y ^ key_lo, pb_lo, pa_hi ^ ctr.w ^ key_hi, pa_lo);
            key_lo += kWeylA;
            key_hi += kWeylB;
        }
        return ctr;
    }

    // The same block with the ten round keys (key + r (kWeylA, kWeylB)) given: a kernel that
    // takes them as launch parameters reads them as constant operands instead of forming them.
    struct RoundKeys {
        uint32_t k[20];   // (lo, hi) of rounds 0..9
    };
    __host__ __device__ static RoundKeys round_keys(uint64_t seed) {
        RoundKeys rk;
        uint32_t lo = (uint32_t)(seed & 0xffffffffu), hi = (uint32_t)(seed >> 32);
        for (int r = 0; r < 10; ++r) {
            rk.k[2 * r] = lo;
            rk.k[2 * r + 1] = hi;
            lo += kWeylA;
            hi += kWeylB;
        }
        return rk;
    }
    __device__ __forceinline__ static uint4 block(uint4 ctr, const RoundKeys &rk) {
#pragma unroll
        for (int round = 0; round < 10; ++round) {
            const uint32_t pa_hi = __umulhi(kMulA, ctr.x);
            const uint32_t pa_lo = kMulA * ctr.x;
            const uint32_t pb_hi = __umulhi(kMulB, ctr.z);
            const uint32_t pb_lo = kMulB * ctr.z;
            ctr = make_uint4(pb_hi ^ ctr.y ^ rk.k[2 * round], pb_lo, pa_hi ^ ctr.w ^ rk.k[2 * round + 1], pa_lo);
        }
        return ctr;
    }

    // Open-interval uniform from the top 23 bits m: (2 m + 1) 2^-24, exact in float.  Formed
    // by bit operations: 1 + m 2^-23 is the float with m as its mantissa, and subtracting
    // 1 - 2^-24 (a float) leaves (2 m + 1) 2^-24, representable, so the subtraction is exact.
    __device__ __forceinline__ static float uniform(uint32_t word) {
        return __int_as_float(0x3f800000u | (word >> 9)) - 0x1.fffffep-1f;
    }

    // Box-Muller on one uniform pair: (sqrt(-2 ln u) cos 2 pi v, sqrt(-2 ln u) sin 2 pi v).
    __device__ __forceinline__ static void gaussian_pair(uint32_t wu, uint32_t wv, float &z0, float &z1) {
        const float u = uniform(wu);
        const float v = uniform(wv);
        const float radius = sqrtf(-2.0f * logf(u));
        float s, c;
        sincospif(2.0f * v, &s, &c);
        z0 = radius * c;
        z1 = radius * s;
    }
};

// ---------------------------------------------------------------------------------------
// Device view of one problem.  Dimensions: D = 2^Q, d = D^2 (packed rho), nx = 4 D^2
// (latent), KD = K*D projectors, d_pad = d rounded up to 64 (operand rows), KD_pad =
// KD rounded up to the contraction's column tile.
// ---------------------------------------------------------------------------------------
// log x for the likelihood terms: the polynomial logarithm (log_poly.h, <= 1 ulp) for
// positive normal x; -inf when x <= 0 (or below the normal range), so a counted outcome
// with p <= 0 makes log L = -inf and the proposal is rejected.  (A NaN or infinite rho
// reaches log L through its trace instead.)
__device__ __forceinline__ float deviance_log(float x) {
    const float r = qst_log_poly(x);
    return (__float_as_int(x) >= 0x00800000) ? r : -INFINITY;
}

// A problem's step counter, kept on the device so that a step's launches have fixed arguments and can
// be captured once in a CUDA graph.  The proposal of step j reads step = j - 1, and its first CTA
// opens the step (j, kept, kept_idx); the accept kernel reads those, and its first CTA closes it (step,
// kept_count).  So neither kernel writes what its own CTAs read, and the order of the launches is all
// the ordering there is.  (A one-thread kernel that opened each step was a node of its dependent
// chain, and advancing the counter in the last accept CTA to finish, by tickets, cost that kernel a
// fence and an atomic's round trip after its last store.  us per step, those two and this: 2567
// three-qubit chains 28.7, 26.7, 24.7; 2885 four-qubit chains 35.9, 35.9, 33.9; 1711 one-qubit chains
// on the tensor cores 18.7, 19.4, 17.5; 16384 three-qubit chains 47.1, 45.8, 45.5.)
struct StepState {
    uint32_t step;       // steps taken
    uint32_t multi;      // the problem runs many steps per launch (advanced by launch_advance_steps)
    int64_t kept_count;  // kept states so far
    uint32_t j;          // the step under way
    int32_t kept;        // it is kept (j % T == 0 and j > burn_in)
    int64_t kept_idx;    // and its index among the kept states (0-based)
    int64_t thin, burn_in;
};
__device__ __forceinline__ void open_step(StepState *st) {
    const uint32_t j = st->step + 1u;
    st->j = j;
    st->kept = (j % (uint32_t)st->thin == 0u) && ((int64_t)j > st->burn_in);
    st->kept_idx = st->kept_count;
}

// Operand kind of the tensor-core projection (the mixed forms).  TC_BF16X3: rho split into
// bf16 hi + mid + lo, P in bf16 (kind::f16).  TC_TF32: rho rounded to TF32 once, P in TF32
// (kind::tf32).  TC_TF32X2: rho = hi + lo, both TF32 (kind::tf32).
enum TcKind { TC_NONE = 0, TC_BF16X3 = 1, TC_TF32 = 2, TC_TF32X2 = 3 };
__host__ __device__ constexpr int tc_splits(int kind) { return kind == TC_BF16X3 ? 3 : kind == TC_TF32X2 ? 2 : 1; }
__host__ __device__ constexpr int tc_elem_bytes(int kind) { return kind == TC_BF16X3 ? 2 : 4; }

struct ProblemView {
    int D, d, nx, KD, KD_pad, d_pad;
    int tc_kind;                 // TcKind of the projection (TC_NONE: the plain FP32 form)
    int KD_tc;                   // columns of the tensor-core operand (multiple of its N tile)
    int64_t R;
    int64_t chain_offset;
    uint64_t seed;
    double C0;     // constant of the deviance form: -sum_{c>0} c log(invf), and for the Poisson
                   // likelihood + sum_{c>0} c log(mu_k) - sum_k mu_k (see the projection kernels)
    double Ntot;   // sum of all counts: weight of log t (trace of the stored rho) in log L
    int poisson;   // 0: the multinomial likelihood (Eq. likelihood); 1: Poisson counts of mean mu_k p_kl

    // packed projector operands and per-column likelihood weights
    const float *P32;            // [d_pad][KD_pad]  (row = packed rho index, contiguous columns)
    const float *sp_val;         // FP32 form at D = 8, 16 (null otherwise): per setting the rows of P where any
                                 //                  of its elements is nonzero, [K][d][D],
    const uint32_t *sp_code;     //                  their row codes [K][d]
    const uint16_t *sp_len;      //                  and the number of rows listed [K];
    int64_t sp_rows;             //                  their sum and the most of one setting, where the host
    int sp_most;                 //                  knows them (0 otherwise)
    const void *Ptc;             // [KD_tc][d_pad]   tensor-core B operand (row = projector, contiguous packed
                                 //                  index): bf16, or FP32 holding TF32 values
    const float *cnt;            // [max(KD_pad, KD_tc)] counts as float, 0 on padding
    const float *invf;           // [max(KD_pad, KD_tc)] P_k / c_kl, Poisson: mu_k / c_kl (1 where c_kl = 0)
    const float *ptot;           // [max(KD_pad, KD_tc) / D] shots P_k of each setting, Poisson: its expected
                                 //                  trials mu_k (0 on padding)
    const float4 *colw;          // [max(KD_pad, KD_tc) / 2] per column pair (invf, invf, add, add), tensor epilogue
    int pauli;                   // the structured Pauli form of the projection (project_pauli.cu)
    const float4 *pauli_wq;      // [KD / 2] deviance weights per output pair in the structured form's order
    const float2 *pauli_wc;      // [KD / 2] and their counts (pauli_weights)
    const int32_t *pauli_perm;   // [KD] tree output k of block p -> setting-major projector index, at [k][p]

    // chain state
    float *y;                    // [2][R][nx] double-buffered latent states
    uint8_t *cur;                // [R] which y buffer holds the current state
    float *rho_cur;              // [R][d_pad] packed rho of the current state
    float *rho_prop;             // [R][d_pad] packed rho of the proposal (FP32 operand)
    void *rho_split;             // [R][tc_splits][d_pad] the same split for the tensor cores: bf16 hi/mid/lo,
                                 //                  or FP32 TF32 hi[, lo]
    double *trace_prop;          // [R] exact FP64 sum of rho_prop's stored diagonal (1 up to rounding)
    double *logl_cur;            // [R]
    double *logl_part;           // [ngroups][R] partial deviance sums of the proposal
    double *beta;                // [R]
    float2 *coef;                // [R] (sqrt(1 - beta^2), beta) rounded to FP32, for the proposal
    int32_t *acc_win;            // [R] accepts in the current adaptation window
    int64_t *acc_total;          // [R]
    double *pool;                // [n_slots][d] FP64 pooled sums, one slot per accept CTA
    int n_slots;
    int accept_cpc;              // chains per accept CTA (n_slots = ceil(R / accept_cpc))
    float *traj;                 // [n_diag][traj_cap][d] kept states of the diagnostic chains
    int n_diag;
    int traj_cap;
    uint8_t *trace_acc;          // [trace_steps][R]
    double *trace_logl;          // [trace_steps][R]
    int trace_steps;
    int ngroups;                 // column groups of the projection (partial sums per group)
    int qr_passes;               // 1 or 2 modified Gram-Schmidt passes, 3: one pass and the refinement; 0: no QR
                                 // (Hilbert-Schmidt prior, W = G)
    int propose_threads = 128;   // CTA size of the proposal kernel at D <= 16 (32, 64 or 128; autotuned)
    bool propose_fixed = false;  // that size was asked for
    int64_t beside = 0;          // chains of the handle's other problems of three qubits or more
};

struct SamplerParams {
    int32_t adapt_interval;
    double acc_lo, acc_hi, adapt_factor, beta_max;
};

// ---------------------------------------------------------------------------------------
// Launchers (each returns the CUDA launch error).
// ---------------------------------------------------------------------------------------
// step_dev: when not null the step is the one after it (MODE_STEP) and is opened, else `step` is used
cudaError_t launch_propose(const ProblemView &p, int mode, uint32_t step, StepState *step_dev, const float *x_eval, int64_t n_eval,
                           bool want_split, float *rho_norm_out, uint32_t *status, cudaStream_t s);
// two groups of lanes per chain (32 / D chains per CTA), in a step or in a call by itself
bool propose_split(const ProblemView &p, int64_t rows, bool step);
cudaError_t launch_project_fp32(const ProblemView &p, const float *A, int64_t rows, double *out_part,
                                float *p_out, cudaStream_t s);
// step_dev, MODE_STEP: the counter whose open step this closes
cudaError_t launch_accept(const ProblemView &p, const SamplerParams &sp, int mode, StepState *step_dev, uint32_t *status,
                          cudaStream_t s);
cudaError_t launch_pool_reduce(const ProblemView &p, double *out, cudaStream_t s);
// ACF sums of the diagnostic chains: part [n_diag][acf_slabs(d)][lmax + 1], then acf_raw [n_diag][lmax + 1]
int acf_slabs(int d);
cudaError_t launch_acf(const ProblemView &p, int n_kept, int lmax, double *part, cudaStream_t s);
cudaError_t launch_acf_reduce(const ProblemView &p, int lmax, const double *part, double *acf_raw, cudaStream_t s);
cudaError_t launch_logl_combine(const ProblemView &p, int64_t rows, double *out, cudaStream_t s);
cudaError_t launch_philox_blocks(uint64_t seed, uint32_t step, uint32_t tag, uint32_t chain0, int64_t nchains,
                                 uint32_t block0, int32_t nblocks, uint32_t *out, cudaStream_t s);
cudaError_t launch_inject_nan(const ProblemView &p, int64_t chain, cudaStream_t s);

// Many steps of a one- or two-qubit problem in one launch (fused_small.cu).  `base`: the problem's step
// counter, as it was before the qst_run_chains call, `off` the steps of its earlier launches; the
// launch covers nsteps steps with at most fused_kept_steps(p) kept ones, whose states go to `hist`
// ([kept step][R][d] floats) for launch_fused_pool.
bool fused_supported(const ProblemView &p);
// the same before the projection's form is chosen (may_be_pauli: the structured form is one of the choices)
bool fused_possible(const ProblemView &p, bool may_be_pauli);
int fused_kept_steps(const ProblemView &p);
cudaError_t launch_fused_steps(const ProblemView &p, const SamplerParams &sp, const StepState *base, uint32_t off,
                               int nsteps, int thin, int64_t burn_in, float *hist, cudaStream_t s);
cudaError_t launch_fused_pool(const ProblemView &p, const StepState *base, uint32_t off, int nsteps, int thin,
                              int64_t burn_in, const float *hist, cudaStream_t s);
cudaError_t launch_fork(cudaStream_t s);   // a kernel that does nothing: the node a step graph's branches leave
// n steps at once for those of the `count` problems that run many steps per launch
cudaError_t launch_advance_steps(StepState *st, int count, uint32_t n, cudaStream_t s);

// tcgen05 projection in the view's tc_kind (sm_103a).  Returns cudaErrorNotSupported if the
// shape is outside what the kernel handles.
struct TcPlan;
cudaError_t tc_plan_create(const ProblemView &p, const void *A_split, int64_t rows, TcPlan **plan);
void tc_plan_destroy(TcPlan *plan);
cudaError_t launch_project_tc(const TcPlan *plan, const ProblemView &p, int64_t rows, double *out_part,
                              float *p_out, uint32_t *status, cudaStream_t s);
int tc_ngroups(const ProblemView &p, int64_t rows);
int tc_column_tile(int D, int KD);       // N tile of the tensor-core contraction for KD columns (0 = unsupported)
bool tc_supported(int kind, int D);      // the tensor-core kernels handle this operand kind at this D
// test hook: one bounded mbarrier wait that nothing satisfies (sets STATUS_TIMEOUT after limit_ns)
cudaError_t launch_wait_timeout_probe(uint32_t *status, uint64_t limit_ns, cudaStream_t s);
int fp32_ngroups(const ProblemView &p, int64_t rows);
// The FP32 form's lists of used rows per setting (project_fp32.cu): whether a call of `rows` rows takes
// the list kernel (else the tiled one), whether this size has them, the
// floats, codes and lengths they take, and the kernel that makes them from P ([d][ld], device).
bool fp32_list_form(const ProblemView &p, int64_t rows);
int fp32_list_groups(const ProblemView &p, int64_t rows);   // partial sums per row of the list kernel
bool fp32_lists(const ProblemView &p);
size_t fp32_list_values(const ProblemView &p);
size_t fp32_list_codes(const ProblemView &p);
size_t fp32_list_lengths(const ProblemView &p);
cudaError_t launch_fp32_lists(const ProblemView &p, const float *P, int ld, float *val, uint32_t *code, uint16_t *len,
                              cudaStream_t s);
// Structured Pauli form: log L partials [rows] (one column group) and optionally p [rows][KD].
cudaError_t launch_project_pauli(const ProblemView &p, const float *A, int64_t rows, double *out, float *p_out,
                                 cudaStream_t s);
void pauli_tree_order(int Q, std::vector<int32_t> &perm);   // perm[o] = k D + l of tree output o
// the structured form's per-pair weights from the setting-major counts and P_k / c
void pauli_weights(int Q, const std::vector<int32_t> &perm, const float *cnt, const float *invf,
                   std::vector<float4> &wq, std::vector<float2> &wc);
void set_last_error(const char *msg);   // message returned by qst_last_error()
// chains per accept CTA for R chains of d packed floats each (a power of two, 8..128)
int accept_chains_per_cta(int64_t R, int d);

}  // namespace qst
