// k_misc.cuh -- declarations of the support kernels' launchers.
#pragma once
#include "sre_internal.cuh"

namespace sre {

// slots of the device scalar block
enum { SCAL_NORM2 = 0, SCAL_S = 1, SCAL_N = 8 };
constexpr int NORM_BLOCKS = 1216;          // 152 SMs x 8
constexpr unsigned long long SCAN_CHUNK = 4096;
// totals of an exact sweep (per state): sum over families of c^2, c^4, c^6,
// c^2 log2 c^2 sums, candidate count, sum over x != 0 of (sum_z c^4)^2, and
// the x = 0 family's sum_z c^4 (the last two give the fluctuation ratio r_2)
constexpr int TOT_N = 7;

struct DrawInfo {
    unsigned long long range;   // z-range (size 2^RL) of the draw
    double t;                   // target within the range, in units of c^2
    double wr;                  // the range's weight (sum of its c^2)
    double pad;
};

constexpr int NORM_ONE_NMAX = 13;          // one block and one launch up to here
// sum |psi|^2 and its inverse into scal; *launches receives the kernels issued;
// zero (or NULL): two words that the launch clears
cudaError_t launch_norm2(const float2 *psi, int N, double *scal, double *partial, cudaStream_t st, int *launches,
                         unsigned long long *zero = nullptr);

// Totals of the family sums of states s0 .. s0 + ns - 1 (N qubits each; family
// f of state st at fm[(st << N) + f - fm_first]) into out[TOT_N st ..] (slot 4
// is unused). flags / n_flag (or NULL): list and count of the candidate
// families. partial: 5 totals_blocks(N, ns) doubles a state; done: a zeroed
// counter a state. norm2 (one state only, or NULL): the norm, which then goes to
// out[TOT_N] with the number of flagged families in out[TOT_N + 1].
constexpr int TOTALS_BLOCKS = 304;
inline int totals_blocks(int N, int ns) {
    const long long want = (1LL << N) / 256, most = ns > 0 ? (TOTALS_BLOCKS + ns - 1) / ns : 1;
    return (int)(want < 1 ? 1 : want < most ? want : most);
}
struct TotalsArgs {
    const FamMoments *fm;
    long long fm_first;
    int N, s0;
    double *out, *partial;
    unsigned *done;
    unsigned long long *flags, *n_flag;
    const double *norm2;
};
cudaError_t launch_totals(const TotalsArgs &a, int ns, cudaStream_t st);

// FP64 recount of flagged families at their listed candidates (k_null.cu).
// Family i of the launch is xs[fam_base + i] (F = (state << N) | x when
// psi_list is set); its candidate count and list come from the FP32
// DST_CANDLIST pass. counts[i] receives the family's stabilizer count, or 0
// when it had no candidate or more than kdirect (<= cand_max, <=
// NULL_CAND_MAX) of them; in the latter case F is appended to ovf (ovf_n).
constexpr int NULL_CAND_MAX = 64;
struct NullDirectArgs {
    const float2 *psi;
    const double *s_ptr;
    const float2 *const *psi_list;
    const double *s_list;
    int N;
    const unsigned long long *xs;
    long long fam_base;
    const unsigned *cand_cnt;
    const unsigned *cand_z;
    int cand_max, kdirect;
    double eps;
    unsigned long long *counts, *ovf, *ovf_n;
    unsigned long long *total;        // sum of the counts of every launch (zeroed before the first), or NULL
};
cudaError_t launch_null_direct(const NullDirectArgs &a, long long n_fam, cudaStream_t st);
// per-family sums of a launch's tile partials into fm[fm_base + slot], or,
// with perm (processing order -> family index), into fm[perm[fam_base + slot]]
cudaError_t launch_fam_reduce(const TilePartial *tp, long long n_fam, int tiles, const unsigned long long *xs,
                              long long fam_base, int N, int M_last, int RL, FamMoments *fm, long long fm_base,
                              float *W, long long nr, cudaStream_t st, const unsigned long long *perm = nullptr);
cudaError_t launch_sum_u64(const unsigned long long *v, long long n, unsigned long long *out, cudaStream_t st);
// bsum: n / SCAN_CHUNK + 1 doubles (chunks rounded up), the exclusive prefix of p's
// chunk sums and the total; tot: 32 doubles of scratch; cdf (or NULL): the
// inclusive CDF of p
cudaError_t launch_scan(const double *p, unsigned long long n, double *cdf, double *bsum, double *tot, int *launches,
                        cudaStream_t st);
// mode 0: uniform on 1 .. d - 1 (no arrays); 1: from the CDF of p, boff as above
cudaError_t launch_draw_x(const double *cdf, const double *p, const double *boff, int N, long long n_x, int mode,
                          unsigned long long seed, unsigned long long ctr0, unsigned long long *xs, cudaStream_t st);
// marginal draws from p and the prefix of its chunk sums (N >= 12)
cudaError_t launch_draw_x_chunks(const double *p, const double *boff, int N, long long n_x, unsigned long long seed,
                                 unsigned long long ctr0, unsigned long long *xs, cudaStream_t st);
constexpr long long ZSEL_STAGE_MAX = 16384;   // ranges of a row that is staged in shared memory
// sums: 256 doubles per family of a launch (rows of more ranges than that)
cudaError_t launch_zrange_select(const float *Wf, long long nr, long long n_fam, long long fam_base, int z_per_x,
                                 unsigned long long seed, unsigned long long ctr0, DrawInfo *draws,
                                 const unsigned long long *perm, double *sums, int *launches, cudaStream_t st);
cudaError_t launch_mc_stats(const FamMoments *fm, const float *cz, long long n_x, int z_per_x, int N, int mode,
                            double *y, double *out, cudaStream_t st);
cudaError_t launch_norm2_multi(const float2 *const *psi_list, int n_states, int N, double *partial, int nb,
                               double *norm2, double *s, cudaStream_t st);
cudaError_t launch_count_scatter(const unsigned long long *flags, const unsigned long long *counts, long long n,
                                 int N, unsigned long long *state_count, cudaStream_t st);
cudaError_t launch_philox_test(const unsigned long long *ctr_key, unsigned long long *out, int n, cudaStream_t st);

// z sampler (k_sample.cu): recompute the c of each draw's range and pick z by
// the exact fixed-point scan of c^2 over the range. fine: ranges of 2^ZR_FINE z
// recomputed from the folded last-pass tile; else a range is a tile half.
// one warp whose mbarrier wait can only end by its bound (k_sample.cu);
// src16: 16 readable, 16-byte aligned device bytes; err: device word
cudaError_t launch_wait_selftest(const void *src16, int *err, cudaStream_t st);
// z draws of a launch's families (k_sample.cu); perm as for launch_fam_reduce
cudaError_t launch_zsample(int single, int fine, int M, const PassArgs &a, const DrawInfo *draws, int z_per_x,
                           unsigned long long *zs, float *cz, const unsigned long long *perm, cudaStream_t st);

// The x-marginal into p (d doubles) with work (d doubles) as intermediate, for
// N >= MARG_NMIN (k_marg.cu); scal holds the norm (launch_norm2).
constexpr int MARG_ROW_BITS = 11, MARG_STRIDED_MAX = 9;
constexpr int MARG_NMIN = MARG_ROW_BITS + 2;
cudaError_t launch_marginal(const float2 *psi, int N, const double *scal, double *p, double *work, int *launches,
                            cudaStream_t st);

// gates (k_gates.cu)
struct __align__(4) GateRow { unsigned char op, q0, q1, pad; };
constexpr unsigned char GATE_OP_U2 = 6;   // general two-qubit gate (matrix table indexed by row)
constexpr int GATE_BLOCK_MAX_U2 = 512;     // two-qubit matrices per block (64 KB of shared memory)
constexpr int GATE_BLOCK_Q = 13;   // qubits per fused gate block (2^13 amplitudes, 64 KB of shared memory)
constexpr int GATE_BLOCK_LOW = 5;  // qubits 0..4 always in the block (256-byte contiguous runs)
constexpr int GATE_ROUND_SLOTS = 5;   // local qubits that a thread holds in a round (32 amplitudes)
// A round: the gates rows [g0, g0 + ng) with local bits slot[i] in registers
// (bit i of a thread's amplitude index) and thr[i] in bit i of the thread index.
struct GateRound {
    int g0, ng;
    unsigned char slot[GATE_ROUND_SLOTS], thr[GATE_BLOCK_Q - GATE_ROUND_SLOTS];
    unsigned char pad[3];
};
// A block: its global qubits (ascending, 255 = unused), rounds and gate rows.
struct GateBlock {
    int r0, nr, g0, ng;
    unsigned char qubit[GATE_BLOCK_Q];
};
// Codes of the rows of a round (GateRow::op on the device): slot indices for
// H, for a phase gate (q0: the phase in units of pi / 4) and for a CNOT (5
// control + target); with q1 a thread bit, the phase gate and the CNOT
// controlled outside the slots. Two-qubit matrices: slots a < b as b (b - 1) / 2 + a.
enum GateCode { GC_H = 0, GC_PHASE = 5, GC_PHASE_THREAD = 10, GC_CX = 11, GC_CX_THREAD = 36 };
// Whether a list runs gate by gate in shared memory instead of in register
// rounds. A state of fewer than 13 qubits would leave most threads of a round
// idle (32 amplitudes each): a call with 400 random gates at N = 8 takes 109 us in
// place and 178 in rounds, 24 brick-wall layers at N = 12 174 and 188 us. And a
// short list of matrices on a few tiles pays for fetching the rounds' unrolled
// code more than for its barriers: 4 layers (26 to 34 gates) take 72 and 81 us at
// N = 14, 91 and 100 us at N = 18, but 122 and 103 us at N = 20 (128 tiles); N = 13
// 88 and 75 us; 2 N layers 362 and 310 us at N = 14.
inline bool gates_in_place(int N, long long n_gates, bool mats) {
    return N < GATE_BLOCK_Q || (mats && n_gates <= 40 && N > GATE_BLOCK_Q && N <= 18);
}
// A gate list in its blocks; rounds_dev NULL: in place (rows with opcodes and local qubits).
cudaError_t launch_gate_blocks(float2 *psi, int N, const GateRow *gates_dev, const GateRound *rounds_dev,
                               const float2 *mats_dev, const GateBlock *blocks, int n_blocks, cudaStream_t st);

// tcgen05 self-test GEMM (k_tc05.cu): D = A B^T, BF16 in, FP32 out
cudaError_t launch_tc05_gemm_selftest(const void *A, const void *B, float *D, int M, int N, int K, int swizzle,
                                      int *err, cudaStream_t st);

// Gram matrix C = Psi Psi^H of the reduced state on the low N_A qubits
// (k_gram.cu): column-major d_A x d_A complex C; `planes` holds
// gram_plane_bytes(N, N_A) bytes; *launches receives the kernels issued.
size_t gram_plane_bytes(int N, int NA);
cudaError_t launch_gram(const float2 *psi, int N, int NA, float2 *C, void *planes, int *err, int *launches,
                        cudaStream_t st);

} // namespace sre
