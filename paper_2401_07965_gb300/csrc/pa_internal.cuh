// pa_internal.cuh -- device-side definitions shared by the library's kernels.
//
// A context advances a batch of M >= 1 independent runs (same dimension,
// coupling kind, rule and schedule; lattice size, population size, couplings
// and seed-independent identity per run) with the same kernels: one launch per
// phase covers every run.
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11), keyed
// by the 64-bit seed of the context; the counter (c0, c1, c2, c3) carries the
// draw's purpose in the top nibble of c1 and the run's identity:
//   sweep      c0 = global replica group (slot_base + slot) >> 5,
//              c1 = (sweep << 4) | (colour << 3) | plane block, c2 = step, c3 = site
//   init       c0 = word >> 2, c1 = 1 << 28, c2 = 0, c3 = slot_base + replica
//   resample   c0 = index, c1 = (2 << 28) | (run << 8) | rule, c2 = step, c3 = chunk
//   disorder   c0 = bond >> 7, c1 = 3 << 28, c2 = 0, c3 = realization
// slot_base of run m is 32 x (the sweep CTAs of runs 0..m-1); a batch of one
// run has slot_base 0 and run index 0.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pa {

constexpr uint32_t PHILOX_M0 = 0xD2511F53u;
constexpr uint32_t PHILOX_M1 = 0xCD9E8D57u;
constexpr uint32_t PHILOX_W0 = 0x9E3779B9u;
constexpr uint32_t PHILOX_W1 = 0xBB67AE85u;

constexpr uint32_t DOM_SWEEP = 0x00000000u;
constexpr uint32_t DOM_INIT = 0x10000000u;
constexpr uint32_t DOM_RESAMPLE = 0x20000000u;
constexpr uint32_t DOM_DISORDER = 0x30000000u;
constexpr uint32_t RULE_NEAREST = 0u, RULE_SYSTEMATIC = 1u, RULE_MULTINOMIAL = 2u,
                   RULE_RESIDUAL = 3u, RULE_POISSON = 4u;

constexpr int FRAC_BITS = 40;          // tau-hat is carried as a 2^-40 fixed-point integer
// tau-hat_j <= R, so f_j = floor(2^40 tau-hat_j) and T = sum_j f_j <= R 2^40 fit in
// 64 bits only for R < 2^24: the largest nominal population (and capacity)
constexpr uint32_t MAX_POPULATION = (1u << 24) - 1u;
constexpr uint32_t POISSON_KMAX = 256; // per chunk of mean <= 16

enum Method { M_MULTINOMIAL = 0, M_SYSTEMATIC = 1, M_RESIDUAL = 2, M_POISSON = 3, M_NEAREST = 4 };

enum DevStatus { S_OK = 0, S_CAPACITY = 4, S_KMAX = 5, S_TIMEOUT = 6, S_DONE = 8 };

// learned-schedule controller (MLP 8 -> 64 -> 64 -> 2, BF16 parameters)
constexpr int MLP_IN = 8, MLP_HID = 64, MLP_OUT = 2;
constexpr int MLP_NPARAM = MLP_HID * MLP_IN + MLP_HID + MLP_HID * MLP_HID + MLP_HID +
                           MLP_OUT * MLP_HID + MLP_OUT;
constexpr int CTL_UMAX = 8;  // largest step in grid units
constexpr int CLN_TAB = 64;  // family sizes c <= CLN_TAB take c ln c from a table

struct CtlDev {
    uint16_t w[MLP_NPARAM];      // BF16 parameters: W1, b1, W2, b2, W3, b3
    int32_t use_mlp;             // 0: plain steps of plain_units with plain_theta
    int32_t K;                   // grid index of beta_f
    int32_t plain_units;
    uint32_t plain_theta;
    uint32_t theta_min, theta_max;
    uint32_t budget;             // total sweeps
    int32_t u_max;               // <= CTL_UMAX
    float theta_c;               // sweeps per step of the planned step count
    int32_t pad[3];
    const double* beta_grid;     // K + 1
    const uint32_t* thr_grid;    // 4 per grid point
    const double* dbeta_tab;     // (K + 1) x CTL_UMAX: beta[k+u] - beta[k]
    const double* q_tab;         // exp(-4 dbeta_tab)
};

struct uint4x {
    uint32_t x, y, z, w;
};

// One Philox4x32-10 block.  Usable on host (couplings) and device.
__host__ __device__ __forceinline__ uint4x philox(uint32_t c0, uint32_t c1, uint32_t c2,
                                                  uint32_t c3, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t p0 = (uint64_t)PHILOX_M0 * c0;
        uint64_t p1 = (uint64_t)PHILOX_M1 * c2;
        uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
        k0 += PHILOX_W0;
        k1 += PHILOX_W1;
    }
    return {c0, c1, c2, c3};
}

// 32x32 -> 64-bit product as one wide multiply
__device__ __forceinline__ void mulhilo(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
    const uint64_t p = (uint64_t)a * (uint64_t)b;
    hi = (uint32_t)(p >> 32);
    lo = (uint32_t)p;
}

// floor(2^40 x / S), the quotient rounded to FP64 first, for 0 <= x < 2^24 S, y = 1 / S
// rounded.  Two residual corrections of x y give the rounded quotient (Markstein, IBM
// J. Res. Dev. 34, 1990): 5 operations of the FP64 pipe instead of a division's 20.  Below
// 2^-45 S the result is 0, and from there on no operation meets a subnormal unless S is tiny
// (partial resampling alone: a level sum is at least 1).
__device__ __forceinline__ uint64_t fixed_quotient(double x, double S, double y) {
    if (S < 0x1p-900) return __double2ull_rz(__dmul_rn(__ddiv_rn(x, S), 0x1p40));
    if (!(x >= __dmul_rn(S, 0x1p-45))) return 0ull;
    double q = __dmul_rn(x, y);
    q = __fma_rn(__fma_rn(-q, S, x), y, q);
    q = __fma_rn(__fma_rn(-q, S, x), y, q);
    return __double2ull_rz(__dmul_rn(q, 0x1p40));
}

// Device state shared by the kernels of a run (the runs' states stand side by side; a
// cache line each).
struct alignas(128) DevState {
    int32_t step;      // completed temperature steps; during a step its index (k_weights)
    int32_t status;    // DevStatus
    uint32_t R_cur;    // current population size
    uint32_t R_prev;   // size that the last resampling started from
    double sum_lnQ;    // running sum of ln Q_k
    uint32_t lmin;     // lowest occupied energy level of the last resampling
    uint32_t K;        // number of levels spanned
    uint64_t T;        // sum of fixed-point weights f_j
    uint64_t Tres;     // sum of their fractional parts (residual rule)
    uint64_t Rres;     // residual draws
    int32_t kgrid;     // learned schedule: grid index of the current beta
    uint32_t sweeps;   // learned schedule: sweeps spent so far
    int32_t resample;  // partial resampling: this step resamples
    int32_t wexp;      // partial resampling: exponent of the largest new weight
    double S_new;      // sum of the level weights (partial resampling: of the new weights)
    double S_inv;      // 1 / S_new
    double S_old;      // sum of the weights before the step (the population size, mostly)
    uint32_t epoch;    // resampling steps taken (tags the look-back descriptors)
    int32_t hlo, hhi;  // lowest / highest histogram level filled since the last reweighting
};

// Look-back descriptor of one scan block (single-pass scans of the resampling step): the
// block's aggregates, then its inclusive prefixes in their place.  A 64-bit value is two words
// of 32 bits under a 32-bit tag of the step's epoch (2e+1: aggregate, 2e+2: inclusive prefix),
// so one load gives a value and says what it is, without fences.
struct alignas(32) LBDesc {
    unsigned long long w[4];
};

// Per-step accumulators, device-resident (row i = after temperature step i).
struct TraceRow {
    double lnQ;
    double sum_lnQ;
    double c_ln_c;   // sum_k c_k ln c_k over families
    double sv_sum;   // sum_j (r_j - f_j 2^-40)^2 over parents
    unsigned long long sumE, sumE2, sumAbsM, sumM2, sumC2, accepts;  // two's complement
    uint32_t R_i, R_prev;
    float x[8];       // learned schedule: features seen by the controller after this step
    int32_t u_next;   // its choice: grid units of the next step (0 = none)
    uint32_t theta_next;  // and the sweeps of the next step
    // partial resampling: effective size of the reweighted population, whether
    // the step resampled, and the weighted sums sum_j w_j O_j after the sweeps
    double ess;
    int32_t resampled, pad;
    double wsum, wE, wE2, wAM, wM2;
};

// Per-run description, in device memory (one per run of the batch).
struct RunDesc {
    int L, N, W, Wp;         // lattice; W words per replica, Wp padded to 4
    int nlev;                // d*N/2 + 1 histogram levels (level = U >> 1)
    int parity;              // U mod 2, the same for every configuration
    uint32_t R, Rcap;
    uint32_t magicL, shiftL; // fast division by L
    int nblk;                // scan blocks of this run
    uint32_t blk0;           // its first block in the flattened scan grids
    uint32_t grp0;           // its first CTA in the flattened sweep grid (= slot_base / 32)
    uint32_t run;            // run index
    uint32_t cta0;           // column walk: its first CTA in the launch for its side
    double lnR;              // ln max(R, 2), from the host's log (the controller's entropy scale)
    uint32_t* spins[2];
    int32_t* E[2];
    uint32_t* fam[2];
    int32_t* M;
    uint32_t* anc;
    uint32_t* counts;
    uint64_t* C;             // inclusive prefix of f
    uint64_t* G;             // inclusive prefix of the remainders (residual rule)
    uint32_t* hist;          // level histogram of the current population
    uint64_t* flev;          // fixed-point tau-hat per level
    double* tree;            // pairwise-sum scratch (power of two >= nlev)
    double* partD;           // per-block partial sums
    double* partCL;
    double* w;               // partial resampling: replica weights
    double* wpart;           // per-block tree sums of the weights (4 per block)
    double* opart;           // per-block tree sums of the weighted observables (5 per block)
    const uint8_t* jbits;    // bit a of byte s: bond (s, s+e_a) has J = -1
    DevState* st;
    TraceRow* trace;         // n_steps + 1 rows
    // the run's step tables (beta_i, dbeta_i, q_i, thresholds, theta_i): the batch's
    // shared tables, or the run's own under the learned schedule
    double* sbeta;
    double* sdbeta;
    double* sq;
    uint32_t* sthr;
    uint32_t* stheta;
    LBDesc* lb1;             // look-back descriptors: prefix of the expected copies
    LBDesc* lb2;             // and of the copy numbers
    uint32_t* tick;          // tickets of the scan blocks [0], family blocks [1], k_wsums blocks [2]
};

// Geometry of a launch of the column-walk sweep kernel (one side L).
struct WalkPlan {
    int L;
    int NC;           // columns of a group
    int H;            // rows of a column
    int S;            // words from row to row
    int CS, GS;       // words of a colour's array, of a group
    int GP, CPT;      // groups side by side, sets of them per CTA
    int NT;           // threads
    int span;         // rows walked before the second pass (fewer than H: the list's room)
    uint32_t mL, sL;  // division by L
    int flat;         // > 0: a side of pa_sweep3d.cu, GP groups per CTA; -1: k_group takes the side
};

// The group (index within the CTA) whose block keys are entry q of a builder that has gpw
// groups from `first` on in each of the plan's sets, or -1 for an entry past the set's last
// group: the next set's first groups may belong to another warp, which no barrier orders.
__host__ __device__ inline int walk_key_group(const WalkPlan& g, int gpw, int first, int q) {
    const int c = q / gpw;
    const int u = first + q - c * gpw;
    return u < g.GP ? c * g.GP + u : -1;
}

// Batch-wide parameters, passed by value to every kernel.
struct KParams {
    int d, ea, method, n_steps, M;
    int maxN;                // largest lattice of the batch
    uint32_t k0, k1;         // Philox key = seed
    uint32_t rk0[10], rk1[10];  // its round keys k + r*W (round r = 0..9)
    uint32_t nblk_total;     // flattened scan grid
    uint32_t ngrp_total;     // flattened sweep grid
    const RunDesc* runs;
    const uint32_t* blk2run; // scan block -> run
    const uint32_t* grp2run; // sweep CTA -> run
    const double* beta;      // n_steps + 1
    const double* dbeta;     // n_steps
    const double* q;         // exp(-4 dbeta), n_steps
    const uint32_t* thr;     // 4 per step (index 1..d used)
    const uint32_t* theta;   // n_steps
    const CtlDev* ctl;       // null without a controller
    double alpha;            // partial resampling threshold (< 0: resample every step)
    int qcap_limit;          // sweep: cap on the undecided-site queue (< 0: its full size)
    int lb_hold;             // test: scan block 0 withholds its prefix (the waits run out)
    const double* clnc;      // c ln c for c = 0 .. CLN_TAB (0 for c < 2), from the host's log
    int L_all;               // the side L shared by every run of the batch (0 if they differ)
    // sweeps by side: one launch per distinct side (nw = 0: the 2D kernel or, without its plan,
    // the general kernel)
    int nw;
    int g3mul;                 // 3D: sets of groups per CTA, the side's count times this (1 or 2)
    WalkPlan wplan[4];
    int G2, TG2;               // 2D kernel (nw = 0): groups per CTA (0: the general kernel),
                               // threads of each
    int pop;                   // k_pop: CTAs per run (0: the general kernels),
    int pop_threads, pop_levels;  // their threads, entries of their level arrays
    const uint32_t* wmap[4];   // CTA -> run of each launch
    uint32_t wcta[4];
};

// partial resampling: blocks of a run whose tree sums one CTA can finish
constexpr int PARTIAL_MAX_BLOCKS = 16384;
static_assert(PARTIAL_MAX_BLOCKS % 1024 == 0, "leaves per thread of the final trees");

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 2;
constexpr int SCAN_CHUNK = SCAN_THREADS * SCAN_ITEMS;

}  // namespace pa

// Chained launches.  A kernel launched by launch_chained() may be placed on the SMs while
// the kernel before it still runs; it calls chain_wait() before it touches memory that an
// earlier kernel writes or reads, which returns when that kernel has ended.  A kernel calls
// chain_next() where the one after it may be placed: all its own CTAs are on the SMs by
// then, so those waiting take no place from them.  Without that call the next kernel is
// placed when this one ends.  Every CTA of a chained kernel waits before it ends, so the
// end of a kernel is the end of all before it.  Only launches whose predecessor is always a
// kernel of this library are chained, and a sweep only where it finds its places beside k_pop
// (chain_sweep(); chain = false is an ordinary launch).  What it saves is the gap between two launches: the
// sweep after k_pop, 2D L = 16, R = 1000 41.9 -> 40.9 us a step, +-J L = 48, R = 20001 217.6
// -> 212.5; the three sides of a 3D batch 1093 -> 1075; pa_weights_static, 10^5 energies
// 14.4 -> 12.3; the training gradients and their sum, 12040 rows, with Adam 30.6 -> 28.7.
namespace pa {
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_chained(bool chain, void (*kernel)(P...), unsigned grid, unsigned block,
                           size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// kernel launchers (defined in the .cu files)
cudaError_t launch_init_spins(const KParams& p, const RunDesc* host_runs, cudaStream_t s);
cudaError_t launch_measure(const KParams& p, int threads, cudaStream_t s);
cudaError_t launch_resample(const KParams& p, cudaStream_t s, int64_t* launches);
int pop_ctas(uint32_t most_R, int most_levels, int M, int method, int* threads,
             int* levels);
bool pop_fits(const KParams& p);
cudaError_t launch_pop(const KParams& p, cudaStream_t s);
inline bool pop_takes(const KParams& p) { return p.pop && !p.lb_hold; }
cudaError_t launch_weighted_sums(const KParams& p, int mode, cudaStream_t s, int64_t* launches);
cudaError_t launch_partial_init(const KParams& p, cudaStream_t s);
cudaError_t launch_sweep(const KParams& p, int threads, cudaStream_t s);
cudaError_t launch_family_finish(const KParams& p, int mode, cudaStream_t s, int64_t* launches);
cudaError_t prepare_sweep(const KParams& p, int threads);
cudaError_t launch_sweep2d(const KParams& p, cudaStream_t s, bool attr_only, bool chain, bool* done);
double sweep_time(int rows, uint32_t ngrp, int GP, int tg, int regs, int CPT, size_t smem,
                  double alone);
int sweep3d_groups(int L, int gm);
cudaError_t launch_sweep3d(const KParams& p, int L, int G, const uint32_t* cta2run, uint32_t ncta,
                           cudaStream_t s, bool attr_only);
int sweep2d_threads(int L, int threads, uint32_t ngrp);
double group_time(int d, int N, bool ea, uint32_t ngrp, int threads);
WalkPlan walk_plan(int d, int L, bool ea, uint32_t ngrp, uint32_t most_grp, int threads, int general, int gm);
cudaError_t launch_walk(const KParams& p, const WalkPlan& g, const uint32_t* cta2run, uint32_t ncta,
                        cudaStream_t s, bool attr_only, bool chain);
cudaError_t launch_control(const KParams& p, cudaStream_t s);
int sweep_threads(int N);
bool sweep_threads_supported(int t);
}  // namespace pa
