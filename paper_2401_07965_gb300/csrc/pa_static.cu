// pa_static.cu -- pa_weights_static: the reweighting of one temperature step
// (energy-level histogram, Boltzmann weights, Q and the fixed-point expected
// copy numbers) for callers that cannot allocate device memory.
//
// Its scratch (the level histogram, the per-level weights and the pairwise-sum
// tree) lives in one file-scope __device__ array, so the call allocates
// nothing.  The arithmetic is the one of the context path's weights kernel,
// operation for operation, so both give the same bits.
#include <algorithm>
#include <cmath>

#include "../../include/pa.h"
#include "pa_internal.cuh"

namespace {

constexpr int STATIC_MAX_LEVELS = 65536;  // d*N/2 + 1 <= 65536 energy levels
constexpr int STATIC_THREADS = 512;

// zero at load time and between calls, except flev, tree and the call's results
struct StaticScratch {
    uint32_t hist[STATIC_MAX_LEVELS];
    uint64_t flev[STATIC_MAX_LEVELS];
    double tree[STATIC_MAX_LEVELS];
    int32_t bad;       // an energy lies outside the lattice's range
    int32_t lo_c, hi;  // STATIC_MAX_LEVELS - lowest level, highest level + 1
    uint32_t tick;     // CTAs that have added their counts
    int32_t lmin, ok;  // results: lowest level; whether the weights are valid
};

// One copy per device that loads the library (about 1.3 MB), kept until exit.
static __device__ __align__(256) StaticScratch g_scratch;

// q^k as the product of the squares q^(2^m) of k's set bits, least significant first
__device__ __forceinline__ double pow_sq(const double* qsq, uint32_t k) {
    double r = 1.0;
    for (int m = 0; k; ++m, k >>= 1)
        if (k & 1u) r = __dmul_rn(r, qsq[m]);
    return r;
}

constexpr int STATIC_SMEM_TREE = 2048;  // tree entries that fit the smallest shared array
constexpr int STATIC_SMEM_MIN = STATIC_SMEM_TREE * 8;
constexpr int STATIC_SMEM_MAX = (3 * 32768 / 2 + 1) * 4;  // the counts of the most levels (3D, N = 32768)

// Level counts over all CTAs; the last CTA to finish (a ticket) turns them into S, ln Q
// and the fixed-point weights of the levels and leaves the counts at zero.  With one CTA
// for the whole population 10^5 energies took 83 us; the counts are bound by the read of
// E, the last CTA by latency (the FP64 tree and the logarithms, about 5 us).
__global__ void __launch_bounds__(STATIC_THREADS)
k_static_weights(StaticScratch* sc, const int32_t* __restrict__ E, uint32_t R_prev, uint32_t R,
                 int d, int N, int parity, double dbeta, double q, double* lnQ_out,
                 uint64_t* f_out) {
    extern __shared__ __align__(16) uint32_t sh[];  // counts of the nlev levels; then the tree
    __shared__ double qsq[32], S_sh, rS_sh, lnS_sh, lnR_sh;
    __shared__ int s_lo, s_hi, s_bad, s_last;
    const int nlev = d * N / 2 + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pa::chain_next();
    for (int l = threadIdx.x; l < nlev; l += STATIC_THREADS) sh[l] = 0u;
    if (threadIdx.x == 0) {
        s_lo = nlev;
        s_hi = -1;
        s_bad = 0;
    }
    __syncthreads();
    int lo = nlev, hi = -1, bad = 0;
    for (uint64_t j = (uint64_t)blockIdx.x * STATIC_THREADS + threadIdx.x; j < R_prev;
         j += gridDim.x * STATIC_THREADS) {
        // 2U = E + dN (U unsatisfied bonds) in 64 bits: no overflow for any int32 E.
        // A valid energy has 0 <= U <= dN and U = parity (mod 2).
        const long long twoU = (long long)E[j] + (long long)d * N;
        if (twoU < 0 || twoU > 2LL * d * N || (twoU & 1) || (((twoU >> 1) & 1) != parity)) {
            bad = 1;
            continue;
        }
        const int l = (int)(twoU >> 2);
        lo = min(lo, l);
        hi = max(hi, l);
        atomicAdd(&sh[l], 1u);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
        if (hi >= 0) {
            atomicMin(&s_lo, lo);
            atomicMax(&s_hi, hi);
        }
        if (bad) atomicOr(&s_bad, 1);
    }
    __syncthreads();
    for (int l = s_lo + threadIdx.x; l <= s_hi; l += STATIC_THREADS)
        if (sh[l]) atomicAdd(&sc->hist[l], sh[l]);
    if (threadIdx.x == 0) {
        if (s_hi >= 0) {
            atomicMax(&sc->lo_c, STATIC_MAX_LEVELS - s_lo);
            atomicMax(&sc->hi, s_hi + 1);
        }
        if (s_bad) atomicOr(&sc->bad, 1);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&sc->tick, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int lmin = STATIC_MAX_LEVELS - *(volatile int32_t*)&sc->lo_c;
    const int K = *(volatile int32_t*)&sc->hi - lmin;
    const bool valid = *(volatile int32_t*)&sc->hi > 0 && *(volatile int32_t*)&sc->bad == 0;
    volatile uint32_t* hist = sc->hist;
    __syncthreads();
    if (threadIdx.x == 0) {
        sc->tick = 0u;
        sc->lo_c = sc->hi = 0;
        sc->bad = 0;
        sc->lmin = lmin;
        sc->ok = valid;
        if (!valid) *lnQ_out = NAN;  // no valid energy, or an invalid one: no weights
        double b = q;
        const int nb = K > 1 ? 32 - __clz(K - 1) : 0;
        for (int m = 0; m < nb; ++m) {
            qsq[m] = b;
            b = __dmul_rn(b, b);
        }
    }
    __syncthreads();
    if (!valid) {
        for (int l = threadIdx.x; l < nlev; l += STATIC_THREADS) sc->hist[l] = 0u;
        return;
    }
    int P = 1;
    while (P < K) P <<= 1;
    // S = sum_k n_k w_k as the fixed pairwise tree (t_k += t_{k+h}, h = P/2 ... 1)
    const bool tree_sh = P <= STATIC_SMEM_TREE;
    double* ts = reinterpret_cast<double*>(sh);
    volatile double* tg = sc->tree;
    for (int k = threadIdx.x; k < P; k += STATIC_THREADS) {
        const double v = k < K ? __dmul_rn((double)hist[lmin + k], pow_sq(qsq, (uint32_t)k)) : 0.0;
        if (tree_sh) ts[k] = v;
        else tg[k] = v;
    }
    __threadfence_block();
    __syncthreads();
    int h = P >> 1;
    for (; h >= 32; h >>= 1) {
        for (int k = threadIdx.x; k < h; k += STATIC_THREADS) {
            if (tree_sh) ts[k] = __dadd_rn(ts[k], ts[k + h]);
            else tg[k] = __dadd_rn(tg[k], tg[k + h]);
        }
        __threadfence_block();
        __syncthreads();
    }
    if (warp == 0) {  // the last levels by shuffles, the same pairs
        const int live = h > 0 ? 2 * h : 1;
        double v = 0.0;
        if (lane < live) v = tree_sh ? ts[lane] : tg[lane];
        for (; h >= 1; h >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, h));
        if (lane == 0) {
            S_sh = v;
            rS_sh = __ddiv_rn(1.0, v);
        }
    }
    __syncthreads();
    const double S = S_sh;
    if (warp == STATIC_THREADS / 32 - 1) {  // the two logarithms beside the divisions
        const double lx = log(lane == 0 ? S : (double)R_prev);
        if (lane == 0) lnS_sh = lx;
        if (lane == 1) lnR_sh = lx;
    }
    const double Rd = (double)R, rS = rS_sh;
    for (int k = threadIdx.x; k < K; k += STATIC_THREADS) {
        sc->flev[k] = pa::fixed_quotient(__dmul_rn(Rd, pow_sq(qsq, (uint32_t)k)), S, rS);
    }
    __threadfence_block();
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += STATIC_THREADS) sc->hist[lmin + k] = 0u;
    if (f_out)  // one CTA holds the whole population: f at once
        for (uint32_t j = threadIdx.x; j < R_prev; j += STATIC_THREADS)
            f_out[j] = ((volatile uint64_t*)sc->flev)[((E[j] + d * N) >> 2) - lmin];
    if (threadIdx.x == 0) {
        const int32_t Umin = 2 * lmin + parity;
        const int32_t Emin = 2 * Umin - d * N;
        *lnQ_out = __dsub_rn(__dsub_rn(lnS_sh, lnR_sh), __dmul_rn(dbeta, (double)Emin));
    }
}

// f_j of every replica from the level table (a launch of its own: every CTA needs it)
__global__ void __launch_bounds__(256)
k_static_f(const StaticScratch* sc, const int32_t* E, uint32_t R_prev, int dN, uint64_t* f_out) {
    uint64_t j = (uint64_t)blockIdx.x * 256u + threadIdx.x;
    int32_t Ej = j < R_prev ? E[j] : 0;  // not written by the kernel before
    pa::chain_wait();
    if (!sc->ok) return;
    const int lmin = sc->lmin;
    while (j < R_prev) {
        const uint64_t next = j + gridDim.x * 256u;
        const int32_t En = next < R_prev ? E[next] : 0;
        f_out[j] = sc->flev[((Ej + dN) >> 2) - lmin];
        j = next;
        Ej = En;
    }
}

}  // namespace

extern "C" pa_status pa_weights_static(const int32_t* E, uint32_t R_prev, uint32_t R, int32_t dim,
                                       int32_t L, int32_t parity, double dbeta, double* lnQ,
                                       uint64_t* f, void* cuda_stream) {
    if (!E || !lnQ || !f || R_prev == 0 || R == 0 || (parity & ~1)) return PA_ERR_ARG;
    if (dim < 2 || dim > 3 || L < 2 || (L & 1)) return PA_ERR_ARG;
    if (!(dbeta > 0.0) || !std::isfinite(dbeta)) return PA_ERR_ARG;
    long long N = 1;
    for (int a = 0; a < dim && N <= 32768; ++a) N *= L;
    if (N > 32768 || dim * N / 2 + 1 > STATIC_MAX_LEVELS) return PA_ERR_LIMIT;
    if (R > pa::MAX_POPULATION) return PA_ERR_LIMIT;  // 2^40 R must fit in 64 bits
    // The array's device address, looked up with the caller's device current on
    // every call: a cached pointer would outlive a reset of the device's context
    // (the module, and the array with it, is then loaded again elsewhere).  The
    // lookup is a host-side table query; only the first one on a device loads the
    // module.
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) return PA_ERR_CUDA;
    StaticScratch* sc = (StaticScratch*)ptr;
    const double q = std::exp(-(4.0 * dbeta));
    const cudaStream_t st = (cudaStream_t)cuda_stream;
    // four energies per thread, at most one CTA per SM
    const uint32_t per = 4 * STATIC_THREADS;
    const unsigned na = (unsigned)std::min<uint64_t>(((uint64_t)R_prev + per - 1) / per, 152u);
    const int sm = std::max(STATIC_SMEM_MIN, (int)(dim * N / 2 + 1) * 4);  // at most 197 KB
    // (always the largest limit: another thread's call must not lower it before this launch)
    if (sm > 48 * 1024 - 512 &&
        cudaFuncSetAttribute(k_static_weights, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             STATIC_SMEM_MAX) != cudaSuccess)
        return PA_ERR_CUDA;
    k_static_weights<<<na, STATIC_THREADS, sm, st>>>(sc, E, R_prev, R, dim, (int)N, parity, dbeta, q,
                                                     lnQ, na == 1 ? f : nullptr);
    if (na == 1) return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
    const unsigned nf = (unsigned)std::min<uint64_t>(((uint64_t)R_prev + 1023u) / 1024u, 152u * 8u);
    return pa::launch_chained(true, k_static_f, nf, 256u, 0, st, sc, E, R_prev, dim * (int)N, f) == cudaSuccess
               ? PA_OK
               : PA_ERR_CUDA;
}
