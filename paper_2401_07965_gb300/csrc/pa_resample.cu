// pa_resample.cu -- reweighting, Q and copy counts (Sec. 2 step 2, Sec. 3),
// the scan-plus-scatter that builds the ancestor array of the new population,
// and the family / sampling-variance measurements (Eqs. rho_t, sv).
//
// All floating-point work uses explicitly rounded IEEE double operations
// (no fused multiply-add) in a fixed order, so that the fixed-point weights
// and therefore every count are reproducible bit for bit:
//   level l = U >> 1 of a replica (U unsatisfied bonds), E = 2U - dN,
//   w_k = q^k (q = exp(-4 dbeta), binary powering), k = l - l_min,
//   S = fixed pairwise tree sum of n_k w_k over a power-of-two array,
//   ln Q = (ln S - ln R_{i-1}) - dbeta E_min,
//   f_k = floor(2^40 * ((R w_k) / S))  (tau-hat of Eq. taus in 2^-40 units).
// The copy counts are exact integer functions of f and of Philox draws.  Small populations
// take one kernel for all of it (pa_pop.cu); the kernels here take the others.
//
// Partial resampling (alpha >= 0): replicas carry weights w_j.  The step
// multiplies them by the level factors q^(l_j - l_min) (k_pw_update), sums
// old and new weights and the squares in balanced binary trees over the
// replica index (blocks of SCAN_CHUNK aligned replicas, then the blocks:
// k_pw_final), and resamples with f_j = floor(2^40 (R wn_j) / S_new) only if
// (sum wn)^2 / sum wn^2 < alpha R_{i-1}; otherwise every replica is kept once
// and its weight is rescaled by a power of two (k_wsums).  The f_j and their total come
// from k_fsum, the rest from the kernels of the plain step (its look-back scans replaced
// six kernels: 2D L = 64, R = 10^4, 200 steps 52.9 -> 40.4 ms).
#include <climits>

#include "pa_counts.cuh"

namespace pa {

// balanced binary tree sums (adjacent pairs first) in explicitly rounded FP64:
// over 8 or 16 consecutive values, and over the threads of a CTA (thread t =
// leaf t, blockDim a power of two); the root ends in every thread
template <int NL>
__device__ __forceinline__ double tree_regs(const double* a) {
    double t[NL];
#pragma unroll
    for (int k = 0; k < NL; ++k) t[k] = a[k];
#pragma unroll
    for (int w = 1; w < NL; w <<= 1)
#pragma unroll
        for (int k = 0; k + w < NL; k += 2 * w) t[k] = __dadd_rn(t[k], t[k + w]);
    return t[0];
}

// the same tree over the threads of a CTA for NV values at once (sh: NV x 33 doubles), of
// which the first `leaves` threads hold any but zeros (the other warps skip their adds: an
// FP64 operation occupies this part's pipe for 16 cycles per warp); the roots end in every
// thread
template <int NV>
__device__ __forceinline__ void tree_threads(double (&v)[NV], double* sh, int leaves = 1024) {
    // levels inside a warp by shuffles (lane t adds lane t + w for t a multiple
    // of 2w: the same pairs as the tree), then the same over the warps' sums
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (warp * 32 < leaves)
#pragma unroll
        for (int w = 1; w < 32; w <<= 1)
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = __dadd_rn(v[q], __shfl_down_sync(0xffffffffu, v[q], w));
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sh[33 * q + warp] = v[q];
    __syncthreads();
    if (warp < NV) {  // warp q finishes value q
        double u = lane < nw ? sh[33 * warp + lane] : 0.0;
        for (int w = 1; w < nw && w * 32 < leaves; w <<= 1)
            u = __dadd_rn(u, __shfl_down_sync(0xffffffffu, u, w));
        if (lane == 0) sh[33 * warp + 32] = u;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = sh[33 * q + 32];
    __syncthreads();
}

// largest of the first n threads' values (non-negative), in every thread
__device__ __forceinline__ double max_threads(double v, double* sh, int n = 1024) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = min((int)blockDim.x >> 5, (n + 31) / 32);
    if (warp < nw) {  // the bit patterns of non-negative doubles are ordered like the values
        unsigned long long u = (unsigned long long)__double_as_longlong(v);
        for (int w = 16; w >= 1; w >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, u, w);
            u = o > u ? o : u;
        }
        if (lane == 0) sh[warp] = __longlong_as_double((long long)u);
    }
    __syncthreads();
    unsigned long long u = 0ull;
    for (int k = 0; k < nw; ++k) {
        const unsigned long long o = (unsigned long long)__double_as_longlong(sh[k]);
        u = o > u ? o : u;
    }
    __syncthreads();
    return __longlong_as_double((long long)u);
}

// --------------------------------------------------------------------------
// K3: weights, S, ln Q, f table (one CTA)
//
// One CTA of 1024 threads; its time is latency, not work, so the phases are
// kept few: the level counts are read from global memory once, and the logarithms of
// ln Q are left to the kernel that closes the step (finish_run).
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_weights(KParams p) {
    const RunDesc& r = p.runs[blockIdx.x];
    DevState* st = r.st;
    if (st->status != S_OK) return;
    constexpr int TREE_SMEM = 2048;
    // tree and weights; before the tree is built, the counts of the K occupied
    // levels (cached when they fit in its 4 TREE_SMEM words)
    __shared__ double tw[2 * TREE_SMEM];
    double* tsm = tw;
    double* wsm = tw + TREE_SMEM;
    uint32_t* hc = reinterpret_cast<uint32_t*>(tw);
    __shared__ double qsq[32], S_sh, rS_sh;
    const int i = st->step + 1;
    const uint32_t Rprev = st->R_cur;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the occupied level range, recorded by the kernels that filled the histogram
    // (the lowest and highest level any replica took)
    const int lo = st->hlo, hi = st->hhi;
    const int lmin = lo;
    const int K = hi >= lo ? hi - lo + 1 : 0;
    const bool cached = K <= 4 * TREE_SMEM;
    if (cached)
        for (int k = threadIdx.x; k < K; k += blockDim.x) hc[k] = r.hist[lmin + k];
    __syncthreads();
    int P = 1;
    while (P < K) P <<= 1;
    const double q = r.sq[i - 1];
    // the squares q^(2^m) for the bits of k < K
    if (threadIdx.x == 0) {
        const int nb = K > 1 ? 32 - __clz(K - 1) : 0;
        double b = q;
        for (int m = 0; m < nb; ++m) {
            qsq[m] = b;
            b = __dmul_rn(b, b);
        }
    }
    const bool in_smem = P <= TREE_SMEM;
    // the counts of the thread's levels k = threadIdx.x + j blockDim.x, j < 2 (all
    // of them when the tree is in shared memory)
    uint32_t n0 = 0u, n1 = 0u;
    if (in_smem) {
        const int k0 = threadIdx.x, k1 = threadIdx.x + blockDim.x;
        if (k0 < K) n0 = cached ? hc[k0] : r.hist[lmin + k0];
        if (k1 < K) n1 = cached ? hc[k1] : r.hist[lmin + k1];
    }
    __syncthreads();  // qsq written; the count cache is free for the tree
    if (p.alpha >= 0.0) {
        // partial resampling: the level factors q^k; k_pw_final closes the step
        double* wl = reinterpret_cast<double*>(r.flev);
        for (int k = threadIdx.x; k < K; k += blockDim.x) wl[k] = pow_tab(qsq, (uint32_t)k);
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += blockDim.x) r.hist[lmin + k] = 0u;
        if (threadIdx.x == 0) {
            st->step = i;  // the step's other kernels read its index here
            st->R_prev = Rprev;
            st->lmin = (uint32_t)lmin;
            st->K = (uint32_t)K;
            st->hlo = 0x7FFFFFFF;  // the histogram is empty again
            st->hhi = -1;
            TraceRow* tr = r.trace + i;
            tr->c_ln_c = 0.0;
            tr->sv_sum = 0.0;
            tr->sumE = tr->sumE2 = tr->sumAbsM = tr->sumM2 = tr->sumC2 = tr->accepts = 0ull;
            tr->R_prev = Rprev;
            tr->R_i = 0;
        }
        return;
    }
    // S = sum_k n_k w_k as the fixed pairwise tree (t_k += t_{k+h}, h = P/2 ... 1) over
    // the zero-padded array: in shared memory when it fits (the usual case: the
    // occupied levels span a few hundred), else in the run's global scratch; the
    // last five levels by warp shuffles with the same pairs
    int h = P >> 1;
    if (in_smem) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int k = threadIdx.x + j * blockDim.x;
            if (k < P) {
                double v = 0.0;
                if (k < K) {
                    const double wk = pow_tab(qsq, (uint32_t)k);
                    wsm[k] = wk;
                    v = __dmul_rn((double)(j == 0 ? n0 : n1), wk);
                }
                tsm[k] = v;
            }
        }
        __syncthreads();
        for (; h >= 32; h >>= 1) {
            for (int k = threadIdx.x; k < h; k += blockDim.x)
                tsm[k] = __dadd_rn(tsm[k], tsm[k + h]);
            __syncthreads();
        }
    } else {
        volatile double* t = r.tree;
        for (int k = threadIdx.x; k < P; k += blockDim.x)
            t[k] = k < K ? __dmul_rn((double)r.hist[lmin + k], pow_tab(qsq, (uint32_t)k)) : 0.0;
        __threadfence_block();
        __syncthreads();
        for (; h >= 32; h >>= 1) {
            for (int k = threadIdx.x; k < h; k += blockDim.x) t[k] = __dadd_rn(t[k], t[k + h]);
            __threadfence_block();
            __syncthreads();
        }
    }
    if (warp == 0) {
        const int live = h > 0 ? 2 * h : 1;  // entries left after the shared-memory levels
        const volatile double* t = in_smem ? tsm : r.tree;
        double v = lane < live ? t[lane] : 0.0;
        for (; h >= 1; h >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, h));
        if (lane == 0) {
            S_sh = v;
            rS_sh = __ddiv_rn(1.0, v);
        }
    }
    __syncthreads();
    const double S = S_sh;
    const double Rd = (double)r.R, rS = rS_sh;
    // f_k, and the totals T = sum_j f_j = sum_k n_k f_k and of the fractional parts
    // (exact integer sums; the copy-count kernels need them before any scan)
    unsigned long long sT = 0, sTr = 0;
    for (int k = threadIdx.x, j = 0; k < K; k += blockDim.x, ++j) {
        const uint64_t f = fixed_quotient(__dmul_rn(Rd, in_smem ? wsm[k] : pow_tab(qsq, (uint32_t)k)), S, rS);
        r.flev[k] = f;
        const uint64_t n = in_smem ? (j == 0 ? n0 : n1) : r.hist[lmin + k];
        sT += n * f;
        sTr += n * (f & ((1ull << FRAC_BITS) - 1));
    }
    for (int o = 16; o > 0; o >>= 1) {
        sT += __shfl_xor_sync(0xffffffffu, sT, o);
        sTr += __shfl_xor_sync(0xffffffffu, sTr, o);
    }
    __shared__ unsigned long long tsum[2];
    if (threadIdx.x == 0) tsum[0] = tsum[1] = 0ull;
    __syncthreads();
    if (lane == 0) {
        atomicAdd(&tsum[0], sT);
        atomicAdd(&tsum[1], sTr);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) r.hist[lmin + k] = 0u;
    if (threadIdx.x == 0) {
        st->step = i;  // the step's other kernels read its index here
        st->T = tsum[0];
        st->Tres = tsum[1];
        st->Rres = (uint64_t)r.R - ((tsum[0] - tsum[1]) >> FRAC_BITS);
        st->epoch += 1u;
        st->S_new = S;
        st->S_old = (double)Rprev;
        st->R_prev = Rprev;
        st->lmin = (uint32_t)lmin;
        st->K = (uint32_t)K;
        st->hlo = 0x7FFFFFFF;  // the histogram is empty again
        st->hhi = -1;
        TraceRow* tr = r.trace + i;
        tr->c_ln_c = 0.0;
        tr->sv_sum = 0.0;
        tr->sumE = tr->sumE2 = tr->sumAbsM = tr->sumM2 = tr->sumC2 = tr->accepts = 0ull;
        tr->R_prev = Rprev;
        tr->R_i = 0;
    }
}

// --------------------------------------------------------------------------
// partial resampling: new weights and their per-block tree sums
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(SCAN_THREADS) k_pw_update(KParams p) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    const uint32_t b = blockIdx.x - r.blk0;
    const DevState* st = r.st;
    if (st->status != S_OK) return;
    __shared__ double sh[3 * 33];
    const int i = st->step;
    const int32_t* E = r.E[(i - 1) & 1];
    const uint32_t Rprev = st->R_prev, lmin = st->lmin;
    const int dN = p.d * r.N;
    const double* wl = reinterpret_cast<const double*>(r.flev);
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    double wo[SCAN_ITEMS], wn[SCAN_ITEMS], w2[SCAN_ITEMS];
    double mx = 0.0;
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const int j = j0 + e;
        wo[e] = wn[e] = w2[e] = 0.0;
        if ((uint32_t)j < Rprev) {
            wo[e] = r.w[j];
            wn[e] = __dmul_rn(wo[e], wl[level_of(E[j], dN) - (int)lmin]);
            w2[e] = __dmul_rn(wn[e], wn[e]);
            r.w[j] = wn[e];
            mx = fmax(mx, wn[e]);
        }
    }
    double v[3] = {tree_regs<SCAN_ITEMS>(wo), tree_regs<SCAN_ITEMS>(wn), tree_regs<SCAN_ITEMS>(w2)};
    tree_threads(v, sh);
    mx = max_threads(mx, sh);
    if (threadIdx.x == 0) {
        r.wpart[4 * b + 0] = v[0];
        r.wpart[4 * b + 1] = v[1];
        r.wpart[4 * b + 2] = v[2];
        r.wpart[4 * b + 3] = mx;
    }
}

// One CTA per run: tree over the blocks, ln Q, effective size, decision.  Up to 1024
// blocks a thread holds one leaf (the tree over PARTIAL_MAX_BLOCKS leaves is the same: the
// others are zeros) and warps past the last leaf skip their FP64 adds: 29 -> 7.9 us at
// R = 10^4 (16 leaves in every thread, whatever the population, and one sum after the
// other).
__global__ void __launch_bounds__(1024) k_pw_final(KParams p) {
    const RunDesc& r = p.runs[blockIdx.x];
    DevState* st = r.st;
    if (st->status != S_OK) return;
    __shared__ double sh[3 * 33];
    const int i = st->step;
    const int nb = r.nblk;  // <= PARTIAL_MAX_BLOCKS = LEAVES leaves x 1024 threads
    constexpr int LEAVES = PARTIAL_MAX_BLOCKS / 1024;
    double S[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (nb <= 1024) {
            S[q] = (int)threadIdx.x < nb ? r.wpart[4 * threadIdx.x + q] : 0.0;
        } else {
            double x[LEAVES];
#pragma unroll
            for (int k = 0; k < LEAVES; ++k) {
                const int bb = LEAVES * threadIdx.x + k;
                x[k] = bb < nb ? r.wpart[4 * bb + q] : 0.0;
            }
            S[q] = tree_regs<LEAVES>(x);
        }
    }
    double mx = 0.0;
    for (int bb = threadIdx.x; bb < nb; bb += blockDim.x) mx = fmax(mx, r.wpart[4 * bb + 3]);
    tree_threads(S, sh, nb <= 1024 ? nb : 1024);
    mx = max_threads(mx, sh, nb);
    if (threadIdx.x == 0) {
        const uint32_t Rprev = st->R_prev;
        const double ess = __ddiv_rn(__dmul_rn(S[1], S[1]), S[2]);
        const int res = ess < __dmul_rn(p.alpha, (double)Rprev) ? 1 : 0;
        int e = 0;
        frexp(mx, &e);
        st->resample = res;
        st->wexp = e;
        st->S_old = S[0];
        st->S_new = S[1];
        st->S_inv = __ddiv_rn(1.0, S[1]);
        st->T = st->Tres = 0ull;  // summed by k_fsum
        st->epoch += 1u;
        TraceRow* tr = r.trace + i;
        tr->ess = ess;
        tr->resampled = res;
    }
}

// weights of a new run: 1
__global__ void k_pw_init(KParams p) {
    const RunDesc& r = p.runs[blockIdx.y];
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < r.Rcap; j += gridDim.x * blockDim.x)
        r.w[j] = 1.0;
}

// --------------------------------------------------------------------------
// partial resampling, a step that resamples: the expected copies of the replicas (kept
// in C until the prefix takes its place) and their total, which the copy-count kernels
// need before any scan; the run's last block to finish sets the residual draws
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(SCAN_THREADS) k_fsum(KParams p) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    const uint32_t b = blockIdx.x - r.blk0;
    DevState* st = r.st;
    if (st->status != S_OK || !st->resample) return;  // the population is kept
    __shared__ unsigned long long tot[2];
    const uint32_t Rprev = st->R_prev;
    const double S = st->S_new, rS = st->S_inv;
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    unsigned long long sf = 0, sg = 0;
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const int j = j0 + e;
        if ((uint32_t)j < Rprev) {
            const uint64_t f = fixed_quotient(__dmul_rn((double)r.R, r.w[j]), S, rS);
            r.C[j] = f;
            sf += f;
            sg += f & ((1ull << FRAC_BITS) - 1);
        }
    }
    if (threadIdx.x == 0) tot[0] = tot[1] = 0ull;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) {
        sf += __shfl_xor_sync(0xffffffffu, sf, o);
        sg += __shfl_xor_sync(0xffffffffu, sg, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&tot[0], sf);
        atomicAdd(&tot[1], sg);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd((unsigned long long*)&st->T, tot[0]);
        atomicAdd((unsigned long long*)&st->Tres, tot[1]);
        __threadfence();
        if (atomicAdd(&r.tick[0], 1u) == (uint32_t)r.nblk - 1u) {
            __threadfence();
            const uint64_t T = *(volatile uint64_t*)&st->T, G = *(volatile uint64_t*)&st->Tres;
            st->Rres = (uint64_t)r.R - ((T - G) >> FRAC_BITS);
            r.tick[0] = 0u;
        }
    }
}

// multinomial draws (multinomial rule: R draws over C; residual rule: R_res
// draws over the remainders G, or over C if every remainder is zero)
__global__ void __launch_bounds__(SCAN_THREADS) k_draws(KParams p) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    const uint32_t b = blockIdx.x - r.blk0;
    const DevState* st = r.st;
    if (st->status != S_OK) return;
    if (p.alpha >= 0.0 && !st->resample) return;  // partial: no resampling this step
    const int i = st->step;
    const uint32_t Rprev = st->R_prev;
    uint64_t n;
    const uint64_t* box;
    uint64_t total;
    uint32_t rule;
    if (p.method == M_MULTINOMIAL) {
        n = r.R;
        box = r.C;
        total = st->T;
        rule = RULE_MULTINOMIAL;
    } else {
        n = st->Rres;
        const bool use_g = st->Tres > 0;
        box = use_g ? r.G : r.C;
        total = use_g ? st->Tres : st->T;
        rule = RULE_RESIDUAL;
    }
    const uint64_t stride = (uint64_t)r.nblk * SCAN_THREADS;
    for (uint64_t k = (uint64_t)b * SCAN_THREADS + threadIdx.x; k < n; k += stride) {
        const uint4x x = draw_block(p, r, i, k, rule);
        const uint64_t u = (k & 1) ? (((uint64_t)x.w << 32) | x.z) : (((uint64_t)x.y << 32) | x.x);
        const uint64_t pos = __umul64hi(u, total);
        uint32_t lo = 0, hi = Rprev;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (pos < box[mid]) hi = mid;
            else lo = mid + 1;
        }
        atomicAdd(&r.counts[lo], 1u);
    }
}

// --------------------------------------------------------------------------
// family statistics of the new population (families stay sorted by slot)
// --------------------------------------------------------------------------
__device__ void finish_run(const KParams& p, const RunDesc& r, DevState* st, int mode, double* a,
                           double* b);

// Everything here is known once the ancestors are, so the kernel runs beside the step's
// sweep (a branch of the captured step).
__global__ void __launch_bounds__(SCAN_THREADS) k_family(KParams p, int mode) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    const uint32_t b = blockIdx.x - r.blk0;
    DevState* st = r.st;
    if (st->status != S_OK) return;
    __shared__ double sd[SCAN_THREADS], fa[SCAN_THREADS], fb[SCAN_THREADS];
    __shared__ unsigned long long sc2;
    __shared__ int last;
    const int i = st->step;
    const uint32_t Ri = st->R_cur;
    const uint32_t* fam = r.fam[i & 1];
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    // Families stay sorted by slot, so a family is a run of equal values.  The
    // block's slots go to shared memory; each run start finds its end from the
    // 32-slot masks of run starts, and warp 0 searches the array beyond the block
    // for the end of the block's last run, which may go on past it.  c ln c of
    // small families comes from a table the host computes once.
    constexpr int FTAB = CLN_TAB;
    __shared__ uint32_t sf[SCAN_CHUNK];
    __shared__ uint32_t smask[SCAN_CHUNK / 32];
    __shared__ double clt[FTAB + 1];
    const uint32_t B0 = b * SCAN_CHUNK;
    const uint32_t nin = B0 < Ri ? min((uint32_t)SCAN_CHUNK, Ri - B0) : 0u;
    if (threadIdx.x == 0) sc2 = 0ull;
    for (int c = threadIdx.x; c <= FTAB; c += blockDim.x) clt[c] = p.clnc[c];
    for (int l = threadIdx.x; l < SCAN_CHUNK; l += blockDim.x)
        sf[l] = (uint32_t)l < nin ? fam[B0 + l] : 0xFFFFFFFFu;
    __syncthreads();
    const uint32_t before = (B0 > 0 && nin) ? fam[B0 - 1] : 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int rnd = 0; rnd < SCAN_CHUNK / SCAN_THREADS; ++rnd) {
        const int l = rnd * SCAN_THREADS + warp * 32 + lane;
        const bool st_l = (uint32_t)l < nin && (l == 0 ? (B0 == 0 || before != sf[0])
                                                       : sf[l - 1] != sf[l]);
        const uint32_t m = __ballot_sync(0xffffffffu, st_l);
        if (lane == 0) smask[rnd * (SCAN_THREADS / 32) + warp] = m;
    }
    __syncthreads();
    double cl = 0.0;
    unsigned long long c2 = 0;
    __shared__ int slast;  // the block's last run start (-1: no slot in the block)
    if (threadIdx.x == 0) slast = -1;
    __syncthreads();
    for (int rnd = 0; rnd < SCAN_CHUNK / SCAN_THREADS; ++rnd) {
        const int l = rnd * SCAN_THREADS + warp * 32 + lane;
        int q = l >> 5;
        const int bit = l & 31;
        if (!((smask[q] >> bit) & 1u)) continue;  // not a run start (or past R_i)
        uint32_t m = bit == 31 ? 0u : (smask[q] & (0xFFFFFFFFu << (bit + 1)));
        while (m == 0u && q + 1 < SCAN_CHUNK / 32) m = smask[++q];
        if (!m) {  // the block's last run: it may continue past the block (below)
            slast = l;
            continue;
        }
        const uint64_t c = (uint64_t)(q * 32 + __ffs(m) - 1 - l);
        c2 += c * c;
        if (c > 1) cl = __dadd_rn(cl, c <= FTAB ? clt[c] : __dmul_rn((double)c, log((double)c)));
    }
    __syncthreads();
    // The last run ends at the first slot from B0 + nin on whose family differs
    // (families are sorted, so "differs" holds from there on): warp 0 finds it by
    // a 32-way search, each round sampling 32 evenly spaced slots of the interval
    // that holds the end (at most five rounds below 2^24 slots).
    if (warp == 0 && slast >= 0) {
        const uint32_t f = sf[slast];
        uint32_t lo = B0 + nin, hi = Ri;  // the end lies in [lo, hi]
        while (hi - lo > 32u) {
            const uint32_t step = (hi - lo + 31u) / 32u;
            const uint32_t pos = lo + (uint32_t)lane * step;
            const bool ne = pos >= hi || fam[pos] != f;
            const uint32_t bal = __ballot_sync(0xffffffffu, ne);
            const int k = bal ? __ffs(bal) - 1 : 32;
            if (k == 0) {
                hi = lo;
                break;
            }
            const uint32_t nlo = lo + (uint32_t)(k - 1) * step + 1u;
            if (k < 32) hi = min(hi, lo + (uint32_t)k * step);
            lo = nlo;
        }
        if (lo < hi) {
            const uint32_t pos = lo + (uint32_t)lane;
            const bool ne = pos >= hi || fam[pos] != f;
            const uint32_t bal = __ballot_sync(0xffffffffu, ne);
            lo = bal ? min(hi, lo + (uint32_t)(__ffs(bal) - 1)) : hi;
        }
        if (lane == 0) {
            const uint64_t c = (uint64_t)(lo - (B0 + (uint32_t)slast));
            c2 += c * c;
            if (c > 1) cl = __dadd_rn(cl, c <= FTAB ? clt[c] : __dmul_rn((double)c, log((double)c)));
        }
    }
    for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    if ((threadIdx.x & 31) == 0 && c2) atomicAdd(&sc2, c2);
    sd[threadIdx.x] = cl;
    __syncthreads();
    for (int h = SCAN_THREADS / 2; h >= 1; h >>= 1) {
        if ((int)threadIdx.x < h) sd[threadIdx.x] = __dadd_rn(sd[threadIdx.x], sd[threadIdx.x + h]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        r.partCL[b] = sd[0];
        if (sc2) atomicAdd(&r.trace[i].sumC2, sc2);
    }
    // the run's last family block to finish closes the step: its ticket says every
    // other block's partials are written (each fenced them before its ticket)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(&r.tick[1], 1u) == (uint32_t)r.nblk - 1u);
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) r.tick[1] = 0u;
    __threadfence();
    finish_run(p, r, st, mode, fa, fb);
}

// fixed-order sums of the run's per-block partials and ln Q (its logarithms cost 2000 cycles
// each on this part: here they run beside the sweep), close the step (one CTA of
// SCAN_THREADS threads; a, b: shared arrays of SCAN_THREADS doubles)
__device__ void finish_run(const KParams& p, const RunDesc& r, DevState* st, int mode, double* a,
                           double* b) {
    const int i = st->step;
    __shared__ double lg[2];
    if (mode == 0 && threadIdx.x >= SCAN_THREADS - 32) {  // beside the sums
        const int lane = threadIdx.x & 31;
        const double lx = log(lane == 0 ? st->S_new : st->S_old);
        if (lane < 2) lg[lane] = lx;
    }
    const int nb_sv = (mode == 0) ? (int)((st->R_prev + SCAN_CHUNK - 1) / SCAN_CHUNK) : 0;
    const int nb_f = (int)((st->R_cur + SCAN_CHUNK - 1) / SCAN_CHUNK);
    double sa = 0.0, sb = 0.0;
    for (int k = threadIdx.x; k < nb_sv; k += blockDim.x) sa = __dadd_rn(sa, __ldcg(&r.partD[k]));
    for (int k = threadIdx.x; k < nb_f; k += blockDim.x) sb = __dadd_rn(sb, __ldcg(&r.partCL[k]));
    a[threadIdx.x] = sa;
    b[threadIdx.x] = sb;
    __syncthreads();
    for (int h = 128; h >= 1; h >>= 1) {
        if ((int)threadIdx.x < h) {
            a[threadIdx.x] = __dadd_rn(a[threadIdx.x], a[threadIdx.x + h]);
            b[threadIdx.x] = __dadd_rn(b[threadIdx.x], b[threadIdx.x + h]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        TraceRow* tr = r.trace + i;
        if (mode == 0) {
            const int32_t Umin = 2 * (int32_t)st->lmin + r.parity;
            const int32_t Emin = 2 * Umin - p.d * r.N;
            const double lnQ = __dsub_rn(__dsub_rn(lg[0], lg[1]),
                                         __dmul_rn(r.sdbeta[i - 1], (double)Emin));
            const double sum = __dadd_rn(st->sum_lnQ, lnQ);
            st->sum_lnQ = sum;
            tr->lnQ = lnQ;
            tr->sum_lnQ = sum;
        }
        tr->sv_sum = a[0];
        tr->c_ln_c = b[0];
        tr->R_i = st->R_cur;
        if (mode != 0) tr->R_prev = st->R_cur;
    }
}

// Partial resampling, after the sweep: the new population's weighted sums of 1, E, E^2, |M|
// and M^2.  rescale: the weights are still those of the old population (k_pop leaves the new
// ones).  What bounds it: the FP64 pipe (some 55 operations a thread of the CTA's SM).
__global__ void __launch_bounds__(SCAN_THREADS) k_wsums(KParams p, int rescale) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    const uint32_t b = blockIdx.x - r.blk0;
    DevState* st = r.st;
    if (st->status != S_OK) return;
    __shared__ double sd[5 * 33];
    __shared__ int last;
    const int i = st->step;
    const uint32_t Ri = st->R_cur;
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    // the weights are 1 after a resampling, else the kept ones rescaled by 2^-wexp
    const int32_t* Ec = r.E[i & 1];
    double v[5][SCAN_ITEMS];
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const uint32_t d = (uint32_t)(j0 + e);
        double w = 0.0, E = 0.0, M = 0.0;
        if (d < Ri) {
            w = r.w[d];
            if (rescale) {
                w = st->resample ? 1.0 : scalbn(w, -st->wexp);
                r.w[d] = w;
            }
            E = (double)Ec[d];
            M = (double)r.M[d];
        }
        v[0][e] = w;
        v[1][e] = __dmul_rn(w, E);
        v[2][e] = __dmul_rn(w, __dmul_rn(E, E));
        v[3][e] = __dmul_rn(w, fabs(M));
        v[4][e] = __dmul_rn(w, __dmul_rn(M, M));
    }
    double t5[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) t5[q] = tree_regs<SCAN_ITEMS>(v[q]);
    tree_threads(t5, sd);
    if (threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < 5; ++q) r.opart[5 * b + q] = t5[q];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(&r.tick[2], 1u) == (uint32_t)r.nblk - 1u);
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) r.tick[2] = 0u;
    __threadfence();
    // the run's last block: tree over the blocks' sums (PARTIAL_MAX_BLOCKS leaves in all, zero
    // past the run's blocks)
    const int nb = r.nblk;
    constexpr int LEAVES = PARTIAL_MAX_BLOCKS / 256;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        if (nb <= 256) {  // a leaf per thread; the leaves past it are zeros
            t5[q] = (int)threadIdx.x < nb ? __ldcg(&r.opart[5 * threadIdx.x + q]) : 0.0;
        } else {  // the thread's LEAVES leaves as a tree, in eighths
            double x8[8];
            for (int h = 0; h < 8; ++h) {
                double x[LEAVES / 8];
#pragma unroll
                for (int k = 0; k < LEAVES / 8; ++k) {
                    const int bb = LEAVES * threadIdx.x + LEAVES / 8 * h + k;
                    x[k] = bb < nb ? __ldcg(&r.opart[5 * bb + q]) : 0.0;
                }
                x8[h] = tree_regs<LEAVES / 8>(x);
            }
            t5[q] = tree_regs<8>(x8);
        }
    }
    tree_threads(t5, sd, nb <= 256 ? nb : 256);
    if (threadIdx.x == 0) {
        TraceRow* tr = r.trace + i;
        double* dst[5] = {&tr->wsum, &tr->wE, &tr->wE2, &tr->wAM, &tr->wM2};
#pragma unroll
        for (int q = 0; q < 5; ++q) *dst[q] = t5[q];
    }
}

// --------------------------------------------------------------------------
// Single-pass scans (look-back).  A scan block takes a ticket for its logical
// index b within its run, computes its block sums, publishes them, and obtains
// the sum over blocks 0..b-1 from its predecessors' descriptors: the nearest
// inclusive prefix plus the aggregates after it.  Blocks only wait on blocks
// with earlier tickets, which are already running, so the waits end; each wait
// is bounded all the same (a run that exceeds it reports PA_ERR_TIMEOUT).
// --------------------------------------------------------------------------
constexpr uint32_t LB_SPIN_LIMIT = 1u << 22;

// a value of a descriptor: its words are written and read one by one, each with its tag
__device__ __forceinline__ void put_tagged(unsigned long long* w, unsigned long long v, uint32_t tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(w), "l"(t | (v & 0xFFFFFFFFull)),
                 "l"(t | (v >> 32))
                 : "memory");
}
__device__ __forceinline__ bool get_tagged(const unsigned long long* w, unsigned long long& v,
                                           uint32_t& tag) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(w) : "memory");
    v = (x & 0xFFFFFFFFull) | (y << 32);
    tag = (uint32_t)(x >> 32);
    return tag == (uint32_t)(y >> 32);
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Called by the whole block.  Publishes the NV values a of block b and returns in pre their
// sums over blocks 0..b-1 (every thread); false if a wait gave up.  A thread waits for one
// predecessor, SCAN_THREADS of them in one round.  publish = false (a test of the bounded
// waits) leaves block b's descriptor unset.  One warp looking back over 32 flags at a time,
// with a fence and a second load for the value, took 8 to 10 k cycles of a block; with two of
// them per block k_resample took 93 us for 24 runs of R = 50000 (systematic), now 54, and the
// residual rule at R = 1024000 103 us in its two scans, now 74.
template <int NV>
__device__ bool look_back(LBDesc* d, int b, const unsigned long long (&a)[NV], uint32_t ep,
                          unsigned long long (&pre)[NV], bool publish = true) {
    constexpr int NW = SCAN_THREADS / 32;
    __shared__ unsigned long long part[NV][NW];
    __shared__ int first[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t FA = 2u * ep + 1u, FI = 2u * ep + 2u;
    if (threadIdx.x < NV && publish) put_tagged(&d[b].w[2 * threadIdx.x], a[threadIdx.x & (NV - 1)], b == 0 ? FI : FA);
#pragma unroll
    for (int q = 0; q < NV; ++q) pre[q] = 0ull;
    for (int j0 = b - 1; j0 >= 0; j0 -= SCAN_THREADS) {
        const int j = j0 - (int)threadIdx.x;
        uint32_t f = FI;  // before block 0: nothing
        unsigned long long v[NV] = {};
        bool ok = true;
        if (j >= 0) {
            uint32_t spins = 0;
            while (true) {
                bool got = get_tagged(&d[j].w[0], v[0], f) && (f == FA || f == FI);
                if (NV == 2) {
                    uint32_t f1;
                    got = get_tagged(&d[j].w[2], v[NV - 1], f1) && f1 == f && got;
                }
                if (got) break;
                if (++spins > LB_SPIN_LIMIT) {
                    ok = false;
                    break;
                }
                __nanosleep(32);
            }
        }
        const uint32_t incl = __ballot_sync(0xffffffffu, f == FI);
        if (lane == 0) first[warp] = incl ? warp * 32 + __ffs(incl) - 1 : SCAN_THREADS;
        if (!__syncthreads_and(ok)) return false;
        int k = SCAN_THREADS;  // the nearest block with its inclusive prefix
#pragma unroll
        for (int w = 0; w < NW; ++w) k = min(k, first[w]);
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const unsigned long long u = warp_sum_u64((int)threadIdx.x <= k ? v[q] : 0ull);
            if (lane == 0) part[q][warp] = u;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q)
#pragma unroll
            for (int w = 0; w < NW; ++w) pre[q] += part[q][w];
        if (k < SCAN_THREADS) break;
        __syncthreads();
    }
    if (threadIdx.x < NV && b > 0 && publish) {
        const int q = threadIdx.x & (NV - 1);
        put_tagged(&d[b].w[2 * q], pre[q] + a[q], FI);
    }
    __syncthreads();  // the shared arrays are free again
    return true;
}

// the block's ticket: its logical index within the run
__device__ __forceinline__ int take_ticket(uint32_t* tick, int* sb) {
    if (threadIdx.x == 0) *sb = (int)atomicAdd(tick, 1u);
    __syncthreads();
    return *sb;
}

// The ancestor scatter of a block whose slots are [pre, pre + tot), ex of them before the
// thread's, and its sampling-variance partial; the last block sets the new population size
// (or the capacity error) and resets the tickets.
__device__ __forceinline__ void scatter(const KParams& p, const RunDesc& r, DevState* st, int b,
                                        const uint32_t (&rc)[SCAN_ITEMS], uint64_t ex, uint64_t pre,
                                        uint64_t tot, double* sd, const uint64_t (&fv)[SCAN_ITEMS],
                                        bool kmax = false) {
    const int i = st->step;
    const uint32_t Rprev = st->R_prev;
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    // The block's slots [pre, pre + tot): the total over blocks is known only to the last
    // block, so slots past the capacity are not written (the last block then stops the run
    // with the capacity error).
    const uint32_t* fam0 = r.fam[(i - 1) & 1];
    uint32_t* fam1 = r.fam[i & 1];
    const uint64_t room = pre < (uint64_t)r.Rcap ? (uint64_t)r.Rcap - pre : 0ull;
    const uint32_t nslot = (uint32_t)(tot < room ? tot : room);
    __shared__ uint32_t so[SCAN_CHUNK], sfam[SCAN_CHUNK];  // first slot and family of each parent
    uint32_t o = (uint32_t)(ex < 0xFFFFFFFFull ? ex : 0xFFFFFFFFull);
    double sv = 0.0;
    int skew = 0;
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const int j = j0 + e, l = threadIdx.x * SCAN_ITEMS + e;
        const bool in = (uint32_t)j < Rprev;
        so[l] = o;
        sfam[l] = in && rc[e] ? fam0[j] : 0u;
        o += rc[e];
        skew |= rc[e] > 4u;
        if (!in) continue;
        const double dl = count_excess(rc[e], fv[e]);
        sv = __dadd_rn(sv, __dmul_rn(dl, dl));
    }
    // Parents of at most four copies write their slots themselves; a block with a larger
    // one gives every slot a thread, which finds its parent in the offsets (a thread that
    // wrote hundreds of copies one by one held up its block and, by the look-back, the
    // run: +-J L = 4, 6, 8, R = 50000, beta step 0.15: 499 -> 89 us for 24 runs).
    if (!__syncthreads_or(skew)) {
#pragma unroll
        for (int e = 0; e < SCAN_ITEMS; ++e) {
            const int l = threadIdx.x * SCAN_ITEMS + e;
#pragma unroll
            for (uint32_t c = 0; c < 4u; ++c)
                if (c < rc[e] && so[l] + c < nslot) {
                    r.anc[pre + so[l] + c] = (uint32_t)(j0 + e);
                    fam1[pre + so[l] + c] = sfam[l];
                }
        }
    } else {
        for (uint32_t q = threadIdx.x; q < nslot; q += SCAN_THREADS) {
            int lo = 0;  // the last parent whose first slot is not after q
#pragma unroll
            for (int w = SCAN_CHUNK / 2; w >= 1; w >>= 1)
                if (so[lo + w] <= q) lo += w;
            r.anc[pre + q] = (uint32_t)(b * SCAN_CHUNK + lo);
            fam1[pre + q] = sfam[lo];
        }
    }
    // fixed-order tree reduction of the block's sampling-variance terms
    sd[threadIdx.x] = sv;
    __syncthreads();
    for (int h = SCAN_THREADS / 2; h >= 1; h >>= 1) {
        if ((int)threadIdx.x < h) sd[threadIdx.x] = __dadd_rn(sd[threadIdx.x], sd[threadIdx.x + h]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        r.partD[b] = __dmul_rn(sd[0], 0x1p-80);
        if (b == r.nblk - 1) {
            const uint64_t Ri = pre + tot;
            // a population that outgrows its capacity, or dies out, stops the run
            if (kmax) st->status = S_KMAX;
            else if (Ri > (uint64_t)r.Rcap || Ri == 0) st->status = S_CAPACITY;
            else st->R_cur = (uint32_t)Ri;
            r.tick[0] = 0u;
        }
    }
}

// Copy numbers' exclusive scan (look-back over lb2) and the scatter.
__device__ __forceinline__ void count_scan_scatter(const KParams& p, const RunDesc& r, DevState* st,
                                                   int b, const uint32_t (&rc)[SCAN_ITEMS],
                                                   uint64_t* sh, double* sd,
                                                   const uint64_t (&fv)[SCAN_ITEMS],
                                                   bool kmax = false, bool publish = true) {
    uint64_t sum = 0;
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) sum += rc[e];
    uint64_t tot;
    const uint64_t ex = block_excl_scan(sum, sh, &tot);
    // the second value counts the blocks with a Poisson inversion at its limit
    const unsigned long long own[2] = {tot, (unsigned long long)(__syncthreads_or(kmax) != 0)};
    unsigned long long pre[2];
    if (!look_back(r.lb2, b, own, st->epoch, pre, publish)) {
        if (threadIdx.x == 0) atomicCAS(&st->status, S_OK, S_TIMEOUT);
        return;
    }
    scatter(p, r, st, b, rc, ex, pre[0], tot, sd, fv, pre[1] + own[1] != 0);
}

// Expected copies f_j and the copy numbers of the rules that need no search.  A rule needs one
// look-back here (5 us of waiting each): PREFIX (multinomial, residual) stores the prefix C of
// the f_j (and G of their fractional parts) for k_draws, by lb1; SYSTEMATIC has the number of
// labels below C_j for first slots, by lb1; LOCAL (nearest, Poisson) needs no prefix of the
// f_j, and scans its counts by lb2.
enum { PREFIX, SYSTEMATIC, LOCAL };
template <int RULE>
__global__ void __launch_bounds__(SCAN_THREADS, 4) k_resample(KParams p) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    DevState* st = r.st;
    if (st->status != S_OK) return;
    if (p.alpha >= 0.0 && !st->resample) {
        // partial resampling keeps every replica once: identity counts, ancestors and
        // families, no sampling variance
        const int i = st->step;
        const uint32_t b = blockIdx.x - r.blk0, Rprev = st->R_prev;
        for (uint32_t j = b * SCAN_CHUNK + threadIdx.x; j < min(Rprev, (b + 1) * SCAN_CHUNK);
             j += SCAN_THREADS) {
            r.counts[j] = 1u;
            r.anc[j] = j;
            r.fam[i & 1][j] = r.fam[(i - 1) & 1][j];
        }
        if (threadIdx.x == 0) r.partD[b] = 0.0;
        return;
    }
    __shared__ uint64_t sh[33];
    __shared__ double sd[SCAN_THREADS];
    __shared__ int sb;
    const int b = take_ticket(&r.tick[0], &sb);
    const int i = st->step;
    const int32_t* E = r.E[(i - 1) & 1];
    const int dN = p.d * r.N;
    const uint32_t Rprev = st->R_prev, lmin = st->lmin;
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    uint64_t f[SCAN_ITEMS];
    uint64_t sf = 0, sg = 0;
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const int j = j0 + e;
        f[e] = 0ull;
        if ((uint32_t)j < Rprev) f[e] = p.alpha >= 0.0 ? r.C[j] : r.flev[level_of(E[j], dN) - (int)lmin];
        sf += f[e];
        sg += f[e] & ((1ull << FRAC_BITS) - 1);
    }
    const int method = p.method;
    uint32_t rc[SCAN_ITEMS];
    if constexpr (RULE == LOCAL) {
        bool kmax = false;
#pragma unroll 1
        for (int e = 0; e < SCAN_ITEMS; ++e) {
            const uint32_t j = (uint32_t)(j0 + e);
            rc[e] = 0u;
            if (j >= Rprev) continue;
            rc[e] = method == M_NEAREST ? nearest_count(p, r, i, j, f[e])
                                        : poisson_count(p, r, i, j, f[e], kmax);
            r.counts[j] = rc[e];
        }
        count_scan_scatter(p, r, st, b, rc, sh, sd, f, kmax, !(p.lb_hold && b == 0));
        return;
    }
    const uint64_t T = st->T;
    uint64_t tf, tg = 0ull, eg = 0ull;
    const uint64_t ef = block_excl_scan(sf, sh, &tf);
    if (RULE == PREFIX) eg = block_excl_scan(sg, sh, &tg);
    constexpr int NV = RULE == PREFIX ? 2 : 1;
    unsigned long long own[NV], pr[NV];
    own[0] = tf;
    if (NV == 2) own[NV - 1] = tg;
    if (!look_back(r.lb1, b, own, st->epoch, pr, !(p.lb_hold && b == 0))) {
        if (threadIdx.x == 0) atomicCAS(&st->status, S_OK, S_TIMEOUT);
        return;
    }
    uint64_t cf = pr[0] + ef, cg = pr[NV - 1] + eg;
    if constexpr (RULE == PREFIX) {
#pragma unroll
        for (int e = 0; e < SCAN_ITEMS; ++e) {
            const int j = j0 + e;
            if ((uint32_t)j >= Rprev) continue;
            cf += f[e];
            cg += f[e] & ((1ull << FRAC_BITS) - 1);
            r.C[j] = cf;
            if (method == M_RESIDUAL) r.G[j] = cg;
            r.counts[j] = method == M_RESIDUAL ? (uint32_t)(f[e] >> FRAC_BITS) : 0u;
        }
        if (threadIdx.x == 0 && b == r.nblk - 1) r.tick[0] = 0u;
    } else {
        // labels below the running boundary, carried from item to item: the first slots
        const uint32_t usys = systematic_offset(p, r, i);
        const uint64_t first = sys_below(cf, r.R, T, usys);
        uint64_t below = first;
#pragma unroll 1
        for (int e = 0; e < SCAN_ITEMS; ++e) {
            const int j = j0 + e;
            rc[e] = 0u;
            if ((uint32_t)j >= Rprev) continue;
            cf += f[e];
            const uint64_t bn = sys_below(cf, r.R, T, usys);
            rc[e] = (uint32_t)(bn - below);
            below = bn;
            r.counts[j] = rc[e];
        }
        if (threadIdx.x == 0) sh[0] = first;
        if (threadIdx.x == SCAN_THREADS - 1) sh[1] = below;
        __syncthreads();
        const uint64_t pre = sh[0];
        scatter(p, r, st, b, rc, first - pre, pre, sh[1] - pre, sd, f);
    }
}

// multinomial / residual: the copy numbers are complete after k_draws
__global__ void __launch_bounds__(SCAN_THREADS) k_cscan(KParams p) {
    const RunDesc& r = p.runs[p.blk2run[blockIdx.x]];
    DevState* st = r.st;
    if (st->status != S_OK || (p.alpha >= 0.0 && !st->resample)) return;
    __shared__ uint64_t sh[33];
    __shared__ double sd[SCAN_THREADS];
    __shared__ int sb;
    const int b = take_ticket(&r.tick[0], &sb);
    const uint32_t Rprev = st->R_prev;
    const int j0 = b * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    uint32_t rc[SCAN_ITEMS];
    uint64_t f[SCAN_ITEMS];  // from the prefix C
#pragma unroll
    for (int e = 0; e < SCAN_ITEMS; ++e) {
        const int j = j0 + e;
        const bool in = (uint32_t)j < Rprev;
        rc[e] = in ? r.counts[j] : 0u;
        f[e] = in ? r.C[j] - (j > 0 ? r.C[j - 1] : 0ull) : 0ull;
    }
    count_scan_scatter(p, r, st, b, rc, sh, sd, f);
}

// --------------------------------------------------------------------------
cudaError_t launch_resample(const KParams& p, cudaStream_t s, int64_t* launches) {
    if (pop_takes(p)) {
        if (launches) *launches += 1;
        return launch_pop(p, s);
    }
    k_weights<<<p.M, 1024, 0, s>>>(p);
    int n = 1;
    if (p.alpha >= 0.0) {
        // partial resampling: the expected copies depend on per-replica weights, so
        // their total comes from a sum over the replicas
        k_pw_update<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        k_pw_final<<<p.M, 1024, 0, s>>>(p);
        k_fsum<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        n += 3;
    }
    if (p.method == M_MULTINOMIAL || p.method == M_RESIDUAL) {
        k_resample<PREFIX><<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        k_draws<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        k_cscan<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        n += 3;
    } else {
        if (p.method == M_SYSTEMATIC) k_resample<SYSTEMATIC><<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        else k_resample<LOCAL><<<p.nblk_total, SCAN_THREADS, 0, s>>>(p);
        n += 1;
    }
    if (launches) *launches += n;
    return cudaGetLastError();
}

cudaError_t launch_partial_init(const KParams& p, cudaStream_t s) {
    k_pw_init<<<dim3(64, (unsigned)p.M), 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_family_finish(const KParams& p, int mode, cudaStream_t s, int64_t* launches) {
    k_family<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p, mode);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_weighted_sums(const KParams& p, int mode, cudaStream_t s, int64_t* launches) {
    k_wsums<<<p.nblk_total, SCAN_THREADS, 0, s>>>(p, mode == 0 && !pop_takes(p));
    if (launches) *launches += 1;
    return cudaGetLastError();
}

}  // namespace pa
