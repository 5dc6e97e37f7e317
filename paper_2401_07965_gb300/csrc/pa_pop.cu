// pa_pop.cu -- the whole resampling of a small population in one launch: weights, (partial
// resampling: effective size and decision), copy numbers, ancestors and families
// (pa_resample.cu's kernels, same results bit for bit).
//
// A run is one thread-block cluster of 1 to 16 CTAs, each with POP_CHUNK replicas, two per
// thread.  Every CTA computes the level weights for itself; block totals, the multinomial
// searches and their counts go through the cluster's shared memory, so the look-backs, the
// prefix arrays and the launches between the phases are gone.
// What bounds it: latency, 14 to 20 thousand cycles (8 to 11 us) of short phases: a block scan
// with its cluster barrier 2 (one for the rules that need one prefix, three for the drawn
// ones), the level weights 5, the draws or the copy numbers 3 to 6, the scatter 2, the
// variance's tree 1.5.  Temperature steps with ten sweeps, the general kernels -> this one, both
// without chained launches: 2D L = 16, R = 1000, multinomial 57 -> 42 us; L = 64, R = 3000,
// systematic, with the learned schedule 60 -> 53; +-J L = 48, R = 20001, Poisson 231 -> 219;
// L = 64, R = 10^4, systematic, partial resampling 202 -> 185.
#include <cooperative_groups.h>

#include <algorithm>

#include "pa_counts.cuh"

namespace pa {

namespace cg = cooperative_groups;

constexpr int POP_CTAS = 16;
constexpr int POP_LEVELS = 8192;  // entries of the level arrays, at most
static_assert(SCAN_CHUNK == 2 * SCAN_THREADS && SCAN_THREADS == 256, "two adjacent replicas per thread");

// the run's state and trace row after its weights (threads t < n of one CTA)
__device__ __forceinline__ void close_step(const RunDesc& r, DevState* st, int i, uint32_t Rprev,
                                           int lmin, int K, double S, double S_old, int t, int n) {
    for (int k = t; k < K; k += n) r.hist[lmin + k] = 0u;
    if (t != n - 1) return;
    st->step = i;  // the step's other kernels read its index here
    st->epoch += 1u;
    st->S_new = S;
    st->S_old = S_old;
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

template <int POP_THREADS, bool PARTIAL>
__global__ void __launch_bounds__(POP_THREADS, 1) k_pop(KParams p) {
    constexpr int POP_CHUNK = 2 * POP_THREADS;  // replicas of a CTA
    cg::cluster_group cl = cg::this_cluster();
    const unsigned cs = cl.num_blocks(), rank = cl.block_rank();
    chain_next();  // the sweep's CTAs
    const auto sync = [&] {  // one CTA needs no cluster barrier (1000 cycles)
        if (cs == 1) __syncthreads();
        else cl.sync();
    };
    DevState* st = p.runs[blockIdx.x / cs].st;
    if (st->status != S_OK) return;  // written by this cluster alone, after its last barrier
    cl.barrier_arrive();  // waited for before the first access to another CTA's shared memory
    extern __shared__ __align__(16) unsigned char dyn[];
    double* ta = reinterpret_cast<double*>(dyn);  // level tree; later the variance terms
    double* tb = ta + p.pop_levels;               // level weights, then fixed-point weights
    __shared__ __align__(16) RunDesc r;           // the run's pointers, a load away
    __shared__ uint32_t cnt[POP_CHUNK], so[POP_CHUNK], sfam[POP_CHUNK];
    __shared__ uint64_t sh[33], xf[POP_CTAS], xg[POP_CTAS], xc[POP_CTAS];
    __shared__ double qsq[32], S_sh, rS_sh;
    __shared__ double pw[PARTIAL ? 3 : 1][33], xw[PARTIAL ? 3 : 1][POP_CTAS * 4];
    __shared__ unsigned long long pm[32], xm[POP_CTAS];
    __shared__ int wexp_sh;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    static_assert(sizeof(RunDesc) % 8 == 0 && sizeof(RunDesc) / 8 <= 256, "one word per thread");
    if (t < (int)(sizeof(RunDesc) / 8))
        reinterpret_cast<uint64_t*>(&r)[t] = reinterpret_cast<const uint64_t*>(p.runs + blockIdx.x / cs)[t];
    const int i = st->step + 1, method = p.method;
    const uint32_t Rprev = st->R_cur;
    const int lmin = st->hlo, hi = st->hhi;
    __syncthreads();
    const int dN = p.d * r.N;
    const int K = hi >= lmin ? hi - lmin + 1 : 0;
    const uint32_t j0 = rank * POP_CHUNK + 2 * t;
    const int32_t* E = r.E[(i - 1) & 1];
    const uint32_t* fam0 = r.fam[(i - 1) & 1];
    int32_t Ej[2];
    uint32_t fj[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const bool in = j0 + e < Rprev;
        Ej[e] = in ? E[j0 + e] : 0;
        fj[e] = in ? fam0[j0 + e] : 0u;
    }
    // ---- level weights: S = sum_k n_k w_k by the fixed pairwise tree, f_k (k_weights) ----
    if (t == 0) {
        const int nb = max(5, K > 1 ? 32 - __clz(K - 1) : 0);
        double b = r.sq[i - 1];
        for (int m = 0; m < nb; ++m) {
            qsq[m] = b;
            b = __dmul_rn(b, b);
        }
    }
    int P = 1;
    while (P < K) P <<= 1;
    const uint32_t n0 = !PARTIAL && t < K ? r.hist[lmin + t] : 0u;
    double wj[2];
    if (PARTIAL) {
#pragma unroll
        for (int e = 0; e < 2; ++e) wj[e] = j0 + e < Rprev ? r.w[j0 + e] : 0.0;
    }
    __syncthreads();
    double wlow = 1.0;  // the low five bits of k are the lane's: pow_tab's product so far
    if (warp * 32 < K) {
#pragma unroll
        for (int m = 0; m < 5; ++m)
            if ((lane >> m) & 1) wlow = __dmul_rn(wlow, qsq[m]);
    }
    for (int k = t; k < P; k += POP_THREADS) {
        double v = 0.0;
        if (k < K) {
            double w = wlow;
            for (uint32_t m = 5, hk = (uint32_t)k >> 5; hk; ++m, hk >>= 1)
                if (hk & 1u) w = __dmul_rn(w, qsq[m]);
            tb[k] = w;
            if (!PARTIAL) v = __dmul_rn((double)(k == t ? n0 : r.hist[lmin + k]), w);
        }
        if (!PARTIAL) ta[k] = v;
    }
    __syncthreads();
    double S, S_old = (double)Rprev;
    uint64_t f[2];
    if constexpr (PARTIAL) {
        // ---- new weights, their tree sums (blocks of SCAN_CHUNK, then the blocks: k_pw_update
        // and k_pw_final), effective size, decision ----
        double wn[2], v[3], mx;
        {
            double wo[2], w2[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool in = j0 + e < Rprev;
                wo[e] = in ? wj[e] : 0.0;
                wn[e] = in ? __dmul_rn(wo[e], tb[level_of(Ej[e], dN) - lmin]) : 0.0;
                w2[e] = __dmul_rn(wn[e], wn[e]);
            }
            v[0] = __dadd_rn(wo[0], wo[1]);
            v[1] = __dadd_rn(wn[0], wn[1]);
            v[2] = __dadd_rn(w2[0], w2[1]);
            mx = fmax(wn[0], wn[1]);
        }
#pragma unroll
        for (int w = 1; w < 32; w <<= 1) {
#pragma unroll
            for (int q = 0; q < 3; ++q) v[q] = __dadd_rn(v[q], __shfl_down_sync(0xffffffffu, v[q], w));
        }
        // the bit patterns of non-negative doubles are ordered like the values
        unsigned long long um = (unsigned long long)__double_as_longlong(mx);
        for (int w = 16; w >= 1; w >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, um, w);
            um = o > um ? o : um;
        }
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) pw[q][warp] = v[q];
            pm[warp] = um;
        }
        __syncthreads();
        cl.barrier_wait();
        constexpr int NW = POP_THREADS / 32, BW = SCAN_THREADS / 32;
        if (warp < 3) {  // the blocks' roots, to every CTA
            double u = lane < NW ? pw[warp][lane] : 0.0;
            for (int w = 1; w < BW; w <<= 1) u = __dadd_rn(u, __shfl_down_sync(0xffffffffu, u, w));
            if (lane < NW && lane % BW == 0)
                for (unsigned q = 0; q < cs; ++q)
                    cl.map_shared_rank(&xw[warp][0], q)[rank * (NW / BW) + lane / BW] = u;
        } else if (warp == 3) {
            unsigned long long u = lane < NW ? pm[lane] : 0ull;
            for (int w = 16; w >= 1; w >>= 1) {
                const unsigned long long o = __shfl_xor_sync(0xffffffffu, u, w);
                u = o > u ? o : u;
            }
            if (lane < (int)cs) cl.map_shared_rank(xm, lane)[rank] = u;
        }
        sync();
        if (warp < 3) {  // up to 64 blocks, the rest of the tree's leaves are zeros
            const int nb = (int)cs * (NW / BW);
            double u = __dadd_rn(2 * lane < nb ? xw[warp][2 * lane] : 0.0,
                                 2 * lane + 1 < nb ? xw[warp][2 * lane + 1] : 0.0);
            for (int w = 1; w < 32; w <<= 1) u = __dadd_rn(u, __shfl_down_sync(0xffffffffu, u, w));
            if (lane == 0) {
                pw[warp][0] = u;
                if (warp == 1) rS_sh = __ddiv_rn(1.0, u);
            }
        } else if (warp == 3) {
            unsigned long long u = lane < (int)cs ? xm[lane] : 0ull;
            for (int w = 16; w >= 1; w >>= 1) {
                const unsigned long long o = __shfl_xor_sync(0xffffffffu, u, w);
                u = o > u ? o : u;
            }
            int e = 0;
            frexp(__longlong_as_double((long long)u), &e);
            if (lane == 0) wexp_sh = e;
        }
        __syncthreads();
        S_old = pw[0][0];
        S = pw[1][0];
        const double ess = __ddiv_rn(__dmul_rn(S, S), pw[2][0]);
        const bool res = ess < __dmul_rn(p.alpha, (double)Rprev);
        if (rank == 0 && t == 0) {
            st->resample = res;
            st->wexp = wexp_sh;
            r.trace[i].ess = ess;
            r.trace[i].resampled = res;
        }
        if (!res) {  // every replica is kept once, with its weight rescaled by a power of two
            const int we = wexp_sh;
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (j0 + e < Rprev) {
                    r.w[j0 + e] = scalbn(wn[e], -we);
                    r.counts[j0 + e] = 1u;
                    r.anc[j0 + e] = j0 + e;
                    r.fam[i & 1][j0 + e] = fj[e];
                }
            const int b = (int)(rank * (POP_CHUNK / SCAN_CHUNK)) + t / SCAN_THREADS;
            if (t % SCAN_THREADS == 0 && b < r.nblk) r.partD[b] = 0.0;
            if (rank == 0) close_step(r, st, i, Rprev, lmin, K, S, S_old, t, POP_THREADS);
            return;
        }
        const double rS = rS_sh;
#pragma unroll
        for (int e = 0; e < 2; ++e)
            f[e] = j0 + e < Rprev ? fixed_quotient(__dmul_rn((double)r.R, wn[e]), S, rS) : 0ull;
    } else {
        int h = P >> 1;
        for (; h >= 32; h >>= 1) {
            for (int k = t; k < h; k += POP_THREADS) ta[k] = __dadd_rn(ta[k], ta[k + h]);
            __syncthreads();
        }
        if (warp == 0) {
            const int live = h > 0 ? 2 * h : 1;
            double v = lane < live ? ta[lane] : 0.0;
            for (; h >= 1; h >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, h));
            if (lane == 0) {
                S_sh = v;
                rS_sh = __ddiv_rn(1.0, v);
            }
        }
        __syncthreads();
        S = S_sh;
        const double Rd = (double)r.R, rS = rS_sh;
        uint64_t* fl = reinterpret_cast<uint64_t*>(tb);
        for (int k = t; k < K; k += POP_THREADS) fl[k] = fixed_quotient(__dmul_rn(Rd, tb[k]), S, rS);
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 2; ++e) f[e] = j0 + e < Rprev ? fl[level_of(Ej[e], dN) - lmin] : 0ull;
    }
    // ---- expected copies, their prefix and total over the cluster ----
    constexpr uint64_t FMASK = (1ull << FRAC_BITS) - 1;
    const bool local = method == M_NEAREST || method == M_POISSON;  // no prefix needed
    uint64_t tg = 0ull, ef = 0ull, eg = 0ull, T = 0ull, G = 0ull, pf = 0ull, pg = 0ull;
    if (!PARTIAL) cl.barrier_wait();
    if (!local) {
        uint64_t tf;
        ef = block_excl_scan(f[0] + f[1], sh, &tf);
        if (method == M_RESIDUAL) eg = block_excl_scan((f[0] & FMASK) + (f[1] & FMASK), sh, &tg);
        if (t < (int)cs) {
            cl.map_shared_rank(xf, t)[rank] = tf;
            cl.map_shared_rank(xg, t)[rank] = tg;
        }
        sync();
        for (unsigned q = 0; q < cs; ++q) {
            if (q == rank) {
                pf = T;
                pg = G;
            }
            T += xf[q];
            G += xg[q];
        }
    }
    // ---- copy numbers ----
    uint32_t rc[2] = {0u, 0u};
    bool kmax = false;
    uint64_t first = 0ull, below = 0ull;  // systematic: labels below the thread's replicas, through them
    if (method == M_MULTINOMIAL || method == M_RESIDUAL) {
        const bool residual = method == M_RESIDUAL, useg = residual && G > 0;
        // every CTA gets the whole population's prefix, over its level arrays (read by now):
        // a search in another CTA's memory takes 250 cycles a step
        uint64_t* box = reinterpret_cast<uint64_t*>(dyn);
        const uint32_t nbox = cs * POP_CHUNK, me = rank * POP_CHUNK + 2 * t;
        uint64_t c[2];
        c[0] = (useg ? pg + eg : pf + ef) + (useg ? f[0] & FMASK : f[0]);
        c[1] = c[0] + (useg ? f[1] & FMASK : f[1]);
        for (unsigned q = 0; q < cs; ++q) {
            uint64_t* bx = q == rank ? box : cl.map_shared_rank(box, q);
            *reinterpret_cast<ulonglong2*>(bx + me) = make_ulonglong2(c[0], c[1]);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) cnt[2 * t + e] = residual ? (uint32_t)(f[e] >> FRAC_BITS) : 0u;
        sync();
        const uint64_t n = residual ? (uint64_t)r.R - ((T - G) >> FRAC_BITS) : (uint64_t)r.R;
        const uint64_t total = useg ? G : T;
        const uint32_t rule = residual ? RULE_RESIDUAL : RULE_MULTINOMIAL;
        for (uint64_t k = 2 * (rank * POP_THREADS + t); k < n; k += 2 * cs * POP_THREADS) {
            // two draws of one Philox block; the first replica whose prefix exceeds each (the
            // prefix is flat past the last replica, and the draws lie below its end)
            const uint4x x = draw_block(p, r, i, k, rule);
            const uint64_t p0 = __umul64hi(((uint64_t)x.y << 32) | x.x, total);
            const uint64_t p1 = __umul64hi(((uint64_t)x.w << 32) | x.z, total);
            uint32_t l0 = 0, l1 = 0;
            for (uint32_t w = nbox / 2; w >= 1; w >>= 1) {
                if (box[l0 + w - 1] <= p0) l0 += w;
                if (box[l1 + w - 1] <= p1) l1 += w;
            }
            const unsigned q0 = l0 / POP_CHUNK, q1 = l1 / POP_CHUNK;
            atomicAdd((q0 == rank ? cnt : cl.map_shared_rank(cnt, q0)) + l0 % POP_CHUNK, 1u);
            if (k + 1 < n)
                atomicAdd((q1 == rank ? cnt : cl.map_shared_rank(cnt, q1)) + l1 % POP_CHUNK, 1u);
        }
        sync();
        rc[0] = cnt[2 * t];
        rc[1] = cnt[2 * t + 1];
    } else {
        uint32_t usys = 0u;
        uint64_t cf = pf + ef;
        if (method == M_SYSTEMATIC) {
            usys = systematic_offset(p, r, i);
            first = below = sys_below(cf, r.R, T, usys);
        }
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            const uint32_t j = j0 + e;
            if (j >= Rprev) continue;
            const uint64_t fe = e ? f[1] : f[0];
            uint32_t c;
            if (method == M_NEAREST) {
                c = nearest_count(p, r, i, j, fe);
            } else if (method == M_SYSTEMATIC) {
                cf += fe;
                const uint64_t bn = sys_below(cf, r.R, T, usys);
                c = (uint32_t)(bn - below);
                below = bn;
            } else {
                c = poisson_count(p, r, i, j, fe, kmax);
            }
            if (e) rc[1] = c;
            else rc[0] = c;
        }
    }
    // ---- first slot of every replica over the cluster ----
    uint64_t tot, ex, Ri = r.R, pre = 0ull;
    bool anyk = false;
    if (method == M_SYSTEMATIC) {  // the labels below its lower boundary
        if (t == 0) sh[0] = first;
        if (t == POP_THREADS - 1) sh[1] = below;
        __syncthreads();
        pre = sh[0];
        ex = first - pre;
        tot = sh[1] - pre;
    } else {
        ex = block_excl_scan((uint64_t)rc[0] + rc[1], sh, &tot);
        const int km = __syncthreads_or(kmax);
        if (t < (int)cs) cl.map_shared_rank(xc, t)[rank] = tot | (km ? 1ull << 63 : 0ull);
        sync();
        Ri = 0ull;
        for (unsigned q = 0; q < cs; ++q) {
            if (q == rank) pre = Ri;
            Ri += xc[q] & ~(1ull << 63);
            anyk |= (xc[q] >> 63) != 0;
        }
    }
    // ---- ancestors and families (slots past the capacity are not written), the variance ----
    uint32_t* fam1 = r.fam[i & 1];
    const uint64_t room = pre < (uint64_t)r.Rcap ? (uint64_t)r.Rcap - pre : 0ull;
    const uint32_t nslot = (uint32_t)(tot < room ? tot : room);
    uint32_t o = (uint32_t)(ex < 0xFFFFFFFFull ? ex : 0xFFFFFFFFull);
    double sv = 0.0;
    int skew = 0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        so[2 * t + e] = o;
        sfam[2 * t + e] = fj[e];
        o += rc[e];
        skew |= rc[e] > 4u;
        if (j0 + e >= Rprev) continue;
        r.counts[j0 + e] = rc[e];
        const double dl = count_excess(rc[e], f[e]);
        sv = __dadd_rn(sv, __dmul_rn(dl, dl));
    }
    ta[t] = sv;
    if (!__syncthreads_or(skew)) {  // as in k_resample: at most four copies each, or by slots
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (uint32_t c = 0; c < 4u; ++c) {
                const uint32_t q = so[2 * t + e] + c;
                if (c < rc[e] && q < nslot) {
                    r.anc[pre + q] = j0 + e;
                    fam1[pre + q] = fj[e];
                    if (PARTIAL) r.w[pre + q] = 1.0;
                }
            }
    } else {
        for (uint32_t q = t; q < nslot; q += POP_THREADS) {
            int lo = 0;
#pragma unroll
            for (int w = POP_CHUNK / 2; w >= 1; w >>= 1)
                if (so[lo + w] <= q) lo += w;
            r.anc[pre + q] = rank * POP_CHUNK + lo;
            fam1[pre + q] = sfam[lo];
            if (PARTIAL) r.w[pre + q] = 1.0;
        }
    }
    // the scan blocks' partials, each over its SCAN_THREADS threads in the same pairs
    const int u = t & (SCAN_THREADS - 1);
    for (int w = SCAN_THREADS / 2; w >= 32; w >>= 1) {
        if (u < w) ta[t] = __dadd_rn(ta[t], ta[t + w]);
        __syncthreads();
    }
    if (u < 32) {
        double v = ta[t];
        for (int w = 16; w >= 1; w >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, w));
        const int b = (int)(rank * (POP_CHUNK / SCAN_CHUNK)) + t / SCAN_THREADS;
        if (u == 0 && b < r.nblk) r.partD[b] = __dmul_rn(v, 0x1p-80);
    }
    // the run's state, which every CTA of the cluster has read; ln Q is left to the kernel
    // that closes the step
    if (rank == 0) {
        close_step(r, st, i, Rprev, lmin, K, S, S_old, t, POP_THREADS);
        if (t == POP_THREADS - 1) {
            // a population that outgrows its capacity, or dies out, stops the run
            if (anyk) st->status = S_KMAX;
            else if (Ri > (uint64_t)r.Rcap || Ri == 0) st->status = S_CAPACITY;
            else st->R_cur = (uint32_t)Ri;
        }
    }
}

// CTAs per run (a power of two), or 0 where the general kernels take the batch.  The fewest
// threads per CTA that hold the population in POP_CTAS CTAs: an SM's FP64 pipe and its
// shared-memory banks are what the phases share (2D L = 16 / 32, one sweep, us per step with
// 256, 512 and 1024 threads: multinomial R = 2000 29, 31, 33, R = 4000 31, 36, 41; systematic
// R = 4000 23, 25, 27, R = 8000 26, 27, 30).  General kernels for more than 32768 replicas,
// for the drawn rules beyond 512 threads (R = 30000: 61 general, 80 here; residual 59, 64;
// systematic 48, 44; Poisson 51, 47; nearest 47, 42), for more levels than shared memory
// holds and for more runs than fit at a time.
int pop_ctas(uint32_t most_R, int most_levels, int M, int method, int* threads, int* levels) {
    const int most = method == M_MULTINOMIAL || method == M_RESIDUAL ? 512 : 1024;
    int nt = 256, cs = 1;
    while (nt < most && (uint64_t)POP_CTAS * 2 * nt < most_R) nt <<= 1;
    while ((uint64_t)cs * 2 * nt < most_R) cs <<= 1;
    int P = 1024;
    while (P < most_levels) P <<= 1;
    if (most == 512) P = std::max(P, cs * nt);  // two words per level hold a prefix per replica
    *threads = nt;
    *levels = P;
    return cs <= POP_CTAS && P <= POP_LEVELS && (int64_t)M * cs <= 128 ? cs : 0;
}

// one launch, or (fits != nullptr) how many of its clusters the device holds at a time
template <int NT, bool PARTIAL>
static cudaError_t launch(const KParams& p, cudaStream_t s, int* fits) {
    // the limit is the kernel's, whoever launches it: always the largest, so that a context on
    // another thread never lowers it between this call and the launch
    cudaError_t e = cudaFuncSetAttribute(k_pop<NT, PARTIAL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         2 * (int)sizeof(double) * POP_LEVELS);
    if (e == cudaSuccess && p.pop > 8)
        e = cudaFuncSetAttribute(k_pop<NT, PARTIAL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)p.pop;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)(p.M * p.pop));
    c.blockDim = dim3(NT);
    c.dynamicSmemBytes = 2 * sizeof(double) * (size_t)p.pop_levels;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    if (fits) return cudaOccupancyMaxActiveClusters(fits, k_pop<NT, PARTIAL>, &c);
    return cudaLaunchKernelEx(&c, k_pop<NT, PARTIAL>, p);
}

template <bool PARTIAL>
static cudaError_t launch(const KParams& p, cudaStream_t s, int* fits) {
    return p.pop_threads == 256   ? launch<256, PARTIAL>(p, s, fits)
           : p.pop_threads == 512 ? launch<512, PARTIAL>(p, s, fits)
                                  : launch<1024, PARTIAL>(p, s, fits);
}

// Whether the device can place the context's clusters.  Up to eight CTAs every device can; for
// more, SMs of one GPC must be free for all of them, which a partition of a GPU may not have.
bool pop_fits(const KParams& p) {
    if (p.pop <= 8) return true;
    int plain = 0, partial = 0;
    const bool known = launch<false>(p, nullptr, &plain) == cudaSuccess &&
                       launch<true>(p, nullptr, &partial) == cudaSuccess;
    if (!known) cudaGetLastError();  // not an error of the caller's: the general kernels run
    return known && plain > 0 && partial > 0;
}

cudaError_t launch_pop(const KParams& p, cudaStream_t s) {
    return p.alpha >= 0.0 ? launch<true>(p, s, nullptr) : launch<false>(p, s, nullptr);
}

}  // namespace pa
