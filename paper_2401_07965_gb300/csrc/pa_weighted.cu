// pa_weighted.cu -- weighted averages of repeated runs (Sec. 4 of the paper).
//
// Runs that repeat one system (same lattice and couplings, any population
// size) carry weights omega_i^(m) proportional to R_i^(m) exp(-beta_i F_i^(m))
// (Eq. weighted-averages), where -beta_i F_i^(m) = ln Z_0 + sum_k ln Q_k^(m)
// (Eq. free-energy-estimator); ln Z_0 is common to the runs and cancels.
// From each run's exact per-step sums the kernel forms, per temperature step,
//   W[e], W[e^2], W[|m|], W[m^2]                      (Eq. weighted-averages)
//   Wvar[c] = beta^2 N (W[e^2] - W[e]^2)              (Eq. Wvar_C)
//   Wvar[chi] = beta N (W[m^2] - W[|m|]^2)            (Eq. Wvar_Chi)
//   the naive weighting sum_m omega c^(m), sum_m omega chi^(m), the plain
//   means over runs, and the combined estimate of ln(Z_i / Z_0) as
//   ln( sum_m R^(m) Zhat_m / sum_m R^(m) ).
// One CTA per step; the sums over runs have a fixed order.  The
// same combination serves the runs of one batch (k_weighted, from the trace
// rows) and runs summarised anywhere else, e.g. on other GPUs
// (k_weighted_rows, from rows the caller passes in).
#include <cmath>

#include "../../include/pa.h"
#include "pa_internal.cuh"

namespace pa {

// what the combination needs of one run at one step
struct RunMoments {
    double Ri, Rnom, slnq;  // R_i, nominal R, sum of ln Q
    double e, e2, am, m2;   // per-run averages (weighted under partial resampling)
};

// block sums of NV values (fixed order: lanes by shuffles, then the warps); every thread
// gets the totals
constexpr int WT = 128;
template <int NV>
__device__ __forceinline__ void block_sums(double (&v)[NV], double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[NV * warp + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        v[k] = sh[k];
        for (int w = 1; w < WT / 32; ++w) v[k] += sh[NV * w + k];
    }
}

__device__ __forceinline__ double block_max(double v, double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    v = sh[0];
    for (int w = 1; w < WT / 32; ++w) v = fmax(v, sh[w]);
    return v;
}

// The combination of n_runs runs at one step, by one CTA of WT threads: a thread takes the
// runs threadIdx.x, + WT, ...  (One thread per step over all runs, three passes with a
// logarithm and an exponential each, took 896 us for 80 runs and 41 steps.)  The result is
// thread 0's.
template <class Get>
__device__ pa_weighted_obs combine_runs(int n_runs, double N, double beta, int step, Get get) {
    __shared__ double sh[WT / 32 * 12];
    double amax = -INFINITY, bmax = -INFINITY;
    double a0 = 0.0, b0 = 0.0;  // of the thread's first run
    for (int k = threadIdx.x; k < n_runs; k += WT) {
        const RunMoments r = get(k);
        const double a = log(r.Ri) + r.slnq, b = r.Rnom == r.Ri ? a : log(r.Rnom) + r.slnq;
        if (k < WT) {
            a0 = a;
            b0 = b;
        }
        amax = fmax(amax, a);
        bmax = fmax(bmax, b);
    }
    amax = block_max(amax, sh);
    bmax = block_max(bmax, sh);
    // 0 S, 1 Sb, 2 Rnom, then unnormalised sums: 3 e, 4 e2, 5 am, 6 m2, 7 c, 8 x; plain 9 e,
    // 10 c, 11 x
    double v[12] = {};
    double w2 = 0.0, wmax = 0.0;
    for (int k = threadIdx.x; k < n_runs; k += WT) {
        const RunMoments r = get(k);
        const double a = k < WT ? a0 : log(r.Ri) + r.slnq;
        const double b = k < WT ? b0 : (r.Rnom == r.Ri ? a : log(r.Rnom) + r.slnq);
        const double w = exp(a - amax);
        const double c = beta * beta * N * (r.e2 - r.e * r.e);
        const double x = beta * N * (r.m2 - r.am * r.am);
        v[0] += w;
        v[1] += exp(b - bmax);
        v[2] += r.Rnom;
        v[3] += w * r.e;
        v[4] += w * r.e2;
        v[5] += w * r.am;
        v[6] += w * r.m2;
        v[7] += w * c;
        v[8] += w * x;
        v[9] += r.e;
        v[10] += c;
        v[11] += x;
        w2 += w * w;
        wmax = fmax(wmax, w);
    }
    block_sums(v, sh);
    double t[1] = {w2};
    block_sums(t, sh);
    wmax = block_max(wmax, sh);
    const double S = v[0];
    const double We = v[3] / S, We2 = v[4] / S, Wam = v[5] / S, Wm2 = v[6] / S;
    pa_weighted_obs o;
    if (threadIdx.x != 0) return o;
    o.step = step;
    o.n_runs = n_runs;
    o.beta = beta;
    o.lnZ = bmax + log(v[1]) - log(v[2]);
    o.minus_beta_F = N * log(2.0) + o.lnZ;
    o.w_max = wmax / S;
    o.eff_runs = S * S / t[0];
    o.e = We;
    o.e2 = We2;
    o.absm = Wam;
    o.m2 = Wm2;
    o.c = beta * beta * N * (We2 - We * We);
    o.chi = beta * N * (Wm2 - Wam * Wam);
    o.c_naive = v[7] / S;
    o.chi_naive = v[8] / S;
    o.e_plain = v[9] / n_runs;
    o.c_plain = v[10] / n_runs;
    o.chi_plain = v[11] / n_runs;
    return o;
}

// per-run averages from the exact sums, or from the weighted sums if wsum > 0
__device__ __forceinline__ RunMoments moments(double Ri, double Rnom, double slnq, double N,
                                              long long sE, long long sE2, long long sAM,
                                              long long sM2, double wsum, double wE,
                                              double wE2, double wAM, double wM2) {
    RunMoments m;
    m.Ri = Ri;
    m.Rnom = Rnom;
    m.slnq = slnq;
    const bool wtd = wsum > 0.0;
    m.e = wtd ? wE / (wsum * N) : (double)sE / (Ri * N);
    m.e2 = wtd ? wE2 / (wsum * N * N) : (double)sE2 / (Ri * N * N);
    m.am = wtd ? wAM / (wsum * N) : (double)sAM / (Ri * N);
    m.m2 = wtd ? wM2 / (wsum * N * N) : (double)sM2 / (Ri * N * N);
    return m;
}

__global__ void __launch_bounds__(WT) k_weighted(KParams p, const int32_t* run_ids, int n_runs,
                                                 pa_weighted_obs* out) {
    const int i = blockIdx.x;
    const double N = (double)p.runs[run_ids[0]].N;
    const bool partial = p.alpha >= 0.0;
    const pa_weighted_obs o = combine_runs(n_runs, N, p.beta[i], i, [&](int k) {
        const RunDesc& r = p.runs[run_ids[k]];
        const TraceRow& t = r.trace[i];
        return moments((double)t.R_i, (double)r.R, t.sum_lnQ, N, (long long)t.sumE,
                       (long long)t.sumE2, (long long)t.sumAbsM, (long long)t.sumM2,
                       partial ? t.wsum : 0.0, t.wE, t.wE2, t.wAM, t.wM2);
    });
    if (threadIdx.x == 0) out[i] = o;
}

__global__ void __launch_bounds__(WT) k_weighted_rows(const pa_run_row* rows, int n_runs, int N,
                                                      double beta, int32_t step,
                                                      pa_weighted_obs* out) {
    const double Nd = (double)N;
    const pa_weighted_obs o = combine_runs(n_runs, Nd, beta, step, [&](int k) {
        const pa_run_row& r = rows[k];
        return moments((double)r.R_i, (double)r.R, r.sum_lnQ, Nd, (long long)r.sumE,
                       (long long)r.sumE2, (long long)r.sumAbsM, (long long)r.sumM2, r.wsum,
                       r.wE, r.wE2, r.wAM, r.wM2);
    });
    if (threadIdx.x == 0) out[0] = o;
}

cudaError_t launch_weighted(const KParams& p, const int32_t* run_ids, int n_runs, int n_rows,
                            pa_weighted_obs* out, cudaStream_t s) {
    k_weighted<<<n_rows, WT, 0, s>>>(p, run_ids, n_runs, out);
    return cudaGetLastError();
}

}  // namespace pa

using namespace pa;

extern "C" pa_status pa_weighted_rows(const pa_run_row* rows, int32_t n_runs, int32_t N,
                                      double beta, int32_t step, pa_weighted_obs* out,
                                      void* cuda_stream) {
    if (!rows || !out || n_runs < 1 || N < 1) return PA_ERR_ARG;
    for (int k = 0; k < n_runs; ++k)
        if (rows[k].R_i == 0 || rows[k].R == 0) return PA_ERR_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    pa_run_row* d_rows = nullptr;
    pa_weighted_obs* d_out = nullptr;
    if (cudaMalloc(&d_rows, sizeof(pa_run_row) * n_runs) != cudaSuccess) return PA_ERR_NOMEM;
    if (cudaMalloc(&d_out, sizeof(pa_weighted_obs)) != cudaSuccess) {
        cudaFree(d_rows);
        return PA_ERR_NOMEM;
    }
    cudaError_t e = cudaMemcpyAsync(d_rows, rows, sizeof(pa_run_row) * n_runs,
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        k_weighted_rows<<<1, WT, 0, s>>>(d_rows, n_runs, N, beta, step, d_out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(out, d_out, sizeof(pa_weighted_obs), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d_rows);
    cudaFree(d_out);
    return e == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}
