// pa_control.cu -- the learned schedule controller (adaptive temperature steps
// and sweep numbers, cited as established practice in Sec. 5 of the paper) and
// the kernels that train its network.
//
// Network: 8 population statistics -> 64 -> 64 -> 2 (ReLU), BF16 parameters,
// FP32 accumulation in a fixed order (bias added last), no fused multiply-add.
// Outputs: s, the step size relative to the average remaining step, and t,
// the sweeps relative to the planned sweeps per step.
//
// Inference (pa_control.cuh, k_control) runs when the controller is switched on and
// then after every temperature step: it writes the next step's entries of the step
// tables from tables precomputed on the host, so the PA step itself is unchanged and
// stays bit-exact.
#include <algorithm>
#include <cmath>
#include <cuda_bf16.h>

#include "../../include/pa.h"
#include "pa_control.cuh"

namespace pa {

namespace {
constexpr int ROWS = 32;  // rows per CTA of the training kernels
}  // namespace

__device__ __forceinline__ float bf_round(float v) {
    return __bfloat162float(__float2bfloat16_rn(v));
}

// --------------------------------------------------------------------------
// controller step: the first decision of a run (at pa_set_controller) and the one after
// every step.  In the family kernel's last CTA it saved a launch, but the family statistics
// now run beside the sweep and the decision has to wait for both (learned schedule, L = 64,
// R = 3000: 24.6 -> 22.5 ms for 240 steps).
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(32 * MLP_IN) k_control(KParams p) {
    const RunDesc& r = p.runs[blockIdx.x];  // one CTA per run of the batch
    control_after_step(p, r, r.st);
}

cudaError_t launch_control(const KParams& p, cudaStream_t s) {
    k_control<<<p.M, 32 * MLP_IN, 0, s>>>(p);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// inference over a batch (BF16 parameters; one product after the other in index
// order, bias last, no fused multiply-add: the order of the controller's step)
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(64) k_mlp_fwd(const uint16_t* __restrict__ params,
                                                const float* __restrict__ X, int B,
                                                float* __restrict__ Y) {
    __shared__ float xs[ROWS][MLP_IN], a1[ROWS][MLP_HID], a2[ROWS][MLP_HID];
    __shared__ float W2s[MLP_HID * MLP_HID];
    const int t = threadIdx.x, r0 = blockIdx.x * ROWS;
    auto P = [&](int idx) -> float { return bf(params[idx]); };
    for (int e = t; e < ROWS * MLP_IN; e += 64) {
        const int rr = e / MLP_IN, k = e % MLP_IN;
        xs[rr][k] = (r0 + rr < B) ? X[(size_t)(r0 + rr) * MLP_IN + k] : 0.0f;
    }
    for (int e = t; e < MLP_HID * MLP_HID; e += 64) W2s[e] = P(OFF_W2 + e);
    __syncthreads();
    float w1[MLP_IN];
    for (int k = 0; k < MLP_IN; ++k) w1[k] = P(OFF_W1 + t * MLP_IN + k);
    const float b1 = P(OFF_B1 + t), b2 = P(OFF_B2 + t);
    for (int rr = 0; rr < ROWS; ++rr) {
        float acc = 0.0f;
        for (int k = 0; k < MLP_IN; ++k) acc = __fadd_rn(acc, __fmul_rn(w1[k], xs[rr][k]));
        acc = __fadd_rn(acc, b1);
        a1[rr][t] = acc > 0.0f ? acc : 0.0f;
    }
    __syncthreads();
    for (int rr = 0; rr < ROWS; ++rr) {
        float acc = 0.0f;
        for (int k = 0; k < MLP_HID; ++k) acc = __fadd_rn(acc, __fmul_rn(W2s[t * MLP_HID + k], a1[rr][k]));
        acc = __fadd_rn(acc, b2);
        a2[rr][t] = acc > 0.0f ? acc : 0.0f;
    }
    __syncthreads();
    const int rr = t >> 1, o = t & 1;
    float acc = 0.0f;
    for (int k = 0; k < MLP_HID; ++k) acc = __fadd_rn(acc, __fmul_rn(P(OFF_W3 + o * MLP_HID + k), a2[rr][k]));
    acc = __fadd_rn(acc, P(OFF_B3 + o));
    if (r0 + rr < B) Y[(size_t)(r0 + rr) * MLP_OUT + o] = acc;
}

// --------------------------------------------------------------------------
// Training gradients (FP32, parameters rounded to BF16 as in inference).  A CTA of 8 GR
// threads takes `rows` consecutive rows, GR at a time, through the forward and the backward
// pass in shared memory and adds up its part of every gradient in registers; the parts are
// summed in CTA order by k_mlp_reduce.  The products with W2 and the sum over rows of its
// gradient are 64 x 64 x GR each: a thread holds a 4 x 2 tile of the result and reads a
// 128-bit and a 64-bit word of shared memory per 8 fused multiply-adds.
// What bounds it: shared-memory latency on one CTA per SM (30 k flops per row).  GR = 32, 64
// or 96, the least that takes the rows of one of 152 CTAs in one pass, and passes of 96 from 97
// rows on (14592 rows 24 us, 14593 to 29184 39; with the forward pass in a kernel of its own 63,
// 70 to 96).  12040 rows are 151 CTAs of 80 rows; two passes of 64 with 256 threads took 33 us, one pass 22 us (the whole
// update of 12040 rows: 66 us with the forward pass stored and read back, 31 with one kernel,
// 29 with the reduction chained to it).
// --------------------------------------------------------------------------
constexpr int LDW = MLP_HID + 4;  // padded rows of units: 16-byte aligned

template <int GR>
struct GradSmem {
    static constexpr int LDR = GR + 4;  // padded rows of batch rows
    float w2[MLP_HID * LDW];            // W2[j][k]
    float w2t[MLP_HID * LDW];           // W2 transposed
    float a1t[MLP_HID * LDR];           // H1[k][row]
    float a2t[MLP_HID * LDR];           // H2[j][row]
    float d2t[MLP_HID * LDR];           // dH2[j][row]
    float d1t[MLP_HID * LDR];           // dH1[k][row]
    float d2[GR * LDW];                 // dH2[row][j]
    float a1[GR * LDW];                 // H1[row][k]
    float w1[MLP_HID * MLP_IN], w3[MLP_OUT * MLP_HID], b1[MLP_HID], b2[MLP_HID], b3[MLP_OUT];
    float xs[GR][MLP_IN];
    float dy[GR][MLP_OUT];
    float loss[GR * MLP_OUT];
};

template <int GR>
__global__ void __launch_bounds__(8 * GR) k_mlp_grad(const float* __restrict__ params,
                                                     const float* __restrict__ X,
                                                     const float* __restrict__ Yt,
                                                     const float* __restrict__ mask, int B, int rows,
                                                     float norm, float* __restrict__ part) {
    constexpr int GT = 8 * GR, LDR = GradSmem<GR>::LDR;
    extern __shared__ __align__(16) unsigned char raw[];
    GradSmem<GR>& s = *reinterpret_cast<GradSmem<GR>*>(raw);
    const int t = threadIdx.x, ti = t % (GR / 2), tj = t / (GR / 2);  // rows 2 ti.., units 4 tj..
    chain_next();
    for (int e = t; e < MLP_HID * MLP_HID; e += GT) {
        const float v = bf_round(params[OFF_W2 + e]);
        s.w2[(e >> 6) * LDW + (e & 63)] = v;
        s.w2t[(e & 63) * LDW + (e >> 6)] = v;
    }
    for (int e = t; e < MLP_HID * MLP_IN; e += GT) s.w1[e] = bf_round(params[OFF_W1 + e]);
    if (t < MLP_OUT * MLP_HID) s.w3[t] = bf_round(params[OFF_W3 + t]);
    if (t < MLP_HID) {
        s.b1[t] = bf_round(params[OFF_B1 + t]);
        s.b2[t] = bf_round(params[OFF_B2 + t]);
    }
    if (t < MLP_OUT) s.b3[t] = bf_round(params[OFF_B3 + t]);
    // W2's gradient: tiles of 4 rows and WC columns on the first 1024 / WC threads
    constexpr int WC = GR == 32 ? 4 : 2, WT2 = 16 * (MLP_HID / WC);
    const int wi = t % (MLP_HID / WC), wj = t / (MLP_HID / WC);
    constexpr int N1 = GT >= 512 ? 1 : 2;  // W1 elements of a thread (t < 512 / N1)
    const int q = t - (GT - 256);          // the last 256 threads: W3, b1, b2; b3 and the loss
    float g2[4][WC] = {}, g1[N1] = {};
    float g3 = 0.0f, gl = 0.0f;
    const int r0 = blockIdx.x * rows, r1 = min(r0 + rows, B);
    for (int base = r0; base < r1; base += GR) {
        const int n = min(GR, r1 - base);
        __syncthreads();
        {
            const int rr = t / MLP_IN;  // GR x 8 values, one per thread
            s.xs[rr][t % MLP_IN] = rr < n ? X[(size_t)(base + rr) * MLP_IN + t % MLP_IN] : 0.0f;
        }
        __syncthreads();
        // H1: unit t & 63 of rows t >> 6, + GR / 8, ...; 0 in rows past the last
        {
            const int k = t & 63;
            float w[MLP_IN];
#pragma unroll
            for (int c = 0; c < MLP_IN; ++c) w[c] = s.w1[k * MLP_IN + c];
            const float bb = s.b1[k];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int rr = (t >> 6) + GR / 8 * m;
                float acc = 0.0f;
#pragma unroll
                for (int c = 0; c < MLP_IN; ++c) acc = __fmaf_rn(w[c], s.xs[rr][c], acc);
                acc += bb;
                const float h = acc > 0.0f && rr < n ? acc : 0.0f;
                s.a1[rr * LDW + k] = h;
                s.a1t[k * LDR + rr] = h;
            }
        }
        __syncthreads();
        // H2[j][row] = relu(sum_k W2[j][k] H1[k][row] + b2[j])
        {
            float acc[4][2] = {};
#pragma unroll 8
            for (int k = 0; k < MLP_HID; ++k) {
                const float4 w = *reinterpret_cast<const float4*>(&s.w2t[k * LDW + 4 * tj]);
                const float2 h = *reinterpret_cast<const float2*>(&s.a1t[k * LDR + 2 * ti]);
                const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[u][0] = __fmaf_rn(wv[u], h.x, acc[u][0]);
                    acc[u][1] = __fmaf_rn(wv[u], h.y, acc[u][1]);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float bb = s.b2[4 * tj + u];
                float2 h;
                h.x = 2 * ti + 0 < n ? fmaxf(acc[u][0] + bb, 0.0f) : 0.0f;
                h.y = 2 * ti + 1 < n ? fmaxf(acc[u][1] + bb, 0.0f) : 0.0f;
                *reinterpret_cast<float2*>(&s.a2t[(4 * tj + u) * LDR + 2 * ti]) = h;
            }
        }
        __syncthreads();
        // outputs, their errors and gradients: two threads per row
        if (t < GR * MLP_OUT) {
            const int rr = t >> 1, o = t & 1;
            float acc = 0.0f;
#pragma unroll 16
            for (int j = 0; j < MLP_HID; ++j) acc = __fmaf_rn(s.w3[o * MLP_HID + j], s.a2t[j * LDR + rr], acc);
            acc += s.b3[o];
            float g = 0.0f, l = 0.0f;
            if (rr < n) {
                const size_t id = (size_t)(base + rr) * MLP_OUT + o;
                const float diff = acc - Yt[id], mk = mask[id];
                g = 2.0f * mk * (diff * norm);
                l = mk * (diff * diff);
            }
            s.dy[rr][o] = g;
            s.loss[t] = l;
        }
        __syncthreads();
        // dH2 (unit t & 63 of rows t >> 6, + GR / 8, ...); zero past the last row (dY = 0)
        {
            const int j = t & 63;
            const float w30 = s.w3[j], w31 = s.w3[MLP_HID + j];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int rr = (t >> 6) + GR / 8 * m;
                const float v = __fmaf_rn(s.dy[rr][1], w31, s.dy[rr][0] * w30);
                const float d = s.a2t[j * LDR + rr] > 0.0f ? v : 0.0f;
                s.d2t[j * LDR + rr] = d;
                s.d2[rr * LDW + j] = d;
            }
        }
        __syncthreads();
        // dH1[k][row] = [H1 > 0] sum_j W2[j][k] dH2[j][row]; W2's gradient [j][k] += sum_row
        {
            float acc[4][2] = {};
#pragma unroll 8
            for (int j = 0; j < MLP_HID; ++j) {
                const float4 w = *reinterpret_cast<const float4*>(&s.w2[j * LDW + 4 * tj]);
                const float2 d = *reinterpret_cast<const float2*>(&s.d2t[j * LDR + 2 * ti]);
                const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[u][0] = __fmaf_rn(wv[u], d.x, acc[u][0]);
                    acc[u][1] = __fmaf_rn(wv[u], d.y, acc[u][1]);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int o = (4 * tj + u) * LDR + 2 * ti;
                const float2 h = *reinterpret_cast<const float2*>(&s.a1t[o]);
                float2 d;
                d.x = h.x > 0.0f ? acc[u][0] : 0.0f;
                d.y = h.y > 0.0f ? acc[u][1] : 0.0f;
                *reinterpret_cast<float2*>(&s.d1t[o]) = d;
            }
        }
        if (t < WT2) {
#pragma unroll 8
            for (int rr = 0; rr < GR; ++rr) {
                const float4 d = *reinterpret_cast<const float4*>(&s.d2[rr * LDW + 4 * wj]);
                const float dv[4] = {d.x, d.y, d.z, d.w};
                float hv[WC];
#pragma unroll
                for (int c = 0; c < WC; c += 2) {
                    const float2 h = *reinterpret_cast<const float2*>(&s.a1[rr * LDW + WC * wi + c]);
                    hv[c] = h.x;
                    hv[c + 1] = h.y;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int c = 0; c < WC; ++c) g2[u][c] = __fmaf_rn(dv[u], hv[c], g2[u][c]);
            }
        }
        __syncthreads();
        if (t < 512 / N1)
#pragma unroll
            for (int m = 0; m < N1; ++m) {
                const int e = t + GT * m, j = e / MLP_IN, k = e % MLP_IN;
                float acc = 0.0f;
#pragma unroll 16
                for (int rr = 0; rr < GR; ++rr) acc = __fmaf_rn(s.d1t[j * LDR + rr], s.xs[rr][k], acc);
                g1[m] += acc;
            }
        if (q >= 0) {
            float acc = 0.0f;
            if (q < MLP_OUT * MLP_HID) {  // W3
                const int o = q >> 6, j = q & 63;
#pragma unroll 16
                for (int rr = 0; rr < GR; ++rr) acc = __fmaf_rn(s.dy[rr][o], s.a2t[j * LDR + rr], acc);
            } else {  // b1, b2
                const int u = q - 128;
                const float* row = u < 64 ? &s.d1t[u * LDR] : &s.d2t[(u - 64) * LDR];
#pragma unroll 16
                for (int rr = 0; rr < GR; ++rr) acc += row[rr];
            }
            g3 += acc;
            if (q < 64) {  // two warps: b3 (lanes o, o + 2, ...) and the loss
                float v = 0.0f;
                const int l = q & 31;
                if (q < 32) {
                    for (int rr = l >> 1; rr < GR; rr += 16) v += s.dy[rr][l & 1];
                } else {
                    for (int e = l; e < GR * MLP_OUT; e += 32) v += s.loss[e];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                }
                for (int o = 16; o >= 2; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                gl += v;
            }
        }
    }
    float* g = part + (size_t)blockIdx.x * (MLP_NPARAM + 1);
    if (t < WT2)
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < WC; ++c) g[OFF_W2 + (4 * wj + u) * MLP_HID + WC * wi + c] = g2[u][c];
    if (t < 512 / N1)
#pragma unroll
        for (int m = 0; m < N1; ++m) g[OFF_W1 + t + GT * m] = g1[m];
    if (q >= 0) {
        g[q < 128 ? OFF_W3 + q : (q < 192 ? OFF_B1 - 128 : OFF_B2 - 192) + q] = g3;
        if (q < MLP_OUT) g[OFF_B3 + q] = gl;
        if (q == 32) g[MLP_NPARAM] = gl * norm;
    }
}

template <int GR>
cudaError_t launch_grad(const float* params, const float* X, const float* Yt, const float* mask,
                        int B, int rows, unsigned nb, float norm, float* part, cudaStream_t s) {
    const cudaError_t e = cudaFuncSetAttribute(
        k_mlp_grad<GR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem<GR>));
    if (e != cudaSuccess) return e;
    k_mlp_grad<GR><<<nb, 8 * GR, sizeof(GradSmem<GR>), s>>>(params, X, Yt, mask, B, rows, norm, part);
    return cudaGetLastError();
}

// fixed-order sum of the per-CTA parts: eight warps of a CTA take the parts b = w, w + 8,
// ... of 32 parameters, then the eight sums in order
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* part, int nb, float* grads, float* loss) {
    __shared__ float sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
    float acc = 0.0f;
    chain_wait();
    if (k <= MLP_NPARAM)
#pragma unroll 8
        for (int b = w; b < nb; b += 8) acc += part[(size_t)b * (MLP_NPARAM + 1) + k];
    sh[w][lane] = acc;
    __syncthreads();
    if (w != 0 || k > MLP_NPARAM) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) acc += sh[q][lane];
    if (k < MLP_NPARAM) grads[k] = acc;
    else if (loss) *loss = acc;
}

// Adam (Kingma & Ba) on the FP32 master parameters; writes the BF16 copy
__global__ void k_mlp_adam(float* __restrict__ w, const float* __restrict__ g,
                           float* __restrict__ m, float* __restrict__ v,
                           uint16_t* __restrict__ wbf, float lr, float c1, float c2) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= MLP_NPARAM) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.0f - b1) * gk;
    const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    const float wk = w[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    w[k] = wk;
    if (wbf) wbf[k] = __bfloat16_as_ushort(__float2bfloat16_rn(wk));
}

}  // namespace pa

using namespace pa;

namespace {
size_t mlp_blocks(int B) { return (size_t)(B + ROWS - 1) / ROWS; }
}  // namespace

extern "C" {

// The gradients' parts take a third of it; the rest, a row's activations, is what the call has
// asked for and checked since the forward pass stored them, and stays so for its callers.
size_t pa_mlp_scratch_bytes(int32_t B) {
    if (B <= 0) return 0;
    const size_t nb = mlp_blocks(B);
    return sizeof(float) * ((size_t)B * (2 * MLP_HID + MLP_OUT) + nb * (MLP_NPARAM + 1));
}

pa_status pa_mlp_forward(const uint16_t* params_bf16, const float* X, int32_t B, float* Y,
                         void* cuda_stream) {
    if (!params_bf16 || !X || !Y || B <= 0) return PA_ERR_ARG;
    k_mlp_fwd<<<(unsigned)mlp_blocks(B), 64, 0, (cudaStream_t)cuda_stream>>>(params_bf16, X, B, Y);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

pa_status pa_mlp_gradients(const float* params, const float* X, const float* Yt,
                           const float* mask, int32_t B, float* grads, float* loss,
                           void* scratch, size_t scratch_bytes, void* cuda_stream) {
    if (!params || !X || !Yt || !mask || !grads || B <= 0 || !scratch) return PA_ERR_ARG;
    if (scratch_bytes < pa_mlp_scratch_bytes(B)) return PA_ERR_NOMEM;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // one CTA per SM; the scratch holds a part per ROWS rows, which is never fewer
    const int rows = std::max(ROWS, (B + 151) / 152);
    const unsigned nb = (unsigned)((B + rows - 1) / rows);
    float* part = (float*)scratch;
    const float norm = 1.0f / (float)(B * MLP_OUT);
    const cudaError_t e =
        rows <= 32   ? launch_grad<32>(params, X, Yt, mask, B, rows, nb, norm, part, s)
        : rows <= 64 ? launch_grad<64>(params, X, Yt, mask, B, rows, nb, norm, part, s)
                     : launch_grad<96>(params, X, Yt, mask, B, rows, nb, norm, part, s);
    if (e != cudaSuccess) return PA_ERR_CUDA;
    return launch_chained(true, k_mlp_reduce, (MLP_NPARAM + 1 + 31) / 32, 256u, 0, s, part, (int)nb, grads,
                          loss) == cudaSuccess
               ? PA_OK
               : PA_ERR_CUDA;
}

pa_status pa_mlp_adam(float* params, const float* grads, float* m, float* v, uint16_t* params_bf16,
                      int32_t step, float lr, void* cuda_stream) {
    if (!params || !grads || !m || !v || step < 1 || !(lr > 0.0f)) return PA_ERR_ARG;
    const float c1 = 1.0f - powf(0.9f, (float)step), c2 = 1.0f - powf(0.999f, (float)step);
    k_mlp_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(
        params, grads, m, v, params_bf16, lr, c1, c2);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

}  // extern "C"
