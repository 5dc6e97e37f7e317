// pa_counts.cuh -- what the resampling kernels share: powers of the level factor, the copy
// numbers of a replica under each rule, and block scans.
#pragma once
#include "pa_internal.cuh"

namespace pa {

// q^k by binary powering from a table of the squares qsq[m] = q^(2^m), each the
// rounded square of the one before (qsq[0] = q): the product of the squares of
// the set bits of k, least significant first, every multiply rounded -- the
// same value as squaring and multiplying in one loop, with popc(k) multiplies
// on the dependent chain.
__device__ __forceinline__ double pow_tab(const double* qsq, uint32_t k) {
    double r = 1.0;
    for (int m = 0; k; ++m, k >>= 1)
        if (k & 1u) r = __dmul_rn(r, qsq[m]);
    return r;
}

// exp(x) = 2^n sum_{k<=13} r^k / k!, x = n ln2 + r (Cody-Waite reduction),
// every operation explicitly rounded.  Used for the Poisson rule, x in [-16, 0].
__device__ __forceinline__ double exp_taylor(double x) {
    const double INV_LN2 = 0x1.71547652b82fep+0;
    const double LN2_HI = 0x1.62e42fefa3800p-1;
    const double LN2_LO = 0x1.ef35793c76730p-45;
    const double c[14] = {0x1.0000000000000p+0,  0x1.0000000000000p+0,  0x1.0000000000000p-1,
                          0x1.5555555555555p-3,  0x1.5555555555555p-5,  0x1.1111111111111p-7,
                          0x1.6c16c16c16c17p-10, 0x1.a01a01a01a01ap-13, 0x1.a01a01a01a01ap-16,
                          0x1.71de3a556c734p-19, 0x1.27e4fb7789f5cp-22, 0x1.ae64567f544e4p-26,
                          0x1.1eed8eff8d898p-29, 0x1.6124613a86d09p-33};
    const double nd = floor(__dadd_rn(__dmul_rn(x, INV_LN2), 0.5));
    const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(nd, LN2_HI)), __dmul_rn(nd, LN2_LO));
    double pp = c[13];
#pragma unroll
    for (int k = 12; k >= 0; --k) pp = __dadd_rn(__dmul_rn(pp, r), c[k]);
    return scalbn(pp, (int)nd);
}

// Poisson draw of mean lc = f 2^-40 / M in [0, 16] by sequential inversion of the CDF: the
// first k with u < P_k, u = bits >> 11 in 2^-53 units, P_k summed in explicitly rounded FP64.
// The search runs in FP32 first.  Its P_k is within (k + 4) 4e-7 of the FP64 one: the mean
// and exp(-l) are off by 6 units of 2^-24 (the mean shifts P_k by at most l p_k <= 1.6 times
// that), each later term by 6 more (product, quotient and sum), and the terms sum to 1.  So u
// farther than that from every P_k it passes decides alike; the others (about 1e-5 of the
// draws) repeat it in FP64, whose operations occupy the pipe for 16 cycles per warp and which
// is kept out of line: inlined, it was executed in part by every draw (+-J L = 48, R = 20001:
// the copy numbers took 50 k cycles, now 4 k).
static __device__ __noinline__ uint32_t poisson_exact(uint64_t f, uint32_t M, uint64_t bits, bool& kmax) {
    const double lam = scalbn((double)f, -FRAC_BITS);
    const double lc = M == 1u ? lam : __ddiv_rn(lam, (double)M);
    const double u = scalbn((double)(bits >> 11), -53);
    double pr = exp_taylor(-lc);
    double Pc = pr;
    uint32_t k = 0;
    while (u >= Pc) {
        k += 1;
        if (k > POISSON_KMAX) {
            kmax = true;
            break;
        }
        pr = __ddiv_rn(__dmul_rn(pr, lc), (double)k);
        Pc = __dadd_rn(Pc, pr);
    }
    return k;
}

__device__ __forceinline__ uint32_t poisson_draw(uint64_t f, uint32_t M, uint64_t bits, bool& kmax) {
    const float lf = __ull2float_rn(f) * 0x1p-40f, l = M == 1u ? lf : __fdividef(lf, (float)M);
    const float u = (float)(uint32_t)(bits >> 40) * 0x1p-24f;
    float pr = expf(-l), Pc = pr;
    uint32_t k = 0;
    float m = 1.6e-6f;
    while (u - Pc > m && k < 64u) {
        k += 1;
        pr = __fdividef(pr * l, (float)k);
        Pc += pr;
        m += 4e-7f;
    }
    return u - Pc < -m ? k : poisson_exact(f, M, bits, kmax);
}

struct U128 {
    uint64_t hi, lo;
};
__device__ __forceinline__ U128 mul128(uint64_t a, uint64_t b) { return {__umul64hi(a, b), a * b}; }
__device__ __forceinline__ bool lt128(U128 a, U128 b) {
    return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}
__device__ __forceinline__ bool le128(U128 a, U128 b) { return !lt128(b, a); }

// Systematic rule: number of labels (k + u/2^32) T/R, k in [0,R), below x:
// with xR = aT + b, that is a + [b 2^32 > u T], at most R.
__device__ inline uint64_t sys_below(uint64_t x, uint64_t R, uint64_t T, uint32_t u) {
    const U128 P = mul128(x, R);
    // a = floor(xR / T) <= R < 2^24: an FP32 estimate is within a few units (FP64 is
    // slow on this part), and the 128-bit corrections below make it exact
    uint64_t a = (uint64_t)__fdiv_rn(__fmul_rn((float)x, (float)R), (float)T);
    for (int it = 0; it < 8 && lt128(P, mul128(a, T)); ++it) --a;
    for (int it = 0; it < 8 && le128(mul128(a + 1, T), P); ++it) ++a;
    const uint64_t b = P.lo - a * T;  // < T, exact in the low 64 bits
    const U128 lhs = {b >> 32, b << 32};
    const U128 rhs = mul128((uint64_t)u, T);
    const uint64_t n = a + (lt128(rhs, lhs) ? 1u : 0u);
    return n < R ? n : R;
}

__device__ __forceinline__ int level_of(int32_t E, int dN) {
    return ((E + dN) >> 1) >> 1;  // U = (E + dN)/2, level = U >> 1
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// exclusive block scan of one value per thread (up to 32 warps; sh: 33 values)
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* sh, T* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = warp_incl_scan(v, lane);
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T w = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : (T)0;
        T wi = warp_incl_scan(w, lane);
        sh[lane] = wi - w;
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    T res = sh[warp] + incl - v;
    *total = sh[32];
    __syncthreads();
    return res;
}

// |c - f 2^-40| in 2^-40 units, rounded to FP64 by integer operations (on this part an FP64
// operation or conversion occupies an SM's pipe for 16 cycles per warp; the conversion of f,
// its scaling and the difference took 190 cycles per warp, this 30)
__device__ __forceinline__ double count_excess(uint32_t c, uint64_t f) {
    const int64_t d = (int64_t)(((uint64_t)c << FRAC_BITS) - f);
    const uint64_t a = (uint64_t)(d < 0 ? -d : d);
    if (a == 0) return 0.0;
    const int n = __clzll((long long)a);
    const uint64_t m = a << n, lo = m & 0x7FFull;
    uint64_t bits = ((uint64_t)(1085 - n) << 52) + (m >> 11);
    bits += lo > 0x400ull || (lo == 0x400ull && (bits & 1ull));
    return __longlong_as_double((long long)bits);
}

// copy number of replica j, expected f in 2^-40 units, under the nearest-integer rule
__device__ __forceinline__ uint32_t nearest_count(const KParams& p, const RunDesc& r, int i,
                                                  uint32_t j, uint64_t f) {
    const uint4x x = philox(j, DOM_RESAMPLE | (r.run << 8) | RULE_NEAREST, (uint32_t)i, 0u, p.k0, p.k1);
    const uint64_t u40 = (((uint64_t)x.y << 32) | x.x) >> 24;
    return (uint32_t)(f >> FRAC_BITS) + (u40 < (f & ((1ull << FRAC_BITS) - 1)) ? 1u : 0u);
}

// ... and under the Poisson rule: sequential inversion per chunk of mean lc <= 16
__device__ __forceinline__ uint32_t poisson_count(const KParams& p, const RunDesc& r, int i,
                                                  uint32_t j, uint64_t f, bool& kmax) {
    const uint32_t M = (uint32_t)(f >> 44) + 1u;
    uint32_t total = 0;
    for (uint32_t m = 0; m < M; ++m) {
        const uint4x x = philox(j, DOM_RESAMPLE | (r.run << 8) | RULE_POISSON, (uint32_t)i, m, p.k0, p.k1);
        total += poisson_draw(f, M, ((uint64_t)x.y << 32) | x.x, kmax);
    }
    return total;
}

// draws k and k + 1, k even, of the multinomial and residual rules: 64 bits each, low word first
__device__ __forceinline__ uint4x draw_block(const KParams& p, const RunDesc& r, int i, uint64_t k,
                                             uint32_t rule) {
    return philox((uint32_t)(k >> 1), DOM_RESAMPLE | (r.run << 8) | rule, (uint32_t)i, 0u, p.k0, p.k1);
}

// the systematic rule's offset of a step
__device__ __forceinline__ uint32_t systematic_offset(const KParams& p, const RunDesc& r, int i) {
    return philox(0u, DOM_RESAMPLE | (r.run << 8) | RULE_SYSTEMATIC, (uint32_t)i, 0u, p.k0, p.k1).x;
}

}  // namespace pa
