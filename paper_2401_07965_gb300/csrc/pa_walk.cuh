// pa_walk.cuh -- the site update of the column-walk sweep kernels (pa_sweep2d.cu,
// pa_sweepw.cu): the parts of the Philox draw that do not depend on the site, the two
// unconditional plane blocks of a site, the comparison of the uniforms' top eight planes
// with the thresholds, the later blocks of undecided sites, and the step's sums.
//
// Planes with zero threshold bits.  The thresholds of dE = 4, 8, 12 are the
// powers x, x^2, x^3 of x = exp(-4 beta), so if thr[dE = 4] has V leading zero
// bits the others have at least 2 V and 3 V.  Per plane the threshold word is
// the sum of the (disjoint) class masks times their threshold bits; with V known
// at compile time the terms of a zero bit are left out: planes below V need no
// word at all and are compared with zero three at a time.  The kernels carry one
// copy of the walk for V = 0, 1, 2, 3, 4, 6, 8 and take one by the step's thresholds;
// at V = 0 a 2D site takes 16 multiply-adds and 16 logic operations here, at
// V = 2, 4, 8: 10 + 14, 4 + 11, 0 + 3.
#pragma once

#include "pa_sweep_common.cuh"

namespace pa {

template <int V>
struct IC {
    static constexpr int value = V;
};

// The site-independent round-3 values (c0k, c1, c2k) of plane block g of one replica
// group; h1a: high word of the step's round-1 product; l0a: low word of the group's.
__device__ __forceinline__ uint4 block_key(const KParams& p, uint32_t h1a, uint32_t l0a, uint32_t t,
                                           uint32_t colour, uint32_t g) {
    const uint32_t c1v = DOM_SWEEP | (t << 4) | (colour << 3) | g;
    uint32_t h0b, l0b, h1c, l1c;
    mulhilo(PHILOX_M0, h1a ^ c1v ^ p.rk0[0], h0b, l0b);
    mulhilo(PHILOX_M1, h0b ^ l0a ^ p.rk1[1], h1c, l1c);
    return make_uint4(h1c ^ p.rk0[2], l1c, l0b ^ p.rk1[2], 0u);
}

// the site-dependent halves of rounds 2 and 3 (A2s: round-1 lane 2 with the site)
struct SiteKey {
    uint32_t B1, h0c, l0c;
};

__device__ __forceinline__ SiteKey site_key(uint32_t A2s, uint32_t B1k) {
    SiteKey s;
    uint32_t h1b;
    mulhilo(PHILOX_M1, A2s, h1b, s.B1);
    mulhilo(PHILOX_M0, h1b ^ B1k, s.h0c, s.l0c);
    return s;
}

// rounds 4-10 of one plane block
__device__ __forceinline__ void draw_block(const uint4 e, const SiteKey& s, const KParams& p,
                                           uint32_t (&W)[4]) {
    uint32_t x0 = e.x ^ s.B1, x1 = e.y, x2 = s.h0c ^ e.z, x3 = s.l0c;
#pragma unroll
    for (int rr = 3; rr < 10; ++rr) {
        uint32_t hi0, lo0, hi1, lo1;
        mulhilo(PHILOX_M0, x0, hi0, lo0);
        mulhilo(PHILOX_M1, x2, hi1, lo1);
        x0 = hi1 ^ x1 ^ p.rk0[rr];
        x1 = lo1;
        x2 = hi0 ^ x3 ^ p.rk1[rr];
        x3 = lo0;
    }
    W[0] = x0; W[1] = x1; W[2] = x2; W[3] = x3;
}

// two plane blocks, rounds interleaved; u[0..3], u[4..7]: their plane words
__device__ __forceinline__ void draw_blocks(const uint4 e, const uint4 f, const SiteKey& s,
                                            const KParams& p, uint32_t (&u)[8]) {
    uint32_t x0 = e.x ^ s.B1, x1 = e.y, x2 = s.h0c ^ e.z, x3 = s.l0c;
    uint32_t y0 = f.x ^ s.B1, y1 = f.y, y2 = s.h0c ^ f.z, y3 = s.l0c;
#pragma unroll
    for (int rr = 3; rr < 10; ++rr) {
        uint32_t hi0, lo0, hi1, lo1, gi0, go0, gi1, go1;
        mulhilo(PHILOX_M0, x0, hi0, lo0);
        mulhilo(PHILOX_M1, x2, hi1, lo1);
        mulhilo(PHILOX_M0, y0, gi0, go0);
        mulhilo(PHILOX_M1, y2, gi1, go1);
        x0 = hi1 ^ x1 ^ p.rk0[rr];
        x1 = lo1;
        x2 = hi0 ^ x3 ^ p.rk1[rr];
        x3 = lo0;
        y0 = gi1 ^ y1 ^ p.rk0[rr];
        y1 = go1;
        y2 = gi0 ^ y3 ^ p.rk1[rr];
        y3 = go0;
    }
    u[0] = x0; u[1] = x1; u[2] = x2; u[3] = x3;
    u[4] = y0; u[5] = y1; u[6] = y2; u[7] = y3;
}

// the step's thresholds of dE = 4, 8 (, 12)
template <int D>
struct Thr {
    uint32_t t[D];
};

// largest V <= 8 such that the thresholds of dE = 4 a have at least a V leading
// zero bits (among the top eight), a = 1 .. D
template <int D>
__device__ __forceinline__ int leading_zeros(const Thr<D>& t) {
    int v = 8;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int z = __clz((int)t.t[a]);
        if (z < 8) v = min(v, z / (a + 1));
    }
    return v;
}

// lane m of a 128-bit word
__device__ __forceinline__ uint32_t lane4(const uint4 v, int m) {
    return m == 0 ? v.x : (m == 1 ? v.y : (m == 2 ? v.z : v.w));
}

// b = [u8 < t8], eq = [u8 == t8] per replica, u8 the top eight planes and t8 those
// of the replica's class threshold (0 outside the classes): the borrow of u - t from
// the least significant plane up, b' = (~u & t) | (~(u ^ t) & b).  c[a]: the mask of
// class dE = 4 (a + 1); tb[8 a + g]: bits 31 - 4g .. 28 - 4g of its threshold (0 or 1
// each), in shared memory: read per site, the shared-memory pipe has room and the
// registers have not.
template <int D, int V>
__device__ __forceinline__ void compare_top(const uint32_t (&c)[D], const uint4* tb,
                                            const uint32_t (&u)[8], uint32_t& b, uint32_t& eq) {
    if constexpr (V >= 8) {
        b = 0u;
        eq = lop3<0x01>(lop3<0xFE>(u[0], u[1], u[2]), lop3<0xFE>(u[3], u[4], u[5]), u[6] | u[7]);
        return;
    }
    b = 0u;
    eq = 0xFFFFFFFFu;
#pragma unroll
    for (int g = 1; g >= 0; --g) {
        uint4 B[D];
#pragma unroll
        for (int a = 0; a < D; ++a)
            if ((a + 1) * V <= 4 * g + 3) B[a] = tb[8 * a + g];
#pragma unroll
        for (int m = 3; m >= 0; --m) {
            const int q = 4 * g + m;
            if (q < V) continue;
            uint32_t t = c[0] * lane4(B[0], m);
#pragma unroll
            for (int a = 1; a < D; ++a)
                if (q >= (a + 1) * V) t += c[a] * lane4(B[a], m);
            b = lop3<0x8E>(u[q], t, b);    // (~u & t) | (~(u ^ t) & b)
            eq = lop3<0x82>(u[q], t, eq);  // eq & ~(u ^ t)
        }
    }
    // planes 0 .. V-1: t = 0
    if constexpr (V == 1) {
        b &= ~u[0];
        eq &= ~u[0];
    } else if constexpr (V == 2) {
        b = lop3<0x10>(b, u[0], u[1]);  // b & ~u0 & ~u1
        eq = lop3<0x10>(eq, u[0], u[1]);
    } else if constexpr (V == 3) {
        const uint32_t z = lop3<0xFE>(u[0], u[1], u[2]);
        b &= ~z;
        eq &= ~z;
    } else if constexpr (V >= 4) {
        uint32_t z = lop3<0xFE>(u[0], u[1], u[2]);
        if constexpr (V >= 6) z = lop3<0xFE>(z, u[3], u[4]);
        b = lop3<0x10>(b, z, V >= 6 ? u[5] : u[3]);
        eq = lop3<0x10>(eq, z, V >= 6 ? u[5] : u[3]);
    }
}

// the threshold bits (0 or 1) of the step, in shared memory: tb[8 a + g] holds planes
// 4g .. 4g + 3 of class a.  Written by threads 0 .. 8 D - 1.
template <int D>
__device__ __forceinline__ void store_thr_bits(uint4* tb, const Thr<D>& th) {
    if (threadIdx.x < 8 * D) {
        const int g = threadIdx.x & 7;
        uint32_t t = th.t[0];
#pragma unroll
        for (int a = 1; a < D; ++a)
            if ((int)(threadIdx.x >> 3) == a) t = th.t[a];
        t <<= 4 * g;
        tb[threadIdx.x] = make_uint4(t >> 31, (t >> 30) & 1u, (t >> 29) & 1u, (t >> 28) & 1u);
    }
}

// plane blocks 2 .. 7 of an undecided site from the top: the replicas of `und` leave
// at the first plane where u and thr differ; returns those with u < thr.  key(g): the
// block key of the site's group, tb: the step's threshold bits.  Called by the whole
// warp (und = 0 for lanes without a site), which stays together until all are decided.
template <int D, class KeyOf>
__device__ __forceinline__ uint32_t finish_site(const uint32_t (&c)[D], const uint4* tb,
                                                uint32_t und, const SiteKey& sk, KeyOf key,
                                                const KParams& p) {
    uint32_t lt = 0u;
#pragma unroll 1
    for (int g = 2; g < 8 && __any_sync(0xFFFFFFFFu, und != 0u); ++g) {
        uint32_t W[4];
        draw_block(key(g), sk, p, W);
        uint4 bits[D];
#pragma unroll
        for (int a = 0; a < D; ++a) bits[a] = tb[8 * a + g];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            uint32_t tm = c[0] * lane4(bits[0], m);
#pragma unroll
            for (int a = 1; a < D; ++a) tm += c[a] * lane4(bits[a], m);
            lt |= lop3<0x40>(und, tm, W[m]);  // und & tm & ~W
            und = lop3<0x82>(W[m], tm, und);  // und & ~(W ^ tm)
        }
    }
    return lt;
}

// 32 x 32 bit transpose over the warp (lane i holds row i), the lane's selectors,
// rotations and masks computed once: byte steps by one permute, bit steps by one
// rotation and one select (8 logic operations instead of 20)
struct Transposer {
    uint32_t s16, s8, r4, r2, r1, m4, m2, m1;
    __device__ explicit Transposer(int lane) {
        s16 = (lane & 16) ? 0x3276u : 0x5410u;
        s8 = (lane & 8) ? 0x3715u : 0x6240u;
        r4 = (lane & 4) ? 28u : 4u;
        r2 = (lane & 2) ? 30u : 2u;
        r1 = (lane & 1) ? 31u : 1u;
        m4 = (lane & 4) ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
        m2 = (lane & 2) ? 0xCCCCCCCCu : 0x33333333u;
        m1 = (lane & 1) ? 0xAAAAAAAAu : 0x55555555u;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
        x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 16), s16);
        x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 8), s8);
        uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, 4);
        x = lop3<0xCA>(m4, x, __funnelshift_l(y, y, r4));  // m ? x : y
        y = __shfl_xor_sync(0xFFFFFFFFu, x, 2);
        x = lop3<0xCA>(m2, x, __funnelshift_l(y, y, r2));
        y = __shfl_xor_sync(0xFFFFFFFFu, x, 1);
        return lop3<0xCA>(m1, x, __funnelshift_l(y, y, r1));
    }
};

// full adder per bit position: a := sum bit of a + b + c, returns the carry
__device__ __forceinline__ uint32_t csa(uint32_t& a, uint32_t b, uint32_t c) {
    const uint32_t k = lop3<0xE8>(a, b, c);
    a = lop3<0x96>(a, b, c);
    return k;
}

// counter planes c += the eight words w (per bit position): a tree of full adders and
// one ripple (5 logic operations per two words)
template <int CB>
__device__ __forceinline__ void vc_add8(uint32_t (&c)[CB], const uint32_t (&w)[8]) {
    static_assert(CB >= 4, "eight words need four planes");
    const uint32_t t0 = csa(c[0], w[0], w[1]), t1 = csa(c[0], w[2], w[3]);
    const uint32_t t2 = csa(c[0], w[4], w[5]), t3 = csa(c[0], w[6], w[7]);
    const uint32_t f0 = csa(c[1], t0, t1), f1 = csa(c[1], t2, t3);
    uint32_t carry = csa(c[2], f0, f1);
#pragma unroll
    for (int j = 3; j < CB; ++j) {
        const uint32_t t = c[j] & carry;
        c[j] ^= carry;
        carry = t;
    }
}

// lane r: the sum over the warp's lanes of their counts at bit position r
template <int CB>
__device__ __forceinline__ int32_t vc_sum(const uint32_t (&c)[CB], const Transposer& tr) {
    int32_t u = 0;
#pragma unroll
    for (int j = 0; j < CB; ++j) u += __popc(tr(c[j])) << j;
    return u;
}

// Append (code, und) to the warp's list if the lane's und is not zero.  The word at
// tail_at holds the shared-memory address past the list; the lanes' slots come from an
// atomic add on it, all under one predicate (no branch, no ballot, no prefix count on
// the logic pipe; the entries' order does not matter).
__device__ __forceinline__ void push_undecided(uint32_t tail_at, uint32_t und, uint32_t code) {
    asm volatile(
        "{\n\t"
        ".reg .pred q;\n\t"
        ".reg .u32 at;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "@q atom.shared.add.u32 at, [%0], 8;\n\t"
        "@q st.shared.v2.u32 [at], {%2, %1};\n\t"
        "}" ::"r"(tail_at), "r"(und), "r"(code) : "memory");
}

// energy classes of a site from its word and its four neighbours n (bond signs folded
// in): c[0] = exactly one unsatisfied bond (dE = 4), c[1] = none (dE = 8), two = the
// others (dE <= 0).  With s, m the sum and carry of three neighbours and x the parity
// of all four, one bond is unsatisfied iff x = 1 and m = w, none iff x = 0 and s = m = w.
__device__ __forceinline__ void classes2(uint32_t w, uint32_t n0, uint32_t n1, uint32_t n2,
                                         uint32_t n3, uint32_t& two, uint32_t (&c)[2]) {
    const uint32_t s = lop3<0x96>(n0, n1, n2), m = lop3<0xE8>(n0, n1, n2);
    const uint32_t x = s ^ n3;
    const uint32_t g = lop3<0x81>(w, s, m);  // w == s == m
    c[0] = lop3<0x90>(x, w, m);              // x & ~(w ^ m)
    c[1] = g & ~x;
    two = lop3<0x0B>(c[0], g, x);            // ~(c0 | (g & ~x))
}

// The population sums of a CTA's replicas: each warp adds up its replicas in registers,
// the CTA in shared memory, and one thread per quantity adds to the run's trace row and
// level range (a small lattice has thousands of CTAs on the same few addresses).
struct StepSums {
    unsigned long long e, e2, am, m2, acc;
    int lo, hi;
};

struct LaneSums {
    long long e = 0, e2 = 0, am = 0, m2 = 0;
    int lo = 0x7FFFFFFF, hi = -1;
    __device__ __forceinline__ void add(int32_t E, int32_t M, int level) {
        e += E;
        e2 += (long long)E * E;
        am += M < 0 ? -M : M;
        m2 += (long long)M * M;
        lo = min(lo, level);
        hi = max(hi, level);
    }
    // called by whole warps
    __device__ __forceinline__ void to_cta(StepSums* s, int lane) {
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, o);
            e2 += __shfl_xor_sync(0xffffffffu, e2, o);
            am += __shfl_xor_sync(0xffffffffu, am, o);
            m2 += __shfl_xor_sync(0xffffffffu, m2, o);
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0 && hi >= 0) {
            atomicAdd(&s->e, (unsigned long long)e);
            atomicAdd(&s->e2, (unsigned long long)e2);
            atomicAdd(&s->am, (unsigned long long)am);
            atomicAdd(&s->m2, (unsigned long long)m2);
            atomicMin(&s->lo, lo);
            atomicMax(&s->hi, hi);
        }
    }
};

__device__ __forceinline__ void clear_sums(StepSums* s) {
    s->e = s->e2 = s->am = s->m2 = s->acc = 0ull;
    s->lo = 0x7FFFFFFF;
    s->hi = -1;
}

// by threads 0 .. 6, after a CTA barrier
__device__ __forceinline__ void add_to_trace(const StepSums& s, const RunDesc& r, int i) {
    TraceRow* t = r.trace + i;
    switch (threadIdx.x) {
        case 0: atomicAdd(&t->sumE, s.e); break;
        case 1: atomicAdd(&t->sumE2, s.e2); break;
        case 2: atomicAdd(&t->sumAbsM, s.am); break;
        case 3: atomicAdd(&t->sumM2, s.m2); break;
        case 4: atomicAdd(&t->accepts, s.acc); break;
        case 5: atomicMin(&r.st->hlo, s.lo); break;  // the occupied level range for the reweighting
        case 6: atomicMax(&r.st->hhi, s.hi); break;
        default: break;
    }
}

// the all-ones mask of byte B's sign bit of v
template <int B>
__device__ __forceinline__ uint32_t byte_sign(uint32_t v) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(r) : "r"(v), "n"(0x8888 + 0x1111 * B));
    return r;
}

}  // namespace pa
