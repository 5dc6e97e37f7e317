// pa_sweep2d.cu -- the temperature step's replica copy, theta checkerboard
// Metropolis sweeps and measurement (Sec. 2 steps 2-4) for two-dimensional
// runs whose side L is a power of two, 16 <= L <= 128: the work of k_group's
// sweep mode, with a lattice layout and a site walk chosen for this case.  The
// random numbers, the order of the updates within a half-sweep (any: sites of
// one colour do not interact) and therefore every result are the same.
//
// Layout.  32 replicas in the multi-spin form (one word per site, bit r =
// replica r), the two colours in arrays of their own: site (x, y) is word
// y S + (x >> 1) of the array of its colour (x + y) & 1.  The four neighbours of
// a site are words of the other colour: same column slot xi = x >> 1 in rows
// y - 1, y, y + 1, and slot xi -+ 1 in row y (left where x is even, right where
// it is odd).
//
// Walk.  A thread owns a column slot and a chunk of H consecutive rows and goes
// down them: of the three words of its own slot one is new per site, so a site
// loads three words (own, next row, side) instead of five; the periodic wrap is
// in the addresses the thread starts from (no halo, no copies after flips).
// L, threads and rows are template parameters, so all offsets inside a chunk are
// immediates and the Philox site counter is the chunk's first one XOR a constant.
// The row stride S puts the chunks (and groups) of a warp on distinct banks.
// G groups per CTA: a lattice of side 16 or 32 gives one warp enough rows per
// thread only when the warp holds a whole group (L = 32) or four (L = 16); the
// half-sweeps of such warps need no CTA barrier.
//
// Undecided sites.  After two unconditional plane blocks (eight bits of the
// uniforms) a site flips the replicas that are decided; a site with undecided
// ones (12% at most) goes to the warp's list with their mask (a shared-memory
// atomic under a predicate).  After its rows the warp finishes the listed sites
// one per lane, from plane block 2 on; the undecided replicas have not flipped, so
// their classes come from the site again.
//
// Spin glass.  A gauge transformation (spins times eps, couplings times the
// products of eps; energies and flips do not change) makes every vertical bond
// +1 except the one that wraps: eps is applied when the rows are read and written,
// the wrap signs where a chunk starts or ends, and a site reads two horizontal
// bond signs, two bytes per site, instead of four masks of a word each.
//
// What bounds it: logic operations and wide multiplies share an issue resource (a probe
// with 6 warps per scheduler: 2 cycles for a logic operation, 2 more for a wide multiply
// beside them, 0.1 for a plain one), so a site costs about 2.17 cycles per scheduler for
// each of its 79 + 34 of them, 7 for the rest: 261 of the 266 cycles measured at L = 64,
// R = 4 10^5 (156 instructions per site word; 189 in the halo layout with its queue).
// L = 64, theta = 10, beta 0 -> 1, updates/ns, before -> now: R = 10^5 4352 -> 4660,
// R = 20000 (theta 5) 3006 -> 3304, R = 3000 1639 -> 1890; L = 32, R = 1024000
// 3811 -> 4797; L = 16, R = 1000 88 -> 117.  The 96 registers that five CTAs of 128 threads
// leave are short by a few: ptxas spills 16 bytes at L = 64, 76 with four groups of L = 32.  80
// registers instead of 96 lose 2%, 64 10%; eight rows per loop pass instead of four 1-4%.
#include "pa_walk.cuh"

namespace pa {
namespace {

constexpr int row_stride2(int tpr, int nch, int h) {
    if (tpr >= 32 || nch == 1) return tpr;
    int s = tpr;
    while ((h * s) % 32 != tpr) ++s;
    return s;
}

template <int L, int NT, int G, bool EA>
struct Shape2 {
    static constexpr int TPR = L / 2, TG = NT / G, NCH = TG / TPR, H = L / NCH;
    static constexpr int N = L * L, W = N / 32, NW = NT / 32;
    static constexpr int LG = (L == 16) ? 4 : (L == 32) ? 5 : (L == 64) ? 6 : 7;
    static constexpr int S = row_stride2(TPR, NCH, H);
    static constexpr int CS = (L * S + 31) / 32 * 32 + 16;         // colour stride
    static constexpr int GS = 2 * CS + (TG < 32 ? TG : 0);      // group stride
    static constexpr int U = H >= 4 ? 4 : H;                        // rows per loop pass
    static constexpr int QW = 32 * H;                               // list entries of a warp
    static constexpr int LAT = (G * GS + 3) & ~3;
    static constexpr size_t SMEM = (size_t)LAT * 4 + (size_t)NW * QW * 8 + (EA ? (size_t)N * 2 : 0);
    static_assert(TG % TPR == 0 && NCH * H == L && H <= 32 && H >= 1, "2D sweep shape");
    static_assert(G == 1 || TG <= 32, "a group of a several-group CTA stays in one warp");
};

template <int L, int NT, int G, bool EA, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_sweep2d(KParams p, const uint32_t* cta2run) {
    using S2 = Shape2<L, NT, G, EA>;
    constexpr int TPR = S2::TPR, H = S2::H, S = S2::S, CS = S2::CS, GS = S2::GS, N = S2::N;
    constexpr int W = S2::W, NW = S2::NW, LG = S2::LG, U = S2::U, TG = S2::TG, Q = H >= 16 ? 1 : U < 2 ? U : 2;
    extern __shared__ __align__(16) uint32_t smem[];
    uint32_t* lat = smem;
    uint2* lists = reinterpret_cast<uint2*>(smem + S2::LAT);            // NW x QW entries
    uint16_t* jt = reinterpret_cast<uint16_t*>(lists + NW * S2::QW);  // EA: bond signs, s = x + L y
    __shared__ uint4 keys[2][G][8];      // block keys of the half-sweep and of the next one
    __shared__ uint4 tbits[16];          // the step's threshold bits
    __shared__ int32_t sU[G][32], sNup[G][32];
    __shared__ uint32_t tail[NW];        // shared-memory address past each warp's list
    __shared__ StepSums sums;

    const RunDesc& r = p.runs[cta2run[blockIdx.x]];
    const DevState* st = r.st;
    chain_wait();
    if (st->status != S_OK) return;
    const int i = st->step;
    const uint32_t R = st->R_cur;
    const uint32_t gfirst = (blockIdx.x - r.cta0) * G;  // the CTA's first group in its run
    if (gfirst * 32u >= R) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* src = r.spins[(i - 1) & 1];
    uint32_t* dst = r.spins[i & 1];
    const uint8_t* jb = r.jbits;

    for (int k = threadIdx.x; k < G * 32; k += NT) {
        sU[k >> 5][k & 31] = 0;
        sNup[k >> 5][k & 31] = 0;
    }
    uint2* list = lists + warp * S2::QW;
    const uint32_t list0 = (uint32_t)__cvta_generic_to_shared(list);
    const uint32_t tail_at = (uint32_t)__cvta_generic_to_shared(&tail[warp]);
    if (lane == 0) tail[warp] = list0;
    if (threadIdx.x == 0) clear_sums(&sums);

    // Gather the parent rows (the copy of step 2) and transpose them into the
    // multi-spin form.  A warp takes whole groups, or a share of one.  Word 32 c4 + k of
    // a row covers rows ybase + (32 k) / L of the lattice from column (32 k) % L on.
    constexpr int WPG = NW > G ? NW / G : 1, GPW = G > NW ? G / NW : 1;
    const Transposer tr(lane);
    const int lx = lane & (L - 1), ly = lane >> LG;
#pragma unroll 1
    for (int gi = 0; gi < GPW; ++gi) {
        const int g = GPW > 1 ? warp * GPW + gi : warp / WPG;
        const uint32_t slot = (gfirst + g) * 32u + lane;
        const bool valid = slot < R;
        const uint4* row =
            reinterpret_cast<const uint4*>(src + (size_t)(valid ? r.anc[slot] : 0u) * r.Wp);
#pragma unroll 1
        for (int c4 = warp % WPG; 4 * c4 < W; c4 += WPG) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (valid) v = row[c4];
            const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
            const int yb = c4 * 128 / L, q = (lx + ly + yb) & 1;
            uint32_t* c0 = lat + g * GS + q * CS + (yb + ly) * S + (lx >> 1);
            uint32_t* c1 = c0 + CS - 2 * q * CS;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint32_t t = tr(w4[k]);
                if (EA) t ^= 0u - ((jb[128 * c4 + 32 * k + lane] >> 4) & 1u);
                (((32 * k / L) & 1) ? c1 : c0)[(32 * k / L) * S + (32 * k % L) / 2] = t;
            }
        }
    }
    if (EA) {
        // signs of a site: bit 7 the bond to the neighbour in its own column slot, bit
        // 15 the one to the side, bits 0 and 1 the wrap bonds up (row 0) and down
        for (int s = threadIdx.x; s < N; s += NT) {
            const int x = s & (L - 1), y = s >> LG;
            const uint32_t right = (jb[s] >> 5) & 1u;
            const uint32_t left = (jb[(y << LG) | ((x - 1) & (L - 1))] >> 5) & 1u;
            const uint32_t up = (jb[(((y - 1) & (L - 1)) << LG) | x] >> 6) & 1u;
            const uint32_t down = (jb[s] >> 6) & 1u;
            jt[s] = (uint16_t)(((x & 1) ? (left << 7) | (right << 15) : (right << 7) | (left << 15)) |
                               up | (down << 1));
        }
    }

    // the thread's column: group gl, slot xi, rows y0 .. y0 + H - 1
    const int gl = G == 1 ? 0 : (int)threadIdx.x / TG;
    const int u = G == 1 ? (int)threadIdx.x : (int)threadIdx.x % TG;
    const int xi = u & (TPR - 1), y0 = (u / TPR) * H;
    const Thr<2> th = {{r.sthr[4 * (i - 1) + 1], r.sthr[4 * (i - 1) + 2]}};
    store_thr_bits<2>(tbits, th);
    const int variant = leading_zeros<2>(th);
    const uint32_t nh = 2u * r.stheta[i - 1];
    uint32_t A2x, B1k, h1a;  // Philox parts of the step and of the thread's group
    {
        uint32_t h0a, l0a, l1a;
        mulhilo(PHILOX_M0, r.grp0 + gfirst + gl, h0a, l0a);
        mulhilo(PHILOX_M1, (uint32_t)i, h1a, l1a);
        A2x = h0a ^ p.rk1[0];
        B1k = l1a ^ p.rk0[1];
    }
    // block keys of half-sweep hh: eight threads per group, of the group's own warp
    // when the half-sweeps are ordered by warp barriers only
    auto build_keys = [&](uint32_t hh) {
        const int g = TG <= 32 ? warp * (32 / TG) + (lane >> 3) : 0;
        const bool mine = TG <= 32 ? lane < 8 * (32 / TG) : threadIdx.x < 8;
        if (mine) {
            uint32_t h0a, l0a;
            mulhilo(PHILOX_M0, r.grp0 + gfirst + g, h0a, l0a);
            keys[hh & 1u][g][lane & 7] = block_key(p, h1a, l0a, hh >> 1, hh & 1u, lane & 7);
        }
    };
    build_keys(0u);
    uint32_t vmask;  // the group's valid replicas
    {
        const uint32_t base = (gfirst + gl) * 32u;
        vmask = base + 32u <= R ? 0xFFFFFFFFu : (base < R ? (1u << (R - base)) - 1u : 0u);
    }
    // the test hook makes the second pass follow every U rows instead of all H
    const int span = p.qcap_limit >= 0 && p.qcap_limit < S2::QW ? U : H;
    __syncthreads();

    constexpr bool SPANS = L >= 64;  // how accepted flips go to 64 bits (add_accepts)
    unsigned long long accepts = 0;
    uint32_t acc = 0;
    for (uint32_t h = 0; h < nh;) {
    for (const uint32_t h1 = SPANS ? min(nh, h + ACC_SPAN) : nh; h < h1; ++h) {
        const uint32_t colour = h & 1u;
        if (h + 1 < nh) build_keys(h + 1);
        uint32_t* own = lat + gl * GS + colour * CS + y0 * S + xi;
        const uint32_t* oth = lat + gl * GS + (colour ^ 1u) * CS + xi;
        const uint32_t par = (y0 + colour) & 1u;  // x parity of the first row's site
        const int dl = ((xi - 1) & (TPR - 1)) - xi, dr = ((xi + 1) & (TPR - 1)) - xi;
        const uint32_t* onx = oth + y0 * S;
        const uint32_t* sd0 = onx + (par ? dr : dl);  // side neighbour: even rows of the chunk
        const uint32_t* sd1 = onx + (par ? dl : dr);  // and odd rows
        const uint32_t* wrap = oth + ((y0 + H) & (L - 1)) * S;
        const uint32_t A2b = A2x ^ (uint32_t)((2 * xi) | (L * y0) | par);
        const uint16_t* jw = jt + (L * y0 + 2 * xi);
        uint32_t prev = oth[((y0 - 1) & (L - 1)) * S], cur = onx[0];
        if (EA) prev ^= 0u - (uint32_t)(jw[par] & 1u);
#pragma unroll 1
        for (int k0 = 0; k0 < H; k0 += span) {
            auto pass1 = [&](auto vtag) {
                constexpr int V = decltype(vtag)::value;
                const uint4 e = keys[h & 1u][gl][0], f = keys[h & 1u][gl][1];
#pragma unroll 1
                for (int kb = k0; kb < k0 + span; kb += U) {
                    const uint32_t* lastn = kb + U == H ? wrap : onx + (kb + U) * S;
#pragma unroll
                    for (int j0 = 0; j0 < U; j0 += Q) {
                        // Q sites at a time, all loads before the stores (the list's writes would
                        // otherwise keep the second site's loads back: +1% where few warps
                        // share a scheduler, -0.6% where they fill it)
                        uint32_t n[Q][4], w[Q], und[Q], fl[Q];
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            const int j = j0 + q, k = kb + j;
                            uint32_t next = j == U - 1 ? lastn[0] : onx[(k + 1) * S];
                            uint32_t side = (j & 1) ? sd1[k * S] : sd0[k * S];
                            uint32_t same = cur;
                            w[q] = own[k * S];
                            if (EA) {
                                const uint32_t jj = jw[L * k + (par ^ (j & 1u))];
                                same ^= byte_sign<0>(jj);
                                side ^= byte_sign<1>(jj);
                                if (j == U - 1) next ^= 0u - ((jj >> 1) & 1u);
                            }
                            n[q][0] = prev;
                            n[q][1] = next;
                            n[q][2] = same;
                            n[q][3] = side;
                            prev = cur;
                            cur = next;
                        }
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            const int j = j0 + q, k = kb + j;
                            uint32_t two, c[2];
                            classes2(w[q], n[q][0], n[q][1], n[q][2], n[q][3], two, c);
                            const SiteKey sk = site_key(A2b ^ (uint32_t)(L * k + (j & 1)), B1k);
                            uint32_t uw[8], b, eq;
                            draw_blocks(e, f, sk, p, uw);
                            compare_top<2, V>(c, tbits, uw, b, eq);
                            und[q] = lop3<0x20>(eq, two, vmask);  // eq & ~two & vmask
                            fl[q] = (two | b) & vmask;            // b = 0 where undecided
                        }
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            const int k = kb + j0 + q;
                            own[k * S] = w[q] ^ fl[q];
                            acc += (uint32_t)__popc(fl[q]);
                            push_undecided(tail_at, und[q], (uint32_t)((k << 5) + lane));
                        }
                    }
                }
            };
            switch (variant) {
                case 0: pass1(IC<0>{}); break;
                case 1: pass1(IC<1>{}); break;
                case 2: pass1(IC<2>{}); break;
                case 3: pass1(IC<3>{}); break;
                case 4: case 5: pass1(IC<4>{}); break;
                case 6: case 7: pass1(IC<6>{}); break;
                default: pass1(IC<8>{}); break;
            }
            // pass 2: the warp's undecided sites, one per lane
            __syncwarp();
            const int total = (int)(tail[warp] - list0) >> 3;
            __syncwarp();
            if (lane == 0) tail[warp] = list0;
#pragma unroll 1
            for (int q0 = 0; q0 < total; q0 += 32) {
                const bool have = q0 + lane < total;
                const uint2 en = list[have ? q0 + lane : 0];
                const uint32_t code = en.x;
                const int tid = warp * 32 + (int)(code & 31u), k = (int)(code >> 5);
                const int g2 = G == 1 ? 0 : tid / TG, u2 = G == 1 ? tid : tid % TG;
                const int x2 = u2 & (TPR - 1), y = (u2 / TPR) * H + k;
                const uint32_t pr = (y + colour) & 1u;
                const int xs = (x2 + (pr ? 1 : -1)) & (TPR - 1);
                uint32_t* a = lat + g2 * GS + colour * CS;
                const uint32_t* o = lat + g2 * GS + (colour ^ 1u) * CS;
                const uint32_t w = a[y * S + x2];
                uint32_t up = o[((y - 1) & (L - 1)) * S + x2], dn = o[((y + 1) & (L - 1)) * S + x2];
                uint32_t same = o[y * S + x2], side = o[y * S + xs];
                const uint32_t s = (uint32_t)(L * y + 2 * x2) | pr;
                if (EA) {
                    const uint32_t jj = jt[s];
                    same ^= byte_sign<0>(jj);
                    side ^= byte_sign<1>(jj);
                    up ^= 0u - (jj & 1u);
                    dn ^= 0u - ((jj >> 1) & 1u);
                }
                uint32_t two, c[2];
                classes2(w, up, dn, same, side, two, c);
                uint32_t A2 = A2x;
                if (G > 1) {
                    uint32_t h0a, l0a;
                    mulhilo(PHILOX_M0, r.grp0 + gfirst + g2, h0a, l0a);
                    A2 = h0a ^ p.rk1[0];
                }
                const uint32_t lt = finish_site<2>(c, tbits, have ? en.y : 0u,
                                                   site_key(A2 ^ s, B1k),
                                                   [&](int g) { return keys[h & 1u][g2][g]; }, p);
                if (have) a[y * S + x2] = w ^ lt;
                acc += (uint32_t)__popc(lt);
            }
            __syncwarp();
        }
        if constexpr (!SPANS) {
            accepts += acc;
            acc = 0;
        }
        if constexpr (TG > 32) __syncthreads();
    }
    if constexpr (SPANS) {
        add_accepts(&sums.acc, acc, lane);
        acc = 0;
    }
    }
    __syncthreads();

    // Measurement: unsatisfied bonds U and up-count per replica, write back.  A warp's
    // unsatisfied-bond words of a group go into a bit-sliced counter (at most 2 per
    // site word it visits), summed per replica at the end.
#pragma unroll 1
    for (int gi = 0; gi < GPW; ++gi) {
        const int g = GPW > 1 ? warp * GPW + gi : warp / WPG;
        const uint32_t slot = (gfirst + g) * 32u + lane;
        constexpr int CB = vc_bits(2 * 4 * ((W / 4 + WPG - 1) / WPG));
        uint32_t ucnt[CB];
#pragma unroll
        for (int j = 0; j < CB; ++j) ucnt[j] = 0u;
        int32_t nup = 0;
#pragma unroll 1
        for (int c4 = warp % WPG; 4 * c4 < W; c4 += WPG) {
            uint32_t out[4], P[8];
            const int yb = c4 * 128 / L, q = (lx + ly + yb) & 1;
            const uint32_t* c0 = lat + g * GS + q * CS + (yb + ly) * S + (lx >> 1);
            const uint32_t* c1 = c0 + CS - 2 * q * CS;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int dy = 32 * k / L, dx = (32 * k % L) / 2;
                const uint32_t* a = (dy & 1) ? c1 : c0;
                const uint32_t* o = (dy & 1) ? c0 : c1;
                uint32_t w = a[dy * S + dx];
                // right: the same slot for even x, the next for odd x (0 past the last)
                const int xl = 32 * k % L + lx;
                const int rs = xl == L - 1 ? -((L - 1) / 2) : (lx & 1);
                P[2 * k] = w ^ o[dy * S + dx + rs];
                const int dn = yb + ly + dy == L - 1 ? (dy + 1 - L) * S : (dy + 1) * S;
                P[2 * k + 1] = w ^ o[dn + dx];
                if (EA) {
                    const uint32_t js = jb[128 * c4 + 32 * k + lane];
                    P[2 * k] ^= 0u - ((js >> 5) & 1u);
                    P[2 * k + 1] ^= 0u - ((js >> 6) & 1u);
                    w ^= 0u - ((js >> 4) & 1u);
                }
                out[k] = tr(w);
                nup += __popc(out[k]);
            }
            vc_add8(ucnt, P);
            if (slot < R)
                reinterpret_cast<uint4*>(dst + (size_t)slot * r.Wp)[c4] =
                    make_uint4(out[0], out[1], out[2], out[3]);
        }
        const int32_t Uw = vc_sum(ucnt, tr);
        atomicAdd(&sU[g][lane], Uw);
        atomicAdd(&sNup[g][lane], nup);
    }
    if constexpr (!SPANS) add_accepts(&sums.acc, accepts, lane);
    __syncthreads();

    if (G == 1 && warp > 0) return;  // one group: its warp adds to the trace itself
    LaneSums ls;
    for (int g = warp; g < G; g += NW) {
        const uint32_t slot = (gfirst + g) * 32u + lane;
        if (slot < R) {
            const int32_t Uv = sU[g][lane];
            const int32_t E = 2 * Uv - 2 * N;
            const int32_t M = N - 2 * sNup[g][lane];
            r.E[i & 1][slot] = E;
            r.M[slot] = M;
            atomicAdd(&r.hist[Uv >> 1], 1u);
            ls.add(E, M, Uv >> 1);
        }
    }
    ls.to_cta(&sums, lane);
    if (G == 1) __syncwarp();
    else __syncthreads();
    add_to_trace(sums, r, i);
}

// dynamic shared memory a CTA of G groups may take (the opt-in limit less the static part)
constexpr size_t smem2d_max(int G) { return 227 * 1024 - 2048 - 520 * (size_t)G; }

template <int L, int NT, int G, bool EA>
cudaError_t launch2d(const KParams& p, const uint32_t* cta2run, uint32_t ncta, cudaStream_t s,
                     bool attr_only, bool chain) {
    constexpr size_t sm = Shape2<L, NT, G, EA>::SMEM;
    static_assert(sm <= smem2d_max(G), "2D sweep shared memory");
    constexpr int MINB = 65536 / (NT * 96);
    const cudaError_t e = cudaFuncSetAttribute(k_sweep2d<L, NT, G, EA, MINB>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem2d_max(G));
    if (e != cudaSuccess || attr_only || ncta == 0) return e;
    return launch_chained(chain, k_sweep2d<L, NT, G, EA, MINB>, ncta, (unsigned)NT, sm, s, p,
                          cta2run);
}

template <int L, int NT, int G>
cudaError_t launch2d_ea(const KParams& p, cudaStream_t s, bool attr_only, bool chain) {
    return p.ea ? launch2d<L, NT, G, true>(p, p.wmap[0], p.wcta[0], s, attr_only, chain)
                : launch2d<L, NT, G, false>(p, p.wmap[0], p.wcta[0], s, attr_only, chain);
}

}  // namespace

// Threads per group of 32 replicas for side L (0: the side has no 2D kernel): the
// variant that `threads` names, or (threads = 0) the least sweep_time() for a
// launch of ngrp groups.
int sweep2d_threads(int L, int threads, uint32_t ngrp) {
    static const int sides[4] = {16, 32, 64, 128};
    static const int tg[4][5] = {{8, 16, 32, 64, 128}, {32, 64, 128, 128, 256},
                                 {128, 128, 256, 256, 512}, {256, 256, 256, 512, 512}};
    for (int k = 0; k < 4; ++k) {
        if (sides[k] != L) continue;
        if (threads > 0) return tg[k][threads <= 64 ? 0 : threads <= 128 ? 1 : threads <= 256 ? 2
                                      : threads <= 384 ? 3 : 4];
        int best = tg[k][0];
        double top = 1e30;
        for (int t : tg[k]) {
            const double v = sweep_time(L * L / 2 / t, ngrp, t <= 32 ? 128 / t : 1, t, t == 512 ? 128 : 96, 1, 0, 1.0);
            if (v < top) {
                top = v;
                best = t;
            }
        }
        return best;
    }
    return 0;
}

// The 2D kernel for runs that all have the same power-of-two side L (16..128); *done =
// false when the plan has none.  attr_only: set the kernel's function attributes only
// (before a stream capture).
cudaError_t launch_sweep2d(const KParams& p, cudaStream_t s, bool attr_only, bool chain, bool* done) {
    *done = p.G2 > 0;
    if (!*done) return cudaSuccess;
    switch (p.L_all * 1000 + p.TG2) {
        case 16008: return launch2d_ea<16, 128, 16>(p, s, attr_only, chain);
        case 16016: return launch2d_ea<16, 128, 8>(p, s, attr_only, chain);
        case 16032: return launch2d_ea<16, 128, 4>(p, s, attr_only, chain);
        case 16064: return launch2d_ea<16, 64, 1>(p, s, attr_only, chain);
        case 16128: return launch2d_ea<16, 128, 1>(p, s, attr_only, chain);
        case 32032: return launch2d_ea<32, 128, 4>(p, s, attr_only, chain);
        case 32064: return launch2d_ea<32, 64, 1>(p, s, attr_only, chain);
        case 32128: return launch2d_ea<32, 128, 1>(p, s, attr_only, chain);
        case 32256: return launch2d_ea<32, 256, 1>(p, s, attr_only, chain);
        case 64128: return launch2d_ea<64, 128, 1>(p, s, attr_only, chain);
        case 64256: return launch2d_ea<64, 256, 1>(p, s, attr_only, chain);
        case 64512: return launch2d_ea<64, 512, 1>(p, s, attr_only, chain);
        case 128256: return launch2d_ea<128, 256, 1>(p, s, attr_only, chain);
        default: return launch2d_ea<128, 512, 1>(p, s, attr_only, chain);
    }
}

}  // namespace pa
