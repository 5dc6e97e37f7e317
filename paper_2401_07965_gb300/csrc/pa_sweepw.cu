// pa_sweepw.cu -- the temperature step's replica copy, theta checkerboard
// Metropolis sweeps and measurement (Sec. 2 steps 2-4) by column walks, for 3D
// lattices (except L = 10, 12, 14) and 2D lattices of the sides that pa_sweep2d.cu
// does not take, where walk_plan() finds them faster than the general kernel.  Random numbers, decisions and results are those of k_group's sweep mode.
//
// Layout.  32 replicas in the multi-spin form (one word per site, bit r =
// replica r), the two colours in arrays of their own: the site of column slot
// xi = x >> 1 of a row is word row S + col of the array of its colour, where the
// rows are the lines y = const (2D, col = xi) or the planes z = const (3D,
// col = y L/2 + xi).  The neighbours of a site are words of the other colour: its
// own column in the rows before, of and after it, the slot beside it in its row
// (left where x is even, right where it is odd) and, in 3D, the columns y -+ 1.
//
// Walk.  A thread owns a column (3D: all L planes; 2D: one of NCH chunks of H
// rows) and goes along it: of its own column's words one is new per site, so a
// site loads 3 (2D) or 5 (3D) words instead of 5 or 7, with the periodic wraps in
// the addresses the thread starts from: no halo, no copies after flips, no site
// table.  GP groups of 32 replicas stand side by side in the threads of a CTA and a
// thread takes the column of CPT such sets, one after the other, before the warp
// finishes its undecided sites (small lattices have few sites per column).
//
// Undecided sites after eight planes go to a list of the warp (shared-memory
// atomics under a predicate) and are finished one per lane from plane block 2 on;
// their undecided replicas have not flipped, so their classes come from the site.
//
// Spin glass.  In a gauge in which every bond along the walk is +1 except the
// one that wraps (bits 4-7 of the coupling bytes) a site reads the signs of 2 (2D)
// or 4 (3D) bonds from one byte, spread over the bytes of a word by a multiplication.
//
// What bounds it: as in pa_sweep2d.cu the issue of logic operations and wide multiplies
// (L = 8: about 150 of them per site word, 171 with the halo layout and its site tables).
// +-J, theta = 10, beta 0 -> 3, updates/ns, before -> now: 64 runs of L = 4 2676 -> 3240,
// 32 of L = 6 3225 -> 3526, 16 of L = 8 3474 -> 3742 (R = 50000 each), 4 of L = 16,
// R = 20000 2643 -> 3514; one run of L = 6, R = 10^5 1798 -> 2497 (its level counts and
// sums now leave the CTA once); ferromagnet L = 20, 4 runs of R = 10^4 2558 -> 2689.
// L = 10, 12, 14, whose columns do not fill warps, stay with pa_sweep3d.cu (L = 10,
// one run of R = 10^5: 2631 here, 2922 there; L = 12, R = 30000: 1849 and 2515).
#include "pa_walk.cuh"

#include <algorithm>
#include <cstring>

namespace pa {

namespace {

__host__ __device__ constexpr int walk_cs(int words) { return (words + 31) / 32 * 32 + 16; }

// classes of d = 3 from the site word and its six bond partners: n unsatisfied bonds
// as a bit-sliced count; c[0], c[1], c[2] = 2, 1, 0 of them (dE = 4, 8, 12), two = the
// others.  The sum and carry of a triple of bonds are w ^ (a ^ b ^ c) and
// w ^ maj(a, b, c), so w cancels from the sums and enters the carries only.
__device__ __forceinline__ void classes3(uint32_t w, const uint32_t (&a)[6], uint32_t& two,
                                         uint32_t (&c)[3]) {
    const uint32_t x3 = lop3<0x96>(a[0], a[1], a[2]), ma = lop3<0xE8>(a[0], a[1], a[2]);
    const uint32_t y3 = lop3<0x96>(a[3], a[4], a[5]), mb = lop3<0xE8>(a[3], a[4], a[5]);
    const uint32_t n0 = x3 ^ y3;
    const uint32_t kc = lop3<0x18>(w, x3, y3);                           // (w^x3)&(w^y3)
    const uint32_t n1 = lop3<0x96>(ma, mb, kc);
    const uint32_t n2 = lop3<0x18>(w, ma, mb) | lop3<0x60>(kc, ma, mb);  // carry of the carries
    two = lop3<0xF8>(n2, n1, n0);                                        // n2 | (n1 & n0)
    c[2] = lop3<0x01>(n0, n1, n2);
    c[1] = lop3<0x10>(n0, n1, n2);
    c[0] = lop3<0x04>(n0, n1, n2);
}

template <int D>
__device__ __forceinline__ void classes(uint32_t w, const uint32_t (&a)[6], uint32_t& two,
                                        uint32_t (&c)[D]) {
    if constexpr (D == 3) classes3(w, a, two, c);
    else classes2(w, a[0], a[1], a[2], a[3], two, c);
}

// bits 0 .. 3 of v as the sign bits of bytes 0 .. 3 (the four copies do not overlap)
__device__ __forceinline__ uint32_t spread_signs(uint32_t v) { return v * 0x10204080u; }

// the group-independent round-2 values of a plane block: (h0b with its key, c2k)
__device__ __forceinline__ uint2 block_part(const KParams& p, uint32_t h1a, uint32_t t,
                                            uint32_t colour, uint32_t b) {
    const uint32_t c1v = DOM_SWEEP | (t << 4) | (colour << 3) | b;
    uint32_t h0b, l0b;
    mulhilo(PHILOX_M0, h1a ^ c1v ^ p.rk0[0], h0b, l0b);
    return make_uint2(h0b ^ p.rk1[1], l0b ^ p.rk1[2]);
}

// a group's block key from it (l0a: low word of the group counter's round-1 product)
__device__ __forceinline__ uint4 block_key_of(const KParams& p, uint2 bp, uint32_t l0a) {
    uint32_t h1c, l1c;
    mulhilo(PHILOX_M1, bp.x ^ l0a, h1c, l1c);
    return make_uint4(h1c ^ p.rk0[2], l1c, bp.y, 0u);
}

// byte offsets of the dynamic shared memory
struct WalkSmem {
    int lists, jt, keys, bpart, tbits, grp, total;
};
__host__ __device__ inline WalkSmem walk_smem(const WalkPlan& g, int D, bool ea) {
    WalkSmem m;
    const int G = g.GP * g.CPT;
    int o = (G * g.GS * 4 + 15) & ~15;
    m.lists = o;  // undecided sites; after the sweeps the per-replica sums sU, sNup
    // ... and the CTA's level counts where the lattice is small (L = 4, 8 runs of R = 50000,
    // four groups per CTA, where the lists leave no room: 150 us a step of ten sweeps with
    // every replica counted in global memory, 126 with room)
    const int nlev = D * (D == 3 ? g.L * g.L * g.L : g.L * g.L) / 2 + 1;
    const int list = (g.NT / 32) * 32 * g.span * g.CPT * 8;
    const int sums = G * 64 * 4 + (nlev <= 1024 ? nlev * 4 : 0);
    o += ((list > sums ? list : sums) + 15) & ~15;
    m.jt = o;
    if (ea) o += 2 * g.CS;
    o = (o + 15) & ~15;
    m.keys = o;
    o += 2 * G * 2 * 16;
    m.bpart = o;
    o += 2 * 8 * 8 * (g.NT / 32);
    m.tbits = o;
    o += 8 * D * 16;
    m.grp = o;  // per group: A2x, l0a, valid replicas
    o += G * 3 * 4;
    m.total = o;
    return m;
}

// LT: the side at compile time (0: any, from the plan).  At most 512 threads are
// launched; the bound of 640 only caps the registers at 96.
template <int D, int LT, bool EA>
__global__ void __launch_bounds__(640) k_walk(const __grid_constant__ KParams p,
                                              const __grid_constant__ WalkPlan pl,
                                              const uint32_t* cta2run) {
    constexpr bool CT = LT > 0 && D == 3;  // compile-time walk
    const int L = LT ? LT : pl.L, TPR = L / 2;
    const int NC = CT ? TPR * L : pl.NC, H = CT ? L : pl.H, S = CT ? TPR * L : pl.S;
    const int CS = CT ? walk_cs(TPR * L * L) : pl.CS;
    constexpr int U = 2;
    const int N = D == 3 ? L * L * L : L * L;
    const int GP = pl.GP, CPT = pl.CPT, G = GP * CPT;
    extern __shared__ __align__(16) unsigned char smraw[];
    const WalkSmem m = walk_smem(pl, D, EA);
    uint32_t* lat = reinterpret_cast<uint32_t*>(smraw);
    uint8_t* jt = smraw + m.jt;  // bond signs, by the cell index of a group
    uint4* keys = reinterpret_cast<uint4*>(smraw + m.keys);    // [2][G][2] blocks 0, 1
    uint2* bpart = reinterpret_cast<uint2*>(smraw + m.bpart);  // [2][8] (a copy per warp)
    uint4* tbits = reinterpret_cast<uint4*>(smraw + m.tbits);
    uint32_t* sA2x = reinterpret_cast<uint32_t*>(smraw + m.grp);
    uint32_t *sL0a = sA2x + G, *sVm = sL0a + G;
    int32_t* sU = reinterpret_cast<int32_t*>(smraw + m.lists);  // [G][32], after the sweeps
    int32_t* sNup = sU + 32 * G;
    __shared__ uint32_t tail[16];
    __shared__ StepSums sums;

    const RunDesc& r = p.runs[cta2run[blockIdx.x]];
    const DevState* st = r.st;
    chain_wait();
    if (st->status != S_OK) return;
    const int i = st->step;
    const uint32_t R = st->R_cur;
    const uint32_t gfirst = (blockIdx.x - r.cta0) * (uint32_t)G;
    if (gfirst * 32u >= R) return;
    const int gact = (int)min((uint32_t)G, (R - gfirst * 32u + 31u) / 32u);  // groups in use
    const int NT = (int)blockDim.x, NW = NT / 32;
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t* src = r.spins[(i - 1) & 1];
    uint32_t* dst = r.spins[i & 1];
    const uint8_t* jb = r.jbits;
    const int Wp4 = r.Wp / 4, W = r.W;
    auto div_L = [&](int s) -> int {
        return LT ? s / LT : (int)(((uint64_t)(uint32_t)s * pl.mL) >> pl.sL);
    };
    // the cell of site s (colour, row, column) within its group
    auto cell_of = [&](int s) -> int {
        const int q = div_L(s), x = s - q * L;
        if (D == 2) return ((x + q) & 1) * CS + q * S + (x >> 1);
        const int z = div_L(q), y = q - z * L;
        return ((x + y + z) & 1) * CS + z * S + y * TPR + (x >> 1);
    };

    // Philox parts of the step and the groups
    uint32_t B1k, h1a;
    {
        uint32_t l1a;
        mulhilo(PHILOX_M1, (uint32_t)i, h1a, l1a);
        B1k = l1a ^ p.rk0[1];
    }
    for (int g = tid; g < G; g += NT) {
        const uint32_t base = (gfirst + g) * 32u;
        sVm[g] = base + 32u <= R ? 0xFFFFFFFFu : (base < R ? (1u << (R - base)) - 1u : 0u);
        uint32_t h0a, l0a;
        mulhilo(PHILOX_M0, r.grp0 + gfirst + g, h0a, l0a);
        sA2x[g] = h0a ^ p.rk1[0];
        sL0a[g] = l0a;
    }
    Thr<D> th;
#pragma unroll
    for (int a = 0; a < D; ++a) th.t[a] = r.sthr[4 * (i - 1) + 1 + a];
    store_thr_bits<D>(tbits, th);
    const int variant = leading_zeros<D>(th);
    if (tid == 0) clear_sums(&sums);
    // gather the parent rows (the copy of step 2) and transpose them
    const Transposer tr(lane);
#pragma unroll 1
    for (int k = warp; k < gact * Wp4; k += NW) {
        const int g = k / Wp4, c4 = k - g * Wp4;
        const uint32_t slot = (gfirst + g) * 32u + lane;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (slot < R) v = reinterpret_cast<const uint4*>(src + (size_t)r.anc[slot] * r.Wp)[c4];
        const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int s = 32 * (4 * c4 + q) + lane;
            if (4 * c4 + q < W) {  // warp-uniform
                uint32_t t = tr(w4[q]);
                if (s < N) {
                    if (EA) t ^= 0u - ((jb[s] >> 4) & 1u);
                    lat[g * pl.GS + cell_of(s)] = t;
                }
            }
        }
    }
    if (EA) {
        // signs of a site: bit 0 the bond in its own column of the row, bit 1 the one to
        // the side, bits 2, 3 those to y - 1, y + 1 (3D); bits 4, 5 the wrap bonds back
        // (first row) and on (last row)
        for (int s = tid; s < N; s += NT) {
            const int q = div_L(s), x = s - q * L;
            const int z = D == 3 ? div_L(q) : q, y = D == 3 ? q - z * L : q;
            const uint32_t j = jb[s];
            const uint32_t right = (j >> 5) & 1u;
            const uint32_t left = (jb[x == 0 ? s + L - 1 : s - 1] >> 5) & 1u;
            const int e = N / L;  // a row of the walk: L (2D) or L^2 (3D) sites
            const uint32_t back = (jb[z == 0 ? s + (L - 1) * e : s - e] >> (4 + D)) & 1u;
            uint32_t v = ((x & 1) ? left | (right << 1) : right | (left << 1)) | (back << 4) |
                         (((j >> (4 + D)) & 1u) << 5);
            if (D == 3)
                v |= (((uint32_t)jb[y == 0 ? s + (L - 1) * L : s - L] >> 6) & 1u) << 2 |
                     ((j >> 6) & 1u) << 3;
            jt[cell_of(s)] = (uint8_t)v;
        }
    }

    // the thread's column u of set c: group c GP + gl
    const int gl = tid / NC, u = tid - gl * NC;
    const bool in_set = gl < GP;
    const int xi = D == 3 ? u % TPR : u % TPR, yy = D == 3 ? u / TPR : (u / TPR) * H;
    const int col = D == 3 ? u : xi, row0 = D == 3 ? 0 : yy;
    const int dl = xi == 0 ? TPR - 1 : -1, dr = xi == TPR - 1 ? 1 - TPR : 1;
    const int dym = yy == 0 ? (L - 1) * TPR : -TPR, dyp = yy == L - 1 ? (1 - L) * TPR : TPR;
    const uint32_t info = (uint32_t)xi | ((uint32_t)yy << 8) | ((uint32_t)gl << 16);
    const int rowm = (row0 == 0 ? L - 1 : row0 - 1) * S, rowp = (row0 + H == L ? 0 : row0 + H) * S;
    const int LS = D == 3 ? L * L : L;  // sites from row to row
    const uint32_t nh = 2u * r.stheta[i - 1];
    const int QW = 32 * pl.span * CPT;
    uint2* list = reinterpret_cast<uint2*>(smraw + m.lists) + warp * QW;
    const uint32_t list0 = (uint32_t)__cvta_generic_to_shared(list);
    const uint32_t tail_at = (uint32_t)__cvta_generic_to_shared(&tail[warp]);
    if (lane == 0) tail[warp] = list0;
    // the test hook makes the second pass follow every U rows
    const int span = p.qcap_limit >= 0 && p.qcap_limit < QW ? U : pl.span;
    const int csets = (gact + GP - 1) / GP;
    __syncthreads();
    // Groups that lie within a warp (L = 4, 8) need no CTA barrier between half-sweeps:
    // each warp then keeps the keys of its own groups and a block table of its own.
    const bool local = 32 % NC == 0;
    const int gpw = local ? 32 / NC : GP;  // groups of a set that the builders share
    bpart += local ? 16 * warp : 0;
    auto build_keys = [&](uint32_t hh) {
        const int n = 2 * gpw * CPT;
        for (int k = local ? lane : tid; k < 8 + n; k += local ? 32 : NT) {
            const int b = k < 8 ? k : k & 1;
            const uint2 bp = block_part(p, h1a, hh >> 1, hh & 1u, (uint32_t)b);
            if (k < 8) {
                bpart[8 * (hh & 1u) + k] = bp;
            } else {
                const int g = walk_key_group(pl, gpw, local ? warp * gpw : 0, (k - 8) >> 1);
                if (g >= 0) keys[2 * G * (hh & 1u) + 2 * g + b] = block_key_of(p, bp, sL0a[g]);
            }
        }
    };
    if (nh > 0) build_keys(0u);
    __syncthreads();

    uint32_t acc = 0;
    for (uint32_t h = 0; h < nh;) {
    for (const uint32_t h1 = min(nh, h + ACC_SPAN); h < h1; ++h) {
        const uint32_t colour = h & 1u;
        if (h + 1 < nh) build_keys(h + 1);
        const uint32_t par = ((uint32_t)yy + colour) & 1u;  // x parity of the column's first site
        const int da = par ? dr : dl, db = par ? dl : dr;   // side neighbour of even, odd rows
        const uint32_t s0 = (uint32_t)(2 * xi + (D == 3 ? L * yy : 0) + row0 * LS);
        const uint8_t* jc = jt + colour * CS + row0 * S + col;
#pragma unroll 1
        for (int k0 = 0; k0 < H; k0 += span) {
            const int k1 = min(k0 + span, H);
            auto pass1 = [&](auto vtag) {
                constexpr int V = decltype(vtag)::value;
#pragma unroll 1
                for (int c = 0; c < csets; ++c) {
                    const bool act = in_set && c * GP + gl < gact;
                    const int g = act ? c * GP + gl : 0;
                    const uint32_t vmask = act ? sVm[g] : 0u, A2x = sA2x[g];
                    const uint4 e = keys[2 * G * colour + 2 * g], f = keys[2 * G * colour + 2 * g + 1];
                    uint32_t* own = lat + g * pl.GS + colour * CS + row0 * S + col;
                    const uint32_t* oc = lat + g * pl.GS + (colour ^ 1u) * CS + col;
                    const uint32_t* oth = oc + row0 * S;
                    uint32_t prev = k0 == 0 ? oc[rowm] : oth[(k0 - 1) * S], cur = oth[k0 * S];
                    if (EA && k0 == 0) prev ^= 0u - (uint32_t)((jc[0] >> 4) & 1u);
#pragma unroll 1
                    for (int kb = k0; kb < k1; kb += U) {
                        const uint32_t* lastn = kb + U == H ? oc + rowp : oth + (kb + U) * S;
#pragma unroll
                        for (int j0 = 0; j0 < U; j0 += 2) {
                            // two sites at a time, all loads before the stores (the list's
                            // writes would otherwise keep the second site's loads back)
                            uint32_t a[2][6] = {}, w[2], und[2], fl[2];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int j = j0 + q, k = kb + j;
                                uint32_t next = j == U - 1 ? lastn[0] : oth[(k + 1) * S];
                                a[q][2] = cur;
                                a[q][3] = oth[k * S + (q ? db : da)];
                                if (D == 3) {
                                    a[q][4] = oth[k * S + dym];
                                    a[q][5] = oth[k * S + dyp];
                                }
                                w[q] = own[k * S];
                                if (EA) {
                                    const uint32_t jv = jc[k * S], jj = spread_signs(jv);
                                    a[q][2] ^= byte_sign<0>(jj);
                                    a[q][3] ^= byte_sign<1>(jj);
                                    if (D == 3) {
                                        a[q][4] ^= byte_sign<2>(jj);
                                        a[q][5] ^= byte_sign<3>(jj);
                                    }
                                    if (j == U - 1) next ^= 0u - ((jv >> 5) & 1u);
                                }
                                a[q][0] = prev;
                                a[q][1] = next;
                                prev = cur;
                                cur = next;
                            }
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int k = kb + j0 + q;
                                uint32_t two, cm[D];
                                classes<D>(w[q], a[q], two, cm);
                                const uint32_t s = s0 + (uint32_t)(k * LS) + (par ^ (uint32_t)q);
                                const SiteKey sk = site_key(A2x ^ s, B1k);
                                uint32_t uw[8], b, eq;
                                draw_blocks(e, f, sk, p, uw);
                                compare_top<D, V>(cm, tbits, uw, b, eq);
                                und[q] = lop3<0x20>(eq, two, vmask);  // eq & ~two & vmask
                                fl[q] = (two | b) & vmask;            // b = 0 where undecided
                            }
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int k = kb + j0 + q;
                                if (act) own[k * S] = w[q] ^ fl[q];
                                acc += (uint32_t)__popc(fl[q]);
                                push_undecided(tail_at, und[q], (uint32_t)((k << 5) + lane + (c << 16)));
                            }
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
                const uint32_t inf = __shfl_sync(0xFFFFFFFFu, info, (int)(en.x & 31u));
                const int k = (int)((en.x >> 5) & 255u);
                const int x2 = (int)(inf & 255u), y2 = (int)((inf >> 8) & 255u);
                const int g2 = (int)(en.x >> 16) * GP + (int)(inf >> 16);
                const int row = D == 3 ? k : y2 + k, c2 = D == 3 ? y2 * TPR + x2 : x2;
                const uint32_t pr = (uint32_t)(y2 + k + (int)colour) & 1u;
                const int xs = pr ? (x2 == TPR - 1 ? 1 - TPR : 1) : (x2 == 0 ? TPR - 1 : -1);
                uint32_t* aw = lat + g2 * pl.GS + colour * CS + row * S + c2;
                const uint32_t* o = lat + g2 * pl.GS + (colour ^ 1u) * CS + c2;
                uint32_t a[6] = {};
                a[0] = o[(row == 0 ? L - 1 : row - 1) * S];
                a[1] = o[(row == L - 1 ? 0 : row + 1) * S];
                a[2] = o[row * S];
                a[3] = o[row * S + xs];
                if (D == 3) {
                    a[4] = o[row * S + (y2 == 0 ? (L - 1) * TPR : -TPR)];
                    a[5] = o[row * S + (y2 == L - 1 ? (1 - L) * TPR : TPR)];
                }
                const uint32_t w = *aw;
                if (EA) {
                    const uint32_t jv = jt[colour * CS + row * S + c2], jj = spread_signs(jv);
                    a[0] ^= 0u - ((jv >> 4) & 1u);
                    a[1] ^= 0u - ((jv >> 5) & 1u);
                    a[2] ^= byte_sign<0>(jj);
                    a[3] ^= byte_sign<1>(jj);
                    if (D == 3) {
                        a[4] ^= byte_sign<2>(jj);
                        a[5] ^= byte_sign<3>(jj);
                    }
                }
                uint32_t two, cm[D];
                classes<D>(w, a, two, cm);
                const uint32_t s = (uint32_t)(2 * x2 + (D == 3 ? L * y2 : 0) + row * LS) + pr;
                const uint32_t l0a = sL0a[g2];
                const uint32_t lt = finish_site<D>(
                    cm, tbits, have ? en.y : 0u, site_key(sA2x[g2] ^ s, B1k),
                    [&](int g) { return block_key_of(p, bpart[8 * colour + g], l0a); }, p);
                if (have) *aw = w ^ lt;
                acc += (uint32_t)__popc(lt);
            }
            __syncwarp();
        }
        if (local) __syncwarp();
        else __syncthreads();
    }
    add_accepts(&sums.acc, acc, lane);
    acc = 0;
    }
    __syncthreads();

    // Measurement.  Unsatisfied bonds: every bond has one end of colour 0, so the
    // threads walk their columns of colour 0 once and count all bonds of its sites in
    // bit-sliced counters; per plane one transpose gives each replica its lanes' bits.
    uint32_t* shist = reinterpret_cast<uint32_t*>(sU + 64 * G);  // level counts, where they fit
    const int hist_room = (m.jt - m.lists) / 4 - 64 * G;
    for (int k = tid; k < (m.jt - m.lists) / 4; k += NT) sU[k] = 0;
    __syncthreads();
    {
        constexpr int CB = D == 3 ? (LT ? vc_bits(6 * LT) : 8) : 10;
        const int gw0 = warp * 32 / NC, gw1 = min((warp * 32 + 31) / NC, GP - 1);
        const uint32_t par = (uint32_t)yy & 1u;
        const int da = par ? dr : dl, db = par ? dl : dr;
        const uint8_t* jc = jt + row0 * S + col;
#pragma unroll 1
        for (int c = 0; c < csets; ++c) {
            const bool act = in_set && c * GP + gl < gact;
            const int g = act ? c * GP + gl : 0;
            const uint32_t* own = lat + g * pl.GS + row0 * S + col;
            const uint32_t* oc = lat + g * pl.GS + CS + col;
            const uint32_t* oth = oc + row0 * S;
            uint32_t cnt[CB];
#pragma unroll
            for (int j = 0; j < CB; ++j) cnt[j] = 0u;
            uint32_t prev = oc[rowm], cur = oth[0];
            if (act) {
#pragma unroll 1
                for (int k = 0; k < H; ++k) {
                    uint32_t next = k == H - 1 ? oc[rowp] : oth[(k + 1) * S];
                    uint32_t a[6] = {prev, next, cur, oth[k * S + ((k & 1) ? db : da)], 0u, 0u};
                    if (D == 3) {
                        a[4] = oth[k * S + dym];
                        a[5] = oth[k * S + dyp];
                    }
                    const uint32_t w = own[k * S];
                    if (EA) {
                        const uint32_t jv = jc[k * S], jj = spread_signs(jv);
                        a[0] ^= 0u - ((jv >> 4) & 1u);
                        a[1] ^= 0u - ((jv >> 5) & 1u);
                        a[2] ^= byte_sign<0>(jj);
                        a[3] ^= byte_sign<1>(jj);
                        if (D == 3) {
                            a[4] ^= byte_sign<2>(jj);
                            a[5] ^= byte_sign<3>(jj);
                        }
                    }
                    prev = cur;
                    cur = next;
                    const uint32_t t0 = csa(cnt[0], w ^ a[0], w ^ a[1]);
                    const uint32_t t1 = csa(cnt[0], w ^ a[2], w ^ a[3]);
                    uint32_t carry = csa(cnt[1], t0, t1);
                    if (D == 3) {
                        const uint32_t t2 = csa(cnt[0], w ^ a[4], w ^ a[5]);
                        const uint32_t k2 = cnt[1] & t2;
                        cnt[1] ^= t2;
                        carry = csa(cnt[2], carry, k2);
                    } else {
                        const uint32_t k2 = cnt[2] & carry;
                        cnt[2] ^= carry;
                        carry = k2;
                    }
#pragma unroll
                    for (int j = 3; j < CB; ++j) {
                        const uint32_t t = cnt[j] & carry;
                        cnt[j] ^= carry;
                        carry = t;
                    }
                }
            }
            uint32_t T[CB];
#pragma unroll
            for (int j = 0; j < CB; ++j) T[j] = tr(cnt[j]);
            for (int gg = gw0; gg <= gw1; ++gg) {  // the groups that have lanes in this warp
                const int b0 = max(gg * NC - warp * 32, 0), b1 = min((gg + 1) * NC - warp * 32, 32);
                const uint32_t mask = (b1 == 32 ? 0xFFFFFFFFu : (1u << b1) - 1u) & (0xFFFFFFFFu << b0);
                int32_t Uw = 0;
#pragma unroll
                for (int j = 0; j < CB; ++j) Uw += __popc(T[j] & mask) << j;
                if (c * GP + gg < gact) atomicAdd(&sU[32 * (c * GP + gg) + lane], Uw);
            }
        }
    }
    // write the rows back
#pragma unroll 1
    for (int k = warp; k < gact * Wp4; k += NW) {
        const int g = k / Wp4, c4 = k - g * Wp4;
        uint32_t out[4];
        int32_t nup = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int s = 32 * (4 * c4 + q) + lane;
            out[q] = 0u;
            if (4 * c4 + q < W) {  // warp-uniform
                uint32_t w = 0u;
                if (s < N) {
                    w = lat[g * pl.GS + cell_of(s)];
                    if (EA) w ^= 0u - ((jb[s] >> 4) & 1u);
                }
                out[q] = tr(w);
                nup += __popc(out[q]);
            }
        }
        const uint32_t slot = (gfirst + g) * 32u + lane;
        if (slot < R)
            reinterpret_cast<uint4*>(dst + (size_t)slot * r.Wp)[c4] =
                make_uint4(out[0], out[1], out[2], out[3]);
        atomicAdd(&sNup[32 * g + lane], nup);
    }
    __syncthreads();

    // a small lattice's levels are counted in the CTA first
    const bool hist_sm = r.nlev <= hist_room;
    LaneSums ls;
    for (int g = warp; g < gact; g += NW) {
        const uint32_t slot = (gfirst + g) * 32u + lane;
        if (slot < R) {
            const int32_t Uv = sU[32 * g + lane];
            const int32_t E = 2 * Uv - D * N;
            const int32_t M = N - 2 * sNup[32 * g + lane];
            r.E[i & 1][slot] = E;
            r.M[slot] = M;
            atomicAdd(hist_sm ? &shist[Uv >> 1] : &r.hist[Uv >> 1], 1u);
            ls.add(E, M, Uv >> 1);
        }
    }
    ls.to_cta(&sums, lane);
    __syncthreads();
    if (hist_sm)
        for (int l = (sums.hi < 0 ? 0 : sums.lo) + tid; l <= sums.hi; l += NT)
            if (shist[l]) atomicAdd(&r.hist[l], shist[l]);
    add_to_trace(sums, r, i);
}

constexpr int WALK_SMEM_MAX = 227 * 1024 - 1024;

template <int D, int LT, bool EA>
cudaError_t launch_walk_t(const KParams& p, const WalkPlan& g, const uint32_t* cta2run,
                          uint32_t ncta, cudaStream_t s, bool attr_only, bool chain) {
    const cudaError_t e = cudaFuncSetAttribute(
        k_walk<D, LT, EA>, cudaFuncAttributeMaxDynamicSharedMemorySize, WALK_SMEM_MAX);
    if (e != cudaSuccess || attr_only || ncta == 0) return e;
    return launch_chained(chain, k_walk<D, LT, EA>, ncta, (unsigned)g.NT,
                          (size_t)walk_smem(g, D, EA).total, s, p, g, cta2run);
}

template <bool EA>
cudaError_t launch_walk_ea(const KParams& p, const WalkPlan& g, const uint32_t* cta2run,
                           uint32_t ncta, cudaStream_t s, bool attr_only, bool chain) {
    if (p.d == 2) return launch_walk_t<2, 0, EA>(p, g, cta2run, ncta, s, attr_only, chain);
    switch (g.L) {
        case 4: return launch_walk_t<3, 4, EA>(p, g, cta2run, ncta, s, attr_only, chain);
        case 6: return launch_walk_t<3, 6, EA>(p, g, cta2run, ncta, s, attr_only, chain);
        case 8: return launch_walk_t<3, 8, EA>(p, g, cta2run, ncta, s, attr_only, chain);
        default: return launch_walk_t<3, 0, EA>(p, g, cta2run, ncta, s, attr_only, chain);
    }
}

// the plan's strides for its columns, groups, sets and span; returns its shared memory
int finish_plan(WalkPlan& g, int d, bool ea) {
    const int L = g.L, TPR = L / 2;
    g.NT = (g.GP * g.NC + 31) / 32 * 32;
    auto size = [&](int S) {
        g.S = S;
        g.CS = walk_cs(L * S);
        g.GS = 2 * g.CS + ((g.NC - 2 * g.CS) % 32 + 32) % 32;
        return walk_smem(g, d, ea).total;
    };
    // 2D chunks of a warp on distinct banks, where a stride does it and there is room
    int S = d == 3 ? TPR * L : TPR;
    if (d == 2 && g.NC > TPR)
        for (int t = TPR; t < TPR + 32; ++t)
            if ((g.H * t) % 32 == TPR % 32) {
                if (size(t) <= WALK_SMEM_MAX) S = t;
                break;
            }
    return size(S);
}

}  // namespace

// The walk's geometry for the runs of side L of a context: ngrp replica groups in all,
// at most most_grp in one run; threads per group wanted (0: the rule's own choice); general:
// the threads k_group would have.  The least sweep_time() of the plans that fit:
//  - columns: 3D all L^2/2 of a group; 2D L/2 times the number of chunks, a divisor of L
//    with an even chunk height (a wish takes the most columns that stay within `threads`);
//  - groups side by side, up to about 320 threads, and sets of them, up to about 14 rows per
//    thread between two second passes (a small lattice's column has 4 to 8; L = 4: up to 2
//    sets, more cost residency); gm doubles the sets;
//  - the span, rows between two second passes: the list takes 8 bytes for every site of a span,
//    the lattice 4 for every site, so a long column's list costs CTAs of an SM.
WalkPlan walk_plan(int d, int L, bool ea, uint32_t ngrp, uint32_t most_grp, int threads, int general, int gm) {
    WalkPlan g;
    std::memset(&g, 0, sizeof(g));
    const int TPR = L / 2;
    constexpr int regs = 96;
    g.L = L;
    if (d == 3 && (g.flat = sweep3d_groups(L, gm)) > 0) {  // pa_sweep3d.cu takes these sides
        g.GP = g.flat;
        g.CPT = 1;
        return g;
    }
    WalkPlan best = g;
    double least = 1e30;
    auto columns = [&](int n) {
        g.NC = d == 3 ? TPR * L : TPR * n;
        g.H = d == 3 ? L : L / n;
    };
    auto consider = [&](int gp, int cpt) {
        g.GP = gp;
        g.CPT = cpt * gm;
        for (g.span = g.H;; g.span = (g.span / 2 + 1) & ~1) {
            const int sm = finish_plan(g, d, ea);
            if (sm <= WALK_SMEM_MAX) {
                const int rows = g.H / ((g.H + g.span - 1) / g.span) * cpt;
                const double t = sweep_time(rows, ngrp, gp, g.NC, regs, cpt, (size_t)sm, 1.15);
                if (t < least - 1e-9) {
                    least = t;
                    best = g;
                }
            }
            if (g.span <= 4) break;
        }
    };
    // all that fit beside each other, with every number of sets
    auto consider_all = [&](int widest) {
        const int most = std::min<int>((int)std::min<uint32_t>(most_grp, 512u), 512 / g.NC);
        const int sets = L == 4 && d == 3 ? 2 : std::max(1, (14 + g.H / 2) / g.H);
        for (int cpt = 1; cpt <= sets; ++cpt)
            for (int gp = 1; gp == 1 || (gp <= most && (d == 3 || gp <= 16) && gp * g.NC <= widest); ++gp) consider(gp, cpt);
    };
    if (d == 3) {
        columns(1);
        consider_all(352);
    } else {
        int wish = 1;
        for (int n = 1; n <= L / 2 && TPR * n <= 512; ++n) {
            if (L % n != 0 || (L / n) % 2 != 0) continue;
            if (threads > 0) {
                if (TPR * n <= threads) wish = n;
                continue;
            }
            columns(n);
            consider_all(320);
        }
        if (threads > 0) {
            columns(wish);
            consider_all(352);
        }
    }
    // The general kernel where it is faster: sides whose divisors leave few columns (twice a
    // prime has L/2 of all rows, or of two rows each) and few groups of any side without a good
    // split; columns of two or four rows cost 1.45 and 1.15 times what sweep_time() says, and the
    // tiniest lattices' line stands at 1536 groups.  One run, us a step with k_group and with the
    // walk: L = 58, 32 groups 95, 327; L = 24, 141 groups 43, 47, 1563 groups 142, 131; L = 8, 32
    // groups 27, 45, 4688 groups 120, 72; 3D L = 2, 32 groups 26, 67, 4688 groups 124, 78.  Over
    // all those runs the choice costs 0.5%, 13% at most (always the walk: 18% and 275%).
    g = best;
    const double few = g.H == 2 ? 1.45 : g.H == 4 ? 1.15 : 1.0;
    if (d == 2 && L > 8 ? few * least > group_time(d, L * L, ea, ngrp, general)
                        : L <= (d == 2 ? 8 : 2) && ngrp < 1536) {
        g.flat = -1;
        g.GP = g.CPT = 1;
        return g;
    }
    // division by L: (s m) >> sh is exact for s < 2^15 (L <= 180) with sh = 24
    g.sL = 24;
    g.mL = (uint32_t)(((1u << 24) + (uint32_t)L - 1u) / (uint32_t)L);
    return g;
}

// One launch of the walk over the CTAs of the runs of one side (cta2run: their run
// indices, device memory).  attr_only: function attributes only (before a capture).
cudaError_t launch_walk(const KParams& p, const WalkPlan& g, const uint32_t* cta2run, uint32_t ncta,
                        cudaStream_t s, bool attr_only, bool chain) {
    if (g.flat) return launch_sweep3d(p, g.L, g.GP, cta2run, ncta, s, attr_only);
    return p.ea ? launch_walk_ea<true>(p, g, cta2run, ncta, s, attr_only, chain)
                : launch_walk_ea<false>(p, g, cta2run, ncta, s, attr_only, chain);
}

}  // namespace pa
