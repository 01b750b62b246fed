// Step 3 of Algorithm 3 under the static screen on the tensor cores (tcgen05), by sibling
// groups: the pieces and factored sums of apply_oct.cu, k <= 8 (lower orders zero-padded
// to 8), FP16 hi + lo operands as in apply_tc.cu (hi*hi + hi*lo + lo*hi into FP32).
//
// A work unit is one group and one chunk of up to 8 pieces.  Per plane b3 and pair of lines
// (b2, b2 + 1):
//   stage I   D_I[(line, i3, i2)][(a1, piece, c1)] = X F^{t1}: M = 128, N = 128 (64 for at
//             most 4 pieces), K = 16 per pair of input boxes b1;
//   stage II  per piece V[(a1, c1, i3)][(a2, hi or lo, c2)] += W [F_hi^{t2} | F_lo^{t2}] for W hi and
//             W lo: M = 128, N = 32, K = 16 (two lines of i2), accumulated over the plane's lines;
//             the two products are added when V is converted;
//   stage III per piece, plane and a2, Y[(a1, c1, c2)][(a3, c3)] = V F^{t3}: M = 128, N = 16,
//             K = 16 (i3 as hi | lo), read out after the plane and summed over the planes and
//             the chunk's pieces in FP32 registers.  (Summing in the tensor core's accumulator
//             instead truncates at every addition: the hydrogen energy then moves by 7e-7.)
// Every B operand is read in place from the chunk's F tiles: with u = b - a + 1 the tile of
// t = 3 - u serves output a and input b, so (a, b) neighbours are tile neighbours and one
// descriptor (constant strides) covers both outputs and both boxes; a piece's excluded
// translations are zero tiles.
//
// One persistent CTA per SM (216 KB of shared memory, all 512 TMEM columns), 28 warps with roles
// that meet at mbarriers only, so that setting up units, loading, MMAs and conversions overlap:
//   0-15   convert accumulators to the next stage's operands, a pair of pieces per four warps;
//   16-19  load X (two buffers; the blocks' power-of-two scales are made equal on the way);
//   20-23  issue stages II and III of a pair each;
//   24     issues stage I into one of two accumulators;
//   25-27  set up the next unit (pieces, inputs, scales, F tiles) in the other of two slots.
// A warp waits for itself: meeting at a named barrier behind one polling warp cost a conversion 200
// to 300 cycles.  What bounds the kernel is shared memory, 75 % busy (half of it the tensor core's: an
// MMA of stage II or III reads 4 KB of A for 32 or 16 columns), and issue slots, 59 %: the conversions'
// share of them is why scaling and splitting use two-lane FP32.  3-D Poisson k = 8: 0.78 ms; 0.93 ms
// with F_hi and F_lo as products of their own and barriers; 1.38 ms in the version whose units were set
// up and finished by the whole CTA.  Stage I in halves of 4 pieces, or pieces instead of pairs as
// the grain of conversions and MMAs, lose (0.86 and 1.07 ms): A is read or waited for twice.
// Planes and pairs of lines without an input box (outside the cube, or not needed) are passed over: a
// replayed plan of one box at k = 8 takes 45 us, 75 with them.
// Every wait is bounded: one that reaches its limit makes all roles stop, the error word is set
// to 4, what was sent ends, and the kernel frees its tensor memory.
#include <cfloat>
#include <climits>

#include "apply_common.cuh"
#include "oct_pieces.cuh"
#include "tc_ptx.cuh"

namespace mra {

#define OTC_THREADS 896
#define OTC_SETUP 96  // threads that set up units
#define OTC_P 8  // pieces per chunk

struct OtcSmem {
    static constexpr int XBUF = 24576;                 // hi then lo: [box b1 6][line 2] x 1 KB
    static constexpr int X = 0;                        // two buffers
    static constexpr int A2_LBO = 2304, A2_SBO = 144;  // 8 x 16-byte core matrices, 16 bytes apart (bank spread)
    static constexpr int A2_PIECE = 4 * A2_LBO;        // stage II: hi, lo (2 K groups each); stage III: a2' = 0, 1
    static constexpr int A2 = X + 2 * XBUF;
    static constexpr int TAB = 7 * OTC_P * 128;        // hi or lo tiles of a direction
    // per slot and direction: tiles [hi, lo][u 0..6][position], direction 2 [u][hi, lo][position]
    static constexpr int T = A2 + OTC_P * A2_PIECE;
    static constexpr int Z = T + 12 * TAB;             // zeros: two tiles a tile row apart
    static constexpr int TIN = Z + OTC_P * 128 + 128;          // per slot 216 int
    static constexpr int TG = TIN + 2 * 864;           // per slot 216 float
    static constexpr int LIST = TG + 2 * 864;          // pieces of the group being set up
    static size_t bytes(int M) { return LIST + OCT_TERM_PIECES * (size_t)M * sizeof(uint32_t); }
};
static_assert(OtcSmem::LIST + OCT_TERM_PIECES * MRA_MAX_TERMS * 4 + 2048 <= 232448, "shared memory of one CTA");

// a unit as its roles see it
struct OtcUnit {
    int unit;            // -1: no more units
    int npc, ps;         // pieces; positions (4 or 8) of a tile row
    int s1, s2;          // first box of the pieces' pairs of boxes per direction: 0, or 1 (core sets only)
    unsigned m1, m2, m3; // boxes the pieces read, per direction, where the group has inputs
    int nout;
    unsigned leaf;       // leaf outputs
    uint32_t piece[OTC_P];
    float c2[OTC_P], c3[OTC_P], fin[OTC_P];
};

// Pieces i and i + 4 of a unit are pair i's (up to four pieces are one each for the pairs), neighbours
// in the tile rows: position 2 i + r of 8, i of 4.
__device__ __forceinline__ int otc_pieces(int g, int npc) { return (g < npc) + (g + 4 < npc); }

// c x[0..3] (c a power of two) as FP16 hi and lo pairs: hi01, lo01, hi23, lo23
__device__ __forceinline__ void split_scaled(const float* x, float c, uint32_t* w) {
    tc::split_scaled_h2(x[0], x[1], c, w[0], w[1]);
    tc::split_scaled_h2(x[2], x[3], c, w[2], w[3]);
}

__global__ void __launch_bounds__(OTC_THREADS, 1) k_apply_oct_tc(OctTcArgs Q) {
    using L = OtcSmem;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ uint32_t s_tmem;
    // X full / empty, D_I full / empty; per pair: operands full, MMAs done; per slot: set up, done with;
    // the pairs' sums written, read; the issuing warps' MMAs done (after a wait that gave up)
    __shared__ __align__(8) uint64_t b_xf[2], b_xe[2], b_df[2], b_de[2], b_af[4], b_ae[4], b_sf[2], b_se[2], b_y, b_yr, b_end[5];
    __shared__ volatile int s_abort;
    __shared__ int s_unit, s_emin;
    __shared__ unsigned s_xmax, s_there, s_reads;  // (boxes of directions 1, 2, 3 in bytes 0, 1, 2)
    __shared__ OtcUnit s_u[2];
    const OctArgs& P = Q.P;
    if (P.skip && *P.skip != P.run_if) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = tc::smem_u32(sm);
    for (int e = tid; e < L::TIN / 16; e += OTC_THREADS) ((uint4*)sm)[e] = make_uint4(0, 0, 0, 0);
    if (warp == 0) tc::tmem_alloc(&s_tmem, 512);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&b_xf[i], 4);
            tc::mbar_init(&b_xe[i], 1);
            tc::mbar_init(&b_df[i], 1);
            tc::mbar_init(&b_de[i], 16);
            tc::mbar_init(&b_sf[i], OTC_SETUP / 32);
            tc::mbar_init(&b_se[i], 4 + 16 + 5);
        }
        tc::mbar_init(&b_y, 16);
        tc::mbar_init(&b_yr, 16);
        for (int i = 0; i < 5; ++i) tc::mbar_init(&b_end[i], 1);
        for (int i = 0; i < 4; ++i) {
            tc::mbar_init(&b_af[i], 4);
            tc::mbar_init(&b_ae[i], 1);
        }
        s_abort = 0;
    }
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = (uint32_t)tc::uniform((int)s_tmem);
    // TMEM columns: D_I 2 x 128; per piece 32: D_II (a2', product with hi or lo, c2), then D_III 2 a2' x 16
    auto cII = [&](int g, int r) { return tbase + 256u + (uint32_t)(g * 64 + r * 32); };
    auto cIII = [&](int g, int r, int a) { return cII(g, r) + (uint32_t)(a * 16); };
#define OTC_WAIT(bar, parity) tc::mbar_wait_or(bar, parity, Q.wait_limit, &s_abort)
    // waits by a whole warp, whose lanes go on or give up together (what follows is warp-collective)
#define OTC_ALL(expr) __all_sync(0xffffffffu, expr)
#define OTC_WAITW(bar, parity) OTC_ALL(OTC_WAIT(bar, parity))
    // barriers complete once per use; a use's parity is its running number's lowest bit
    uint32_t ln = 0;  // lines (pairs of boxes b2) so far

    // registers by warpgroup: 896 threads x 72 at launch = 512 x 80 + 128 x (72 + 48 + 64)
    if (warp >= 24) {
        tc::reg_dec<64>();
        if (warp > 24) {
        // ================= set up units
        const int t = tid - 800;
        uint32_t* list = (uint32_t*)(sm + L::LIST);
        auto sync = [] { asm volatile("bar.sync 1, 96;" ::: "memory"); };
        for (uint32_t k = 0;; ++k) {
            const int slot = k & 1;
            const bool ok = k < 2 || t != 0 || tc::mbar_wait_or(&b_se[slot], ((k >> 1) - 1) & 1, Q.wait_limit, &s_abort, 500);
            OtcUnit& U = s_u[slot];
            int* tin = (int*)(sm + L::TIN + slot * 864);
            float* tg = (float*)(sm + L::TG + slot * 864);
            int unit, g, np, q0;
            for (;;) {  // the next unit that has pieces and inputs (one without inputs is zero)
                if (t == 0) {
                    int u = ok ? atomicAdd(Q.counter, 1) : Q.nunits;
                    while (u < Q.nunits && (u % P.ns) * OTC_P >= P.np[P.g0 + u / P.ns]) u = atomicAdd(Q.counter, 1);
                    s_unit = u;
                    s_emin = INT_MAX;
                    s_xmax = 0u;
                    s_there = 0u;
                }
                sync();
                unit = s_unit;
                if (unit >= Q.nunits) break;
                g = P.g0 + unit / P.ns;
                q0 = (unit % P.ns) * OTC_P;
                np = P.np[g];
                const int i0 = P.first[g], j = P.coord[4 * i0], nout = j ? 8 : 1;
                const size_t fb = (size_t)j * P.M;
                int in[3] = {-1, -1, -1};
                float sx[3] = {1.0f, 1.0f, 1.0f};
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    if (t + OTC_SETUP * r < 216) in[r] = P.in[(size_t)g * 216 + t + OTC_SETUP * r];
                unsigned there = 0u;
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    if (in[r] >= 0) {
                        sx[r] = Q.sx[in[r]];
                        int e;
                        frexpf(sx[r], &e);
                        atomicMin(&s_emin, e);
                        atomicMax(&s_xmax, __float_as_uint(Q.xmax[in[r]]));  // non-negative floats order as ints
                        const int q = t + OTC_SETUP * r;
                        there |= 1u << (q / 36) | 256u << ((q / 6) % 6) | 65536u << (q % 6);
                    }
                there = __reduce_or_sync(0xffffffffu, there);
                if (lane == 0) atomicOr(&s_there, there);
                if (warp == 25) {
                    const unsigned lf = __ballot_sync(0xffffffffu, lane < nout && P.leaf[i0 + (lane < nout ? lane : 0)]);
                    const int tree = P.node_tree ? P.node_tree[i0] : 0;
                    oct_pieces(P.sched + (size_t)tree * P.sl, P.M, P.lm, j, lf != 0, lf != (1u << nout) - 1u, list);
                    __syncwarp();
                    const int npc = min(OTC_P, np - q0);
                    unsigned m1 = 0, m2 = 0, m3 = 0;
                    for (int pc = 0; pc < npc; ++pc) {
                        const uint32_t p = list[q0 + pc];
                        m1 |= set_boxes((p >> 20) & 3);
                        m2 |= set_boxes((p >> 18) & 3);
                        m3 |= set_boxes((p >> 16) & 3);
                    }
                    if (lane < OTC_P) U.piece[lane] = lane < npc ? list[q0 + lane] : 0u;
                    if (lane == 0) {
                        U.unit = unit;
                        U.npc = npc;
                        U.ps = npc <= 4 ? 4 : 8;
                        U.s1 = m1 == 0x1e;
                        U.s2 = m2 == 0x1e;
                        U.nout = nout;
                        U.leaf = lf;
                        s_reads = m1 | m2 << 8 | m3 << 16;
                    }
                }
                sync();
                const float xmax = __uint_as_float(s_xmax);
                const int es = s_emin - 1;  // the common scale 2^es
                if (!(xmax <= FLT_MAX) && t == 0) atomicExch(Q.err, 5);  // input values beyond FP32's range
                // (boxes that only other chunks' pieces read do not count; planes and pairs of lines without
                // an input are passed over by all roles)
                const unsigned m = s_reads & s_there, m1 = m & 0xffu, m2 = (m >> 8) & 0xffu, m3 = m >> 16;
                if (!(xmax > 0.0f && xmax <= FLT_MAX) || !m1 || !m2 || !m3) {
                    const int k3 = P.k * P.k * P.k;
                    for (int e = t; e < nout * k3; e += OTC_SETUP) ((float*)Q.part)[(size_t)unit * 8 * k3 + e] = 0.0f;
                    sync();
                    continue;
                }
                if (t == 0) {
                    U.m1 = m1;
                    U.m2 = m2;
                    U.m3 = m3;
                }
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    if (t + OTC_SETUP * r < 216) {
                        tin[t + OTC_SETUP * r] = in[r];
                        tg[t + OTC_SETUP * r] = in[r] < 0 ? 0.0f : ldexpf(1.0f, es) / sx[r];
                    }
                // F tiles, masked by the pieces' sets; a lane copies 16 bytes of a position, a warp the 7
                // tiles of 4 positions of a (direction, hi or lo) at once, all loads in flight
                const int v = lane & 7, ps = U.ps;
                for (int r = warp - 25; r < 3 * ps / 2; r += OTC_SETUP / 32) {
                    const int dh = ps == 8 ? r >> 1 : r, pos = (lane >> 3) + (ps == 8 ? 4 * (r & 1) : 0);
                    const uint32_t p = U.piece[ps == 8 ? (pos >> 1) + 4 * (pos & 1) : pos];  // (0 beyond the last: the empty set)
                    const int set = (p >> (20 - 2 * (dh >> 1))) & 3;
                    const uint4* src = (const uint4*)((dh & 1) ? Q.Fl : Q.Fh) + ((fb + (p & 0xffff)) * 7 + 6) * 8 + v;
                    uint4 x[7];
#pragma unroll
                    for (int u = 0; u < 7; ++u)
                        x[u] = set & ((u >= 2 && u <= 4) ? 1 : 2) ? __ldg(src - u * 8) : make_uint4(0, 0, 0, 0);
                    const bool mixed = (dh >> 1) == 1;
                    uint4* dst = (uint4*)(sm + L::T + slot * 6 * L::TAB + (dh >> 1) * 2 * L::TAB) +
                                 ((dh & 1) * (mixed ? ps : 7 * OTC_P) + pos) * 8 + v;
                    const int row = (mixed ? 2 : 1) * ps * 8;
#pragma unroll
                    for (int u = 0; u < 7; ++u) dst[u * row] = x[u];
                }
                // power-of-two scales as in apply_tc.cu: sW = 2^eW, the largest power of two <=
                // 8192 / (48 max|F| max|x|), and sV = 2^eV <= 8192 / (48^2 max|F|^2 max|x|)
                if (t < OTC_P) {
                    float c2 = 0.0f, c3 = 0.0f, fin = 0.0f;
                    if (t < U.npc) {
                        const int m = U.piece[t] & 0xffff;
                        const float mf = Q.maxF[fb + m], sf = Q.sF[fb + m];
                        if (mf > 0.0f) {
                            int em, ex, ef, e1, e2;
                            const float fm = frexpf(mf, &em), fx = frexpf(xmax, &ex);
                            frexpf(sf, &ef);
                            ef -= 1;
                            frexpf(8192.0f / (48.0f * fm * fx), &e1);
                            frexpf(8192.0f / (2304.0f * fm * fm * fx), &e2);
                            const int eW = min(e1 - 1 - em - ex, 126), eV = min(e2 - 1 - 2 * em - ex, 126);
                            // (sW and sV themselves may pass FP32's range where the factors do not)
                            const int a2 = eW - ef - es, a3 = eV - eW - ef;
                            c2 = ldexpf(1.0f, a2);                  // sW / (sF sx)
                            c3 = ldexpf(1.0f, a3);                  // sV / (sW sF)
                            fin = ldexpf((float)P.w[m], -(eV + ef));  // w_m / (sV sF)
                            if (min(a2, a3) < -126 || !(fin <= FLT_MAX)) {  // scales or outputs beyond the FP32 range: refuse
                                atomicExch(Q.err, 5);
                                fin = 0.0f;
                            }
                        }
                    }
                    U.c2[t] = c2;
                    U.c3[t] = c3;
                    U.fin[t] = fin;
                }
                break;
            }
            if (unit >= Q.nunits && t == 0) U.unit = -1;
            tc::fence_async_smem();
            tc::mbar_arrive_warp(&b_sf[slot]);
            if (unit >= Q.nunits) break;
            sync();  // s_unit and the scale words are free again
        }
        } else {
        // ================= stage I
        if (!Q.withhold) {
            bool ok = true;
            for (uint32_t k = 0; ok; ++k) {
                const int slot = k & 1;
                ok = OTC_WAITW(&b_sf[slot], (k >> 1) & 1);
                if (!ok || tc::uniform(s_u[slot].unit) < 0) break;
                const unsigned m2 = tc::uniform(s_u[slot].m2), m3 = tc::uniform(s_u[slot].m3);
                const int s1 = tc::uniform(s_u[slot].s1), s2 = tc::uniform(s_u[slot].s2), n1 = 3 - s1, n2 = 3 - s2;
                const int ps = tc::uniform(s_u[slot].ps);
                const uint32_t id = tc::idesc_f16(128, 16 * ps);
                const uint64_t th = tc::sdesc(sbase + L::T + slot * 6 * L::TAB + s1 * ps * 128, ps * 128, 128);
                int lines = 0;
                for (int q = 0; q < n2; ++q) lines += ((m2 >> (s2 + 2 * q)) & 3u) != 0;
                lines *= __popc(m3);
                for (int l = 0; l < lines && ok; ++l, ++ln) {
                    const int buf = ln & 1;
                    ok = OTC_WAITW(&b_xf[buf], (ln >> 1) & 1) && (ln < 2 || OTC_WAITW(&b_de[buf], ((ln >> 1) - 1) & 1));
                    if (!ok) break;
                    tc::fence_after();
                    const uint32_t d = tbase + buf * 128;
                    const uint64_t xh = tc::sdesc(sbase + L::X + buf * L::XBUF, 2048, 128);
#pragma unroll
                    for (int s = 0; s < 3; ++s) {  // boxes s1 + 2 s, + 1
                        if (s >= n1) break;
                        const uint64_t ah = xh + (uint64_t)(s * (4096 / 16)), al = ah + L::XBUF / 32;
                        const uint64_t bh = th + (uint64_t)(s * 2 * ps * 8), bl = bh + L::TAB / 16;
                        tc::mma_f16_warp(d, ah, bh, id, s > 0);
                        tc::mma_f16_warp(d, ah, bl, id, 1);
                        tc::mma_f16_warp(d, al, bh, id, 1);
                    }
                    tc::commit_warp(&b_xe[buf]);
                    tc::commit_warp(&b_df[buf]);
                }
                tc::commit_warp(&b_se[slot]);
            }
        }
        }
    } else if (warp >= 16 && warp < 20) {
        // ================= X of a pair of lines into a buffer
        const int lt = tid - 512, hl = lt >> 6, v = lt & 63;
        const uint4* src0 = (const uint4*)(hl ? Q.xl : Q.xh) + v;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            const int slot = k & 1;
            ok = OTC_WAITW(&b_sf[slot], (k >> 1) & 1);
            if (!ok || s_u[slot].unit < 0) break;
            const unsigned m1 = s_u[slot].m1, m2 = s_u[slot].m2, m3 = s_u[slot].m3;
            const int s1 = s_u[slot].s1, s2 = s_u[slot].s2, n1 = 3 - s1, n2 = 3 - s2;
            const int* tin = (const int*)(sm + L::TIN + slot * 864);
            const float* tg = (const float*)(sm + L::TG + slot * 864);
            for (int b3 = 0; b3 < 6 && ok; ++b3) {
                if (!((m3 >> b3) & 1u)) continue;
                for (int q = 0; q < n2 && ok; ++q) {
                    const int b2 = s2 + 2 * q, buf = ln & 1;
                    if (!((m2 >> b2) & 3u)) continue;
                    uint4 x[12];
                    float gs[12];
#pragma unroll
                    for (int r = 0; r < 12; ++r) {  // r = (b1, line)
                        const int b1 = s1 + (r >> 1), qq = b1 * 36 + (b2 + (r & 1)) * 6 + b3;
                        gs[r] = 0.0f;
                        x[r] = make_uint4(0, 0, 0, 0);
                        if ((r >> 1) < 2 * n1 && ((m1 >> b1) & 1u)) {
                            const int b = tin[qq];
                            if (b >= 0) {
                                gs[r] = tg[qq];
                                x[r] = __ldg(src0 + (size_t)b * 64);
                            }
                        }
                    }
                    if (ln >= 2) ok = OTC_WAITW(&b_xe[buf], ((ln >> 1) - 1) & 1);
                    if (!ok) break;
                    unsigned char* dst = sm + L::X + buf * L::XBUF + hl * (L::XBUF / 2) + v * 16;
#pragma unroll
                    for (int r = 0; r < 12; ++r) {
                        if ((r >> 1) >= 2 * n1) break;
                        const __half2 g2 = __float2half2_rn(gs[r]);
                        __half2* hv = (__half2*)&x[r];
#pragma unroll
                        for (int i = 0; i < 4; ++i) hv[i] = __hmul2(hv[i], g2);
                        *(uint4*)(dst + r * 1024) = x[r];
                    }
                    tc::fence_async_smem();
                    tc::mbar_arrive_warp(&b_xf[buf]);
                    ++ln;
                }
            }
            tc::mbar_arrive_warp(&b_se[slot]);
        }
    } else if (warp >= 20) {
        // ================= stages II and III of one pair of pieces
        tc::reg_dec<48>();
        const int g = tc::uniform(warp - 20);
        uint32_t bt = 0;  // batches so far
        bool ok = true;
        const uint32_t id2 = tc::idesc_f16(128, 32), id = tc::idesc_f16(128, 16);
        const uint64_t a0 = tc::sdesc(sbase + L::A2 + 2 * g * L::A2_PIECE, L::A2_LBO, L::A2_SBO);
        for (uint32_t k = 0; ok; ++k) {
            const int slot = k & 1;
            ok = OTC_WAITW(&b_sf[slot], (k >> 1) & 1);
            if (!ok || tc::uniform(s_u[slot].unit) < 0) break;
            const unsigned m2 = tc::uniform(s_u[slot].m2), m3 = tc::uniform(s_u[slot].m3);
            const int npc = tc::uniform(s_u[slot].npc), n = otc_pieces(g, npc);
            const int s2 = tc::uniform(s_u[slot].s2), n2 = 3 - s2;
            const int ps = tc::uniform(s_u[slot].ps);
            const uint32_t tab = sbase + L::T + slot * 6 * L::TAB + (ps == 8 ? 2 * g : g) * 128;
            for (int b3 = 0; b3 < 6 && ok && n > 0; ++b3) {
                if (!((m3 >> b3) & 1u)) continue;
                uint32_t acc = 0;
                for (int q = 0; q < n2 && ok; ++q) {
                    const int b2 = s2 + 2 * q;
                    if (!((m2 >> b2) & 3u)) continue;
                    ok = OTC_WAITW(&b_af[g], bt & 1);
                    if (!ok) break;
                    tc::fence_after();
                    // B: (a2', hi or lo, c2), so that A is read once for both products
                    const uint64_t b0 = tc::sdesc(tab + 2 * L::TAB + b2 * 2 * ps * 128, 2 * ps * 128, ps * 128);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        if (r >= n) break;
                        const uint64_t ah = a0 + (uint64_t)(r * (L::A2_PIECE / 16)), bv = b0 + (uint64_t)(r * 8);
                        tc::mma_f16_warp(cII(g, r), ah, bv, id2, acc);
                        tc::mma_f16_warp(cII(g, r), ah + 2 * L::A2_LBO / 16, bv, id2, 1);
                    }
                    tc::commit_warp(&b_ae[g]);
                    ++bt;
                    acc = 1;
                }
                if (!ok) break;
                // B operands of stage III: [F_hi ; F_hi], and [F_lo ; 0] (a tile further on the zeros
                // are a tile nearer)
                const uint32_t tile = tab + 4 * L::TAB + b3 * ps * 128;
                const uint64_t h0 = tc::sdesc(tile, 0, ps * 128);
                const uint64_t l0 = tc::sdesc(tile + L::TAB, sbase + L::Z - tile - L::TAB, ps * 128);
                ok = OTC_WAITW(&b_af[g], bt & 1);
                if (!ok) break;
                tc::fence_after();
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r >= n) break;
                    const uint64_t bh = h0 + (uint64_t)(r * 8), bl = l0 + (uint64_t)(r * 8) - ((uint64_t)(r * 8) << 16);
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        const uint64_t av = a0 + (uint64_t)((r * L::A2_PIECE + a * 2 * L::A2_LBO) / 16);
                        tc::mma_f16_warp(cIII(g, r, a), av, bh, id, 0);
                        tc::mma_f16_warp(cIII(g, r, a), av, bl, id, 1);
                    }
                }
                tc::commit_warp(&b_ae[g]);
                ++bt;
            }
            tc::commit_warp(&b_se[slot]);
        }
    } else {
        // ================= conversions of one pair of pieces, and the outputs
        tc::reg_inc<80>();
        const int g = warp >> 2, w4 = warp & 3;
        const uint32_t lane_off = (uint32_t)(w4 * 32) << 16;
        const int mi = lane >> 3, mr = lane & 7;  // this lane's matrix and row of a stmatrix
        const uint32_t mine = sbase + L::A2 + 2 * g * L::A2_PIECE;
        // D_I: lanes (line, i3, i2) -> rows (a1', c1 | i3), K = (line, i2); matrices hi, lo of two i3
        const uint32_t rowI = mine + (mi & 1) * 2 * L::A2_LBO + (w4 >> 1) * L::A2_LBO + mr * L::A2_SBO +
                              ((w4 & 1) * 4 + (mi >> 1)) * 16;
        // D_II: lanes (a1', c1, i3) -> rows (a1' c1 | c2), K = hi | lo; matrices hi, lo of two (a1', c1)
        const uint32_t rowII = mine + (mi & 1) * L::A2_LBO + (w4 * 4 + (mi >> 1)) * L::A2_SBO + mr * 16;
        uint32_t bt = 0, units = 0;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            const int slot = k & 1;
            ok = OTC_ALL(OTC_WAIT(&b_sf[slot], (k >> 1) & 1));
            const OtcUnit& U = s_u[slot];
            if (!ok || U.unit < 0) break;
            const unsigned m2 = U.m2;
            const int npc = U.npc, nplane = __popc(U.m3), n = otc_pieces(g, npc);
            const int ps = U.ps;
            const int s2 = U.s2, n2 = 3 - s2;
            int lpp = 0;  // lines per plane
            for (int q = 0; q < n2; ++q) lpp += ((m2 >> (s2 + 2 * q)) & 3u) != 0;
            float2 y[2][8];  // [a2'][(a3', c3)] of lane (a1', c1, c2), this pair's pieces
#pragma unroll
            for (int c = 0; c < 8; ++c) y[0][c] = y[1][c] = make_float2(0.0f, 0.0f);
            // y += fin Y after a plane's stage III
            auto add_plane = [&]() {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r >= n) break;
                    const float fin = U.fin[g + 4 * r];
                    const bool leaf_only = (U.piece[g + 4 * r] >> 24) != 0;
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        float t[16];
                        tc::tmem_ld32x16(cIII(g, r, a) + lane_off, t);
#pragma unroll
                        for (int a3 = 0; a3 < 2; ++a3) {
                            const int o = (1 - (w4 >> 1)) * 4 + (1 - a) * 2 + 1 - a3;
                            const float f = leaf_only && !((U.leaf >> o) & 1u) ? 0.0f : fin;
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                y[a][4 * a3 + c] = tc::fma2(make_float2(f, f), make_float2(t[8 * a3 + 2 * c], t[8 * a3 + 2 * c + 1]),
                                                            y[a][4 * a3 + c]);
                        }
                    }
                }
            };
            // the pairs' sums of the unit before have been read out of the operand space
            if (units > 0) ok = OTC_ALL(OTC_WAIT(&b_yr, (units - 1) & 1));
            for (int p = 0; p < nplane && ok; ++p) {
                for (int q = 0; q < lpp && ok; ++q, ++ln) {
                    const int buf = ln & 1;
                    // the last batch is complete: the operands are free, and after a stage III its result
                    // is whole; D_I of the line is there
                    if (n > 0 && p > 0 && q == 0) {
                        ok = OTC_ALL(OTC_WAIT(&b_ae[g], (bt - 1) & 1));
                        if (!ok) break;
                        tc::fence_after();
                        add_plane();
                    }
                    ok = OTC_ALL((n <= 0 || bt == 0 || OTC_WAIT(&b_ae[g], (bt - 1) & 1)) && OTC_WAIT(&b_df[buf], (ln >> 1) & 1));
                    if (!ok) break;
                    if (n <= 0) {  // nothing to convert: only keep step
                        tc::mbar_arrive_warp(&b_de[buf]);
                        continue;
                    }
                    tc::fence_after();
                    const float c20 = U.c2[g], c21 = n > 1 ? U.c2[g + 4] : 0.0f;
                    const uint32_t ad = tbase + buf * 128 + (uint32_t)((ps == 8 ? 2 * g : g) * 8) + lane_off;
#pragma unroll
                    for (int lh = 0; lh < 2; ++lh) {
                        float v[2][2][4];  // [a1'][piece][.]
                        tc::tmem_ld16x256_x2x2(ad + ((uint32_t)(lh * 16) << 16), ad + (uint32_t)(ps * 8) + ((uint32_t)(lh * 16) << 16), v);
                        if (lh) {
                            tc::fence_before();
                            tc::mbar_arrive_warp(&b_de[buf]);  // D_I read
                        }
                        uint32_t w[2][2][4];
#pragma unroll
                        for (int a = 0; a < 2; ++a)
#pragma unroll
                            for (int r = 0; r < 2; ++r) split_scaled(v[a][r], r ? c21 : c20, w[r][a]);
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            if (r >= n) break;
#pragma unroll
                            for (int a = 0; a < 2; ++a)
                                tc::stmatrix_x4_trans(rowI + r * L::A2_PIECE + a * 8 * L::A2_SBO + lh * 32, w[r][a][0], w[r][a][1],
                                                      w[r][a][2], w[r][a][3]);
                        }
                    }
                    tc::fence_async_smem();
                    tc::mbar_arrive_warp(&b_af[g]);
                    ++bt;
                }
                if (!ok || n <= 0) continue;
                // the plane's V
                ok = OTC_ALL(OTC_WAIT(&b_ae[g], (bt - 1) & 1));
                if (!ok) break;
                tc::fence_after();
                const float c30 = U.c3[g], c31 = n > 1 ? U.c3[g + 4] : 0.0f;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r >= n) break;
#pragma unroll
                    for (int lh = 0; lh < 2; ++lh) {
                        float v[2][2][4];  // [a2'][product with hi or lo][.]
                        const uint32_t ad = cII(g, r) + lane_off + ((uint32_t)(lh * 16) << 16);
                        tc::tmem_ld16x256_x2x2(ad, ad + 16u, v);
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            uint32_t w[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) v[a][0][c] += v[a][1][c];
                            split_scaled(v[a][0], r ? c31 : c30, w);
                            tc::stmatrix_x4_trans(rowII + r * L::A2_PIECE + a * 2 * L::A2_LBO + lh * 2 * L::A2_SBO, w[0], w[1], w[2],
                                                  w[3]);
                        }
                    }
                }
                tc::fence_before();
                tc::fence_async_smem();
                tc::mbar_arrive_warp(&b_af[g]);
                ++bt;
            }
            float* ysum = (float*)(sm + L::A2);  // per pair, in its operand space: 32 x 128
            constexpr int YS = 2 * L::A2_PIECE / 4;
            const int r = w4 * 32 + lane;
            if (ok && n > 0) {
                ok = OTC_ALL(OTC_WAIT(&b_ae[g], (bt - 1) & 1));
                if (ok) {
                    tc::fence_after();
                    add_plane();
                    tc::fence_before();
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        ysum[g * YS + (2 * c) * 128 + r] = y[c >> 3][c & 7].x;
                        ysum[g * YS + (2 * c + 1) * 128 + r] = y[c >> 3][c & 7].y;
                    }
                }
            }
            tc::mbar_arrive_warp(&b_y);
            ok = OTC_ALL(ok && OTC_WAIT(&b_y, units & 1));
            if (ok) {  // four warps per (a2', a3') add the pairs' sums in order
                const int a1 = 1 - (r >> 6), c1 = (r >> 3) & 7, c2 = r & 7, kk = P.k;
                const int o = a1 * 4 + (1 - (g >> 1)) * 2 + 1 - (g & 1);
                if (o < U.nout && c1 < kk && c2 < kk) {
                    float* dst = (float*)Q.part + (size_t)U.unit * 8 * kk * kk * kk + (size_t)o * kk * kk * kk + (c1 * kk + c2) * kk;
                    float s[8];
#pragma unroll
                    for (int c3 = 0; c3 < 8; ++c3) {
                        s[c3] = 0.0f;
#pragma unroll
                        for (int gg = 0; gg < 4; ++gg)
                            if (otc_pieces(gg, npc) > 0) s[c3] += ysum[gg * YS + (g * 8 + c3) * 128 + r];
                    }
                    if (kk == 8) {
                        ((float4*)dst)[0] = make_float4(s[0], s[1], s[2], s[3]);
                        ((float4*)dst)[1] = make_float4(s[4], s[5], s[6], s[7]);
                    } else {
#pragma unroll
                        for (int c3 = 0; c3 < 8; ++c3)
                            if (c3 < kk) dst[c3] = s[c3];
                    }
                }
            }
            tc::mbar_arrive_warp(&b_yr);
            tc::mbar_arrive_warp(&b_se[slot]);
            ++units;
        }
    }
#undef OTC_WAIT
#undef OTC_WAITW
#undef OTC_ALL
    tc::fence_before();
    __syncthreads();
    if (s_abort) {
        if (tid == 0) atomicExch(Q.err, 4);
        // a role stops where it stands: what the issuing warps have sent may still write tensor memory
        if (warp >= 20 && warp <= 24) {
            tc::commit_warp(&b_end[warp - 20]);
            tc::mbar_wait(&b_end[warp - 20], 0, TC_WAIT_MIN);
        }
        __syncthreads();
    }
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
}

int oct_tc_configure() {
    MRA_CK(cudaFuncSetAttribute(k_apply_oct_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)OtcSmem::bytes(MRA_MAX_TERMS)));
    return MRA_OK;
}

int oct_slice_tc() { return OTC_P; }

// Q.P, the operands, err, withhold and wait_limit (0: the default) set; part:
// oct_part_alloc(S, oct_slice_tc(), sizeof(float), ...).  oct_tc_configure() first.
int oct_tc_launch(OctTcArgs Q, const ScreenOut& S, void* part, double* out, cudaStream_t st) {
    Q.wait_limit = tc::wait_polls(Q.wait_limit);
    Q.part = part;
    Q.P.ns = std::max(1, (S.max_pieces + OTC_P - 1) / OTC_P);
    const int per = S.oct.batch;
    for (int g0 = 0; g0 < S.oct.n; g0 += per) {
        const int ng = std::min(per, S.oct.n - g0);
        Q.P.g0 = g0;
        Q.nunits = ng * Q.P.ns;
        MRA_CK(cudaMemsetAsync(Q.counter, 0, sizeof(int), st));
        k_apply_oct_tc<<<std::min(Q.nunits, num_sms()), OTC_THREADS, OtcSmem::bytes(Q.P.M), st>>>(Q);
        MRA_CK_LAUNCH();
        MRA_TRY(oct_reduce(Q.P, OTC_P, ng, (const float*)part, out, st));
    }
    return MRA_OK;
}

}  // namespace mra
