// Step 3 of Algorithm 3 under the static screen on the tensor cores (tcgen05), by sibling
// groups: the pieces and factored sums of apply_oct.cu, k <= 8 (lower orders zero-padded
// to 8), FP16 hi + lo operands as in apply_tc.cu (hi*hi + hi*lo + lo*hi into FP32).
//
// A work unit is one group and one chunk of up to 8 pieces.  Per plane b3 and pair of lines
// (b2, b2 + 1):
//   stage I   D_I[(line, i3, i2)][(a1, piece, c1)] = X F^{t1}: M = 128, N = 128 (64 for at
//             most 4 pieces), K = 16 per pair of input boxes b1;
//   stage II  per piece V[(a1, c1, i3)][(a2, c2)] += W F^{t2}: M = 128, N = 16, K = 16 (two
//             lines of i2), accumulated over the plane's lines;
//   stage III per piece, plane and a2, Y[(a1, c1, c2)][(a3, c3)] = V F^{t3}: M = 128, N = 16,
//             K = 16 (i3 as hi | lo), read out after the plane and summed over the planes and
//             the chunk's pieces in FP32 registers.  (Summing in the tensor core's accumulator
//             instead truncates at every addition: the hydrogen energy then moves by 7e-7.)
// Every B operand is read in place from the chunk's F tiles: with u = b - a + 1 the tile of
// t = 3 - u serves output a and input b, so (a, b) neighbours are tile neighbours and one
// descriptor (constant strides) covers both outputs and both boxes; a piece's excluded
// translations are zero tiles.
//
// One CTA per SM (202 KB of shared memory, all 512 TMEM columns), 15 warps with roles, so
// that loading, MMAs and conversions run beside each other: warps 0-7 convert accumulators to
// the next stage's operands (warps 0-3 the chunk's first half of the pieces, 4-7 the second),
// 8-11 load X (two buffers; the blocks' power-of-two scales are made equal on the way),
// 12 issues stage I into one of two accumulators, 13 and 14 issue stages II and III of a half
// each.  Every wait is bounded: one that reaches its limit makes all roles stop, the error
// word is set to 4 and the kernel frees its tensor memory.
#include <cfloat>
#include <climits>

#include "apply_common.cuh"
#include "oct_pieces.cuh"
#include "tc_ptx.cuh"

namespace mra {

#define OTC_THREADS 480
#define OTC_WAIT_LIMIT (1u << 24)
#define OTC_WAIT_MIN 4096u
#define OTC_P 8  // pieces per chunk

struct OtcSmem {
    static constexpr int XBUF = 24576;                 // hi then lo: [box b1 6][line 2] x 1 KB
    static constexpr int X = 0;                        // two buffers
    static constexpr int A2_LBO = 2304, A2_SBO = 144;  // 8 x 16-byte core matrices, 16 bytes apart (bank spread)
    static constexpr int A2_PIECE = 4 * A2_LBO;        // stage II: hi, lo (2 K groups each); stage III: a2' = 0, 1
    static constexpr int A2 = X + 2 * XBUF;
    static constexpr int TAB = 7 * OTC_P * 128;        // tiles [u 0..6][piece]
    static constexpr int T = A2 + OTC_P * A2_PIECE;    // [direction][hi, lo]
    static constexpr int Z = T + 6 * TAB;              // zeros: two tiles a tile row apart
    static constexpr int TIN = Z + OTC_P * 128 + 128;  // 216 int
    static constexpr int TG = TIN + 864;               // 216 float
    static constexpr int LIST = TG + 864;              // pieces
    static size_t bytes(int M) { return LIST + 4 * (size_t)M * sizeof(uint32_t); }
};
static_assert(OtcSmem::LIST + 4 * MRA_MAX_TERMS * 4 + 1024 <= 232448, "shared memory of one CTA");

__global__ void __launch_bounds__(OTC_THREADS, 1) k_apply_oct_tc(OctTcArgs Q) {
    using L = OtcSmem;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t b_xf[2], b_xe[2], b_df[2], b_de[2], b_af[2], b_ae[2], b_vf[2];
    __shared__ volatile int s_abort;
    __shared__ int s_unit, s_emin;
    __shared__ unsigned s_leaf, s_xmax;
    __shared__ float s_c2[OTC_P], s_c3[OTC_P], s_fin[OTC_P];
    const OctArgs& P = Q.P;
    if (P.skip && *P.skip != P.run_if) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = tc::smem_u32(sm);
    int* tin = (int*)(sm + L::TIN);
    float* tg = (float*)(sm + L::TG);
    uint32_t* list = (uint32_t*)(sm + L::LIST);
    for (int e = tid; e < L::TIN / 16; e += OTC_THREADS) ((uint4*)sm)[e] = make_uint4(0, 0, 0, 0);
    if (warp == 0) tc::tmem_alloc(&s_tmem, 512);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&b_xf[i], 128);
            tc::mbar_init(&b_xe[i], 1);
            tc::mbar_init(&b_df[i], 1);
            tc::mbar_init(&b_de[i], 256);
            tc::mbar_init(&b_af[i], 128);
            tc::mbar_init(&b_ae[i], 1);
            tc::mbar_init(&b_vf[i], 1);
        }
        s_abort = 0;
    }
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = s_tmem;
    // TMEM columns: D_I 2 x 128; per half D_II 4 pieces x 16 at 256 + 64 half, and D_III 4 pieces
    // x 2 a2' x 16: the first two pieces' at 384 + 64 half, the others' over D_II, which stage III
    // has no more use for
    auto cII = [&](int h, int lp) { return tbase + 256u + (uint32_t)(h * 64 + lp * 16); };
    auto cIII = [&](int h, int lp, int a) { return tbase + (lp < 2 ? 384u : 256u) + (uint32_t)(h * 64 + (lp & 1) * 32 + a * 16); };
    // running counts of lines, stage II / III batches and planes: every role counts the same
    uint32_t line0 = 0, batch0 = 0, plane0 = 0;
    bool stop = false;
#define OTC_WAIT(bar, parity) tc::mbar_wait_or(bar, parity, Q.wait_limit, &s_abort)
    // the same by a whole warp, whose lanes go on or give up together (what follows is warp-collective)
#define OTC_WAITW(bar, parity) __all_sync(0xffffffffu, OTC_WAIT(bar, parity))

    while (!stop) {
        if (tid == 0) s_unit = atomicAdd(Q.counter, 1);
        __syncthreads();
        const int unit = s_unit;
        if (unit >= Q.nunits) break;
        const int g = P.g0 + unit / P.ns, sl = unit % P.ns, np = P.np[g], q0 = sl * OTC_P;
        if (q0 >= np) {
            __syncthreads();
            continue;
        }
        const int npc = min(OTC_P, np - q0), ps = npc <= 4 ? 4 : 8, ph = ps / 2;
        const int i0 = P.first[g], tree = P.node_tree ? P.node_tree[i0] : 0;
        const int j = P.coord[4 * i0], nout = j ? 8 : 1;
        if (tid == 0) {
            s_emin = INT_MAX;
            s_xmax = 0u;
        }
        if (warp == 14) {
            const unsigned lf = __ballot_sync(0xffffffffu, lane < nout && P.leaf[i0 + (lane < nout ? lane : 0)]);
            if (lane == 0) s_leaf = lf;
            oct_pieces(P.sched + (size_t)tree * P.sl, P.M, P.lm, j, lf != 0, lf != (1u << nout) - 1u, list);
        }
        __syncthreads();
        // the inputs: the neighbourhood's smallest scale and largest value
        int in = -1;
        float sxb = 0.0f;
        if (tid < 216) {
            in = P.in[(size_t)g * 216 + tid];
            tin[tid] = in;
            if (in >= 0) {
                sxb = Q.sx[in];
                int e;
                frexpf(sxb, &e);
                atomicMin(&s_emin, e);
                atomicMax(&s_xmax, __float_as_uint(Q.xmax[in]));  // non-negative floats order as ints
            }
        } else {
            // F tiles of the chunk, masked by the pieces' sets
            for (int e = tid - 216; e < 7 * ps * 8 * 6; e += OTC_THREADS - 216) {
                const int v = e & 7, pc = (e >> 3) % ps, r = (e >> 3) / ps, u = r % 7, dh = r / 7;
                const int d = dh >> 1, hl = dh & 1;
                uint4 x = make_uint4(0, 0, 0, 0);
                if (pc < npc) {
                    const uint32_t p = list[q0 + pc];
                    const int set = (p >> (20 - 2 * d)) & 3;
                    if (set & ((u >= 2 && u <= 4) ? 1 : 2))
                        x = ((const uint4*)(hl ? Q.Fl : Q.Fh))[(((size_t)j * P.M + (p & 0xffff)) * 7 + 6 - u) * 8 + v];
                }
                ((uint4*)(sm + L::T + dh * L::TAB))[(u * ps + pc) * 8 + v] = x;
            }
        }
        __syncthreads();
        const float xmax = __uint_as_float(s_xmax);
        const int es = s_emin - 1;  // the common scale 2^es
        if (!(xmax <= FLT_MAX) && tid == 0) atomicExch(Q.err, 5);  // input values beyond FP32's range
        const bool live = xmax > 0.0f && xmax <= FLT_MAX;
        if (tid < 216) tg[tid] = in < 0 ? 0.0f : ldexpf(1.0f, es) / sxb;
        if (warp == 14 && live) {
            // power-of-two scales as in apply_tc.cu: sW = 2^eW, the largest power of two <=
            // 8192 / (48 max|F| max|x|), and sV = 2^eV <= 8192 / (48^2 max|F|^2 max|x|)
            if (lane < OTC_P) {
                float c2 = 0.0f, c3 = 0.0f, fin = 0.0f;
                if (lane < npc) {
                    const int m = list[q0 + lane] & 0xffff;
                    const size_t jm = (size_t)j * P.M + m;
                    const float mf = Q.maxF[jm], sf = Q.sF[jm];
                    if (mf > 0.0f) {
                        int em, ex, ef, e1, e2;
                        const float fm = frexpf(mf, &em), fx = frexpf(xmax, &ex);
                        frexpf(sf, &ef);
                        ef -= 1;
                        frexpf(8192.0f / (48.0f * fm * fx), &e1);
                        frexpf(8192.0f / (2304.0f * fm * fm * fx), &e2);
                        const int eW = min(e1 - 1 - em - ex, 126), eV = min(e2 - 1 - 2 * em - ex, 126);
                        if (eW >= -126 && eV >= -126) {
                            c2 = ldexpf(1.0f, eW - ef - es);            // sW / (sF sx)
                            c3 = ldexpf(1.0f, eV - eW - ef);            // sV / (sW sF)
                            fin = ldexpf((float)P.w[m], -(eV + ef));    // w_m / (sV sF)
                            if (!(fin <= FLT_MAX)) {  // outputs beyond the FP32 range: refuse
                                atomicExch(Q.err, 5);
                                fin = 0.0f;
                            }
                        }
                    }
                }
                s_c2[lane] = c2;
                s_c3[lane] = c3;
                s_fin[lane] = fin;
            }
        }
        // boxes any piece reads, per direction
        unsigned m1 = 0, m2 = 0, m3 = 0;
        for (int pc = 0; pc < npc; ++pc) {
            const uint32_t p = list[q0 + pc];
            m1 |= set_boxes((p >> 20) & 3);
            m2 |= set_boxes((p >> 18) & 3);
            m3 |= set_boxes((p >> 16) & 3);
        }
        const int s1 = m1 == 0x1e ? 1 : 0, s2 = m2 == 0x1e ? 1 : 0;   // first box of the first pair
        const int n1 = m1 == 0x1e ? 2 : 3, n2 = m2 == 0x1e ? 2 : 3;   // pairs
        tc::fence_async_smem();
        __syncthreads();
        float* part = (float*)Q.part + (size_t)unit * 8 * P.k * P.k * P.k;
        uint32_t nline = 0, nplane = 0;  // lines and planes of this unit
        if (live) {
            for (int b3 = 0; b3 < 6; ++b3) nplane += (m3 >> b3) & 1u;
            for (int q = 0; q < n2; ++q) nline += ((m2 >> (s2 + 2 * q)) & 3u) != 0;
            const uint32_t lpp = nline;  // lines (pairs) per plane
            nline *= nplane;
            float* ysum = (float*)(sm + L::A2 + ph * L::A2_PIECE);  // 32 x 128
            if (warp >= 8 && warp < 12) {
                // ---- X of a pair of lines into a buffer
                const int lt = tid - 256, hl = lt >> 6, v = lt & 63;
                const __half* src0 = hl ? Q.xl : Q.xh;
                uint32_t ln = line0;
                bool ok = true;
                for (int b3 = 0; b3 < 6 && ok; ++b3) {
                    if (!((m3 >> b3) & 1u)) continue;
                    for (int q = 0; q < n2 && ok; ++q) {
                        const int b2 = s2 + 2 * q;
                        if (!((m2 >> b2) & 3u)) continue;
                        const int buf = ln & 1;
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
                                    x[r] = __ldg((const uint4*)(src0 + (size_t)b * 512) + v);
                                }
                            }
                        }
                        if (ln >= 2) ok = OTC_WAIT(&b_xe[buf], ((ln >> 1) - 1) & 1);
                        if (!ok) break;
                        unsigned char* dst = sm + L::X + buf * L::XBUF + hl * (L::XBUF / 2) + v * 16;
#pragma unroll
                        for (int r = 0; r < 12; ++r) {
                            if ((r >> 1) >= 2 * n1) break;
                            const __half2 g2 = __float2half2_rn(gs[r]);
                            __half2* h = (__half2*)&x[r];
#pragma unroll
                            for (int i = 0; i < 4; ++i) h[i] = __hmul2(h[i], g2);
                            *(uint4*)(dst + r * 1024) = x[r];
                        }
                        tc::fence_async_smem();
                        tc::mbar_arrive(&b_xf[buf]);
                        ++ln;
                    }
                }
            } else if (warp == 12) {
                // ---- stage I
                if (lane == 0 && !Q.withhold) {
                    const uint32_t id = tc::idesc_f16(128, 16 * ps);
                    uint32_t ln = line0;
                    for (uint32_t l = 0; l < nline; ++l, ++ln) {
                        const int buf = ln & 1;
                        if (!OTC_WAIT(&b_xf[buf], (ln >> 1) & 1)) break;
                        if (ln >= 2 && !OTC_WAIT(&b_de[buf], ((ln >> 1) - 1) & 1)) break;
                        tc::fence_after();
                        const uint32_t d = tbase + buf * 128;
                        const uint64_t xh = tc::sdesc(sbase + L::X + buf * L::XBUF, 2048, 128);
                        const uint64_t th = tc::sdesc(sbase + L::T + s1 * ps * 128, ps * 128, 128);
                        for (int s = 0; s < n1; ++s) {  // boxes s1 + 2 s, + 1
                            const uint64_t ah = xh + (uint64_t)(s * (4096 / 16)), al = ah + L::XBUF / 32;
                            const uint64_t bh = th + (uint64_t)(s * 2 * ps * 8), bl = bh + L::TAB / 16;
                            tc::mma_f16(d, ah, bh, id, s > 0);
                            tc::mma_f16(d, ah, bl, id, 1);
                            tc::mma_f16(d, al, bh, id, 1);
                        }
                        tc::commit(&b_xe[buf]);
                        tc::commit(&b_df[buf]);
                    }
                }
            } else if (warp >= 13) {
                // ---- stages II and III of one half of the pieces
                if (lane == 0) {
                    const int h = warp - 13, pl = min(npc, h * ph), pe = min(npc, h * ph + ph);
                    const uint32_t id = tc::idesc_f16(128, 16);
                    uint32_t bt = batch0;
                    bool ok = true;
                    for (int b3 = 0; b3 < 6 && ok; ++b3) {
                        if (!((m3 >> b3) & 1u)) continue;
                        bool first = true;
                        for (int q = 0; q < n2 && ok; ++q) {
                            const int b2 = s2 + 2 * q;
                            if (!((m2 >> b2) & 3u)) continue;
                            ok = OTC_WAIT(&b_af[h], bt & 1);
                            if (!ok) break;
                            tc::fence_after();
                            for (int pc = pl; pc < pe; ++pc) {
                                const uint32_t d = cII(h, pc - pl);
                                const uint64_t ah = tc::sdesc(sbase + L::A2 + pc * L::A2_PIECE, L::A2_LBO, L::A2_SBO);
                                const uint64_t al = ah + 2 * L::A2_LBO / 16;
                                const uint64_t bh = tc::sdesc(sbase + L::T + 2 * L::TAB + (b2 * ps + pc) * 128, ps * 128,
                                                              ps * 128);
                                const uint64_t bl = bh + L::TAB / 16;
                                tc::mma_f16(d, ah, bh, id, first ? 0u : 1u);
                                tc::mma_f16(d, ah, bl, id, 1);
                                tc::mma_f16(d, al, bh, id, 1);
                            }
                            first = false;
                            tc::commit(&b_ae[h]);
                            ++bt;
                        }
                        if (!ok) break;
                        tc::commit(&b_vf[h]);
                        ok = OTC_WAIT(&b_af[h], bt & 1);
                        if (!ok) break;
                        tc::fence_after();
                        for (int pc = pl; pc < pe; ++pc) {
                            const uint32_t tile = sbase + L::T + 4 * L::TAB + (b3 * ps + pc) * 128;
                            const uint64_t bh = tc::sdesc(tile, 0, ps * 128);  // [F_hi ; F_hi]
                            const uint64_t bl = tc::sdesc(tile + L::TAB, sbase + L::Z - tile - L::TAB, ps * 128);  // [F_lo ; 0]
                            for (int a = 0; a < 2; ++a) {
                                const uint32_t d = cIII(h, pc - pl, a);
                                const uint64_t av = tc::sdesc(sbase + L::A2 + pc * L::A2_PIECE + a * 2 * L::A2_LBO,
                                                              L::A2_LBO, L::A2_SBO);
                                tc::mma_f16(d, av, bh, id, 0);
                                tc::mma_f16(d, av, bl, id, 1);
                            }
                        }
                        tc::commit(&b_ae[h]);
                        ++bt;
                    }
                }
            } else if (warp < 8) {
                // ---- conversions of one half of the pieces
                const int h = warp >> 2, w4 = warp & 3, pl = min(npc, h * ph), n = min(npc, h * ph + ph) - pl;
                const uint32_t lane_off = (uint32_t)(w4 * 32) << 16;
                const int mi = lane >> 3, mr = lane & 7;  // this lane's matrix and row of a stmatrix
                // D_I: lanes (line, i3, i2) -> rows (a1', c1 | i3), K = (line, i2); matrices hi, lo of two i3
                const uint32_t rowI = sbase + L::A2 + (mi & 1) * 2 * L::A2_LBO + (w4 >> 1) * L::A2_LBO + mr * L::A2_SBO +
                                      ((w4 & 1) * 4 + (mi >> 1)) * 16;
                // D_II: lanes (a1', c1, i3) -> rows (a1' c1 | c2), K = hi | lo; matrices hi, lo of two (a1', c1)
                const uint32_t rowII = sbase + L::A2 + (mi & 1) * L::A2_LBO + (w4 * 4 + (mi >> 1)) * L::A2_SBO + mr * 16;
                uint32_t ln = line0, bt = batch0, pn = plane0;
                bool ok = true;
                float y[2][16];  // [a2'][(a3', c3)] of lane (a1', c1, c2), this half's pieces
#pragma unroll
                for (int c = 0; c < 16; ++c) y[0][c] = y[1][c] = 0.0f;
                // outputs a2', a3' of this lane that are leaves: bit 2 a2' + a3'
                unsigned lf = 0;
                for (int q = 0; q < 4; ++q) lf |= ((s_leaf >> ((1 - (w4 >> 1)) * 4 + (1 - (q >> 1)) * 2 + 1 - (q & 1))) & 1u) << q;
                // y += fin Y of the plane whose stage III has completed
                auto add_plane = [&]() {
#pragma unroll
                    for (int pc = 0; pc < 4; ++pc) {
                        if (pc >= n) break;
                        const float fin = s_fin[pl + pc];
                        const bool leaf_only = (list[q0 + pl + pc] >> 24) != 0;
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            float t[16];
                            tc::tmem_ld32x16(cIII(h, pc, a) + lane_off, t);
#pragma unroll
                            for (int c = 0; c < 16; ++c) {
                                const float f = leaf_only && !((lf >> (2 * a + (c >> 3))) & 1u) ? 0.0f : fin;
                                y[a][c] = fmaf(f, t[c], y[a][c]);
                            }
                        }
                    }
                };
                for (uint32_t p = 0; p < nplane && ok; ++p, ++pn) {
                    for (uint32_t q = 0; q < lpp && ok; ++q, ++ln, ++bt) {
                        const int buf = ln & 1;
                        // the last batch is complete: the operands are free, and after a stage III
                        // its result is whole
                        if (bt > 0) ok = OTC_WAITW(&b_ae[h], (bt - 1) & 1);
                        if (ok && p > 0 && q == 0) {
                            tc::fence_after();
                            add_plane();
                        }
                        ok = ok && OTC_WAITW(&b_df[buf], (ln >> 1) & 1);
                        if (!ok) break;
                        tc::fence_after();
#pragma unroll
                        for (int lh = 0; lh < 2; ++lh) {
                            float v[2][4][4];  // [a1'][piece][.]
                            if (n > 0) {
#pragma unroll
                                for (int a = 0; a < 2; ++a) {
                                    const uint32_t ad = tbase + buf * 128 + (uint32_t)(a * ps * 8 + pl * 8) + lane_off + ((uint32_t)(lh * 16) << 16);
                                    if (ps == 8) tc::tmem_ld16x256_rep<4>(ad, v[a]);
                                    else tc::tmem_ld16x256_rep<2>(ad, v[a]);
                                }
                            }
                            if (lh == 1) {
                                tc::fence_before();
                                tc::mbar_arrive(&b_de[buf]);
                            }
#pragma unroll
                            for (int pc = 0; pc < 4; ++pc) {
                                if (pc >= n) break;
                                const float c2 = s_c2[pl + pc];
#pragma unroll
                                for (int a = 0; a < 2; ++a) {
                                    const float* x = v[a][pc];
                                    uint32_t h0, l0, h1, l1;
                                    tc::split_h2(x[0] * c2, x[1] * c2, h0, l0);
                                    tc::split_h2(x[2] * c2, x[3] * c2, h1, l1);
                                    tc::stmatrix_x4_trans(rowI + (pl + pc) * L::A2_PIECE + a * 8 * L::A2_SBO + lh * 32, h0,
                                                          l0, h1, l1);
                                }
                            }
                        }
                        tc::fence_before();
                        tc::fence_async_smem();
                        tc::mbar_arrive(&b_af[h]);
                    }
                    if (!ok) break;
                    // the plane's stage II is complete: D_II is whole and the operands are free
                    ok = OTC_WAITW(&b_vf[h], pn & 1) && OTC_WAITW(&b_ae[h], (bt - 1) & 1);
                    if (!ok) break;
                    tc::fence_after();
                    if (n > 0) {
#pragma unroll
                        for (int lh = 0; lh < 2; ++lh) {
                            float v[2][4][4];  // [piece pair][2 piece' + a2'][.]
#pragma unroll
                            for (int pp = 0; pp < 2; ++pp)
                                if (2 * pp < n) tc::tmem_ld16x256_rep<4>(cII(h, 2 * pp) + lane_off + ((uint32_t)(lh * 16) << 16), v[pp]);
#pragma unroll
                            for (int pc = 0; pc < 4; ++pc) {
                                if (pc >= n) break;
                                const float c3 = s_c3[pl + pc];
#pragma unroll
                                for (int a = 0; a < 2; ++a) {
                                    const float* x = v[pc >> 1][2 * (pc & 1) + a];
                                    uint32_t h0, l0, h1, l1;
                                    tc::split_h2(x[0] * c3, x[1] * c3, h0, l0);
                                    tc::split_h2(x[2] * c3, x[3] * c3, h1, l1);
                                    tc::stmatrix_x4_trans(rowII + (pl + pc) * L::A2_PIECE + a * 2 * L::A2_LBO + lh * 2 * L::A2_SBO,
                                                          h0, l0, h1, l1);
                                }
                            }
                        }
                    }
                    tc::fence_before();
                    tc::fence_async_smem();
                    tc::mbar_arrive(&b_af[h]);
                    ++bt;
                }
                if (ok) ok = OTC_WAITW(&b_ae[h], (bt - 1) & 1);
                if (ok) {
                    tc::fence_after();
                    add_plane();
                    tc::fence_before();
                    // the second half's sum waits in its operand space for the first half's
                    if (h == 1 && n > 0)
#pragma unroll
                        for (int c = 0; c < 32; ++c) ysum[c * 128 + w4 * 32 + lane] = y[c >> 4][c & 15];
                }
                // (after the barrier every thread of the first half writes the sums out)
                __syncthreads();
                if (h == 0 && ok && !s_abort) {
                    const int r = w4 * 32 + lane, a1 = 1 - (r >> 6), c1 = (r >> 3) & 7, c2 = r & 7, k = P.k;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int o = a1 * 4 + (1 - (q >> 1)) * 2 + 1 - (q & 1);
                        if (o < nout && c1 < k && c2 < k) {
                            float* dst = part + (size_t)o * k * k * k + (c1 * k + c2) * k;
#pragma unroll
                            for (int c3 = 0; c3 < 8; ++c3) {
                                const int c = q * 8 + c3;
                                if (c3 < k) dst[c3] = y[c >> 4][c & 15] + (npc > ph ? ysum[c * 128 + r] : 0.0f);
                            }
                        }
                    }
                }
            }
            if (warp >= 8) __syncthreads();
            line0 += nline;
            batch0 += nline + nplane;
            plane0 += nplane;
        } else {
            for (int e = tid; e < nout * P.k * P.k * P.k; e += OTC_THREADS) part[e] = 0.0f;
        }
        __syncthreads();
        tc::fence_after();
        if (s_abort) {
            stop = true;
            if (tid == 0) atomicExch(Q.err, 4);
        }
    }
#undef OTC_WAIT
#undef OTC_WAITW
    tc::fence_before();
    __syncthreads();
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
    const int k = Q.P.k;
    Q.wait_limit = Q.wait_limit ? std::max(Q.wait_limit, OTC_WAIT_MIN) : OTC_WAIT_LIMIT;
    Q.part = part;
    Q.P.ns = std::max(1, (S.max_pieces + OTC_P - 1) / OTC_P);
    const int per = oct_part_groups(S, OTC_P, sizeof(float), k);
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
