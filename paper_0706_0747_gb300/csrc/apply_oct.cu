// Step 3 of Algorithm 3 under the static screen, by sibling groups.
//
// The band of an output box a (eq. fine_scale_band, t_d in [-3, 2] for even a_d and
// [-2, 3] for odd) is made of the children of its parent's 27 neighbours.  So the 8
// siblings of a group have the same 6 x 6 x 6 input boxes; with b_d in 0..5 the input's
// and a_d in {0, 1} the output's place, t_d = a_d + 2 - b_d, and |t_d| <= 1 ("core"
// in direction d) reads a_d = 0: b_d in {1, 2, 3}, a_d = 1: b_d in {2, 3, 4}.
//
// The static schedule (Sec. 4) keeps term m at a scale for a set of classes S = number
// of core directions, the core itself left out at internal boxes when J_m > j.  Such a
// set of translations is a disjoint union of products T1 x T2 x T3 with each T_d the core
// translations, the off-core ones, or all (at most four products): a piece is a term with
// one such product, optionally for the leaf outputs only.  For a piece the sum over its
// translations factors by direction,
//   ghat_a += w_m sum_{t3 in T3} F^{t3} x_3 [ sum_{t2 in T2} F^{t2} x_2 [ sum_{t1 in T1} F^{t1} x_1 f ] ],
// and the bracketed sums belong to box positions, not to one output: the inner one to
// (a1, b2, b3), shared by the four siblings with that a1, the middle one to (a1, a2, b3).
// A full-band piece costs 72 * 6 + 24 * 6 + 8 * 6 = 624 mode products for eight outputs
// where the nested sums of one output at a time cost 8 (216 + 36 + 6) = 2064; a core
// piece 168 where they cost 312.  The items are the static screen's, none more or fewer.
//
// Also F^{-t}[c][i] = (-1)^{c+i} F^t[c][i] (Appendix, Proposition 1: the cross-correlations'
// symmetry), so a pair of translations t, -t of one sum takes
//   F^t x + F^{-t} x' = E (x + x') + O (x - x'),   E / O: the entries with c + i even / odd,
// half the multiplications of the two products, and F^0 = E alone.
#include <algorithm>

#include "apply_common.cuh"
#include "oct_pieces.cuh"

namespace mra {

#define OCT_SLICE 4  // pieces per work unit: one partial sum each, added up in order afterwards

// ------------------------------------------------------------------ groups of a forest
// Group of node i of tree b, whose root is node r: r is a group of its own, and the other
// nodes come in sibling groups of eight in node order; tree b's first group is (r + 7 b) / 8.
__global__ void k_oct_first(Forest F, int32_t* first) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < F.n; i += gridDim.x * blockDim.x) {
        const int b = F.node_tree ? F.node_tree[i] : 0;
        const int r = F.off[b * (F.lm + 1)], l = i - r;
        if (l == 0) first[(r + 7 * b) / 8] = i;
        else if ((l & 7) == 1) first[(r + 7 * b) / 8 + 1 + (l >> 3)] = i;
    }
}

// Warp per group: its input boxes (node index; -2 - slot of the parent in the Step-2 set
// where the box is missing; -1 where no output needs it or it lies outside the domain),
// the pairs and items of its outputs, and its number of pieces.  A parent's eight children
// are consecutive nodes, so 27 searches (lane per neighbour of the group's parent) find
// the 216 inputs.  (The pair lists need 216 searches for each of the eight outputs.)
__global__ void k_oct_screen(ScreenArgs A, OctGroups O, int32_t* max_pieces) {
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int lm = A.F.lm;
    for (int g = warp; g < O.n; g += nwarps) {
        const int i0 = O.first[g], b = A.F.node_tree ? A.F.node_tree[i0] : 0;
        const int32_t* sched = A.sched + (size_t)b * A.sl;
        const int32_t* off = A.F.off + b * (lm + 1);
        const int j = A.F.coord[4 * i0];
        const int nout = j ? 8 : 1;
        const unsigned leafm = __ballot_sync(0xffffffffu, lane < nout && A.F.leaf[i0 + (lane < nout ? lane : 0)]);
        const int32_t* cnt = sched + A.M + 8 * lm + 8 * j;  // [S][core at an internal box]
        int c[8];
        for (int q = 0; q < 8; ++q) c[q] = cnt[q];
        unsigned pairs = 0, items = 0;
        if (lane < 27) {
            const int d1 = lane / 9, d2 = (lane / 3) % 3, d3 = lane % 3;  // neighbour + 1 per direction
            int base = -1;
            bool inside;
            int p1 = 0, p2 = 0, p3 = 0;
            if (j == 0) {
                inside = lane == 13;
                base = i0;
            } else {
                const int N = 1 << (j - 1);
                p1 = (A.F.coord[4 * i0 + 1] >> 1) + d1 - 1;
                p2 = (A.F.coord[4 * i0 + 2] >> 1) + d2 - 1;
                p3 = (A.F.coord[4 * i0 + 3] >> 1) + d3 - 1;
                inside = p1 >= 0 && p2 >= 0 && p3 >= 0 && p1 < N && p2 < N && p3 < N;
                if (inside) base = find_key_exact(A.F.key, off[j], off[j + 1], morton3(p1, p2, p3) << 3);
            }
            unsigned need = 0;
            if (inside)
                for (int o = 0; o < (j ? 8 : 1); ++o) {
                    const int b1 = 2 * d1 + (o >> 2), b2 = 2 * d2 + ((o >> 1) & 1), b3 = 2 * d3 + (o & 1);
                    for (int a = 0; a < nout; ++a) {
                        const int S = band_core(a >> 2, b1) + band_core((a >> 1) & 1, b2) + band_core(a & 1, b3);
                        const int n = (S == 3 && !((leafm >> a) & 1u)) ? c[7] : (S == 3 ? c[6] : (S == 2 ? c[4] : (S == 1 ? c[2] : c[0])));
                        if (n > 0) {
                            need |= 1u << o;
                            ++pairs;
                            items += n;
                        }
                    }
                }
            int slot = 0;
            if (need && base < 0) {
                slot = ghost_insert(A.gtab, A.gcap, ghost_key(j, b, p1, p2, p3));
                if (slot < 0) {
                    atomicExch(A.err, 1);
                    slot = 0;
                } else {
                    atomicOr(&A.gmask[slot], need);
                }
            }
            for (int o = 0; o < 8; ++o) {
                const int q = (2 * d1 + (o >> 2)) * 36 + (2 * d2 + ((o >> 1) & 1)) * 6 + 2 * d3 + (o & 1);
                O.in[(size_t)g * 216 + q] = !((need >> o) & 1u) ? -1 : (base >= 0 ? base + o : -2 - slot);
            }
        }
        const int np = oct_pieces(sched, A.M, lm, j, leafm != 0, leafm != (1u << nout) - 1u, nullptr);
        for (int o = 16; o > 0; o >>= 1) {
            pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
            items += __shfl_xor_sync(0xffffffffu, items, o);
        }
        if (lane == 0) {
            O.np[g] = np;
            atomicMax(max_pieces, np);
            atomicAdd(&O.pairs[b], (unsigned long long)pairs);
            atomicAdd(&O.items[b], (unsigned long long)items);
        }
    }
}

// the Step-2 blocks' places (node count + id) once the ids are known
__global__ void k_oct_ghosts(int total, int n, const uint32_t* gmask, const int32_t* gid, int32_t* in) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int v = in[e];
        if (v > -2) continue;
        const int q = e % 216, slot = -2 - v;
        const unsigned oct = (((q / 36) & 1) << 2) | (((q / 6) & 1) << 1) | ((q % 6) & 1);
        in[e] = n + gid[slot] + __popc(gmask[slot] & ((1u << oct) - 1u));
    }
}

int oct_alloc(const Forest& F, const Alloc& A, OctGroups* O) {
    O->n = (F.n + 7 * F.ntrees) / 8;
    MRA_TRY(dalloc(A, &O->first, O->n));
    MRA_TRY(dalloc(A, &O->in, (size_t)O->n * 216));
    MRA_TRY(dalloc(A, &O->np, O->n));
    return MRA_OK;
}

void oct_release(const Alloc& A, OctGroups* O) {
    A.put(O->first); A.put(O->in); A.put(O->np);
    *O = OctGroups();
}

int oct_screen(const ScreenArgs& sa, const OctGroups& O, int32_t* max_pieces, cudaStream_t st) {
    const int nb = std::max(1, std::min(num_sms() * 16, (sa.F.n + 255) / 256));
    k_oct_first<<<nb, 256, 0, st>>>(sa.F, O.first);
    MRA_CK_LAUNCH();
    const int ng = std::max(1, std::min(num_sms() * 16, (O.n + 3) / 4));
    k_oct_screen<<<ng, 128, 0, st>>>(sa, O, max_pieces);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

int oct_place_ghosts(const ScreenOut& S, int n, cudaStream_t st) {
    if (S.nghost <= 0) return MRA_OK;
    const int total = S.oct.n * 216;
    k_oct_ghosts<<<std::max(1, std::min(num_sms() * 8, (total + 255) / 256)), 256, 0, st>>>(total, n, S.gmask, S.gid,
                                                                                          S.oct.in);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

__global__ void k_oct_items(int ntrees, const unsigned long long* items, const int32_t* skip, unsigned long long* out) {
    if (skip && *skip != 0) return;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < ntrees; b += gridDim.x * blockDim.x) out[b] = items[b];
}

int oct_items(const ScreenOut& S, int ntrees, const int32_t* skip, unsigned long long* n_items, cudaStream_t st) {
    k_oct_items<<<std::max(1, std::min(num_sms(), (ntrees + 127) / 128)), 128, 0, st>>>(ntrees, S.oct.items, skip,
                                                                                      n_items);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

// ------------------------------------------------------------------ Step 3, SIMT
// FP64 runs on two multiply-adds per clock and SM, so what counts is their number: the
// factored sums and the even / odd halves above.  Block per (group, slice of OCT_SLICE
// pieces); per plane b3, PC pieces at a time:
//   stage I   thread (b2, i2, i3): the six input fibers along direction 1 in registers,
//             W[a1][b2] = sum_{t1 in T1} F^{t1} x for both a1 and the PC pieces;
//   stage II  thread (piece, a1, c1, i3): V[a1][a2] = sum_{t2 in T2} F^{t2} x_2 W, both a2;
//   stage III thread (a1, a2, c1, c2), the same one for every plane and piece: the two
//             output fibers a3 = 0, 1 stay in registers.
// A slice's sum goes to its own place and k_oct_reduce adds a group's slices in order, so
// the result does not depend on how the slices are scheduled.  Lines and planes without an input box
// (outside the cube, or not needed) are passed over, and the outputs that a root does not have:
// they are most of a coarse level's 216 inputs, where a box at a time had no work for them either (an
// FP64 apply of one box at k = 12: 8.97 ms with them, 0.41 ms without; a box at a time 1.14 ms; of
// 89 boxes at k = 8 2.00, 1.56 and 2.82 ms).
template <typename T, int K>
struct OctCfg {
    static constexpr int K2 = K * K, K3 = K2 * K;
    static constexpr int W1 = K2 + K, WB = K * W1;    // a block of W: c1 stride padded
    static constexpr int V2 = K + 1, VB = K2 * V2;    // a block of V: c2 stride padded
    static constexpr bool ONE = sizeof(T) == 8 && K > 11;  // one a1 at a time (shared memory)
    static constexpr int NA = ONE ? 1 : 2;
    static constexpr int PER = NA * (6 * WB + 2 * VB) + 14 * K2;  // elements per piece in flight
    static constexpr int FIT = 100 * 1024 / (PER * (int)sizeof(T));
    static constexpr int PC = FIT >= 4 ? 4 : (FIT >= 2 ? 2 : 1);
    static constexpr int NT = (4 * K2 + 31) / 32 * 32 < 64 ? 64 : (4 * K2 + 31) / 32 * 32;
    // lines without an input are passed over, planes always; not in FP32 at k = 8, where the test costs
    // the second block of an SM (148 registers for 128: 64 Gaussians 3.86 -> 5.56 ms)
    static constexpr bool BY_LINE = sizeof(T) == 8 || K != 8;
    static size_t smem(int M) { return (size_t)PC * PER * sizeof(T) + 216 * sizeof(int) + OCT_TERM_PIECES * (size_t)M * sizeof(uint32_t); }
};

template <typename T, int K>
__global__ void __launch_bounds__(OctCfg<T, K>::NT) k_apply_oct(OctArgs P) {
    using C = OctCfg<T, K>;
    constexpr int K2 = C::K2, K3 = C::K3, PC = C::PC, NT = C::NT, NA = C::NA;
    extern __shared__ __align__(16) unsigned char oct_sm[];
    T* W = (T*)oct_sm;                              // [PC][NA][6] blocks (c1, i2, i3)
    T* V = W + PC * NA * 6 * C::WB;                 // [PC][NA][2] blocks (c1, c2, i3)
    T* Ft = V + PC * NA * 2 * C::VB;                // [PC][7] tiles
    T* Fw = Ft + PC * 7 * K2;                       // [PC][7] tiles times w_m (FP64), or the same
    int* tin = (int*)(Fw + PC * 7 * K2);            // 216
    uint32_t* list = (uint32_t*)(tin + 216);
    __shared__ unsigned s_leaf;
    __shared__ __align__(8) unsigned s_there[12];  // input boxes: 64 bits per plane b3, bit 6 b2 + b1
    __shared__ float s_wh[PC], s_wl[PC];
    if (P.skip && *P.skip != P.run_if) return;
    const int g = P.g0 + blockIdx.x / P.ns, sl = blockIdx.x % P.ns, tid = threadIdx.x;
    const int np = P.np[g], q0 = sl * OCT_SLICE;
    if (q0 >= np) return;
    const int i0 = P.first[g], tree = P.node_tree ? P.node_tree[i0] : 0;
    const int j = P.coord[4 * i0], nout = j ? 8 : 1;
    for (int e = tid; e < 384; e += NT) {
        const int b3 = e >> 6, b2 = (e & 63) / 6, b1 = (e & 63) % 6, q = b1 * 36 + b2 * 6 + b3;
        const int in = b2 < 6 ? P.in[(size_t)g * 216 + q] : -1;
        if (b2 < 6) tin[q] = in;
        const unsigned there = __ballot_sync(0xffffffffu, in >= 0);
        if ((e & 31) == 0) s_there[e >> 5] = there;
    }
    if (tid < 32) {
        const unsigned lf = __ballot_sync(0xffffffffu, tid < nout && P.leaf[i0 + (tid < nout ? tid : 0)]);
        if (tid == 0) s_leaf = lf;
        oct_pieces(P.sched + (size_t)tree * P.sl, P.M, P.lm, j, lf != 0, lf != (1u << nout) - 1u, list);
    }
    __syncthreads();
    const unsigned leafm = s_leaf;
    // the boxes b1 of line (b2, b3) that are there, read where it is asked for: registers are short
    auto line_boxes = [&](int b3, int b2) {
        return (unsigned)(*(const unsigned long long*)(s_there + 2 * b3) >> (6 * b2)) & 63u;
    };
    // this thread's output fibers (stage III): a1, a2, c1, c2; a3 = 0, 1
    const bool mine = tid < 4 * K2;
    const int oa = tid / K2, oc = tid % K2;  // a1 a2; c1 c2
    const bool exists = mine && oa < (j ? 4 : 1);
    T y[2][K], ylo[2][K];  // FP32: a pair of floats (sum and rounding error)
#pragma unroll
    for (int c = 0; c < K; ++c) y[0][c] = y[1][c] = ylo[0][c] = ylo[1][c] = (T)0;
    const T* Ftab = (const T*)P.F;
    const int q1 = min(np, q0 + OCT_SLICE);
    for (int qb = q0; qb < q1; qb += PC) {
        const int npc = min(PC, q1 - qb);
        for (int e = tid; e < npc * 7 * K2; e += NT) {
            const int pc = e / (7 * K2), m = list[qb + pc] & 0xffff;
            const T f = Ftab[((size_t)j * P.M + m) * 7 * K2 + e % (7 * K2)];
            Ft[e] = f;
            Fw[e] = sizeof(T) == 8 ? (T)(P.w[m] * f) : f;
        }
        if (tid < npc) {
            const double w = P.w[list[qb + tid] & 0xffff];
            s_wh[tid] = (float)w;
            s_wl[tid] = (float)(w - (double)(float)w);
        }
        // boxes any of the pieces reads, per direction
        unsigned m1 = 0, m2 = 0, m3 = 0;
        for (int pc = 0; pc < npc; ++pc) {
            const int box = (list[qb + pc] >> 16) & 0xff;
            m1 |= set_boxes(box >> 4);
            m2 |= set_boxes((box >> 2) & 3);
            m3 |= set_boxes(box & 3);
        }
        for (int b3 = 0; b3 < 6; ++b3) {
            if (!((m3 >> b3) & 1u)) continue;
            if (!(s_there[2 * b3] | s_there[2 * b3 + 1])) continue;  // a plane without an input adds nothing
            for (int a1p = 0; a1p < (j ? 2 / NA : 1); ++a1p) {
                __syncthreads();
                for (int task = tid; task < 6 * K2; task += NT) {
                    const int b2 = task / K2, r = task % K2;
                    const unsigned have = line_boxes(b3, b2);
                    if (!((m2 >> b2) & 1u) || (C::BY_LINE && !have)) continue;
                    T x[6][K];
#pragma unroll
                    for (int b1 = 0; b1 < 6; ++b1) {
                        const int in = tin[b1 * 36 + b2 * 6 + b3];
                        if (in >= 0 && ((m1 >> b1) & 1u)) {
                            const double* src = (in < P.n ? P.s + (size_t)in * K3 : P.gblk + (size_t)(in - P.n) * K3) + r;
#pragma unroll
                            for (int i = 0; i < K; ++i) x[b1][i] = (T)src[i * K2];
                        } else {
#pragma unroll
                            for (int i = 0; i < K; ++i) x[b1][i] = (T)0;
                        }
                    }
#pragma unroll 1
                    for (int pc = 0; pc < npc; ++pc) {
                        const int box = (list[qb + pc] >> 16) & 0xff;
#pragma unroll
                        for (int a = 0; a < NA; ++a) {
                            if (a && !j) break;  // (the root alone has the one output 0, 0, 0)
                            T out[K];
                            band_sum<T, K>(Ft + pc * 7 * K2, box >> 4, NA == 2 ? a : a1p, have & m1, x, out);
                            T* dst = W + ((pc * NA + a) * 6 + b2) * C::WB + r;
#pragma unroll
                            for (int c = 0; c < K; ++c) dst[c * C::W1] = out[c];
                        }
                    }
                }
                __syncthreads();
                for (int task = tid; task < npc * NA * K2; task += NT) {
                    const int pa = task / K2, r = task % K2, c1 = r / K, i3 = r % K, pc = pa / NA;
                    const int set = (list[qb + pc] >> 18) & 3;
                    unsigned boxes = set_boxes(set);  // of the lines that stage I has written
                    if (C::BY_LINE)
#pragma unroll
                        for (int b2 = 0; b2 < 6; ++b2)
                            if (!line_boxes(b3, b2)) boxes &= ~(1u << b2);
                    T x[6][K];
#pragma unroll
                    for (int b2 = 0; b2 < 6; ++b2) {
                        const T* src = W + (pa * 6 + b2) * C::WB + c1 * C::W1 + i3;
#pragma unroll
                        for (int i = 0; i < K; ++i) x[b2][i] = ((boxes >> b2) & 1u) ? src[i * K] : (T)0;
                    }
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        if (a && !j) break;
                        T out[K];
                        band_sum<T, K>(Ft + pc * 7 * K2, set, a, boxes, x, out);
                        T* dst = V + (pa * 2 + a) * C::VB + c1 * K * C::V2 + i3;
#pragma unroll
                        for (int c = 0; c < K; ++c) dst[c * C::V2] = out[c];
                    }
                }
                __syncthreads();
                if (exists && (NA == 2 || (oa >> 1) == a1p)) {
#pragma unroll
                    for (int pc = 0; pc < PC; ++pc) {
                        if (pc >= npc) break;
                        const int set = (list[qb + pc] >> 16) & 3;
                        const bool leaf_only = (list[qb + pc] >> 24) != 0;
                        T v[K];
                        const T* src = V + ((pc * NA + (NA == 2 ? oa >> 1 : 0)) * 2 + (oa & 1)) * C::VB + oc * C::V2;
#pragma unroll
                        for (int i = 0; i < K; ++i) v[i] = src[i];
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            const int t = a + 2 - b3;
                            if (a && !j) break;
                            if (!(set & (band_core(a, b3) ? 1 : 2))) continue;
                            if (leaf_only && !((leafm >> (2 * oa + a)) & 1u)) continue;
                            const T* F = Fw + (pc * 7 + t + 3) * K2;
                            if (sizeof(T) == 8) {
                                half_mul<T, K, 0>(F, v, y[a]);
                                if (t != 0) half_mul<T, K, 1>(F, v, y[a]);
                                continue;
                            }
                            // FP32: y += w_m (F v) in two floats, products split by fma, sums by Knuth's
                            // two-sum: about 48 bits (the low words add up in FP32), far below the
                            // rounding of the 24-bit factors in F v
                            T acc[K];
#pragma unroll
                            for (int c = 0; c < K; ++c) acc[c] = (T)0;
                            half_mul<T, K, 0>(F, v, acc);
                            if (t != 0) half_mul<T, K, 1>(F, v, acc);
                            const float wh = s_wh[pc], wl = s_wl[pc];
#pragma unroll
                            for (int c = 0; c < K; ++c) {
                                const float u = (float)acc[c], p = __fmul_rn(wh, u);
                                const float e = __fmaf_rn(wl, u, __fmaf_rn(wh, u, -p));
                                const float s0 = (float)y[a][c], s = __fadd_rn(s0, p), bb = __fsub_rn(s, s0);
                                y[a][c] = (T)s;
                                ylo[a][c] += (T)(__fadd_rn(__fsub_rn(s0, __fsub_rn(s, bb)), __fsub_rn(p, bb)) + e);
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    if (!exists) return;
    double* dst = P.part + ((size_t)blockIdx.x * 8 + 2 * oa) * K3 + (size_t)oc * K;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        if (a && !j) break;
#pragma unroll
        for (int c = 0; c < K; ++c) dst[(size_t)a * K3 + c] = (double)y[a][c] + (double)ylo[a][c];
    }
}

// ghat of a group's outputs: its slices' sums in order.  FP32 slices are added in two floats
// (Knuth's two-sum: about 48 bits, where a slice has 24) and converted once: on this part FP64
// additions and conversions run at 1/64 of the FP32 rate (120 us on 3-D Poisson k = 8 with an FP64
// conversion and addition per slice).
template <typename TP>
__global__ void k_oct_reduce(OctArgs P, int slice, int k3, const TP* part, double* out) {
    if (P.skip && *P.skip != P.run_if) return;
    const int g = P.g0 + blockIdx.x, np = P.np[g], n = (np + slice - 1) / slice;
    const int i0 = P.first[g], total = (P.coord[4 * i0] ? 8 : 1) * k3;
    const TP* src = part + (size_t)blockIdx.x * P.ns * 8 * k3;
    double* dst = out + (size_t)i0 * k3;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        if (sizeof(TP) == 8) {
            double v = 0.0;
            for (int s = 0; s < n; ++s) v += (double)src[(size_t)s * 8 * k3 + e];
            dst[e] = v;
        } else {
            float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
            for (int s = 0; s < n; ++s) {
                const float x = (float)src[(size_t)s * 8 * k3 + e], t = __fadd_rn(hi, x), b = __fsub_rn(t, hi);
                lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(x, b));
                hi = t;
            }
            dst[e] = (double)hi + (double)lo;
        }
    }
}

int oct_reduce(const OctArgs& P, int slice, int ng, const float* part, double* out, cudaStream_t st) {
    k_oct_reduce<float><<<ng, 256, 0, st>>>(P, slice, P.k * P.k * P.k, part, out);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

OctArgs oct_args(const ApplyArgs& A, const ScreenOut& S, const Forest& F) {
    OctArgs P;
    P.k = A.k; P.M = A.M; P.lm = F.lm; P.sl = S.sl; P.n = F.n;
    P.first = S.oct.first; P.in = S.oct.in; P.np = S.oct.np;
    P.coord = F.coord; P.leaf = F.leaf; P.node_tree = F.node_tree; P.sched = S.sched;
    P.s = A.s; P.gblk = A.gblk; P.F = A.F; P.w = A.w;
    return P;
}

// Partial sums of at most OCT_PART_BYTES are in flight; more groups run in batches.  Where the
// allocator has no room for as many, batches shrink by halves, as long as they are of more than
// OCT_PART_LEAST.
#define OCT_PART_BYTES ((size_t)1 << 30)
#define OCT_PART_LEAST ((size_t)64 << 20)

int oct_part_alloc(ScreenOut* S, int slice, size_t elem, int k, const Alloc& A, void** part) {
    const size_t per = (size_t)std::max(1, (S->max_pieces + slice - 1) / slice) * 8 * k * k * k * elem;
    size_t batch = std::max<size_t>(1, std::min<size_t>((size_t)S->oct.n, OCT_PART_BYTES / per));
    unsigned char* p;
    int rc;
    while ((rc = dalloc(A, &p, per * batch)) == MRA_ENOMEM && batch > 1 && per * batch > OCT_PART_LEAST) batch = (batch + 1) / 2;
    MRA_TRY(rc);
    *part = p;
    S->oct.batch = (int)batch;
    return MRA_OK;
}

template <typename T, int K>
static int oct_launch_k(OctArgs P, const ScreenOut& S, double* part, double* out, cudaStream_t st) {
    using C = OctCfg<T, K>;
    const size_t smem = C::smem(P.M);
    auto fn = k_apply_oct<T, K>;
    MRA_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    P.part = part;
    P.ns = std::max(1, (S.max_pieces + OCT_SLICE - 1) / OCT_SLICE);
    const int per = S.oct.batch;
    for (int g0 = 0; g0 < S.oct.n; g0 += per) {
        const int ng = std::min(per, S.oct.n - g0);
        P.g0 = g0;
        fn<<<(unsigned)(ng * P.ns), C::NT, smem, st>>>(P);
        MRA_CK_LAUNCH();
        k_oct_reduce<double><<<ng, 256, 0, st>>>(P, OCT_SLICE, C::K3, part, out);
        MRA_CK_LAUNCH();
    }
    return MRA_OK;
}

template <typename T>
static int oct_launch_t(const OctArgs& P, const ScreenOut& S, double* part, double* out, cudaStream_t st) {
    switch (P.k) {
        case 1: return oct_launch_k<T, 1>(P, S, part, out, st);
        case 2: return oct_launch_k<T, 2>(P, S, part, out, st);
        case 3: return oct_launch_k<T, 3>(P, S, part, out, st);
        case 4: return oct_launch_k<T, 4>(P, S, part, out, st);
        case 5: return oct_launch_k<T, 5>(P, S, part, out, st);
        case 6: return oct_launch_k<T, 6>(P, S, part, out, st);
        case 7: return oct_launch_k<T, 7>(P, S, part, out, st);
        case 8: return oct_launch_k<T, 8>(P, S, part, out, st);
        case 9: return oct_launch_k<T, 9>(P, S, part, out, st);
        case 10: return oct_launch_k<T, 10>(P, S, part, out, st);
        case 11: return oct_launch_k<T, 11>(P, S, part, out, st);
        case 12: return oct_launch_k<T, 12>(P, S, part, out, st);
    }
    set_error("k=%d not supported by the sibling-group apply", P.k);
    return MRA_EINVAL;
}

int oct_slice_simt() { return OCT_SLICE; }

// P.skip / P.run_if as wanted; part: oct_part_alloc(S, oct_slice_simt(), sizeof(double), ...)
int oct_launch(const OctArgs& P, const ScreenOut& S, int precision, double* part, double* out, cudaStream_t st) {
    return precision == MRA_PREC_FP64 ? oct_launch_t<double>(P, S, part, out, st)
                                      : oct_launch_t<float>(P, S, part, out, st);
}

}  // namespace mra
