// The pieces of a sibling group's schedule (see apply_oct.cu).
#pragma once
#include "apply_common.cuh"
#include "band_sum.cuh"

namespace mra {

struct PieceTable {
    PieceSet p[16];
};

constexpr PieceTable make_pieces() {
    PieceTable T{};
    for (int A = 0; A < 16; ++A) piece_split(3, A, 0, T.p[A]);
    return T;
}

// every translation class (bit d of v: core in direction d) is in exactly one piece of A when A has
// its number of core directions, in none otherwise
constexpr bool pieces_cover_classes(int dims) {
    for (int A = 0; A < 1 << (dims + 1); ++A) {
        PieceSet P{};
        piece_split(dims, A, 0, P);
        for (int v = 0; v < 1 << dims; ++v) {
            int S = 0, in = 0;
            for (int d = 0; d < dims; ++d) S += (v >> d) & 1;
            for (int i = 0; i < P.n; ++i) {
                bool all = true;
                for (int d = 0; d < dims; ++d) all = all && ((P.box[i] >> (2 * d)) & (((v >> d) & 1) ? 1 : 2));
                in += all;
            }
            if (in != ((A >> S) & 1)) return false;
        }
    }
    return true;
}
static_assert(pieces_cover_classes(3), "a term's pieces are its kept classes");

// most pieces of a term: its classes' products, or (J_m > j, leaf and internal siblings) those of the
// classes but the core, and the core for the leaves.  {0, 2} beside the core takes five.
constexpr int most_pieces() {
    const PieceTable T = make_pieces();
    int most = 0;
    for (int A = 0; A < 16; ++A) {
        const int n = (A & 8) && T.p[A & 7].n + 1 > T.p[A].n ? T.p[A & 7].n + 1 : T.p[A].n;
        most = n > most ? n : most;
    }
    return most;
}
#define OCT_TERM_PIECES 5  // entries of a group's piece list per term
static_assert(most_pieces() <= OCT_TERM_PIECES, "a group's pieces fit its list");

static __constant__ PieceTable c_pieces = make_pieces();

#define PIECE_CCC 0x15  // core in every direction

// The pieces of a group at level j, by one warp: non-core pieces first, then the core
// ones, each in increasing m.  out[i] = m | box << 16 | leaf_only << 24 (NULL: count only); at most
// OCT_TERM_PIECES M of them.
static __device__ int oct_pieces(const int32_t* sched, int M, int lm, int j, bool any_leaf, bool any_int, uint32_t* out) {
    const int lane = threadIdx.x & 31;
    const int32_t* m1 = sched + M + 4 * j;
    const int32_t* m2 = sched + M + 4 * lm + 4 * j;
    int lo[4], hi[4], first = M, last = -1;
    for (int S = 0; S < 4; ++S) {
        lo[S] = m1[S];
        hi[S] = m2[S];
        if (hi[S] >= lo[S]) {
            first = min(first, lo[S]);
            last = max(last, hi[S]);
        }
    }
    int total = 0;
    for (int pass = 0; pass < 2; ++pass)
        for (int m0 = first; m0 <= last; m0 += 32) {
            const int m = m0 + lane;
            int A = 0;
            bool extra = false;  // the core for the leaf outputs only
            if (m <= last) {
                const int jm = sched[m];
                if (jm >= j) {
                    for (int S = 0; S < 4; ++S) A |= (m >= lo[S] && m <= hi[S]) << S;
                    if (jm > j && any_int && (A & 8)) {
                        A &= 7;
                        extra = any_leaf;
                    }
                }
            }
            const PieceSet& P = c_pieces.p[A];
            int n = 0;
            for (int i = 0; i < P.n; ++i) n += (P.box[i] == PIECE_CCC) == (pass == 1);
            n += pass == 1 && extra;
            int at = n;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += v;
            }
            const int sum = __shfl_sync(0xffffffffu, at, 31);
            if (out) {
                at += total - n;
                for (int i = 0; i < P.n; ++i)
                    if ((P.box[i] == PIECE_CCC) == (pass == 1)) out[at++] = (uint32_t)m | ((uint32_t)P.box[i] << 16);
                if (pass == 1 && extra) out[at++] = (uint32_t)m | ((uint32_t)PIECE_CCC << 16) | (1u << 24);
            }
            total += sum;
        }
    return total;
}

}  // namespace mra
