// One direction of a sibling group's sums: inputs b = 0..5, outputs a = 0, 1, t = a + 2 - b (see
// apply_oct.cu), and the classes of translations as products of per-direction sets.
#pragma once
#include <stdint.h>

namespace mra {

// The classes {S : bit S of A set} of `dims` directions as products of per-direction sets
// (1 core, 2 off, 3 both), two bits per direction from direction 1 at the top.
struct PieceSet {
    int n;
    uint8_t box[4];
};

constexpr void piece_split(int dims, int A, int prefix, PieceSet& P) {
    if (A == 0) return;
    if (A == (1 << (dims + 1)) - 1) {  // every class: all translations of the rest
        int b = prefix;
        for (int d = 0; d < dims; ++d) b = (b << 2) | 3;
        P.box[P.n++] = (uint8_t)b;
        return;
    }
    const int in = A >> 1, off = A & ((1 << dims) - 1);  // classes left with this direction core / off core
    if (in == off) {
        piece_split(dims - 1, in, (prefix << 2) | 3, P);
        return;
    }
    piece_split(dims - 1, in, (prefix << 2) | 1, P);
    piece_split(dims - 1, off, (prefix << 2) | 2, P);
}

// whether input b lies in the core of output a in a direction
__device__ inline bool band_core(int a, int b) { return b >= 1 + a && b <= 3 + a; }

// boxes b of a direction that some a in {0, 1} reaches by a translation of the set
__device__ __forceinline__ unsigned set_boxes(int set) { return set == 1 ? 0x1eu : (set == 2 ? 0x33u : 0x3fu); }

// out += F x over the entries with c + i even (PAR 0) or odd (PAR 1)
template <typename T, int K, int PAR>
__device__ __forceinline__ void half_mul(const T* F, const T* x, T* out) {
#pragma unroll
    for (int c = 0; c < K; ++c)
#pragma unroll
        for (int i = (c + PAR) & 1; i < K; i += 2) out[c] += F[c * K + i] * x[i];
}

// out += F x; FP32 sums each product on its own before adding it (shorter chains of roundings)
template <typename T, int K>
__device__ __forceinline__ void full_mul(const T* F, const T* x, T* out) {
    if (sizeof(T) == 8) {
        half_mul<T, K, 0>(F, x, out);
        half_mul<T, K, 1>(F, x, out);
        return;
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
        T acc = (T)0;
#pragma unroll
        for (int i = 0; i < K; ++i) acc += F[c * K + i] * x[i];
        out[c] += acc;
    }
}

// out += F^t xp + F^{-t} xm.  FP32 takes the two products: the rounding of the sums would
// show in the result (3.7e-8 against 2.9e-8 relative on the k = 5 case).
template <typename T, int K>
__device__ __forceinline__ void pair_mul(const T* Ft, const T* Fm, const T* xp, const T* xm, T* out) {
    if (sizeof(T) == 4) {
        full_mul<T, K>(Ft, xp, out);
        full_mul<T, K>(Fm, xm, out);
        return;
    }
    T s[K], d[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        s[i] = xp[i] + xm[i];
        d[i] = xp[i] - xm[i];
    }
    half_mul<T, K, 0>(Ft, s, out);
    half_mul<T, K, 1>(Ft, d, out);
}

// out = sum over b of F^{a + 2 - b} x[b], the translations of `set` (1 core, 2 off, 3 both);
// F: tiles of t = -3..3; have: the boxes b whose x may differ from zero.  FP64 passes over the others'
// products: near the cube's faces and on coarse levels most boxes are outside (585 boxes at k = 8: apply 2.17
// ms -> 1.81).  Not at k = 12, whose six fibers do not fit the registers: the branches cost more in spills
// than they save (9.1 ms -> 11.0); nor in FP32, whose products cost less than the branches (0.95 of the
// time without them on average over k = 2..10).
template <typename T, int K>
__device__ __forceinline__ void band_sum(const T* F, int set, int a, unsigned have, const T (*x)[K], T* out) {
    constexpr int K2 = K * K;
    if (sizeof(T) == 4 || K == 12) have = 0x3fu;
#pragma unroll
    for (int c = 0; c < K; ++c) out[c] = (T)0;
    if (a == 0) {
        if (set & 1) {
            if (have & 0x0au) pair_mul<T, K>(F + 4 * K2, F + 2 * K2, x[1], x[3], out);
            if (have & 0x04u) half_mul<T, K, 0>(F + 3 * K2, x[2], out);
        }
        if (set & 2) {
            if (have & 0x11u) pair_mul<T, K>(F + 5 * K2, F + K2, x[0], x[4], out);
            if (have & 0x20u) full_mul<T, K>(F, x[5], out);
        }
    } else {
        if (set & 1) {
            if (have & 0x14u) pair_mul<T, K>(F + 4 * K2, F + 2 * K2, x[2], x[4], out);
            if (have & 0x08u) half_mul<T, K, 0>(F + 3 * K2, x[3], out);
        }
        if (set & 2) {
            if (have & 0x22u) pair_mul<T, K>(F + 5 * K2, F + K2, x[1], x[5], out);
            if (have & 0x01u) full_mul<T, K>(F + 6 * K2, x[0], out);
        }
    }
}

}  // namespace mra
