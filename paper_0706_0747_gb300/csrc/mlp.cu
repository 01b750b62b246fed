// The learned schedule's network: a 3 x 128 ReLU MLP with FP16 weights and
// activations, FP32 accumulation, FP32 master weights and Adam, trained and
// run by the kernels below.  The paper has no learned part; the network
// predicts, per output box, the term cut-offs of the exact per-pair screen
// (Sec. 4's term ranges narrowed per box), which the apply then checks.
//
// Parameter order (one FP32 vector): W1 [H][n_in], b1 [H], W2 [H][H], b2,
// W3 [H][H], b3, W4 [n_out][H], b4 [n_out], row-major.  Per layer l the
// FP16 copies hold W_l both row-major ([out][in], for the backward data pass)
// and transposed ([in][out], for the forward pass), so a thread per output
// unit reads a coalesced row either way.
//
// Loss per box (n_out = 12, per class S: [e_S, lo_S, hi_S], targets
// [E_S, LO_S, HI_S]):
//   sum_S softplus(e_S) - E_S e_S + (1 - E_S) ((lo_S - LO_S)^2 + (hi_S - HI_S)^2)
// averaged over the batch.
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "mra_internal.cuh"

#define MLP_H 128
#define MLP_RB 32  // rows per block

struct mra_mlp {
    uint32_t magic = 0;
    int n_in = 0, n_out = 0;
    int64_t np = 0;                 // parameters
    int64_t off_w[4], off_b[4];     // offsets of W_l, b_l in the flat vector
    int din[4], dout[4];
    float* master = nullptr;        // FP32 parameters
    float* grad = nullptr;
    float* m = nullptr;             // Adam moments
    float* v = nullptr;
    __half* w16 = nullptr;          // per layer [out][in] then [in][out], at off_w * 2
    int step = 0;
    // activations of the last training batch (capacity rows)
    int64_t cap = 0;
    __half *h1 = nullptr, *h2 = nullptr, *h3 = nullptr;
    float *y = nullptr, *d3 = nullptr, *d2 = nullptr, *d1 = nullptr, *dy = nullptr;
    float* part = nullptr;          // the row slices' weight gradients (room for part_n floats)
    int64_t part_n = 0;
    double* loss = nullptr;
    mra::Alloc A;
};

namespace mra {

// Rows are independent of each other through the whole network, the loss and the backward
// data pass, so one block carries MLP_RB rows through all of it with the activations in
// shared memory; what bounds it is then the multiply-adds (2 din dout per row and layer) and
// the shared-memory reads that feed them.  A thread's tile is 4 rows x 4 outputs: per input i
// one 16-byte broadcast of activations and one 8-byte weight read for 16 multiply-adds.
// (One output x 32 rows per thread, a launch per layer: one shared read per multiply-add,
// 67 us per 128 x 128 layer at 4,096 rows.)  Each output sums its bias, then the products in
// increasing i, as a chain of fused multiply-adds.
#define MLP_NT 256
#define MLP_XS 36   // activations [i][row], rows padded to a multiple of 4
#define MLP_WI 64   // weight rows staged at a time

struct MlpTile {
    float v[4][4];  // [row][output]
};

// rows 4 warp.., outputs o0 + 4 lane..: bias + sum_i xs[i][row] Wio[i][o]; Wio half [din][dout]
// in global memory (dout a multiple of 4 or read element by element)
__device__ void mlp_layer(const float* xs, int din, const __half* Wio, int dout, int o0, const float* bias, __half* ws,
                          MlpTile& t) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int o = o0 + 4 * lane + q;
        const float b = bias && o < dout ? bias[o] : 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r) t.v[r][q] = b;
    }
    for (int i0 = 0; i0 < din; i0 += MLP_WI) {
        const int ni = min(MLP_WI, din - i0);
        __syncthreads();
        if (dout % 8 == 0 && o0 + 128 <= dout) {  // whole rows of 16-byte words
#pragma unroll
            for (int q = 0; q < MLP_WI * 16 / MLP_NT; ++q) {
                const int e = threadIdx.x + q * MLP_NT, i = e >> 4;
                if (i < ni) ((uint4*)ws)[e] = *(const uint4*)(Wio + (size_t)(i0 + i) * dout + o0 + (e & 15) * 8);
            }
        } else {
            for (int e = threadIdx.x; e < ni * 128; e += MLP_NT) {
                const int i = e >> 7, o = o0 + (e & 127);
                ws[e] = o < dout ? Wio[(size_t)(i0 + i) * dout + o] : __half(0.0f);
            }
        }
        __syncthreads();
        if (o0 + 4 * lane < dout)
#pragma unroll 4
            for (int i = 0; i < ni; ++i) {
                const float4 x = *(const float4*)(xs + (size_t)(i0 + i) * MLP_XS + 4 * warp);
                const uint2 w2 = *(const uint2*)(ws + i * 128 + 4 * lane);
                const float2 wa = __half22float2(*(const __half2*)&w2.x), wb = __half22float2(*(const __half2*)&w2.y);
                const float xr[4] = {x.x, x.y, x.z, x.w}, w[4] = {wa.x, wa.y, wb.x, wb.y};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int q = 0; q < 4; ++q) t.v[r][q] = fmaf(w[q], xr[r], t.v[r][q]);
            }
    }
}

struct MlpArgs {
    int64_t n;
    int n_in, n_out;
    const float* x;
    const __half *wt[4], *wr[4];  // [in][out] and [out][in] copies
    const float* b[4];
    float* y;
    __half* h[3];                 // activations kept for the gradient (NULL: not kept)
    // training: targets, dL/dy, the data gradients of the hidden layers, the loss
    const float* target;
    float *dy, *d[3];
    double* loss;
};

template <bool TRAIN>
__global__ void __launch_bounds__(MLP_NT) k_mlp_rows(MlpArgs A) {
    extern __shared__ __align__(16) float mlp_sm[];
    __shared__ __align__(16) __half ws[MLP_WI * 128];
    __shared__ double red[MLP_NT / 32];
    float* xa = mlp_sm;                                     // [max(n_in, 128)][MLP_XS]
    float* xb = xa + (size_t)max(A.n_in, MLP_H) * MLP_XS;   // [128][MLP_XS]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * MLP_RB;
    const int rows = (int)min((int64_t)MLP_RB, A.n - r0);
    for (int e = tid; e < MLP_RB * A.n_in; e += MLP_NT) {
        const int r = e / A.n_in, i = e - r * A.n_in;
        xa[i * MLP_XS + r] = r < rows ? A.x[(r0 + r) * A.n_in + i] : 0.0f;
    }
    MlpTile t;
    unsigned on[3] = {0, 0, 0};  // hidden units of this thread's tile above zero
    float *in = xa, *out = xb;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        mlp_layer(in, l ? MLP_H : A.n_in, A.wt[l], MLP_H, 0, A.b[l], ws, t);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            __align__(8) __half hv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                hv[q] = __float2half_rn(fmaxf(t.v[r][q], 0.0f));
                t.v[r][q] = __half2float(hv[q]);
                on[l] |= (unsigned)(t.v[r][q] > 0.0f) << (4 * r + q);
            }
            if (TRAIN && 4 * warp + r < rows)
                *(uint2*)(A.h[l] + (r0 + 4 * warp + r) * MLP_H + 4 * lane) = *(const uint2*)hv;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *(float4*)(out + (4 * lane + q) * MLP_XS + 4 * warp) = make_float4(t.v[0][q], t.v[1][q], t.v[2][q], t.v[3][q]);
        float* s = in;
        in = out;
        out = s;
    }
    for (int o0 = 0; o0 < A.n_out; o0 += 128) {
        mlp_layer(in, MLP_H, A.wt[3], A.n_out, o0, A.b[3], ws, t);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int o = o0 + 4 * lane + q;
                if (o < A.n_out && 4 * warp + r < rows) A.y[(r0 + 4 * warp + r) * A.n_out + o] = t.v[r][q];
                if (TRAIN && o < 12) out[o * MLP_XS + 4 * warp + r] = t.v[r][q];
            }
    }
    if (!TRAIN) return;
    // loss and dL/dy (divided by n), FP64: thread (row, class)
    __syncthreads();
    double acc = 0.0;
    if (tid < MLP_RB * 4) {
        const int r = tid >> 2, S = tid & 3;
        float g[3] = {0.0f, 0.0f, 0.0f};
        if (r < rows) {
            const double inv = 1.0 / (double)A.n;
            const float e = out[(3 * S) * MLP_XS + r], lo = out[(3 * S + 1) * MLP_XS + r], hi = out[(3 * S + 2) * MLP_XS + r];
            const float* T = A.target + (r0 + r) * 12 + 3 * S;
            const float E = T[0], LO = T[1], HI = T[2];
            const double z = exp(-fabs((double)e));  // softplus and sigmoid from one exponential
            const double sp = fmax((double)e, 0.0) + log1p(z);
            const double sg = (e > 0.0f ? 1.0 : z) / (1.0 + z);
            acc = sp - (double)E * e + (1.0 - E) * ((double)(lo - LO) * (lo - LO) + (double)(hi - HI) * (hi - HI));
            g[0] = (float)((sg - E) * inv);
            g[1] = (float)(2.0 * (1.0 - E) * (lo - LO) * inv);
            g[2] = (float)(2.0 * (1.0 - E) * (hi - HI) * inv);
            for (int q = 0; q < 3; ++q) A.dy[(r0 + r) * 12 + 3 * S + q] = g[q];
        }
        for (int q = 0; q < 3; ++q) out[(3 * S + q) * MLP_XS + r] = g[q];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < MLP_RB * 4 / 32; ++w) s += red[w];
        atomicAdd(A.loss, s / (double)A.n);
    }
    // back through the layers: d_l = (d_{l+1} W) where the unit was on
    float* g = out;
    float* nx = in;
#pragma unroll
    for (int l = 2; l >= 0; --l) {
        mlp_layer(g, l == 2 ? A.n_out : MLP_H, A.wr[l + 1], MLP_H, 0, nullptr, ws, t);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#pragma unroll
            for (int q = 0; q < 4; ++q) t.v[r][q] = ((on[l] >> (4 * r + q)) & 1u) ? t.v[r][q] : 0.0f;
            if (4 * warp + r < rows)
                *(float4*)(A.d[l] + (r0 + 4 * warp + r) * MLP_H + 4 * lane) = make_float4(t.v[r][0], t.v[r][1], t.v[r][2], t.v[r][3]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *(float4*)(nx + (4 * lane + q) * MLP_XS + 4 * warp) = make_float4(t.v[0][q], t.v[1][q], t.v[2][q], t.v[3][q]);
        float* s = g;
        g = nx;
        nx = s;
    }
}

// Weight gradients gW[o][i] = sum_r d[r][o] h[r][i], gb[o] = sum_r d[r][o] of all layers in one
// launch: block (row slice, layer, tile of 128 x 128), 8 x 8 outputs per thread, 32 rows at a
// time in shared memory; the slices' sums are added in order afterwards, so the result does
// not depend on scheduling.  (A thread per weight walking all rows by itself: 2.7 ms for the
// four layers at 4,096 rows, a serial chain of 4,096 loads.)
struct WgradArgs {
    int64_t n, np;
    int rows;  // rows per slice
    const float* d[4];
    const void* h[4];   // layer 0: float x, else half
    int din[4], dout[4], ti[4];   // ti: tiles along i
    int tile0[5];       // first tile of each layer
    int64_t off_w[4], off_b[4];
    float* part;        // [slices][np]
    bool x16;           // x starts on a 16-byte boundary
};

__global__ void __launch_bounds__(256) k_mlp_wgrad(WgradArgs A) {
    __shared__ __align__(16) float ds[32][128], hs[32][128];
    int l = 0;
    while (l < 3 && (int)blockIdx.y >= A.tile0[l + 1]) ++l;
    const int tile = blockIdx.y - A.tile0[l], o0 = tile / A.ti[l] * 128, i0 = tile % A.ti[l] * 128;
    const int din = A.din[l], dout = A.dout[l], tid = threadIdx.x, to = tid >> 4, ti = tid & 15;
    const int64_t r0 = (int64_t)blockIdx.x * A.rows, r1 = min(A.n, r0 + A.rows);
    float acc[8][8], gb = 0.0f;
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.0f;
    const bool busy = o0 + 4 * to < dout && i0 + 4 * ti < din;
    for (int64_t r = r0; r < r1; r += 32) {
        __syncthreads();
        // four columns at a time (every row starts on a 16-byte boundary when the width is a multiple of 4)
        const bool vd = dout % 4 == 0, vh = din % 4 == 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + q * 256, rr = e >> 5, c = (e & 31) * 4;
            const int64_t row = r + rr;
            float4 dv = make_float4(0.0f, 0.0f, 0.0f, 0.0f), hv = dv;
            if (row < r1) {
                const float* dp = A.d[l] + row * dout + o0 + c;
                if (vd && o0 + c < dout) dv = *(const float4*)dp;
                else if (!vd) {
                    float* v = (float*)&dv;
                    for (int z = 0; z < 4; ++z)
                        if (o0 + c + z < dout) v[z] = dp[z];
                }
                if (vh && i0 + c < din) {
                    if (l) {
                        const uint2 h2 = *(const uint2*)((const __half*)A.h[l] + row * din + i0 + c);
                        const float2 a = __half22float2(*(const __half2*)&h2.x), b = __half22float2(*(const __half2*)&h2.y);
                        hv = make_float4(a.x, a.y, b.x, b.y);
                    } else if (A.x16) {
                        hv = *(const float4*)((const float*)A.h[0] + row * din + i0 + c);
                    }
                }
                if (!vh || (l == 0 && !A.x16)) {
                    float* v = (float*)&hv;
                    for (int z = 0; z < 4; ++z)
                        if (i0 + c + z < din)
                            v[z] = l ? __half2float(((const __half*)A.h[l])[row * din + i0 + c + z]) : ((const float*)A.h[0])[row * din + i0 + c + z];
                }
            }
            *(float4*)&ds[rr][c] = dv;
            *(float4*)&hs[rr][c] = hv;
        }
        __syncthreads();
        if (busy)
#pragma unroll 4
            for (int rr = 0; rr < 32; ++rr) {
                // outputs 4 to + {0..3, 64..67}, inputs 4 ti + {0..3, 64..67}
                const float4 da = *(const float4*)&ds[rr][4 * to], db = *(const float4*)&ds[rr][64 + 4 * to];
                const float4 ha = *(const float4*)&hs[rr][4 * ti], hb = *(const float4*)&hs[rr][64 + 4 * ti];
                const float dv[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
                const float hv[8] = {ha.x, ha.y, ha.z, ha.w, hb.x, hb.y, hb.z, hb.w};
#pragma unroll
                for (int a = 0; a < 8; ++a)
#pragma unroll
                    for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(dv[a], hv[b], acc[a][b]);
            }
        if (i0 == 0 && tid < 128)
            for (int rr = 0; rr < 32; ++rr) gb += ds[rr][tid];
    }
    float* part = A.part + (size_t)blockIdx.x * A.np;
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int o = o0 + 4 * to + (a & 3) + (a >> 2) * 64, i = i0 + 4 * ti + (b & 3) + (b >> 2) * 64;
            if (o < dout && i < din) part[A.off_w[l] + (size_t)o * din + i] = acc[a][b];
        }
    if (i0 == 0 && tid < 128 && o0 + tid < dout) part[A.off_b[l] + o0 + tid] = gb;
}

__global__ void k_mlp_wsum(int64_t np, int slices, const float* part, float* g) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np; e += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int q = 0; q < slices; ++q) s += part[(size_t)q * np + e];
        g[e] = s;
    }
}

__global__ void k_adam(int64_t np, float* p, const float* g, float* m, float* v, float lr, float c1, float c2) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np; e += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[e];
        const float mi = 0.9f * m[e] + 0.1f * gi;
        const float vi = 0.999f * v[e] + 0.001f * gi * gi;
        m[e] = mi;
        v[e] = vi;
        p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    }
}

// FP16 copies of the weight matrices: [out][in] at 2 off_w, [in][out] right after
struct W16Layout {
    int64_t off_w[4];
    int din[4], dout[4];
};

__global__ void k_refresh16(W16Layout L, const float* p, __half* w16) {
    for (int l = 0; l < 4; ++l) {
        const int64_t sz = (int64_t)L.din[l] * L.dout[l];
        __half* rm = w16 + 2 * L.off_w[l];
        __half* tr = rm + sz;
        for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < sz; e += (int64_t)gridDim.x * blockDim.x) {
            const int o = (int)(e / L.din[l]), i = (int)(e % L.din[l]);
            const __half h = __float2half_rn(p[L.off_w[l] + e]);
            rm[e] = h;
            tr[(size_t)i * L.dout[l] + o] = h;
        }
    }
}

static W16Layout w16_layout(const mra_mlp* M) {
    W16Layout L;
    for (int l = 0; l < 4; ++l) {
        L.off_w[l] = M->off_w[l];
        L.din[l] = M->din[l];
        L.dout[l] = M->dout[l];
    }
    return L;
}

static const __half* w_rowmajor(const mra_mlp* M, int l) { return M->w16 + 2 * M->off_w[l]; }
static const __half* w_trans(const mra_mlp* M, int l) {
    return M->w16 + 2 * M->off_w[l] + (int64_t)M->din[l] * M->dout[l];
}

static int refresh16(const mra_mlp* M, cudaStream_t st) {
    k_refresh16<<<num_sms(), 256, 0, st>>>(w16_layout(M), M->master, M->w16);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

static int ensure_cap(mra_mlp* M, int64_t n) {
    if (n <= M->cap) return MRA_OK;
    const Alloc& A = M->A;
    A.put(M->h1); A.put(M->h2); A.put(M->h3); A.put(M->y); A.put(M->d3); A.put(M->d2); A.put(M->d1); A.put(M->dy);
    // a failure below leaves no stale buffer behind (capacity 0, the rest NULL)
    M->h1 = M->h2 = M->h3 = nullptr;
    M->y = M->d3 = M->d2 = M->d1 = M->dy = nullptr;
    M->cap = 0;
    int64_t c = std::max<int64_t>(n, 4096);
    MRA_TRY(dalloc(A, &M->h1, c * MLP_H));
    MRA_TRY(dalloc(A, &M->h2, c * MLP_H));
    MRA_TRY(dalloc(A, &M->h3, c * MLP_H));
    MRA_TRY(dalloc(A, &M->y, c * M->n_out));
    MRA_TRY(dalloc(A, &M->dy, c * M->n_out));
    MRA_TRY(dalloc(A, &M->d3, c * MLP_H));
    MRA_TRY(dalloc(A, &M->d2, c * MLP_H));
    MRA_TRY(dalloc(A, &M->d1, c * MLP_H));
    M->cap = c;
    return MRA_OK;
}

// Rows per slice for a batch of n, and where the slices' gradients go: a buffer that the network keeps,
// as it keeps its activations (a block of the stream it was made on could reach another network
// that trains on another stream); the gradient itself when there is one slice.  It is made for the
// most slices at once, so that a larger batch does not give it back while an earlier step uses it.
// Fewer slices where the allocator has no room for as many.
#define MLP_SLICES 64
static float* slice_room(mra_mlp* M, int64_t n, int* rows) {
    for (int want = MLP_SLICES;; want /= 2) {
        *rows = (int)std::max<int64_t>(32, ((n + want - 1) / want + 31) / 32 * 32);
        const int64_t slices = (n + *rows - 1) / *rows;
        if (slices == 1) return M->grad;
        if (slices * M->np <= M->part_n) return M->part;
        M->A.put(M->part);
        M->part = nullptr;
        M->part_n = 0;
        const int64_t room = (want == MLP_SLICES ? want : slices) * M->np;
        if (dalloc(M->A, &M->part, room) == MRA_OK) {
            M->part_n = room;
            return M->part;
        }
    }
}

static MlpArgs mlp_args(const mra_mlp* M, const float* x, int64_t n, float* y) {
    MlpArgs A{};
    A.n = n;
    A.n_in = M->n_in;
    A.n_out = M->n_out;
    A.x = x;
    for (int l = 0; l < 4; ++l) {
        A.wt[l] = w_trans(M, l);
        A.wr[l] = w_rowmajor(M, l);
        A.b[l] = M->master + M->off_b[l];
    }
    A.y = y;
    return A;
}

template <bool TRAIN>
static int mlp_rows(const MlpArgs& A, cudaStream_t st) {
    if (A.n <= 0) return MRA_OK;
    const int64_t blocks = (A.n + MLP_RB - 1) / MLP_RB;
    const size_t smem = (size_t)(std::max(A.n_in, MLP_H) + MLP_H) * MLP_XS * sizeof(float);
    MRA_CK(cudaFuncSetAttribute(k_mlp_rows<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_mlp_rows<TRAIN><<<(unsigned)blocks, MLP_NT, smem, st>>>(A);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

// forward, loss and gradients of the batch into M->grad (loss into M->loss)
static int mlp_loss_grad_impl(mra_mlp* M, const float* x, const float* t, int64_t n, cudaStream_t st) {
    MRA_TRY(ensure_cap(M, n));
    MlpArgs A = mlp_args(M, x, n, M->y);
    A.h[0] = M->h1; A.h[1] = M->h2; A.h[2] = M->h3;
    A.target = t;
    A.dy = M->dy;
    A.d[0] = M->d1; A.d[1] = M->d2; A.d[2] = M->d3;
    A.loss = M->loss;
    MRA_CK(cudaMemsetAsync(M->loss, 0, sizeof(double), st));
    MRA_TRY(mlp_rows<true>(A, st));
    // row slices: about an SM each for a 128 x 128 layer, at least 32 rows, at most MLP_SLICES
    WgradArgs W{};
    W.n = n;
    W.np = M->np;
    W.part = slice_room(M, n, &W.rows);
    const int slices = (int)((n + W.rows - 1) / W.rows);
    const float* d[4] = {M->d1, M->d2, M->d3, M->dy};
    const void* h[4] = {x, M->h1, M->h2, M->h3};
    for (int l = 0; l < 4; ++l) {
        W.d[l] = d[l];
        W.h[l] = h[l];
        W.din[l] = M->din[l];
        W.dout[l] = M->dout[l];
        W.off_w[l] = M->off_w[l];
        W.off_b[l] = M->off_b[l];
        W.ti[l] = (M->din[l] + 127) / 128;
        W.tile0[l + 1] = W.tile0[l] + W.ti[l] * ((M->dout[l] + 127) / 128);
    }
    W.x16 = ((uintptr_t)x & 15) == 0;
    k_mlp_wgrad<<<dim3(slices, W.tile0[4]), 256, 0, st>>>(W);
    MRA_CK_LAUNCH();
    if (slices == 1) return MRA_OK;
    k_mlp_wsum<<<(unsigned)std::min<int64_t>(num_sms() * 4, (M->np + 255) / 256), 256, 0, st>>>(M->np, slices, W.part, M->grad);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

}  // namespace mra

using namespace mra;

static bool mlp_ok(const mra_mlp* M) { return M && M->magic == MRA_MLP_MAGIC; }

namespace mra {
const mra_mlp* mlp_checked(const void* h) {
    const mra_mlp* M = (const mra_mlp*)h;
    return mlp_ok(M) ? M : nullptr;
}
int mlp_forward(const mra_mlp* M, const float* x, int64_t n, float* y, const Alloc& A, cudaStream_t st) {
    (void)A;
    return mlp_rows<false>(mlp_args(M, x, n, y), st);
}
int mlp_n_in(const mra_mlp* M) { return M->n_in; }
int mlp_n_out(const mra_mlp* M) { return M->n_out; }
}  // namespace mra

// splitmix64: seeded parameter initialisation on the host
static uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

extern "C" {

int mra_mlp_create(int n_in, int n_out, const float* params_host, unsigned long long seed, const mra_alloc* alloc,
                   void* stream, mra_mlp** out) {
    if (!out) { set_error("out is NULL"); return MRA_EINVAL; }
    *out = nullptr;
    if (n_in < 1 || n_in > 1024 || n_out < 1 || n_out > 1024) { set_error("n_in, n_out must lie in [1, 1024]"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    mra_mlp* M = new mra_mlp();
    M->magic = MRA_MLP_MAGIC;
    M->n_in = n_in;
    M->n_out = n_out;
    M->A = make_alloc(alloc, stream);
    const int din[4] = {n_in, MLP_H, MLP_H, MLP_H}, dout[4] = {MLP_H, MLP_H, MLP_H, n_out};
    int64_t o = 0;
    for (int l = 0; l < 4; ++l) {
        M->din[l] = din[l];
        M->dout[l] = dout[l];
        M->off_w[l] = o;
        o += (int64_t)din[l] * dout[l];
        M->off_b[l] = o;
        o += dout[l];
    }
    M->np = o;
    std::vector<float> h(o, 0.0f);
    if (params_host) {
        memcpy(h.data(), params_host, o * sizeof(float));
    } else {
        // He-uniform weights, zero biases
        uint64_t s = seed;
        for (int l = 0; l < 4; ++l) {
            const double a = sqrt(6.0 / din[l]);
            for (int64_t e = 0; e < (int64_t)din[l] * dout[l]; ++e) {
                const double u = (double)(splitmix(s) >> 11) * (1.0 / 9007199254740992.0);
                h[M->off_w[l] + e] = (float)((2.0 * u - 1.0) * a);
            }
        }
    }
    int rc = MRA_OK;
    const Alloc& A = M->A;
    if (rc == MRA_OK) rc = dalloc(A, &M->master, o);
    if (rc == MRA_OK) rc = dalloc(A, &M->grad, o);
    if (rc == MRA_OK) rc = dalloc(A, &M->m, o);
    if (rc == MRA_OK) rc = dalloc(A, &M->v, o);
    if (rc == MRA_OK) rc = dalloc(A, &M->w16, 2 * o);
    if (rc == MRA_OK) rc = dalloc(A, &M->loss, 1);
    if (rc == MRA_OK) {
        cudaError_t e = cudaMemcpyAsync(M->master, h.data(), o * sizeof(float), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(M->m, 0, o * sizeof(float), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(M->v, 0, o * sizeof(float), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(M->w16, 0, 2 * o * sizeof(__half), st);
        if (e != cudaSuccess) { set_error("mlp upload: %s", cudaGetErrorString(e)); rc = MRA_ECUDA; }
    }
    if (rc == MRA_OK) rc = refresh16(M, st);
    if (rc == MRA_OK) {
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { set_error("mlp create: %s", cudaGetErrorString(e)); rc = MRA_ECUDA; }
    }
    if (rc != MRA_OK) {
        mra_mlp_free(M);
        return rc;
    }
    *out = M;
    return MRA_OK;
}

int mra_mlp_num_params(const mra_mlp* M, int64_t* n) {
    if (!mlp_ok(M) || !n) { set_error("invalid network handle"); return MRA_EINVAL; }
    *n = M->np;
    return MRA_OK;
}

int mra_mlp_get_params(const mra_mlp* M, float* params_host, void* stream) {
    if (!mlp_ok(M) || !params_host) { set_error("invalid network handle"); return MRA_EINVAL; }
    MRA_CK(cudaMemcpyAsync(params_host, M->master, M->np * sizeof(float), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    MRA_CK(cudaStreamSynchronize((cudaStream_t)stream));
    return MRA_OK;
}

int mra_mlp_set_params(mra_mlp* M, const float* params_host, void* stream) {
    if (!mlp_ok(M) || !params_host) { set_error("invalid network handle"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    MRA_CK(cudaMemcpyAsync(M->master, params_host, M->np * sizeof(float), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemsetAsync(M->m, 0, M->np * sizeof(float), st));
    MRA_CK(cudaMemsetAsync(M->v, 0, M->np * sizeof(float), st));
    M->step = 0;
    MRA_TRY(refresh16(M, st));
    MRA_CK(cudaStreamSynchronize(st));
    return MRA_OK;
}

int mra_mlp_forward(const mra_mlp* M, const float* x, int64_t n, float* y, void* stream) {
    if (!mlp_ok(M) || (!x && n > 0) || (!y && n > 0) || n < 0) { set_error("invalid network forward arguments"); return MRA_EINVAL; }
    return mlp_forward(M, x, n, y, M->A, (cudaStream_t)stream);
}

int mra_mlp_loss_grad(mra_mlp* M, const float* x, const float* target, int64_t n, float* grad_host, double* loss_host,
                      void* stream) {
    if (!mlp_ok(M) || !x || !target || n < 1) { set_error("invalid network arguments"); return MRA_EINVAL; }
    if (M->n_out != 12) { set_error("the schedule loss needs 12 outputs"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    MRA_TRY(mlp_loss_grad_impl(M, x, target, n, st));
    if (grad_host) MRA_CK(cudaMemcpyAsync(grad_host, M->grad, M->np * sizeof(float), cudaMemcpyDeviceToHost, st));
    if (loss_host) MRA_CK(cudaMemcpyAsync(loss_host, M->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaStreamSynchronize(st));
    return MRA_OK;
}

int mra_mlp_train_step(mra_mlp* M, const float* x, const float* target, int64_t n, float lr, void* stream,
                       double* loss_host) {
    if (!mlp_ok(M) || !x || !target || n < 1 || !(lr > 0.0f)) { set_error("invalid training arguments"); return MRA_EINVAL; }
    if (M->n_out != 12) { set_error("the schedule loss needs 12 outputs"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    MRA_TRY(mlp_loss_grad_impl(M, x, target, n, st));
    M->step++;
    const float c1 = (float)(1.0 - pow(0.9, M->step)), c2 = (float)(1.0 - pow(0.999, M->step));
    k_adam<<<num_sms(), 256, 0, st>>>(M->np, M->master, M->grad, M->m, M->v, lr, c1, c2);
    MRA_CK_LAUNCH();
    MRA_TRY(refresh16(M, st));
    if (loss_host) {
        MRA_CK(cudaMemcpyAsync(loss_host, M->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        MRA_CK(cudaStreamSynchronize(st));
    }
    return MRA_OK;
}

int mra_mlp_free(mra_mlp* M) {
    if (!M) return MRA_OK;
    if (!mlp_ok(M)) { set_error("invalid network handle"); return MRA_EINVAL; }
    const Alloc& A = M->A;
    A.put(M->master); A.put(M->grad); A.put(M->m); A.put(M->v); A.put(M->w16); A.put(M->loss);
    A.put(M->h1); A.put(M->h2); A.put(M->h3); A.put(M->y); A.put(M->d3); A.put(M->d2); A.put(M->d1); A.put(M->dy);
    A.put(M->part);
    M->magic = 0;
    delete M;
    return MRA_OK;
}

}  // extern "C"
