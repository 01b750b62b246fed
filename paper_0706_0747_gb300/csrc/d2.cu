// The d = 2 variant of the method (Sec. 6: the apply was implemented for
// d = 2 and d = 3; Algorithm 3 as the paper illustrates it for d = 2; Sec. 4:
// three subsets Core / Boundary-1 / Boundary-2 in d = 2): quadtrees,
// Algorithm 1, the redundant tree, Algorithm 3 with Step 2, eq. g_assemble and
// the truncation in two dimensions, all FP64.  The operator tables come from
// operator.cu (built with d = 2); the 1-D blocks are the same as in d = 3.
#include <algorithm>
#include <cmath>

#include "band_sum.cuh"
#include "mra_internal.cuh"

namespace mra {

// ------------------------------------------------------------ keys and reductions
__host__ __device__ inline uint64_t spread2(uint32_t v) {
    uint64_t x = v;
    x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
    x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
    x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
    x = (x | (x << 2)) & 0x3333333333333333ull;
    x = (x | (x << 1)) & 0x5555555555555555ull;
    return x;
}
// bit 2b+1 <- a1 bit b, bit 2b <- a2 bit b: child quadrant (p1 p2) appends two bits
__host__ __device__ inline uint64_t morton2(uint32_t a1, uint32_t a2) { return (spread2(a1) << 1) | spread2(a2); }

__device__ double blk2_max(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < nw; ++i) s = fmax(s, red[i]);
    __syncthreads();
    return s;
}

__device__ double blk2_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < nw; ++i) s += red[i];
    __syncthreads();
    return s;
}

struct Offs2 {
    int v[MRA_MAX_LEVEL + 2];
};

// ------------------------------------------------------------ tree arrays
static int tree2_alloc(mra_tree2* t, int n) {
    const Alloc& A = t->A;
    const size_t kk = (size_t)t->k * t->k;
    MRA_TRY(dalloc(A, &t->key, n));
    MRA_TRY(dalloc(A, &t->coord, 3 * (size_t)n));
    MRA_TRY(dalloc(A, &t->leaf, n));
    MRA_TRY(dalloc(A, &t->child, n));
    MRA_TRY(dalloc(A, &t->parent, n));
    MRA_TRY(dalloc(A, &t->s, (size_t)n * kk));
    MRA_TRY(dalloc(A, &t->dnorm, n));
    if (!t->filt) {
        MRA_TRY(dalloc(A, &t->filt, 6 * t->k * t->k));
        MRA_TRY(launch_filters(t->k, t->filt, A.stream));
    }
    t->n = n;
    return MRA_OK;
}

static void tree2_free_arrays(mra_tree2* t) {
    const Alloc& A = t->A;
    A.put(t->key); A.put(t->coord); A.put(t->leaf); A.put(t->child); A.put(t->parent);
    A.put(t->s); A.put(t->dnorm);
    t->key = nullptr; t->coord = nullptr; t->leaf = nullptr; t->child = nullptr; t->parent = nullptr;
    t->s = nullptr; t->dnorm = nullptr;
}

static mra_tree2* tree2_new(int k, const Alloc& A) {
    mra_tree2* t = new mra_tree2();
    t->magic = MRA_TREE2_MAGIC;
    t->k = k;
    t->A = A;
    t->state = MRA_TREE_LEAVES;
    t->depth_hit = 0;
    t->n = 0;
    t->nlev = 0;
    for (int j = 0; j < MRA_MAX_LEVEL + 2; ++j) t->off[j] = 0;
    return t;
}

static void tree2_delete(mra_tree2* t) {
    if (!t) return;
    tree2_free_arrays(t);
    t->A.put(t->filt);
    t->magic = 0;
    delete t;
}

// the tree is freed on every error return of the function holding the guard
struct Tree2Guard {
    mra_tree2* t;
    ~Tree2Guard() { tree2_delete(t); }
};

// host-side validation and linking of an imported node list (coords: 3n)
static int tree2_link_upload(mra_tree2* t, const int32_t* coords, const int32_t* leaf) {
    const int n = t->n;
    std::vector<uint64_t> key(n);
    std::vector<int32_t> child(n, -1), parent(n, -1), lf(n);
    int off[MRA_MAX_LEVEL + 2];
    for (int j = 0; j < MRA_MAX_LEVEL + 2; ++j) off[j] = n;
    int nlev = 0;
    for (int i = 0; i < n; ++i) {
        const int j = coords[3 * i];
        if (j < 0 || j > MRA_MAX_LEVEL) { set_error("node %d: level %d out of range", i, j); return MRA_EINVAL; }
        for (int d = 1; d < 3; ++d)
            if (coords[3 * i + d] < 0 || coords[3 * i + d] >= (1 << j)) {
                set_error("node %d: box index out of range", i);
                return MRA_EINVAL;
            }
        key[i] = morton2(coords[3 * i + 1], coords[3 * i + 2]);
        if (i > 0) {
            const int jp = coords[3 * (i - 1)];
            if (jp > j || (jp == j && key[i - 1] >= key[i])) {
                set_error("nodes not sorted by (level, Morton key) at %d", i);
                return MRA_EINVAL;
            }
        }
        if (off[j] == n) off[j] = i;
        nlev = std::max(nlev, j + 1);
        lf[i] = leaf[i] ? 1 : 0;
    }
    if (n == 0 || coords[0] != 0) { set_error("tree must start with the root (0,0,0)"); return MRA_EINVAL; }
    for (int j = nlev; j >= 0; --j)
        if (off[j] == n && j < nlev) off[j] = off[j + 1];
    for (int j = nlev; j < MRA_MAX_LEVEL + 2; ++j) off[j] = n;
    for (int i = 0; i < n; ++i) {
        const int j = coords[3 * i];
        if (lf[i]) continue;
        if (j + 1 >= nlev) { set_error("internal node %d lacks children", i); return MRA_EINVAL; }
        const uint64_t ck = key[i] << 2;
        const int lo = off[j + 1], hi = off[j + 2];
        const int pos = (int)(std::lower_bound(key.begin() + lo, key.begin() + hi, ck) - key.begin());
        if (pos + 4 > hi) { set_error("internal node %d lacks children", i); return MRA_EINVAL; }
        for (int o = 0; o < 4; ++o)
            if (key[pos + o] != ck + o) { set_error("internal node %d lacks child %d", i, o); return MRA_EINVAL; }
        child[i] = pos;
        for (int o = 0; o < 4; ++o) parent[pos + o] = i;
    }
    for (int i = 1; i < n; ++i)
        if (parent[i] < 0) { set_error("node %d has no parent", i); return MRA_EINVAL; }
    t->nlev = nlev;
    memcpy(t->off, off, sizeof(off));
    cudaStream_t st = t->A.stream;
    MRA_CK(cudaMemcpyAsync(t->key, key.data(), n * sizeof(uint64_t), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->coord, coords, 3 * (size_t)n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->leaf, lf.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->child, child.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->parent, parent.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaStreamSynchronize(st));  // host vectors go out of scope
    return MRA_OK;
}

static int tree2_clone_skeleton(const mra_tree2* src, mra_tree2** out) {
    *out = nullptr;
    mra_tree2* t = tree2_new(src->k, src->A);
    Tree2Guard g{t};
    t->nlev = src->nlev;
    t->state = src->state;
    t->depth_hit = src->depth_hit;
    memcpy(t->off, src->off, sizeof(t->off));
    cudaStream_t st = t->A.stream;
    MRA_TRY(dalloc(t->A, &t->filt, 6 * t->k * t->k));
    MRA_CK(cudaMemcpyAsync(t->filt, src->filt, 6 * t->k * t->k * sizeof(double), cudaMemcpyDeviceToDevice, st));
    MRA_TRY(tree2_alloc(t, src->n));
    const int n = src->n;
    MRA_CK(cudaMemcpyAsync(t->key, src->key, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->coord, src->coord, 3 * (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->leaf, src->leaf, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->child, src->child, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    MRA_CK(cudaMemcpyAsync(t->parent, src->parent, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    g.t = nullptr;
    *out = t;
    return MRA_OK;
}

// ------------------------------------------------------------ Algorithm 1 in d = 2
struct Dens2 {
    int n;
    const double *coef, *r2, *expo, *cen;  // cen: 2 per term
};

__device__ double dens2_eval(const Dens2& D, double x, double y) {
    double f = 0.0;
    for (int g = 0; g < D.n; ++g) {
        const double dx = x - D.cen[2 * g], dy = y - D.cen[2 * g + 1];
        const double r2 = dx * dx + dy * dy;
        f += (D.coef[g] + D.r2[g] * r2) * exp(-D.expo[g] * r2);
    }
    return f;
}

__global__ void k_dens_scale2(Dens2 D, double eps, double* tol) {
    __shared__ double red[32];
    double m = 0.0;
    for (int g = threadIdx.x; g < D.n; g += blockDim.x)
        m = fmax(m, fabs(dens2_eval(D, D.cen[2 * g], D.cen[2 * g + 1])));
    m = blk2_max(m, red);
    if (threadIdx.x == 0) tol[0] = eps * m;
}

// One block per box of level j.  mode: 0 adaptive test, 1 refine, 2 leaf.
// Projection s = 2^{-j} P v P^T from the values v at the box's k x k GL nodes
// (eq. fvals2coefs); the test compares the density with the block's values at
// the 4 children's GL nodes.
__global__ void k_build_level2(int k, int j, Dens2 D, const int32_t* boxes, const double* tolp, int mode, int at_max,
                               double* s_out, int32_t* refine, int32_t* depth_hit) {
    extern __shared__ double sm[];
    const int kk = k * k;
    double* g = sm;
    double* gw = g + k;
    double* P = gw + k;   // [i][q] phi_i(g_q) w_q
    double* Q = P + kk;   // [p][q][i] phi_i((g_q + p)/2)
    double* v = Q + 2 * kk;
    double* t1 = v + kk;
    double* s = t1 + kk;
    __shared__ double red[32];
    const int b = blockIdx.x, tid = threadIdx.x;
    const int a1 = boxes[2 * b], a2 = boxes[2 * b + 1];
    if (tid < k) gauss_legendre01_root(k, tid, g, gw);
    __syncthreads();
    if (tid < k) {
        double tmp[MRA_MAX_K];
        phi_all(k, g[tid], tmp);
        for (int i = 0; i < k; ++i) P[i * k + tid] = tmp[i] * gw[tid];
        for (int p = 0; p < 2; ++p) {
            phi_all(k, 0.5 * (g[tid] + p), tmp);
            for (int i = 0; i < k; ++i) Q[p * kk + tid * k + i] = tmp[i];
        }
    }
    const double h = exp2(-(double)j);
    for (int e = tid; e < kk; e += blockDim.x) v[e] = dens2_eval(D, (g[e / k] + a1) * h, (g[e % k] + a2) * h);
    __syncthreads();
    for (int e = tid; e < kk; e += blockDim.x) {
        const int i1 = e / k, q2 = e % k;
        double acc = 0.0;
        for (int q1 = 0; q1 < k; ++q1) acc += P[i1 * k + q1] * v[q1 * k + q2];
        t1[e] = acc;
    }
    __syncthreads();
    const double sc = exp2(-(double)j);
    for (int e = tid; e < kk; e += blockDim.x) {
        const int i1 = e / k, i2 = e % k;
        double acc = 0.0;
        for (int q2 = 0; q2 < k; ++q2) acc += t1[i1 * k + q2] * P[i2 * k + q2];
        s[e] = acc * sc;
    }
    __syncthreads();
    int ref = (mode == 1);
    if (mode == 0) {
        double err = 0.0;
        const double hc = 0.5 * h, up = exp2((double)j);
        for (int o = 0; o < 4; ++o) {
            const int p1 = o >> 1, p2 = o & 1;
            for (int e = tid; e < kk; e += blockDim.x) {
                const int a = e / k, i2 = e % k;
                double acc = 0.0;
                for (int i1 = 0; i1 < k; ++i1) acc += Q[p1 * kk + a * k + i1] * s[i1 * k + i2];
                t1[e] = acc;
            }
            __syncthreads();
            for (int e = tid; e < kk; e += blockDim.x) {
                const int a = e / k, c = e % k;
                double acc = 0.0;
                for (int i2 = 0; i2 < k; ++i2) acc += t1[a * k + i2] * Q[p2 * kk + c * k + i2];
                const double f = dens2_eval(D, (g[a] + 2 * a1 + p1) * hc, (g[c] + 2 * a2 + p2) * hc);
                err = fmax(err, fabs(f - up * acc));
            }
            __syncthreads();
        }
        err = blk2_max(err, red);
        ref = err > tolp[0];
        if (ref && at_max) {
            ref = 0;
            if (tid == 0) atomicExch(depth_hit, 1);
        }
    }
    for (int e = tid; e < kk; e += blockDim.x) s_out[(size_t)b * kk + e] = s[e];
    if (tid == 0) refine[b] = ref;
}

__global__ void k_make_children2(int nb, const int32_t* boxes, const int32_t* refine, const int32_t* pos,
                                 int32_t* next, int32_t* parent_local) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb || !refine[b]) return;
    const int p = pos[b];
    parent_local[p] = b;
    for (int o = 0; o < 4; ++o) {
        const int c = 4 * p + o;
        next[2 * c] = 2 * boxes[2 * b] + (o >> 1);
        next[2 * c + 1] = 2 * boxes[2 * b + 1] + (o & 1);
    }
}

struct Tree2Dev {
    uint64_t* key;
    int32_t *coord, *leaf, *child, *parent;
    double* s;
};

__global__ void k_place_level2(int nb, int j, int base, int next_base, const int32_t* boxes, const int32_t* refine,
                               const int32_t* pos, const int32_t* parent_local, int prev_base, int kk,
                               const double* s_lvl, Tree2Dev T) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const int i = base + b;
    T.key[i] = morton2(boxes[2 * b], boxes[2 * b + 1]);
    T.coord[3 * i] = j;
    T.coord[3 * i + 1] = boxes[2 * b];
    T.coord[3 * i + 2] = boxes[2 * b + 1];
    T.leaf[i] = refine[b] ? 0 : 1;
    T.child[i] = refine[b] ? next_base + 4 * pos[b] : -1;
    T.parent[i] = (j == 0) ? -1 : prev_base + parent_local[b / 4];
    // (the level's blocks are copied as one contiguous range by the caller)
}

static int build_tree2_impl(const mra_density* f, int k, double eps, int max_level, int uniform_level, int init_level,
                            const Alloc& A, mra_tree2** out) {
    cudaStream_t st = A.stream;
    const int kk = k * k, ng = f->n;
    Scratch tmp(A);
    double* dd;
    MRA_TRY(tmp.get(&dd, 5 * (size_t)ng + 1));
    std::vector<double> h(5 * (size_t)ng + 1, 0.0);
    for (int g = 0; g < ng; ++g) {
        h[g] = f->coef_host[g];
        h[ng + g] = f->r2coef_host ? f->r2coef_host[g] : 0.0;
        h[2 * ng + g] = f->expo_host[g];
        h[3 * ng + 2 * g] = f->center_host[2 * g];
        h[3 * ng + 2 * g + 1] = f->center_host[2 * g + 1];
    }
    MRA_CK(cudaMemcpyAsync(dd, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    Dens2 D{ng, dd, dd + ng, dd + 2 * ng, dd + 3 * ng};
    double* tol;
    int32_t* flags;  // [0] depth_hit, [1] refined count
    MRA_TRY(tmp.get(&tol, 2));
    MRA_TRY(tmp.get(&flags, 4));
    MRA_CK(cudaMemsetAsync(flags, 0, 4 * sizeof(int32_t), st));
    k_dens_scale2<<<1, 256, 0, st>>>(D, eps, tol);
    MRA_CK_LAUNCH();
    struct Level {
        int n;
        int32_t *boxes, *refine, *pos, *parent_local;
        double* s;
    };
    std::vector<Level> L;
    int32_t* boxes0;
    MRA_TRY(tmp.get(&boxes0, 2));
    MRA_CK(cudaMemsetAsync(boxes0, 0, 2 * sizeof(int32_t), st));
    int nb = 1;
    int32_t* cur = boxes0;
    int32_t* plocal_prev = nullptr;
    const size_t smem = (2 * (size_t)k + 6 * (size_t)kk) * sizeof(double);
    for (int j = 0; j <= max_level; ++j) {
        Level lv{nb, cur, nullptr, nullptr, plocal_prev, nullptr};
        MRA_TRY(tmp.get(&lv.refine, nb));
        MRA_TRY(tmp.get(&lv.pos, nb));
        MRA_TRY(tmp.get(&lv.s, (size_t)nb * kk));
        int mode;
        if (uniform_level >= 0) mode = (j < uniform_level) ? 1 : 2;
        else mode = (j < init_level) ? 1 : 0;
        if (j == max_level && mode == 1) mode = 2;
        k_build_level2<<<nb, 64, smem, st>>>(k, j, D, cur, tol, mode, j >= max_level, lv.s, lv.refine, flags);
        MRA_CK_LAUNCH();
        MRA_TRY(scan_exclusive(lv.refine, lv.pos, nb, flags + 1, st));
        int32_t nref = 0;
        MRA_CK(cudaMemcpyAsync(&nref, flags + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        MRA_CK(cudaStreamSynchronize(st));
        L.push_back(lv);
        if (nref == 0) break;
        int32_t *next, *plocal;
        MRA_TRY(tmp.get(&next, 2 * 4 * (size_t)nref));
        MRA_TRY(tmp.get(&plocal, nref));
        k_make_children2<<<(nb + 255) / 256, 256, 0, st>>>(nb, cur, lv.refine, lv.pos, next, plocal);
        MRA_CK_LAUNCH();
        cur = next;
        nb = 4 * nref;
        plocal_prev = plocal;
    }
    mra_tree2* t = tree2_new(k, A);
    Tree2Guard tg{t};
    int n = 0;
    for (auto& lv : L) n += lv.n;
    MRA_TRY(tree2_alloc(t, n));
    t->nlev = (int)L.size();
    for (int j = 0; j < MRA_MAX_LEVEL + 2; ++j) t->off[j] = n;
    int base = 0;
    for (int j = 0; j < t->nlev; ++j) {
        t->off[j] = base;
        base += L[j].n;
    }
    base = 0;
    const Tree2Dev T{t->key, t->coord, t->leaf, t->child, t->parent, t->s};
    for (int j = 0; j < t->nlev; ++j) {
        const int nbj = L[j].n, next_base = base + nbj, prev_base = j ? t->off[j - 1] : 0;
        k_place_level2<<<(nbj + 127) / 128, 128, 0, st>>>(nbj, j, base, next_base, L[j].boxes, L[j].refine, L[j].pos,
                                                           L[j].parent_local, prev_base, kk, L[j].s, T);
        MRA_CK_LAUNCH();
        MRA_CK(cudaMemcpyAsync(t->s + (size_t)base * kk, L[j].s, (size_t)nbj * kk * sizeof(double),
                               cudaMemcpyDeviceToDevice, st));
        base = next_base;
    }
    MRA_CK(cudaMemsetAsync(t->dnorm, 0, n * sizeof(double), st));
    int32_t hit = 0;
    MRA_CK(cudaMemcpyAsync(&hit, flags, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaStreamSynchronize(st));
    t->depth_hit = hit;
    tg.t = nullptr;
    *out = t;
    return hit ? MRA_EDEPTH : MRA_OK;
}

// ------------------------------------------------------------ two-scale transforms in d = 2
// A warp per sibling group (the groups of level j+1 are its nodes by fours, in the order of
// their parents), a lane per fiber.  Both halves of the filter come from H^(0) by parity:
// H^(1)_{ia} = (-1)^{i+a} H^(0)_{ia}, zero for a > i (the d = 3 transforms' identities).  The
// wavelet norm is ||children - upsampled parent|| = ||d|| (the filter matrix is orthogonal), for all
// levels in one launch, the last one, whose first block also computes the root's scaling block (a launch
// of its own for the norms cost trees of two or three levels more than the rest saved: 5 boxes at
// k = 8 21 us -> 29 a call, now 25).  k = 8: 1,250 FP64 operations a group for the scaling block and as many
// for the norm, where the full filter matrix took 8,192 (12 us per level, a block per node).

// src (2 fibers' worth of K at stride st, the second half at src + h) -> y
template <int K>
__device__ __forceinline__ void down2_fiber(const double* H, const double* src, int st, int h, double* y) {
    double p[K], m[K];
#pragma unroll
    for (int a = 0; a < K; ++a) {
        const double x0 = src[a * st], x1 = (a & 1) ? -src[a * st + h] : src[a * st + h];
        p[a] = x0 + x1;
        m[a] = x0 - x1;
    }
#pragma unroll
    for (int i = 0; i < K; ++i) {
        double acc = 0.0;
#pragma unroll
        for (int a = 0; a <= i; ++a) acc += H[i * K + a] * ((i & 1) ? m[a] : p[a]);
        y[i] = acc;
    }
}

// s (K values at stride st) -> x0[K], x1[K]: the children's fibers
template <int K>
__device__ __forceinline__ void up2_fiber(const double* H, const double* src, int st, double* x0, double* x1) {
    double v[K];
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = src[i * st];
#pragma unroll
    for (int a = 0; a < K; ++a) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int i = a; i < K; i += 2) s0 += H[i * K + a] * v[i];
#pragma unroll
        for (int i = a + 1; i < K; i += 2) s1 += H[i * K + a] * v[i];
        x0[a] = s0 + s1;
        x1[a] = s0 - s1;
    }
}

// MODE 0: scaling block of the parent; 1: the parent's wavelet norm, the first group's scaling block
// before it; 2: children += upsampled parent
template <int K, int MODE>
__global__ void __launch_bounds__(32) k_scale2(int cbase, const int32_t* parent, double* s, double* dnorm, const double* filt) {
    constexpr int KK = K * K, K1 = K + 1;
    __shared__ double H[KK];
    __shared__ double t[2 * K * K1];  // (2k, k), rows padded
    const int lane = threadIdx.x, c0 = cbase + 4 * blockIdx.x, par = parent[c0];
    for (int e = lane; e < KK; e += 32) H[e] = filt[e];
    __syncwarp();
    double* ch = s + (size_t)c0 * KK;
    if (MODE == 0 || (MODE == 1 && blockIdx.x == 0)) {
        // direction 1: fiber of column c (0..2k-1) of the children's square, rows r of both halves
        if (lane < 2 * K) {
            double y[K];
            down2_fiber<K>(H, ch + (lane / K) * KK + lane % K, K, 2 * KK, y);
#pragma unroll
            for (int i = 0; i < K; ++i) t[lane * K1 + i] = y[i];  // (column, i1)
        }
        __syncwarp();
        if (lane < K) {  // direction 2: row i1
            double y[K];
            down2_fiber<K>(H, t + lane, K1, K * K1, y);
#pragma unroll
            for (int i = 0; i < K; ++i) s[(size_t)par * KK + lane * K + i] = y[i];
        }
        if (MODE == 0) return;
        __syncwarp();
    }
    // direction 1 of the parent's block: column i2 -> rows 0..2k-1
    if (lane < K) {
        double x0[K], x1[K];
        up2_fiber<K>(H, s + (size_t)par * KK + lane, K, x0, x1);
#pragma unroll
        for (int a = 0; a < K; ++a) {
            t[a * K1 + lane] = x0[a];
            t[(K + a) * K1 + lane] = x1[a];
        }
    }
    __syncwarp();
    double acc = 0.0;
    if (lane < 2 * K) {  // direction 2: row `lane` of the square
        double x0[K], x1[K];
        up2_fiber<K>(H, t + lane * K1, 1, x0, x1);
        double* d0 = ch + (lane / K) * 2 * KK + (lane % K) * K;
#pragma unroll
        for (int a = 0; a < K; ++a) {
            if (MODE == 2) {
                d0[a] += x0[a];
                d0[KK + a] += x1[a];
            } else {
                const double e0 = d0[a] - x0[a], e1 = d0[KK + a] - x1[a];
                acc += e0 * e0 + e1 * e1;
            }
        }
    }
    if (MODE == 1) {
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) dnorm[par] = sqrt(acc);
    }
}

template <int K>
static int compress2_t(mra_tree2* t, cudaStream_t st) {
    for (int j = t->nlev - 2; j >= 1; --j) {
        const int ng = (t->off[j + 2] - t->off[j + 1]) / 4;
        if (ng <= 0) continue;
        k_scale2<K, 0><<<ng, 32, 0, st>>>(t->off[j + 1], t->parent, t->s, t->dnorm, t->filt);
        MRA_CK_LAUNCH();
    }
    const int ng = (t->n - 1) / 4;
    if (ng > 0) {
        k_scale2<K, 1><<<ng, 32, 0, st>>>(1, t->parent, t->s, t->dnorm, t->filt);
        MRA_CK_LAUNCH();
    }
    return MRA_OK;
}

template <int K>
static int assemble2_t(mra_tree2* t, cudaStream_t st) {
    for (int j = 0; j + 1 < t->nlev; ++j) {
        const int ng = (t->off[j + 2] - t->off[j + 1]) / 4;
        if (ng <= 0) continue;
        k_scale2<K, 2><<<ng, 32, 0, st>>>(t->off[j + 1], t->parent, t->s, t->dnorm, t->filt);
        MRA_CK_LAUNCH();
    }
    return MRA_OK;
}


static int compress2_impl(mra_tree2* t, cudaStream_t st) {
    static int (*const fn[])(mra_tree2*, cudaStream_t) = FOR_EVERY_K(compress2_t);
    MRA_TRY(fn[t->k](t, st));
    t->state = MRA_TREE_REDUNDANT;
    return MRA_OK;
}

// eq. g_assemble
static int assemble2_impl(mra_tree2* t, cudaStream_t st) {
    static int (*const fn[])(mra_tree2*, cudaStream_t) = FOR_EVERY_K(assemble2_t);
    MRA_TRY(fn[t->k](t, st));
    t->state = MRA_TREE_LEAVES;
    return MRA_OK;
}

// sum of the squares of the leaf blocks: fixed 256 partial sums, then one warp
// adds them in a fixed order (the result does not depend on scheduling)
#define NORM_PARTS 256
__global__ void k_leaf_sq_partial2(int n, int kk, const int32_t* leaf, const double* s, double* part) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        if (!leaf[i]) continue;
        for (int e = threadIdx.x; e < kk; e += blockDim.x) acc += s[(size_t)i * kk + e] * s[(size_t)i * kk + e];
    }
    acc = blk2_sum(acc, red);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

__global__ void k_sum_parts2(int np, const double* part, double* out) {
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += 32) s += part[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *out = s;
}

static int leaf_norm2(const mra_tree2* t, double* part, double* out, cudaStream_t st) {
    k_leaf_sq_partial2<<<NORM_PARTS, 128, 0, st>>>(t->n, t->k * t->k, t->leaf, t->s, part);
    MRA_CK_LAUNCH();
    k_sum_parts2<<<1, 32, 0, st>>>(NORM_PARTS, part, out);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

// ------------------------------------------------------------ truncation in d = 2
__global__ void k_trunc_thr2(double eps, int n, const double* norm2, double* thr) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *thr = eps * sqrt(*norm2) / sqrt((double)n);
}

// an internal node of the level whose 4 children are leaves and whose wavelet
// norm is below the threshold becomes a leaf; its children are dropped
__global__ void k_merge2_level(int lo, int hi, const int32_t* child, int32_t* leaf, const double* dnorm,
                               const double* thr, int32_t* alive, double* removed2) {
    const int i = lo + blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= hi || leaf[i]) return;
    const int c = child[i];
    if (!(leaf[c] && leaf[c + 1] && leaf[c + 2] && leaf[c + 3])) return;
    if (!(dnorm[i] < *thr)) return;
    leaf[i] = 1;
    for (int o = 0; o < 4; ++o) alive[c + o] = 0;
    atomicAdd(removed2, dnorm[i] * dnorm[i]);
}

__global__ void k_compact2(int n, int kk, const int32_t* alive, const int32_t* newidx, Tree2Dev src,
                           const double* dnorm_src, Tree2Dev dst, double* dnorm_dst) {
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        if (!alive[i]) continue;
        const int ni = newidx[i];
        if (threadIdx.x == 0) {
            dst.key[ni] = src.key[i];
            for (int d = 0; d < 3; ++d) dst.coord[3 * ni + d] = src.coord[3 * i + d];
            dst.leaf[ni] = src.leaf[i];
            dst.child[ni] = src.leaf[i] ? -1 : newidx[src.child[i]];
            dst.parent[ni] = src.parent[i] < 0 ? -1 : newidx[src.parent[i]];
            dnorm_dst[ni] = src.leaf[i] ? 0.0 : dnorm_src[i];
        }
        for (int e = threadIdx.x; e < kk; e += blockDim.x) dst.s[(size_t)ni * kk + e] = src.s[(size_t)i * kk + e];
    }
}

__global__ void k_new_offsets2(Offs2 off, int nlev, int n, const int32_t* newidx, const int32_t* total, int32_t* out) {
    const int j = threadIdx.x;
    if (j >= MRA_MAX_LEVEL + 2) return;
    out[j] = (j < nlev && off.v[j] < n) ? newidx[off.v[j]] : *total;
}

__global__ void k_ones2(int n, int32_t* p) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 1;
}

static int truncate2_impl(mra_tree2* t, double eps, cudaStream_t st, double* removed_host) {
    const int n = t->n, kk = t->k * t->k;
    Scratch tmp(t->A);
    double *part, *sc;  // sc: [0] norm^2, [1] threshold, [2] removed^2
    int32_t *alive, *newidx, *total, *offs;
    MRA_TRY(tmp.get(&part, NORM_PARTS));
    MRA_TRY(tmp.get(&sc, 4));
    MRA_TRY(tmp.get(&alive, n));
    MRA_TRY(tmp.get(&newidx, n));
    MRA_TRY(tmp.get(&total, 1));
    MRA_TRY(tmp.get(&offs, MRA_MAX_LEVEL + 2));
    MRA_TRY(leaf_norm2(t, part, sc, st));
    k_trunc_thr2<<<1, 32, 0, st>>>(eps, n, sc, sc + 1);
    MRA_CK_LAUNCH();
    MRA_CK(cudaMemsetAsync(sc + 2, 0, sizeof(double), st));
    k_ones2<<<(n + 255) / 256, 256, 0, st>>>(n, alive);
    MRA_CK_LAUNCH();
    for (int j = t->nlev - 2; j >= 0; --j) {
        const int lo = t->off[j], hi = t->off[j + 1];
        if (hi <= lo) continue;
        k_merge2_level<<<(hi - lo + 127) / 128, 128, 0, st>>>(lo, hi, t->child, t->leaf, t->dnorm, sc + 1, alive,
                                                               sc + 2);
        MRA_CK_LAUNCH();
    }
    MRA_TRY(scan_exclusive(alive, newidx, n, total, st));
    Offs2 off;
    memcpy(off.v, t->off, sizeof(off.v));
    k_new_offsets2<<<1, 32, 0, st>>>(off, t->nlev, n, newidx, total, offs);
    MRA_CK_LAUNCH();
    int32_t hoffs[MRA_MAX_LEVEL + 2];
    double removed2 = 0.0;
    MRA_CK(cudaMemcpyAsync(hoffs, offs, sizeof(hoffs), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaMemcpyAsync(&removed2, sc + 2, sizeof(double), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaStreamSynchronize(st));
    if (removed_host) *removed_host = sqrt(removed2);
    const int nn = hoffs[MRA_MAX_LEVEL + 1];
    if (nn == n) return MRA_OK;
    // the compacted arrays, swapped into t
    mra_tree2 fresh = {};
    fresh.k = t->k;
    fresh.A = t->A;
    fresh.filt = t->filt;  // kept, not reallocated
    const int rc = tree2_alloc(&fresh, nn);
    if (rc != MRA_OK) {
        tree2_free_arrays(&fresh);
        return rc;
    }
    const Tree2Dev src{t->key, t->coord, t->leaf, t->child, t->parent, t->s};
    const Tree2Dev dst{fresh.key, fresh.coord, fresh.leaf, fresh.child, fresh.parent, fresh.s};
    k_compact2<<<std::max(1, std::min(n, num_sms() * 8)), 64, 0, st>>>(n, kk, alive, newidx, src, t->dnorm, dst,
                                                                        fresh.dnorm);
    cudaError_t e = cudaGetLastError();
    count_launch();
    if (e != cudaSuccess) {
        fresh.filt = nullptr;
        tree2_free_arrays(&fresh);
        set_error("compaction launch: %s", cudaGetErrorString(e));
        return MRA_ECUDA;
    }
    tree2_free_arrays(t);
    t->key = fresh.key; t->coord = fresh.coord; t->leaf = fresh.leaf; t->child = fresh.child;
    t->parent = fresh.parent; t->s = fresh.s; t->dnorm = fresh.dnorm;
    t->n = nn;
    int nlev = 0;
    for (int j = 0; j < MRA_MAX_LEVEL + 1; ++j)
        if (hoffs[j] < hoffs[j + 1]) nlev = j + 1;
    t->nlev = nlev;
    for (int j = 0; j < MRA_MAX_LEVEL + 2; ++j) t->off[j] = (j <= nlev) ? hoffs[j] : nn;
    return MRA_OK;
}

// ------------------------------------------------------------ Algorithm 3 in d = 2
// ||T_0 f_0||: y = sum_m w_m F_m X F_m^T on the root block (j = 0, t = 0): block per term, then
// the terms summed per coefficient in order and the norm taken; dv[1]
__global__ void k_pilot2_terms(int k, const double* w, const double* F, const double* s_root, double* ym) {
    __shared__ double X[MRA_MAX_K * MRA_MAX_K], Z[MRA_MAX_K * MRA_MAX_K], Fm[MRA_MAX_K * MRA_MAX_K];
    const int kk = k * k, m = blockIdx.x, e = threadIdx.x;
    if (e < kk) {
        X[e] = s_root[e];
        Fm[e] = F[((size_t)m * 7 + 3) * kk + e];
    }
    __syncthreads();
    const int a = e / k, c = e % k;
    if (e < kk) {
        double acc = 0.0;
        for (int i = 0; i < k; ++i) acc += Fm[a * k + i] * X[i * k + c];
        Z[e] = acc;
    }
    __syncthreads();
    if (e < kk) {
        double acc = 0.0;
        for (int i = 0; i < k; ++i) acc += Z[a * k + i] * Fm[c * k + i];
        ym[(size_t)m * kk + e] = w[m] * acc;
    }
}

__global__ void k_pilot2_sum(int kk, int M, const double* ym, double* dv) {
    __shared__ double red[32], part[4][MRA_MAX_K * MRA_MAX_K];
    const int e = threadIdx.x % 160, q = threadIdx.x / 160;  // four quarters of the terms
    double y = 0.0;
    if (e < kk)
        for (int m = q * M / 4; m < (q + 1) * M / 4; ++m) y += ym[(size_t)m * kk + e];
    if (e < kk) part[q][e] = y;
    __syncthreads();
    y = threadIdx.x < kk ? ((part[0][threadIdx.x] + part[1][threadIdx.x]) + part[2][threadIdx.x]) + part[3][threadIdx.x] : 0.0;
    const double nrm = blk2_sum(y * y, red);
    if (threadIdx.x == 0) dv[1] = sqrt(nrm);
}

// eta = eps sigma / ||f||; J_m; per scale j and subset S = 0, 1, 2 the range
// [m1, m2] trimmed from both ends while the cumulative w_m c^S b^(2-S) stays
// <= eta / 72 (c, b: the largest N_F over |l| <= 1 and over 2 <= |l| <= 3).
// Layout: Jm[M] | m1[nlev*3] | m2[nlev*3].
// (The bounds of all (j, S, m) are formed in parallel in shared memory; a term with J_m < j
// gets 0, which the serial scans pass over as they skip it.)
__global__ void k_schedule2(int M, int nlev, double eps, const double* w, const double* nF, const double* est,
                            double* dv, int32_t* sched) {
    extern __shared__ double sched2_sm[];
    double* ev = sched2_sm;                // [nlev * 3][M]
    int* Js = (int*)(ev + (size_t)nlev * 3 * M);
    int32_t* Jm = sched;
    int32_t* m1 = Jm + M;
    int32_t* m2 = m1 + nlev * 3;
    const double fn = sqrt(dv[0]);
    const double eta = fn > 0.0 ? eps * dv[1] / fn : 0.0;
    if (threadIdx.x == 0) dv[2] = eta;
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        int jm = 0;
        for (int j = 1; j < nlev; ++j)
            if (w[m] * est[(size_t)j * M + m] > eta / M) jm = j;
        Jm[m] = jm;
        Js[m] = jm;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nlev * M; e += blockDim.x) {
        const int j = e / M, m = e - j * M;
        const double* r = nF + (size_t)e * 7;
        const double c = fmax(fmax(r[2], r[3]), r[4]);
        const double bb = fmax(fmax(r[0], r[1]), fmax(r[5], r[6]));
        const bool on = Js[m] >= j;
        ev[((size_t)j * 3 + 0) * M + m] = on ? w[m] * bb * bb : 0.0;
        ev[((size_t)j * 3 + 1) * M + m] = on ? w[m] * c * bb : 0.0;
        ev[((size_t)j * 3 + 2) * M + m] = on ? w[m] * c * c : 0.0;
    }
    __syncthreads();
    const double budget = eta / (2.0 * 36.0);
    for (int js = threadIdx.x; js < nlev * 3; js += blockDim.x) {
        const int j = js / 3;
        int lo_m = 0, hi_m = -1, first = -1, last = -1;
        for (int m = 0; m < M; ++m)
            if (Js[m] >= j) {
                if (first < 0) first = m;
                last = m;
            }
        if (first >= 0) {
            const double* e_js = ev + (size_t)js * M;
            double acc = 0.0;
            int lo = first;
            for (; lo <= last; ++lo) {
                const double e = e_js[lo];
                if (acc + e <= budget) acc += e;
                else break;
            }
            acc = 0.0;
            int hi = last;
            for (; hi >= lo; --hi) {
                const double e = e_js[hi];
                if (acc + e <= budget) acc += e;
                else break;
            }
            if (hi >= lo && lo <= last) {
                lo_m = lo;
                hi_m = hi;
            }
        }
        m1[js] = lo_m;
        m2[js] = hi_m;
    }
}

// Algorithm 3 in d = 2.  The four siblings of a group have the same 6 x 6 inputs (b = 0..5 a
// direction, t = a + 2 - b), and whether a translation is core depends on |t1| and |t2| alone.
// So the kept terms of a level sum to one k^2 x k^2 matrix per translation,
//   D^t[c][i] = sum_m w_m F^{t1}[c1][i1] F^{t2}[c2][i2],
// and with F^{-t}[c][i] = (-1)^{c+i} F^t[c][i] the matrices of |t1|, |t2| = 0..3 suffice: output c takes
// from input i the sum of the (up to four) inputs at +-t1, +-t2 with signs (-1)^{c1+i1}, (-1)^{c2+i2}.
// FP64 multiply-adds are the bound: a group takes 4 x 12.25 k^4 of them whatever the number of
// terms (k = 8: 0.2 M; the terms one at a time, by separable sums shared by the four siblings, took
// 33 K each, 1.1 M on the bench's quadtree: apply 1.69 ms, 2.7 ms an output box at a time).
//
// A level of 2^j boxes a direction has no translations beyond 2^j - 1: of levels 0 and 1 only the
// planes within reach are formed and read.
//
// Planes of a level: 4 |t1| + |t2|, the core x core ones (|t| <= 1) with the terms that a leaf
// keeps (J_m >= j); 16 + 2 |t1| + |t2| those ones with the terms an internal box keeps (J_m = j).
#define D2_PLANES 20
__device__ __forceinline__ int d2_reach(int j) { return j > 1 ? 3 : j; }  // largest |t| of a level
#define D2_Q 8     // entries of F^{t1} a block
#define D2_MB 16   // terms staged at a time
#define D2_LEAST ((size_t)1 << 20)

// One block per (level, plane |t1| <= |t2|, D2_Q entries (c1, i1)); thread (i2, c2), the sums in
// registers.  The plane with |t1| and |t2| exchanged is the same matrix with directions exchanged.
// Layout [i][c]: the apply's threads read consecutive c.
template <int K>
__global__ void __launch_bounds__((K * K + 31) / 32 * 32) k_dense2(int M, int nlev, int j0, const double* F, const double* w,
                                                                  const int32_t* sched, double* D) {
    constexpr int KK = K * K;
    constexpr int U1[13] = {0, 0, 0, 0, 1, 1, 1, 2, 2, 3, 0, 0, 1}, U2[13] = {0, 1, 2, 3, 1, 2, 3, 2, 3, 3, 0, 1, 1};
    __shared__ double f1[D2_MB][D2_Q], f2[D2_MB][KK];
    const int j = j0 + blockIdx.x, q0 = blockIdx.z * D2_Q, tid = threadIdx.x, lane = tid & 31;
    int u1 = 0, u2 = 0;
#pragma unroll
    for (int p = 0; p < 13; ++p)
        if ((int)blockIdx.y == p) u1 = U1[p], u2 = U2[p];
    if (u2 > d2_reach(j)) return;  // (u1 <= u2)
    const bool inner = blockIdx.y >= 10;
    const int S = (u1 <= 1) + (u2 <= 1);
    const int lo = sched[M + 3 * j + S], hi = sched[M + 3 * nlev + 3 * j + S];
    unsigned use = 0;  // entries that are not zero by parity (|t1| = 0: c1 + i1 even)
    for (int q = 0; q < D2_Q; ++q)
        if (q0 + q < KK && (u1 || !(((q0 + q) / K + (q0 + q) % K) & 1))) use |= 1u << q;
    double acc[D2_Q];
#pragma unroll
    for (int q = 0; q < D2_Q; ++q) acc[q] = 0.0;
    for (int mb = lo; mb <= hi; mb += 32) {
        const int ml = mb + lane;
        unsigned mask = __ballot_sync(0xffffffffu, ml <= hi && (inner ? sched[ml] == j : sched[ml] >= j));
        while (mask) {  // the same in every warp
            unsigned take = 0;
            for (int n = 0; n < D2_MB && mask; ++n) {
                take |= mask & -mask;
                mask &= mask - 1;
            }
            const int nb = __popc(take);
            __syncthreads();
            for (int n = 0; n < nb; ++n, take &= take - 1) {
                const int m = mb + __ffs(take) - 1;
                const double* Fm = F + ((size_t)j * M + m) * 7 * KK;
                if (tid < D2_Q && q0 + tid < KK) f1[n][tid] = w[m] * Fm[(3 + u1) * KK + q0 + tid];
                if (tid < KK) f2[n][tid] = Fm[(3 + u2) * KK + (tid % K) * K + tid / K];
            }
            __syncthreads();
            if (tid < KK)
                for (int n = 0; n < nb; ++n) {
                    const double y = f2[n][tid];
#pragma unroll
                    for (int q = 0; q < D2_Q; ++q)
                        if ((use >> q) & 1u) acc[q] += f1[n][q] * y;
                }
        }
    }
    if (tid >= KK) return;
    const int i2 = tid / K, c2 = tid % K;
    double* D0 = D + ((size_t)blockIdx.x * D2_PLANES + (inner ? 16 + 2 * u1 + u2 : 4 * u1 + u2)) * KK * KK;
    double* D1 = D + ((size_t)blockIdx.x * D2_PLANES + (inner ? 16 + 2 * u2 + u1 : 4 * u2 + u1)) * KK * KK;
#pragma unroll
    for (int q = 0; q < D2_Q; ++q) {
        if (q0 + q >= KK) break;
        const int c1 = (q0 + q) / K, i1 = (q0 + q) % K;
        D0[(size_t)(i1 * K + i2) * KK + c1 * K + c2] = acc[q];
        if (u1 != u2) D1[(size_t)(i2 * K + i1) * KK + c2 * K + c1] = acc[q];
    }
}

// The apply.  Block per sibling group: the 36 inputs are gathered into shared memory, missing ones
// refined from their covering leaf (Step 2, a warp per missing parent); then per |t1| the sums Y of
// inputs at +-t1, per |t2| those of Y at +-t2, and the plane's product: thread (c, part of the i)
// for the four outputs, a matrix entry read once per group (k = 8: 0.5 MB a group out of L2).
// counters: [0] items, [1] pairs, [2] Step-2 refinements an output box at a time would make, [3]
// lookups that found no ancestor (0 for a valid tree)
#define A2_NT 256
template <int K>
struct Apply2Smem {
    static constexpr int KK = K * K, PARTS = A2_NT / KK < KK ? A2_NT / KK : KK;
    static constexpr size_t bytes = (size_t)(36 + 24 + 16) * KK * sizeof(double);
};

template <int K>
__global__ void __launch_bounds__(A2_NT) k_apply2(int M, int nlev, int j0, int g0, Offs2 off, const uint64_t* key,
                                                              const int32_t* coord, const int32_t* leaf, const double* s,
                                                              const double* D, const int32_t* sched,
                                                              const double* filt, double* gout, unsigned long long* counters) {
    constexpr int KK = K * K, NT = A2_NT, PARTS = Apply2Smem<K>::PARTS;
    extern __shared__ __align__(16) double sm[];
    double* X = sm;            // [6][6] blocks
    double* Y = X + 36 * KK;   // [parity of c1 + i1][a1][6] blocks
    double* Z = Y + 24 * KK;   // [parities][i][a]
    double* H = Z;             // H^(0), H^(1) while inputs are refined
    __shared__ int s_cnt[4], s_base[9], s_anc[9], s_lev[9], s_nout;
    __shared__ unsigned s_leaf, s_need[9];
    const int tid = threadIdx.x, lane = tid & 31, g = g0 + blockIdx.x;
    const int i0 = g == 0 ? 0 : 1 + 4 * (g - 1);
    const int j = coord[3 * i0], nout = j ? 4 : 1;
    const int p1 = coord[3 * i0 + 1] >> 1, p2 = coord[3 * i0 + 2] >> 1;
    const int32_t *m1 = sched + M + 3 * j, *m2 = sched + M + 3 * nlev + 3 * j;
    for (int e = tid; e < 2 * KK; e += NT) H[e] = filt[e];
    if (tid < 32) {
        const unsigned leafm = __ballot_sync(0xffffffffu, lane < nout && leaf[i0 + (lane < nout ? lane : 0)]);
        // the kept terms per class (S; the core at an internal box: index 3)
        int cnt[4] = {0, 0, 0, 0};
        for (int S = 0; S < 3; ++S)
            for (int m = m1[S] + lane; m <= m2[S]; m += 32) {
                cnt[S] += sched[m] >= j;
                if (S == 2) cnt[3] += sched[m] == j;
            }
        for (int S = 0; S < 4; ++S)
            for (int o = 16; o > 0; o >>= 1) cnt[S] += __shfl_xor_sync(0xffffffffu, cnt[S], o);
        // lane per neighbour of the parent: its children at level j, or the leaf that covers it
        unsigned long long items = 0, pairs = 0, ghosts = 0, lost = 0;
        if (lane < 9) {
            const int d1 = lane / 3, d2 = lane % 3;
            const int q1 = p1 + d1 - 1, q2 = p2 + d2 - 1, N = j ? 1 << (j - 1) : 1;
            int base = -1, anc = -1, lev = -1;
            bool inside = j ? q1 >= 0 && q2 >= 0 && q1 < N && q2 < N : lane == 4;
            if (j == 0) base = inside ? i0 : -1;
            else if (inside) base = find_key_exact(key, off.v[j], off.v[j + 1], morton2(q1, q2) << 2);
            unsigned need = 0;
            if (inside)
                for (int o = 0; o < (j ? 4 : 1); ++o) {
                    const int b1 = 2 * d1 + (o >> 1), b2 = 2 * d2 + (o & 1);
                    for (int a = 0; a < nout; ++a) {
                        const int S = band_core(a >> 1, b1) + band_core(a & 1, b2);
                        const int n = S == 2 ? (((leafm >> a) & 1u) ? cnt[2] : cnt[3]) : (S ? cnt[1] : cnt[0]);
                        if (n <= 0) continue;
                        need |= 1u << o;
                        ++pairs;
                        items += n;
                        ghosts += base < 0;
                    }
                }
            if (need && base < 0) {
                for (lev = j - 1; lev >= 0 && anc < 0; --lev)
                    anc = find_key_exact(key, off.v[lev], off.v[lev + 1], morton2(q1 >> (j - 1 - lev), q2 >> (j - 1 - lev)));
                ++lev;
                if (anc < 0) ++lost;  // impossible for a complete tree; counted, read as zero
            }
            s_base[lane] = base;
            s_need[lane] = need;
            s_anc[lane] = anc;
            s_lev[lane] = lev;
        }
        for (int o = 16; o > 0; o >>= 1) {
            items += __shfl_xor_sync(0xffffffffu, items, o);
            pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
            ghosts += __shfl_xor_sync(0xffffffffu, ghosts, o);
            lost += __shfl_xor_sync(0xffffffffu, lost, o);
        }
        if (lane == 0) {
            for (int S = 0; S < 4; ++S) s_cnt[S] = cnt[S];
            s_leaf = leafm;
            s_nout = nout;
            atomicAdd(&counters[0], items);
            atomicAdd(&counters[1], pairs);
            atomicAdd(&counters[2], ghosts);
            if (lost) atomicAdd(&counters[3], lost);
        }
    }
    __syncthreads();
    const unsigned leafm = s_leaf;
    // the inputs that are nodes; the others zero until refined
    for (int e = tid; e < 36 * KK; e += NT) {
        const int q = e / KK, b1 = q / 6, b2 = q % 6, pi = (b1 >> 1) * 3 + (b2 >> 1), o = (b1 & 1) * 2 + (b2 & 1);
        X[e] = s_base[pi] >= 0 && ((s_need[pi] >> o) & 1u) ? s[(size_t)(s_base[pi] + o) * KK + e % KK] : 0.0;
    }
    __syncthreads();
    // Step 2, a warp per missing parent: down the path to the parent, then its four children
    for (int pi = tid >> 5; pi < 9; pi += NT / 32) {
        if (!s_need[pi] || s_base[pi] >= 0 || s_anc[pi] < 0) continue;
        const int q1 = p1 + pi / 3 - 1, q2 = p2 + pi % 3 - 1, lev0 = s_lev[pi];
        double *x = Y + (tid >> 5) * 3 * KK, *y = x + KK, *z = y + KK;
        __syncwarp();
        for (int e = lane; e < KK; e += 32) x[e] = s[(size_t)s_anc[pi] * KK + e];
        __syncwarp();
        for (int lev = lev0; lev < j - 1; ++lev) {
            const int sh = j - 2 - lev;
            const double *H1 = H + ((q1 >> sh) & 1) * KK, *H2 = H + ((q2 >> sh) & 1) * KK;
            for (int e = lane; e < KK; e += 32) {
                const int a = e / K, c = e % K;
                double acc = 0.0;
                for (int i = a; i < K; ++i) acc += H1[i * K + a] * x[i * K + c];
                y[e] = acc;
            }
            __syncwarp();
            for (int e = lane; e < KK; e += 32) {
                const int a = e / K, b = e % K;
                double acc = 0.0;
                for (int c = b; c < K; ++c) acc += y[a * K + c] * H2[c * K + b];
                x[e] = acc;
            }
            __syncwarp();
        }
        if (lane < K) {
            double x0[K], x1[K];
            up2_fiber<K>(H, x + lane, K, x0, x1);
#pragma unroll
            for (int a = 0; a < K; ++a) {
                y[a * K + lane] = x0[a];
                z[a * K + lane] = x1[a];
            }
        }
        __syncwarp();
        if (lane < 2 * K) {
            double x0[K], x1[K];
            up2_fiber<K>(H, (lane < K ? y : z) + (lane % K) * K, 1, x0, x1);
            double* d0 = X + (size_t)((2 * (pi / 3) + lane / K) * 6 + 2 * (pi % 3)) * KK + (lane % K) * K;
#pragma unroll
            for (int a = 0; a < K; ++a) {
                d0[a] = x0[a];
                d0[KK + a] = x1[a];
            }
        }
    }
    const int c = tid % KK, part = tid / KK, pc1 = (c / K) & 1, pc2 = (c % K) & 1;
    const double* Dj = D + (size_t)(j - j0) * D2_PLANES * KK * KK;
    const bool inner = s_cnt[3] > 0 && leafm != 0xfu;  // some internal output keeps core terms
    double y[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int u1 = 0; u1 <= d2_reach(j); ++u1) {
        __syncthreads();
        for (int e = tid; e < 12 * KK; e += NT) {  // (a1, b2, i)
            const int a1 = e / (6 * KK), r = e % (6 * KK);
            const double xp = a1 + 2 - u1 >= 0 ? X[(a1 + 2 - u1) * 6 * KK + r] : 0.0;
            const double xm = u1 && a1 + 2 + u1 < 6 ? X[(a1 + 2 + u1) * 6 * KK + r] : 0.0;
            Y[e] = xp + xm;
            Y[12 * KK + e] = xp - xm;
        }
#pragma unroll 1
        for (int u2 = 0; u2 <= d2_reach(j); ++u2) {
            const int S = (u1 <= 1) + (u2 <= 1);
            if (!s_cnt[S]) continue;
            __syncthreads();
            for (int e = tid; e < 8 * KK; e += NT) {  // (p1, i, a)
                const int a = e & 3, i = (e >> 2) % KK, p = e / (4 * KK), a2 = a & 1;
                const double* Yr = Y + (p * 2 + (a >> 1)) * 6 * KK + i;
                // (an internal output without core terms reads zeros)
                const bool on = S < 2 || ((leafm >> a) & 1u) || inner;
                const double yp = on && a2 + 2 - u2 >= 0 ? Yr[(a2 + 2 - u2) * KK] : 0.0;
                const double ym = on && u2 && a2 + 2 + u2 < 6 ? Yr[(a2 + 2 + u2) * KK] : 0.0;
                Z[((2 * p) * KK + i) * 4 + a] = yp + ym;
                Z[((2 * p + 1) * KK + i) * 4 + a] = yp - ym;
            }
            __syncthreads();
            if (part < PARTS) {
                const double* Dp = Dj + (size_t)(4 * u1 + u2) * KK * KK + c;
                // F^0 has no entries with c + i odd
                const int s1 = u1 ? 1 : 2, s2 = u2 ? 1 : 2, o1 = u1 ? 0 : pc1, o2 = u2 ? 0 : pc2;
                const int n2 = (K - o2 + s2 - 1) / s2, nq = ((K - o1 + s1 - 1) / s1) * n2;
                if (S < 2 || !inner) {
#pragma unroll 4
                    for (int q = part; q < nq; q += PARTS) {
                        const int i1 = (q / n2) * s1 + o1, i2 = (q % n2) * s2 + o2, i = i1 * K + i2;
                        const double d = Dp[(size_t)i * KK];
                        const double2* z = (const double2*)(Z + ((2 * ((i1 + pc1) & 1) + ((i2 + pc2) & 1)) * KK + i) * 4);
                        const double2 z0 = z[0], z1 = z[1];
                        y[0] += d * z0.x;
                        y[1] += d * z0.y;
                        y[2] += d * z1.x;
                        y[3] += d * z1.y;
                    }
                } else {
                    const double* Di = Dj + (size_t)(16 + 2 * u1 + u2) * KK * KK + c;
#pragma unroll 4
                    for (int q = part; q < nq; q += PARTS) {
                        const int i1 = (q / n2) * s1 + o1, i2 = (q % n2) * s2 + o2, i = i1 * K + i2;
                        const double dl = Dp[(size_t)i * KK], di = Di[(size_t)i * KK];
                        const double2* z = (const double2*)(Z + ((2 * ((i1 + pc1) & 1) + ((i2 + pc2) & 1)) * KK + i) * 4);
                        const double2 z0 = z[0], z1 = z[1];
                        y[0] += ((leafm & 1u) ? dl : di) * z0.x;
                        y[1] += ((leafm & 2u) ? dl : di) * z0.y;
                        y[2] += ((leafm & 4u) ? dl : di) * z1.x;
                        y[3] += ((leafm & 8u) ? dl : di) * z1.y;
                    }
                }
            }
        }
    }
    // the parts' sums in order
    __syncthreads();
    double* ys = X;  // [part][a][c]
    if (part < PARTS)
#pragma unroll
        for (int a = 0; a < 4; ++a) ys[(part * 4 + a) * KK + c] = y[a];
    __syncthreads();
    for (int e = tid; e < s_nout * KK; e += NT) {
        double v = ys[e];
        for (int p = 1; p < PARTS; ++p) v += ys[p * 4 * KK + e];
        gout[(size_t)i0 * KK + e] = v;
    }
}

// levels j0 .. j1 - 1, whose matrices D holds
template <int K>
static int apply2_launch(int j0, int j1, int M, const mra_tree2* f, const mra_op* op, const int32_t* sched, double* D,
                         double* gout, unsigned long long* counters, cudaStream_t st) {
    constexpr int KK = K * K;
    constexpr size_t bytes = Apply2Smem<K>::bytes;
    Offs2 off;
    memcpy(off.v, f->off, sizeof(off.v));
    k_dense2<K><<<dim3(j1 - j0, 13, (KK + D2_Q - 1) / D2_Q), (KK + 31) / 32 * 32, 0, st>>>(M, f->nlev, j0, op->F, op->w, sched, D);
    MRA_CK_LAUNCH();
    MRA_CK(cudaFuncSetAttribute(k_apply2<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    const int g0 = (f->off[j0] + 3) / 4, ng = (f->off[j1] + 3) / 4 - g0;  // the root alone, then fours
    k_apply2<K><<<ng, A2_NT, bytes, st>>>(M, f->nlev, j0, g0, off, f->key, f->coord, f->leaf, f->s, D, sched, f->filt, gout, counters);
    MRA_CK_LAUNCH();
    return MRA_OK;
}

static int apply2_impl(const mra_op* op, const mra_tree2* f, cudaStream_t st, mra_tree2** gout,
                       mra_apply_stats* stats) {
    *gout = nullptr;
    const int k = op->k, kk = k * k, M = op->M, n = f->n, nlev = f->nlev;
    if (f->k != k) { set_error("tree order k=%d differs from operator k=%d", f->k, k); return MRA_EINVAL; }
    if (nlev - 1 > op->J) { set_error("tree depth %d exceeds operator max_level %d", nlev - 1, op->J); return MRA_EINVAL; }
    if (f->state != MRA_TREE_REDUNDANT) { set_error("apply_ns2 needs a compressed (redundant) tree"); return MRA_ESTATE; }
    Scratch tmp(f->A);
    double *part, *dv;
    int32_t* sched;
    unsigned long long* counters;
    MRA_TRY(tmp.get(&part, NORM_PARTS));
    MRA_TRY(tmp.get(&dv, 4));
    MRA_TRY(tmp.get(&sched, (size_t)M + 6 * nlev));
    MRA_TRY(tmp.get(&counters, 4));
    MRA_CK(cudaMemsetAsync(counters, 0, 4 * sizeof(unsigned long long), st));
    MRA_TRY(leaf_norm2(f, part, dv, st));
    double* ym;
    MRA_TRY(tmp.get(&ym, (size_t)M * kk));
    // the matrices of all levels; of fewer at a time where the allocator has no room for them, as long
    // as they take more than D2_LEAST bytes (k = 12: 3.3 MB a level)
    double* D;
    int per = nlev, rc;
    while ((rc = tmp.get(&D, (size_t)per * D2_PLANES * kk * kk)) == MRA_ENOMEM && per > 1 &&
           (size_t)per * D2_PLANES * kk * kk * sizeof(double) > D2_LEAST)
        per = (per + 1) / 2;
    MRA_TRY(rc);
    k_pilot2_terms<<<M, (kk + 31) / 32 * 32, 0, st>>>(k, op->w, op->F, f->s, ym);
    MRA_CK_LAUNCH();
    k_pilot2_sum<<<1, 640, 0, st>>>(kk, M, ym, dv);
    MRA_CK_LAUNCH();
    const size_t ssm = (size_t)M * (3 * nlev * sizeof(double) + sizeof(int));
    MRA_CK(cudaFuncSetAttribute(k_schedule2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssm));
    k_schedule2<<<1, 256, ssm, st>>>(M, nlev, op->eps, op->w, op->nF, op->est, dv, sched);
    MRA_CK_LAUNCH();
    mra_tree2* g = nullptr;
    MRA_TRY(tree2_clone_skeleton(f, &g));
    Tree2Guard tg{g};
    g->state = MRA_TREE_NSFORM;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    MRA_CK(cudaEventCreate(&e0));
    struct Ev {
        cudaEvent_t& a;
        cudaEvent_t& b;
        ~Ev() {
            if (a) cudaEventDestroy(a);
            if (b) cudaEventDestroy(b);
        }
    } ev{e0, e1};
    MRA_CK(cudaEventCreate(&e1));
    MRA_CK(cudaEventRecord(e0, st));
    using Fn = int (*)(int, int, int, const mra_tree2*, const mra_op*, const int32_t*, double*, double*, unsigned long long*, cudaStream_t);
    static const Fn fn[] = FOR_EVERY_K(apply2_launch);
    for (int j = 0; j < nlev; j += per) MRA_TRY(fn[k](j, std::min(nlev, j + per), M, f, op, sched, D, g->s, counters, st));
    MRA_CK(cudaEventRecord(e1, st));
    MRA_CK(cudaMemsetAsync(g->dnorm, 0, n * sizeof(double), st));
    unsigned long long hc[4];
    double hdv[4];
    MRA_CK(cudaMemcpyAsync(hc, counters, sizeof(hc), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaMemcpyAsync(hdv, dv, sizeof(hdv), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaStreamSynchronize(st));
    if (hc[3]) { set_error("%llu input boxes without an ancestor (tree not complete)", hc[3]); return MRA_ECUDA; }
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->n_items = (int64_t)hc[0];
        stats->n_pairs = (int64_t)hc[1];
        stats->n_ghosts = (int64_t)hc[2];
        stats->n_out_nodes = n;
        stats->fnorm = sqrt(hdv[0]);
        stats->sigma = hdv[1];
        stats->eta = hdv[2];
        float ms = 0.0f;
        MRA_CK(cudaEventElapsedTime(&ms, e0, e1));
        stats->ms_apply = ms;
    }
    tg.t = nullptr;
    *gout = g;
    return MRA_OK;
}

}  // namespace mra

using namespace mra;

static bool tree2_ok(const mra_tree2* t) { return t && t->magic == MRA_TREE2_MAGIC; }
static bool op2_ok(const mra_op* o) { return o && o->magic == MRA_OP_MAGIC && o->d == 2; }

int mra_build_tree2(const mra_density* f, int k, double eps, int max_level, int uniform_level, int init_level,
                    const mra_alloc* alloc, void* stream, mra_tree2** out) {
    if (!out) { set_error("out is NULL"); return MRA_EINVAL; }
    *out = nullptr;
    if (!f || f->n <= 0 || !f->coef_host || !f->expo_host || !f->center_host) {
        set_error("empty or invalid density");
        return MRA_EINVAL;
    }
    if (k < 1 || k > MRA_MAX_K) { set_error("k=%d outside [1, %d]", k, MRA_MAX_K); return MRA_EINVAL; }
    if (!(eps > 0.0)) { set_error("eps must be > 0"); return MRA_EINVAL; }
    if (max_level < 0 || max_level > MRA_MAX_LEVEL) { set_error("max_level outside [0, %d]", MRA_MAX_LEVEL); return MRA_EINVAL; }
    for (int g = 0; g < f->n; ++g)
        if (!(f->expo_host[g] > 0.0)) { set_error("exponent %d is not positive", g); return MRA_EINVAL; }
    return build_tree2_impl(f, k, eps, max_level, uniform_level, init_level, make_alloc(alloc, stream), out);
}

int mra_tree2_import(int k, int n, const int32_t* coords_host, const int32_t* leaf_host, const double* blocks_host,
                     const mra_alloc* alloc, void* stream, mra_tree2** out) {
    if (!out) { set_error("out is NULL"); return MRA_EINVAL; }
    *out = nullptr;
    if (k < 1 || k > MRA_MAX_K || n < 1 || !coords_host || !leaf_host || !blocks_host) {
        set_error("invalid import arguments");
        return MRA_EINVAL;
    }
    mra_tree2* t = tree2_new(k, make_alloc(alloc, stream));
    Tree2Guard g{t};
    MRA_TRY(tree2_alloc(t, n));
    MRA_TRY(tree2_link_upload(t, coords_host, leaf_host));
    cudaStream_t st = t->A.stream;
    MRA_CK(cudaMemcpyAsync(t->s, blocks_host, (size_t)n * k * k * sizeof(double), cudaMemcpyHostToDevice, st));
    MRA_CK(cudaMemsetAsync(t->dnorm, 0, n * sizeof(double), st));
    MRA_CK(cudaStreamSynchronize(st));
    g.t = nullptr;
    *out = t;
    return MRA_OK;
}

int mra_tree2_export(const mra_tree2* t, int32_t* coords_host, int32_t* leaf_host, double* blocks_host,
                     double* dnorm_host, void* stream) {
    if (!tree2_ok(t)) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    const int n = t->n;
    if (coords_host) MRA_CK(cudaMemcpyAsync(coords_host, t->coord, 3 * (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    if (leaf_host) MRA_CK(cudaMemcpyAsync(leaf_host, t->leaf, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    if (blocks_host) MRA_CK(cudaMemcpyAsync(blocks_host, t->s, (size_t)n * t->k * t->k * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (dnorm_host) MRA_CK(cudaMemcpyAsync(dnorm_host, t->dnorm, (size_t)n * sizeof(double), cudaMemcpyDeviceToHost, st));
    MRA_CK(cudaStreamSynchronize(st));
    return MRA_OK;
}

int mra_tree2_get_info(const mra_tree2* t, mra_tree_info* info) {
    if (!tree2_ok(t) || !info) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    info->k = t->k;
    info->n_nodes = t->n;
    info->n_levels = t->nlev;
    info->state = t->state;
    info->depth_hit = t->depth_hit;
    memcpy(info->level_offset, t->off, sizeof(t->off));
    return MRA_OK;
}

int mra_compress2(mra_tree2* t, void* stream) {
    if (!tree2_ok(t)) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    if (t->state == MRA_TREE_NSFORM) { set_error("compress needs leaf data; assemble an ns-form tree first"); return MRA_ESTATE; }
    return compress2_impl(t, (cudaStream_t)stream);
}

int mra_apply_ns2(const mra_op* op, const mra_tree2* f, void* stream, mra_tree2** g_ns, mra_apply_stats* stats) {
    if (!g_ns) { set_error("g_ns is NULL"); return MRA_EINVAL; }
    *g_ns = nullptr;
    if (!op2_ok(op)) { set_error("invalid operator handle or not a d = 2 operator"); return MRA_EINVAL; }
    if (!tree2_ok(f)) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    return apply2_impl(op, f, (cudaStream_t)stream, g_ns, stats);
}

int mra_reconstruct2(mra_tree2* t, int truncate, double eps, void* stream, double* truncation_l2_host) {
    if (!tree2_ok(t)) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    if (truncation_l2_host) *truncation_l2_host = 0.0;
    if (t->state != MRA_TREE_NSFORM) { set_error("reconstruct2 needs an ns-form tree"); return MRA_ESTATE; }
    if (truncate && !(eps > 0.0)) { set_error("truncation eps must be > 0"); return MRA_EINVAL; }
    cudaStream_t st = (cudaStream_t)stream;
    MRA_TRY(assemble2_impl(t, st));
    MRA_TRY(compress2_impl(t, st));
    if (truncate) MRA_TRY(truncate2_impl(t, eps, st, truncation_l2_host));
    return MRA_OK;
}

int mra_free_tree2(mra_tree2* t) {
    if (!t) return MRA_OK;
    if (!tree2_ok(t)) { set_error("invalid d = 2 tree handle"); return MRA_EINVAL; }
    tree2_delete(t);
    return MRA_OK;
}
