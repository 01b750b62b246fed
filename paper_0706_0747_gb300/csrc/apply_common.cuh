// Worklist records shared by the apply kernels (apply.cu, apply_fact.cu).
#pragma once
#include <cuda_fp16.h>

#include "mra_internal.cuh"

namespace mra {

struct Pair {
    int32_t out;    // output node
    int32_t in;     // input node (>= 0) or -1 - ghost id
    int16_t m_lo, m_hi;
    int8_t t1, t2, t3;
    uint8_t flags;  // bit 0: core translation at an internal node
};
static_assert(sizeof(Pair) == 16, "Pair is 16 bytes");

struct ApplyArgs {
    int k, M, n;
    const Pair* pairs;
    const int32_t* pair_off;
    const int32_t* coord;
    const double* s;
    const double* gblk;
    const double* w;
    const void* F;         // double or float table [j][m][l+3][k][k]
    const double* nF;
    const int32_t* Jm;     // per-tree term schedules: J_m of tree b at Jm[b * jm_stride + m]
    const int32_t* node_tree = nullptr;  // tree of each node (NULL: one tree)
    int jm_stride = 0;
    double eta_blk;        // < 0: no per-block screen
    double* out;
    unsigned long long* n_items;  // items applied, per tree
    const int32_t* skip = nullptr;  // run only when *skip == run_if (NULL: always)
    int run_if = 0;
};

// tensor-core apply (apply_tc.cu)
struct TcArgs {
    ApplyArgs A;           // A.n: number of node blocks (Step-2 blocks follow them)
    const __half* xh;      // FP16 hi/lo input blocks in the stage-I layout
    const __half* xl;
    const float* sx;       // per-block power-of-two scale
    const float* xmax;     // per-block max |x|
    const float* xnrm;     // per-block ||x||_2
    const __half* Fh;      // FP16 hi/lo operator blocks, 8 x 8, per (j, m, t)
    const __half* Fl;
    const float* sF;       // per-(j, m) scale
    const float* maxF;
    const double* lpb;     // per-tree error budget of one node for single-FP16 terms (NULL: all hi+lo)
    unsigned long long* n_lowp;  // items done with single FP16 operands (may be NULL)
    int* err;              // set to 4 when a completion wait reaches its limit
    unsigned wait_limit;   // polls of one completion wait
    int withhold;          // test hook: the first MMA group and its commit are not sent
    int* counter;          // work counter (zeroed by tc_launch)
    const int* order;      // node order (NULL: 0..nwork-1)
    int nwork;
    int kr;                // basis order (<= 8; padded to 8 inside)
};

struct TcBuffers {
    __half *xh = nullptr, *xl = nullptr, *Fh = nullptr, *Fl = nullptr;
    float *sx = nullptr, *xmax = nullptr, *xnrm = nullptr, *sF = nullptr, *maxF = nullptr;
    int* counter = nullptr;
};

// The screen works on a forest: one tree, or many trees whose node arrays are
// concatenated (tree b owns a contiguous node range, level-major and Morton
// sorted within a level, its root first).  Per tree: level offsets as
// absolute node indices (lm + 1 entries), its number of levels, and in the
// outputs its norms and schedule.
struct Forest {
    int k, ntrees, n, lm;        // order; trees; nodes in all; levels of the per-tree layouts
    const int32_t* coord;        // [n][4]: (j, a1, a2, a3)
    const int32_t* leaf;         // [n]
    const uint64_t* key;         // [n]
    const int32_t* off;          // [ntrees][lm + 1]
    const int32_t* node_tree;    // [n] (NULL: one tree)
    const int32_t* nlev;         // [ntrees] (NULL: lm)
    const double* s;             // [n][k^3]
    const double* filt;          // H0, H1 (k x k each)
};

// ---- the Step-2 set and the screen's arguments
#define GH_EMPTY 0xffffffffffffffffull
#define GH_TREE_BITS 22

// level (6 bits) | tree (22 bits) | Morton key of the box (36 bits, level <= 12)
__device__ inline uint64_t ghost_key(int j, int tree, int b1, int b2, int b3) {
    return ((uint64_t)j << 58) | ((uint64_t)tree << 36) | morton3(b1, b2, b3);
}

__device__ inline uint32_t hash64(uint64_t k) {
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return (uint32_t)k;
}

// returns the slot (>= 0) or -1 when the probe limit is exceeded
__device__ inline int ghost_insert(uint64_t* tab, uint32_t cap, uint64_t key) {
    uint32_t h = hash64(key) & (cap - 1);
    for (uint32_t it = 0; it < cap && it < 4096; ++it) {
        uint64_t prev = atomicCAS((unsigned long long*)&tab[h], (unsigned long long)GH_EMPTY,
                                  (unsigned long long)key);
        if (prev == GH_EMPTY || prev == key) return (int)h;
        h = (h + 1) & (cap - 1);
    }
    return -1;
}

__device__ inline int ghost_find(const uint64_t* tab, uint32_t cap, uint64_t key) {
    uint32_t h = hash64(key) & (cap - 1);
    for (uint32_t it = 0; it < cap && it < 4096; ++it) {
        uint64_t v = tab[h];
        if (v == key) return (int)h;
        if (v == GH_EMPTY) return -1;
        h = (h + 1) & (cap - 1);
    }
    return -1;
}

// The Step-2 set is keyed by the missing box's parent: slot -> parent key, an
// 8-bit mask of the octants needed, and (after k_ghost_ids) the id of the
// parent's first needed child.  A group's children get consecutive ids in
// octant order, so no sort is needed to find siblings.
struct ScreenArgs {
    Forest F;
    int M, sl;
    const int32_t* sched;  // per tree: Jm | m1 | m2 | cnt
    uint64_t* gtab;
    uint32_t gcap;
    uint32_t* gmask;       // slot -> octants needed (count pass)
    const int32_t* gid;    // slot -> id of its first needed child (fill pass)
    int32_t* count;        // per node pair count (count pass)
    const int32_t* pair_off;
    Pair* pairs;
    int32_t* err;          // [0] hash overflow
    // [n][216] (optional): the count pass's lookup per band position -- the input node,
    // or -1 - slot of the missing box's parent in the Step-2 set -- so that the fill
    // pass searches nothing
    int32_t* qin;
};

// Sibling groups of a forest (apply_oct.cu): the root of a tree alone, then its other nodes
// by eights in node order.
struct OctGroups {
    int n = 0;
    int32_t* first = nullptr;            // [n] first output node
    int32_t* in = nullptr;               // [n][216] input blocks (node, or node count + Step-2 id; -1 none)
    int32_t* np = nullptr;               // [n] pieces
    unsigned long long* pairs = nullptr; // [ntrees] static pairs and items (in ScreenOut's report)
    unsigned long long* items = nullptr;
    int batch = 0;                       // groups a launch takes (oct_part_alloc)
};

// what a screen leaves: pair lists per output node, sibling groups, or both
#define SCREEN_PAIRS 1
#define SCREEN_GROUPS 2

// The host reads what a screen and an apply count in as few copies as it needs the numbers at
// (each copy is a round trip of about 10 us): all counters lie in one allocation that starts at dv,
//   dv [ntrees][4] | group pairs [ntrees] | group items [ntrees] | nitems [2] | total [4] | err [2].
struct ScreenReport {  // of one tree
    double dv[4];
    unsigned long long group_pairs, group_items, nitems[2];
    int32_t total[4], err[2];
};

// device results of the screen over a forest (screen_forest in apply.cu)
struct ScreenOut {
    double* dv = nullptr;         // [ntrees][4]: ||f_b||^2, sigma_b, eta_b, unused; the report's start
    unsigned long long* nitems = nullptr;  // [2] for an apply of one tree: items, items with single FP16 operands
    int32_t* sched = nullptr;     // [ntrees][sl]: Jm | m1 | m2 | cnt
    int sl = 0;
    int32_t* count = nullptr;     // [n + 1] pairs per output node
    int32_t* pair_off = nullptr;  // [n + 1]
    int32_t* total = nullptr;     // [3]: pairs, Step-2 blocks, most pieces of a group
    int32_t* err = nullptr;       // [0] screen, [1] Step 2 / apply
    uint64_t* gtab = nullptr;     // Step-2 set: parent keys of the missing boxes
    int32_t* gid = nullptr;       // slot -> id of its first needed child
    uint32_t* gmask = nullptr;    // slot -> octants needed
    uint64_t* gkeys = nullptr;    // [nghost] level | tree | Morton key of each child, by id
    uint32_t gcap = 0;
    Pair* pairs = nullptr;        // [npairs], out and in are forest node indices
    int npairs = 0, nghost = 0, max_pieces = 0;
    OctGroups oct;
};

// the sibling-group apply (apply_oct.cu)
struct OctArgs {
    int k, M, lm, sl, n;   // n: node blocks (Step-2 blocks follow them)
    int g0 = 0, ns = 1;    // first group of the launch, slices per group
    const int32_t *first, *in, *np;
    const int32_t *coord, *leaf, *node_tree, *sched;
    const double *s, *gblk;
    const void* F;
    const double* w;
    double* part = nullptr;
    const int32_t* skip = nullptr;  // run only when *skip == run_if (NULL: always)
    int run_if = 0;
};

// tensor-core apply by sibling groups (apply_oct_tc.cu)
struct OctTcArgs {
    OctArgs P;
    const __half *xh, *xl, *Fh, *Fl;   // as in TcArgs
    const float *sx, *xmax, *sF, *maxF;
    int* err;
    unsigned wait_limit;
    int withhold;
    int* counter;
    void* part;
    int nunits;
};

int oct_alloc(const Forest& F, const Alloc& A, OctGroups* O);
void oct_release(const Alloc& A, OctGroups* O);
int oct_screen(const ScreenArgs& sa, const OctGroups& O, int32_t* max_pieces, cudaStream_t st);
int oct_place_ghosts(const ScreenOut& S, int n, cudaStream_t st);
int oct_items(const ScreenOut& S, int ntrees, const int32_t* skip, unsigned long long* n_items, cudaStream_t st);
OctArgs oct_args(const ApplyArgs& A, const ScreenOut& S, const Forest& F);
int oct_slice_simt();
int oct_part_alloc(ScreenOut* S, int slice, size_t elem, int k, const Alloc& A, void** part);
int oct_reduce(const OctArgs& P, int slice, int ng, const float* part, double* out, cudaStream_t st);
int oct_tc_configure();
int oct_slice_tc();
int oct_tc_launch(OctTcArgs Q, const ScreenOut& S, void* part, double* out, cudaStream_t st);
int oct_launch(const OctArgs& P, const ScreenOut& S, int precision, double* part, double* out, cudaStream_t st);

int screen_forest(const mra_op* op, const Forest& F, int unscreened, int what, const Alloc& A, cudaStream_t st,
                  ScreenOut* S);
void screen_release(const Alloc& A, ScreenOut* S);
// Step 2 for every missing input block of a forest.  Its blocks: FP64, or floats from arithmetic in two floats or one, in the same memory
enum GhostBlocks { GHOST_FP64, GHOST_TWO_FLOATS, GHOST_FP32 };
// floats where the blocks only become the tensor cores' FP16 operands and no screen reads them
inline GhostBlocks ghost_blocks_of(int precision, int screen_mode) {
    if (screen_mode != MRA_SCREEN_STATIC) return GHOST_FP64;
    return precision == MRA_PREC_TC_SPLIT ? GHOST_TWO_FLOATS : (precision == MRA_PREC_TC_FAST ? GHOST_FP32 : GHOST_FP64);
}
int ghost_refine_forest(const Forest& F, const ScreenOut& S, double* gblk, cudaStream_t st, GhostBlocks as = GHOST_FP64);
Forest forest_of_tree(const mra_tree* f);

int tc_alloc(const mra_op* op, int nb, TcBuffers* B);            // nb: node + Step-2 blocks
int tc_prep_F(const mra_op* op, const TcBuffers& B, cudaStream_t st);
int tc_prep_blocks(int nb, int kr, int n, const double* s, const double* gblk, GhostBlocks ghosts, const TcBuffers& B,
                   cudaStream_t st);
void tc_release(const mra_op* op, TcBuffers* B);
int tc_configure();
TcArgs tc_args(const ApplyArgs& A, const TcBuffers& B, int* err);
int tc_launch(const TcArgs& T, int mc, int ctas_per_sm, cudaStream_t st);
int tc3_configure();                               // apply_tc3.cu
int tc3_launch(const TcArgs& T, cudaStream_t st);  // counter zeroed by the caller

int launch_apply_fact(const ApplyArgs& A, int precision, cudaStream_t st);
OctTcArgs oct_tc_args(const OctArgs& P, const TcBuffers& B, int* err);
// OP: the sibling groups (with their partial sums `part`) and / or the pair lists
int launch_apply_tc(const ApplyArgs& A, const ScreenOut& S, GhostBlocks ghosts, const OctArgs* OP, void* part, bool pairs,
                    const mra_op* op, int* err, const double* lpb, unsigned long long* n_lowp, unsigned wait_limit,
                    int withhold, cudaStream_t st);
int lp_budget(const Forest& F, const ScreenOut& S, double eps, double* lpb, cudaStream_t st);
int schedule_narrow(const mra_op* op, const Forest& F, const ScreenOut& S, const double* gblk, int mode,
                    const void* model, int margin, float* X_out, float* T_out, unsigned long long* counts,
                    int32_t* narrowed, const Alloc& A, cudaStream_t st);
int screen_data_impl(const mra_op* op, const mra_tree* f, float* X, float* T, cudaStream_t st);

}  // namespace mra
