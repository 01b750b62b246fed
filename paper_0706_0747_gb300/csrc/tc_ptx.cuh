// Thin wrappers over the sm_100-family tcgen05 / mbarrier PTX used by the
// tensor-core apply.  Shared-memory operands use the canonical no-swizzle
// K-major layout: 8-row x 16-byte core matrices; LBO = byte distance between
// core matrices adjacent in K, SBO = between core matrices adjacent in M/N.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace mra {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor (no swizzle, version 1 at bit 46)
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor: kind::f16 with FP16 A and B, FP32 D, K-major A/B
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void commit(uint64_t* mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
        smem_u32(mbar)));
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
    asm volatile("fence.mbarrier_init.release.cluster;");
}

// Polls of one completion wait, in every kernel: as the caller asked, at least TC_WAIT_MIN (far
// above the time of the work that is waited for), or the default.  A poll that finds nothing takes
// 3.8 us here (4,096 polls 15.5 ms in the group kernel, 16.0 in the pair-list one), so the default
// is four seconds.
#define TC_WAIT_MIN 4096u
#define TC_WAIT_LIMIT (1u << 20)
inline unsigned wait_polls(unsigned asked) {
    return !asked ? TC_WAIT_LIMIT : (asked < TC_WAIT_MIN ? TC_WAIT_MIN : asked);
}

// Bounded wait for the given phase; returns false when the limit is reached.  A
// poll that finds the phase incomplete puts the thread to sleep for TC_POLL_NS
// nanoseconds before the next, so a waiting warp issues few instructions.
#define TC_POLL_NS 32
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t phase, uint32_t limit) {
    uint32_t done = 0;
    for (uint32_t it = 0; it < limit; ++it) {
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(mbar)), "r"(phase));
        if (done) break;
        __nanosleep(TC_POLL_NS);
    }
    return done != 0;
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// warp-collective TMEM allocation (column count: power of two >= 32)
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

// 16 lanes x 256 bits (8 consecutive 32-bit columns) from lane base `taddr`:
// thread t of the warp gets v[0], v[1] = lane t/4, columns 2(t%4), 2(t%4)+1
// and v[2], v[3] = lane t/4 + 8, the same columns
__device__ __forceinline__ void tmem_ld16x256(uint32_t taddr, float* v) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __uint_as_float(r[q]);
}

// NREP (2 or 4) repetitions of the 16x256b shape over consecutive 8-column
// groups in one instruction and one wait: v[r][0..3] as in tmem_ld16x256 for
// columns taddr + 8 r.  The wait names every destination register, so no use
// can be scheduled before it.
template <int NREP>
__device__ __forceinline__ void tmem_ld16x256_rep(uint32_t taddr, float (*v)[4]);

template <>
__device__ __forceinline__ void tmem_ld16x256_rep<2>(uint32_t taddr, float (*v)[4]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q >> 2][q & 3] = __uint_as_float(r[q]);
}

template <>
__device__ __forceinline__ void tmem_ld16x256_rep<4>(uint32_t taddr, float (*v)[4]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q >> 2][q & 3] = __uint_as_float(r[q]);
}

// 32 lanes x 16 consecutive 32-bit columns: lane l of the warp gets its TMEM lane's values
__device__ __forceinline__ void tmem_ld32x16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

// two loads of 16 lanes x 16 columns (16x256b.x2: v[i][r][0..3] as tmem_ld16x256_rep<2> of
// taddr[i]) in flight together, one wait
__device__ __forceinline__ void tmem_ld16x256_x2x2(uint32_t ta0, uint32_t ta1, float (*v)[2][4]) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta0));
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(ta1));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q >> 3][(q >> 2) & 1][q & 3] = __uint_as_float(r[q]);
}

// move registers between the warpgroups of a CTA (every warp of the warpgroup; N a multiple of 8)
template <int N>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

// one arrival of the calling thread
__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
    asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.shared::cta.b64 t, [%0];\n}\n" ::"r"(smem_u32(mbar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_warp(uint64_t* mbar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(mbar);
}

// As mbar_wait, but also gives up once *abort (shared memory) is set by another waiter; a wait
// that reaches its limit sets it.  A poll suspends the thread in hardware until the phase completes
// or TC_SUSPEND_NS have passed, so that waiting warps leave the issue slots to the others.
#define TC_SUSPEND_NS 1000
__device__ __forceinline__ bool mbar_wait_or(uint64_t* mbar, uint32_t phase, uint32_t limit, volatile int* abort,
                                             uint32_t nap = TC_POLL_NS) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(phase)
        : "memory");
    if (done) return true;
    for (uint32_t it = 0; it < limit; ++it) {
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(mbar)), "r"(phase), "r"((uint32_t)TC_SUSPEND_NS)
            : "memory");
        if (done) return true;
        if (*abort) return false;
        __nanosleep(nap);
    }
    *abort = 1;
    return false;
}

// MMA and commit by one elected lane of a converged warp: called by all lanes with the same
// operands, which then stay in uniform registers (a lone lane's operands are moved there for every
// instruction)
__device__ __forceinline__ void mma_f16_warp(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p, e;\nsetp.ne.b32 p, %4, 0;\nelect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void commit_warp(uint64_t* mbar) {
    asm volatile(
        "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(mbar)));
}

__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// 16-byte asynchronous global -> shared copies (completion by wait_all)
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// four 8x8 b16 matrices from the warp's fragments (thread t holds row t/4, columns 2(t%4)
// and 2(t%4)+1 of each, as one 32-bit register per matrix), stored transposed: memory row
// r of matrix i (16 bytes at the address thread 8 i + r supplies) is column r of fragment i
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0),
                 "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}

// FP32 pair -> FP16 hi + FP16 lo pairs (v ~= hi + lo to about 2^-22 relative), packed as half2
__device__ __forceinline__ void split_h2(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
    hi = *(const uint32_t*)&h;
    lo = *(const uint32_t*)&l;
}

// two FP32 lanes an instruction (as many roundings as the two scalar ones)
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(*(unsigned long long*)&r)
        : "l"(*(const unsigned long long*)&a), "l"(*(const unsigned long long*)&b));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(*(unsigned long long*)&r)
        : "l"(*(const unsigned long long*)&a), "l"(*(const unsigned long long*)&b), "l"(*(const unsigned long long*)&c));
    return r;
}

// c (a, b), c a power of two, as split_h2
__device__ __forceinline__ void split_scaled_h2(float a, float b, float c, uint32_t& hi, uint32_t& lo) {
    const float2 x = mul2(make_float2(a, b), make_float2(c, c));
    const __half2 h = __floats2half2_rn(x.x, x.y);
    const float2 l = fma2(__half22float2(h), make_float2(-1.0f, -1.0f), x);  // exact
    const __half2 l2 = __floats2half2_rn(l.x, l.y);
    hi = *(const uint32_t*)&h;
    lo = *(const uint32_t*)&l2;
}

// FP32 -> FP16 hi + FP16 lo with v ~= hi + lo to about 2^-22 relative
__device__ __forceinline__ void split_h(float v, __half& hi, __half& lo) {
    hi = __float2half_rn(v);
    lo = __float2half_rn(v - __half2float(hi));
}

}  // namespace tc
}  // namespace mra
