// PTX wrappers shared by the tensor-core kernels (mbarrier, bulk copies,
// tcgen05 MMA, tensor-memory loads), written for sm_103a.  Every wait is
// bounded: it gives up after `limit` clock cycles (or when another role of
// the CTA has raised the abort flag) and reports it.
#pragma once

#include <stdint.h>

namespace rdm {
namespace {

constexpr long long kWaitCycles = 4000000000LL;   // default bound of a wait: ~2 s at 2 GHz

// ---------------------------------------------------------------------------
// PTX helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; false on timeout or when another role has aborted
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          long long limit) {
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}
// bounded wait that ignores the abort flag (draining after an abort)
__device__ __forceinline__ bool mbar_wait_drain(uint64_t *bar, uint32_t parity, long long limit) {
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    // K-major, no swizzle; version 1 (tcgen05) in bits 46-47
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(r[c]);
}
// 8 columns, without the wait (tmem_wait_ld comes before the values are used)
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr));
}
// (the operands keep the compiler from using the values before the wait)
__device__ __forceinline__ void tmem_wait_ld(float (&v)[4][8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0][0]), "+f"(v[0][1]), "+f"(v[0][2]), "+f"(v[0][3]), "+f"(v[0][4]), "+f"(v[0][5]), "+f"(v[0][6]), "+f"(v[0][7]),
                   "+f"(v[1][0]), "+f"(v[1][1]), "+f"(v[1][2]), "+f"(v[1][3]), "+f"(v[1][4]), "+f"(v[1][5]), "+f"(v[1][6]), "+f"(v[1][7]),
                   "+f"(v[2][0]), "+f"(v[2][1]), "+f"(v[2][2]), "+f"(v[2][3]), "+f"(v[2][4]), "+f"(v[2][5]), "+f"(v[2][6]), "+f"(v[2][7]),
                   "+f"(v[3][0]), "+f"(v[3][1]), "+f"(v[3][2]), "+f"(v[3][3]), "+f"(v[3][4]), "+f"(v[3][5]), "+f"(v[3][6]), "+f"(v[3][7]));
}

// ---------------------------------------------------------------------------
// The tiles of a persistent CTA, handed from the thread that claims them to the
// warps that work on them through a ring in shared memory.  The first tile is
// the CTA's own, every further one the next that no CTA has taken.
// ---------------------------------------------------------------------------
struct __align__(16) TileEntry {
    int64_t s0, s1;               // K-steps
    int t;                        // >= number of tiles: the end
};
constexpr int kSeq = 4;           // entries kept
struct __align__(16) TileSeq {
    TileEntry e[kSeq];
    uint64_t full[kSeq], empty[kSeq];
};
__device__ __forceinline__ void init_seq(TileSeq *q, int readers) {
    for (int k = 0; k < kSeq; ++k) {
        mbar_init(&q->full[k], 1);
        mbar_init(&q->empty[k], readers);
    }
}
// entry k, by one thread; returns the tile (the end too when the wait is given up)
__device__ __forceinline__ int put_tile(TileSeq *q, uint32_t k, int ntile, const int64_t *step_rng, int *next_tile,
                                        volatile int *abort_flag, long long limit) {
    const int t = k == 0 ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(next_tile, 1);
    const int slot = k % kSeq;
    if (!mbar_wait(&q->empty[slot], ((k / kSeq) & 1) ^ 1, abort_flag, limit)) return ntile;
    volatile TileEntry *e = &q->e[slot];
    e->t = t;
    if (t < ntile) {
        e->s0 = step_rng[2 * t];
        e->s1 = step_rng[2 * t + 1];
    }
    mbar_arrive(&q->full[slot]);
    return t;
}
// Entry k, by a warp (LANES = 32) or by one lane (1).  Every reader takes every
// entry once, in order.  Every lane waits by itself and reads by shared loads of
// one address, which leaves the control flow that follows uniform for the
// compiler: read through a generic pointer, the loops over a tile's K-steps
// and segments were compiled as divergent and 1.7 times slower.
template <int LANES>
__device__ __forceinline__ bool take_tile(TileSeq *q, uint32_t k, int lane, volatile int *abort_flag, long long limit,
                                          TileEntry &e) {
    const int slot = k % kSeq;
    if (!mbar_wait(&q->full[slot], (k / kSeq) & 1, abort_flag, limit)) return false;
    const uint32_t at = smem_u32(&q->e[slot]);
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(e.s0), "=l"(e.s1) : "r"(at) : "memory");
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(e.t) : "r"(at + 16) : "memory");
    if (LANES > 1) __syncwarp();
    if (LANES == 1 || lane == 0) mbar_arrive(&q->empty[slot]);
    return true;
}

}  // namespace
}  // namespace rdm
