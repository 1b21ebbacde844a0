// PTX building blocks of the tensor-core kernels on sm_103a: mbarriers with
// bounded waits, TMA tile loads, tcgen05 TMEM allocation, MMA issue, commit
// and loads, and the shared-memory matrix / instruction descriptors.
// Included by each translation unit that runs tcgen05 contractions.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace dstd {
namespace tc {

constexpr int BM = 128;
constexpr int BK = 64;  // bf16 elements per 128-byte swizzled row
constexpr unsigned long long WAIT_NS = 2000000000ull;

static __device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

static __device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

static __device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static __device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

static __device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// try_wait with a suspend-time hint: the thread parks in hardware until the
// phase completes or about 1 ms passes, instead of spinning on issue slots
static __device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(1000000u)
        : "memory");
    return ok != 0;
}

// try_wait without a suspend-time hint: returns after the implementation's
// own short time limit, so a thread that polls in a loop reacts to the
// phase change within a few cycles
static __device__ __forceinline__ bool mbar_try_wait_now(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded spin wait for the threads on a pipeline's critical path (TMA
// producer, MMA issuer, operand generators): false after limit_ns
static __device__ __forceinline__ bool mbar_wait_spin(uint64_t *bar, uint32_t parity,
                                                      unsigned long long limit_ns = WAIT_NS) {
    if (mbar_try_wait_now(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (;;) {
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait_now(bar, parity)) return true;
        if (globaltimer() - t0 > limit_ns) return false;
    }
}

// bounded wait: false if the phase did not complete within limit_ns
static __device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          unsigned long long limit_ns = WAIT_NS) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer() - t0 > limit_ns) return false;
    }
}

// bounded wait with a sleep between polls, for warps that have nothing else
// to do (the epilogue warps during the main loop)
static __device__ __forceinline__ bool mbar_wait_sleep(uint64_t *bar, uint32_t parity,
                                                unsigned long long limit_ns = WAIT_NS) {
    const uint64_t t0 = globaltimer();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer() - t0 > limit_ns) return false;
        __nanosleep(256);
    }
}

static __device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

static __device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
static __device__ __forceinline__ uint32_t cluster_id_x() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
static __device__ __forceinline__ uint32_t cluster_count_x() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
    return r;
}
// every thread of both CTAs of the cluster calls it once, converged
static __device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

static __device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

static __device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

static __device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
static __device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

static __device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

static __device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

// ---------------------------------------------------------------------------
// Issue by a whole warp. tcgen05.mma, its commit and TMA copies take their
// descriptors, addresses and coordinates from uniform registers. In a branch
// that one lane takes, with an exit that depends on a wait's result, the
// compiler cannot tell that they are uniform: an MMA then costs 102 clocks to
// issue whatever its size (measured: M = 128, N = 64, 4 MMAs per wait; the
// tensor core itself takes 48, and 64 with N = 128). So every lane runs the
// loop, waits end it by a warp vote, and only the instructions are left to the
// elected lane (68 clocks with 4 MMAs per wait, 54 with 36).
// ---------------------------------------------------------------------------
static __device__ __forceinline__ uint32_t elect_one() {
    uint32_t p;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(p));
    return p;
}

// a value that is the same in every lane, through a warp reduction, whose
// result the compiler knows to be uniform
static __device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(0xffffffffu, x); }

// bounded wait of a whole warp: the same answer in every lane
static __device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity) {
    return !__any_sync(0xffffffffu, !mbar_wait_spin(bar, parity));
}

// An MMA (inside a branch of the elected lane) with descriptors given by their
// low words (start address / 16, and the encoded leading offset): the high word of a K-major 128-byte-swizzle
// descriptor is a constant, so stepping an operand is one addition
constexpr uint32_t SDESC_KK_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
static __device__ __forceinline__ uint32_t sdesc_kk_lo(uint32_t saddr) {
    return ((saddr & 0x3FFFFu) >> 4) | (1u << 16);
}
// (the MN-major 128-byte-swizzle descriptor has the same high word)
static __host__ __device__ constexpr uint32_t sdesc_sw128_mn_hi() { return SDESC_KK_HI; }
template <uint32_t HI>
static __device__ __forceinline__ void mma_lo(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                              uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b64 da, db;\n"
        "mov.b64 da, {%1, %3};\n"
        "mov.b64 db, {%2, %3};\n"
        "setp.ne.b32 p, %5, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(alo), "r"(blo), "r"(HI), "r"(idesc), "r"(accumulate)
        : "memory");
}
static __device__ __forceinline__ void mma_kk(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                              uint32_t accumulate) {
    mma_lo<SDESC_KK_HI>(d_tmem, alo, blo, idesc, accumulate);
}

static __device__ __forceinline__ void mma_commit_if(uint32_t lead, uint64_t *bar) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(smem_u32(bar)),
        "r"(lead)
        : "memory");
}

static __device__ __forceinline__ void mbar_expect_tx_if(uint32_t lead, uint64_t *bar, uint32_t bytes) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %2, 0;\n"
        "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
        "}\n" ::"r"(smem_u32(bar)),
        "r"(bytes), "r"(lead)
        : "memory");
}

static __device__ __forceinline__ void tma_load_2d_if(uint32_t lead, uint32_t dst, const CUtensorMap *map, uint64_t *bar,
                                                      int x, int y) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
        "}\n" ::"r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar)), "r"(lead)
        : "memory");
}

static __device__ __forceinline__ void tma_load_5d_if(uint32_t lead, uint32_t dst, const CUtensorMap *map, uint64_t *bar,
                                                      int c, int m, int x, int y, int b) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %8, 0;\n"
        "@q cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n"
        "}\n" ::"r"(dst),
        "l"((uint64_t)map), "r"(c), "r"(m), "r"(x), "r"(y), "r"(b), "r"(smem_u32(bar)), "r"(lead)
        : "memory");
}

// 32 lanes x 32 consecutive fp32 columns; the wait is in the same asm block
// so the registers are valid when the statement completes.
static __device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
          "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
          "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor (tcgen05 format): K-major operand tile with
// 128-byte rows in 128-byte-swizzle layout; 8-row core-matrix groups are
// 1024 bytes apart (SBO); LBO is not used by swizzled K-major layouts.
static __device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address >> 4
    d |= (uint64_t)1 << 16;                     // LBO (encoded, ignored)
    d |= (uint64_t)(1024u >> 4) << 32;          // SBO
    d |= (uint64_t)1 << 46;                     // descriptor version
    d |= (uint64_t)2 << 61;                     // 128-byte swizzle
    return d;
}

// MN-major operand in 128-byte-swizzle layout: 64 consecutive MN elements
// fill a 128-byte row, one row per k; 8 rows form a 1024-byte atom. SBO =
// 1024 bytes between the 8-row groups along K, LBO = the distance between
// the 64-wide atom columns along MN.
static __device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address >> 4
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;  // LBO: next 64 MN elements
    d |= (uint64_t)(1024u >> 4) << 32;          // SBO: next 8 k
    d |= (uint64_t)1 << 46;                     // descriptor version
    d |= (uint64_t)2 << 61;                     // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B both bf16 (format 1)
// or both fp16 (format 0); A K-major, B K-major or (b_mn) MN-major.
static __host__ __device__ constexpr uint32_t idesc_16bit(int M, int N, bool f16, bool b_mn = false) {
    return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

}  // namespace tc
}  // namespace dstd
