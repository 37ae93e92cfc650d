// Inline-PTX wrappers shared by the kernels: shared-memory barriers with bounded waits, tensor
// memory, asynchronous copies, tcgen05 matrix instructions.
#pragma once
#include <cstdint>

namespace patconv {

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void tmem_ld8(uint32_t ta, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t ta, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(ta) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t ta, uint32_t *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(ta) : "memory");
}
// 32 lanes x 16 columns as matrix fragments: lane t gets columns 8 i + 2 (t % 4) + e of rows 16 h + 8 r + t / 4 as
// r[8 h + 4 i + 2 r + e].
__device__ __forceinline__ void tmem_ld_quad(uint32_t ta, uint32_t *r) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
        asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[8 * h]), "=r"(r[8 * h + 1]), "=r"(r[8 * h + 2]), "=r"(r[8 * h + 3]), "=r"(r[8 * h + 4]), "=r"(r[8 * h + 5]),
                       "=r"(r[8 * h + 6]), "=r"(r[8 * h + 7])
                     : "r"(ta + (uint32_t)h * (16u << 16)) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t ta, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(ta), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t ta, const uint32_t *r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(ta), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_ready(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Whether a phase is over, without waiting.
template <bool CLUSTER> __device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    if (CLUSTER)
        asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    else
        asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    return ok != 0;
}
// The same, the thread asleep meanwhile for up to kSleepNs.
constexpr uint32_t kSleepNs = 20000;
template <bool CLUSTER> __device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    if (CLUSTER)
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(mbar), "r"(parity), "r"(kSleepNs) : "memory");
    else
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(mbar), "r"(parity), "r"(kSleepNs) : "memory");
    return ok != 0;
}

// Wait for an mbarrier phase with a bound in time (limit_us microseconds and three tries of kSleepNs; in case
// the timer stands still, a cap on the tries: 80 seconds at most): on expiry the block-wide abort flag and the device
// status word are set.  Every later wait of the block is given 100 microseconds and those tries, more than
// any copy or matrix instruction takes, so that a launch that gave up ends soon (nothing else rests on it).  The kernel
// still runs to its end (releasing tensor memory) with results the host can tell are invalid.
// CLUSTER: what other blocks of the cluster wrote before they arrived is seen too.
template <bool CLUSTER>
__device__ __noinline__ bool mbar_wait_long(uint32_t mbar, uint32_t parity, volatile int *abort_flag, int *status,
                                            uint32_t limit_us) {
    if (mbar_try<CLUSTER>(mbar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0; it < 4000000u; ++it) {
        if (mbar_try<CLUSTER>(mbar, parity)) return true;
        if (global_ns() - t0 > (uint64_t)(*abort_flag ? min(limit_us, 100u) : limit_us) * 1000ull) break;
    }
    if (!*abort_flag) {
        *abort_flag = 1;
        if (status) atomicExch(status, 1);
    }
    return false;
}
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, volatile int *abort_flag, int *status,
                                          uint32_t limit_us) {
    return mbar_try<CLUSTER>(mbar, parity) || mbar_wait_long<CLUSTER>(mbar, parity, abort_flag, status, limit_us);
}

__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(e));
    return e != 0;
}
// 16 bytes global -> shared, of which `bytes` (0 or 16) are read and the rest filled with zeros.
__device__ __forceinline__ void copy16(uint32_t dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// Ask for `bytes` (a multiple of 16, from a multiple of 16) to be brought into L2.
__device__ __forceinline__ void prefetch_l2(const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING> __device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Clusters: the address of the same shared-memory location in another block, and what goes there.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
    uint32_t far;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(far) : "r"(addr), "r"(rank));
    return far;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t far) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(far) : "memory");
}
// `bytes` (a multiple of 16) of this block's shared memory to another block's, counted by a barrier there.
__device__ __forceinline__ void copy_cluster(uint32_t far, uint32_t src, uint32_t bytes, uint32_t far_bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(far), "r"(src), "r"(bytes), "r"(far_bar) : "memory");
}
// The two halves of a meeting, each thread on its own.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_meet() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Matrix instructions, by one block (128 rows) or by a pair of blocks (256 rows: each holds its own
// half of the rows and half of the columns' operand; the even block of the pair issues).
template <bool PAIR> __device__ __forceinline__ void tc_commit(uint32_t mbar, uint16_t mask) {
    if (PAIR)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(mbar), "h"(mask) : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// Operand descriptors as (low word, high word): only the low word, which holds the address, moves.
#define XGEN_MMA(GROUP, KIND)                                                                                             \
    asm volatile("{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.u32 p, %6, 0;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n" \
                 " tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], a, b, %5, p;\n}"                                   \
                 ::"r"(d), "r"(a), "r"(a_hi), "r"(b), "r"(b_hi), "r"(idesc), "r"(acc) : "memory")
template <bool PAIR>
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc) {
    if (PAIR) XGEN_MMA("2", "f16"); else XGEN_MMA("1", "f16");
}
template <bool PAIR>
__device__ __forceinline__ void mma_i8(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc) {
    if (PAIR) XGEN_MMA("2", "i8"); else XGEN_MMA("1", "i8");
}
#undef XGEN_MMA
template <bool PAIR> __device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t cols) {
    if (PAIR) asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols) : "memory");
    else asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols) : "memory");
}
template <bool PAIR> __device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
    if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tensor_load4(uint32_t dst, const void *map, int c0, int c1, int c2, int c3, uint32_t mbar) {
    if (PAIR)          // the barrier may be the other block's
        asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4, %5}], [%6];"
                     ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(mbar) : "memory");
    else
        asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                     ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(mbar) : "memory");
}
// The same with rows of 128 bytes of K, 16-byte pieces swizzled by the row (address bits 4..6 xor 7..9):
// 8 rows are 1024 contiguous bytes, the next 8 follow `sbo` bytes on.  The swizzle is one of addresses,
// so a start at any row is allowed; K advances by 32 bytes inside the row.
__device__ __forceinline__ uint64_t operand_desc_swizzled(uint32_t addr, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
// Shared-memory operand of a matrix instruction, K-major without swizzle: 8 rows of 16 bytes are
// contiguous, the next 8 rows follow `sbo` bytes on, the next 16 bytes of K `lbo` bytes on.
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

}  // namespace patconv
