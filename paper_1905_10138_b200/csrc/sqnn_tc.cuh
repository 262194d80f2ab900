// Building blocks of the tensor-core kernels: mbarriers with bounded waits, tensor memory, tcgen05.mma with
// the A operand in tensor memory, and the expansion of packed mask and plane bits into bf16.
#pragma once
#include "sqnn_decode.cuh"

#include <cuda.h>

namespace sqnn {

SQNN_DEV void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(bar), "r"(count) : "memory");
}
SQNN_DEV void mbar_arrive(uint32_t bar)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" :: "r"(bar) : "memory");
}
SQNN_DEV void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
                 :: "r"(bar), "r"(bytes) : "memory");
}
SQNN_DEV bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false if the wait was abandoned (limit reached or another role gave up).
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status, uint64_t limit)
{
    const long long t0 = clock64();
    while (true) {
        for (uint32_t k = 0; k < 16; ++k)
            if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if ((uint64_t)(clock64() - t0) > limit) {
            *abort_flag = 1u;
            if (status) atomicMax(status, (uint32_t)(-SQNN_E_TIMEOUT));
            return false;
        }
    }
}
SQNN_DEV bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status, uint64_t limit)
{
    for (uint32_t k = 0; k < 4; ++k)
        if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, status, limit);
}
// The same for a converged warp: true in all lanes or in none.  (One instruction of a converged warp gives all
// its lanes the same answer, so only the slow way needs a vote.)
SQNN_DEV bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status, uint64_t limit)
{
    for (uint32_t k = 0; k < 4; ++k)
        if (mbar_try(bar, parity)) return true;
    return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, abort_flag, status, limit));
}
// The same without a report, for copies that must land before the kernel may leave.
SQNN_DEV void mbar_drain(uint32_t bar, uint32_t parity, uint64_t limit)
{
    const long long t0 = clock64();
    while (!mbar_try(bar, parity) && (uint64_t)(clock64() - t0) <= limit) {}
}
SQNN_DEV void tma_load_2d(uint32_t sdst, const CUtensorMap *map, uint32_t bar, int32_t x, int32_t y)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n"
                 :: "r"(sdst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}
SQNN_DEV void tmem_alloc(uint32_t *slot, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                 :: "r"(smem_addr(slot)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
SQNN_DEV void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(taddr), "r"(cols) : "memory");
}
SQNN_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
SQNN_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// The tcgen05.mma of one A slot (4 or 8 slices of K = 16) and the commit that frees it, by one elected lane of
// a converged warp: A from tensor memory (128 lanes x 16 bf16 each, two per column), B from shared memory.
// Issued from converged code the operands are uniform registers; issued under a lane test they were moved
// there one by one and a step of 64 columns took over 800 cycles instead of the 256 the tensor cores need at
// N = 128.  `bdesc_hi`: descriptor step from the first four slices (one box of 64 columns) to the next four.
#define SQNN_MMA(D, A, B, P) " @e tcgen05.mma.cta_group::1.kind::f16 [" D "], [" A "], " B ", %3, " P ";\n"
template <uint32_t SLICES>
SQNN_DEV void mma_slot(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate, uint32_t free_a,
                       uint64_t bdesc_hi)
{
    static_assert(SLICES == 4 || SLICES == 8, "slots of 64 or 128 columns");
    if constexpr (SLICES == 8) {
        asm volatile("{\n .reg .pred e, p, t;\n .reg .b32 a1, a2, a3, a4, a5, a6, a7;\n .reg .b64 b1, b2, b3, b4, b5, b6, b7;\n"
                     " elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, %4, %4;\n"
                     " add.u32 a1, %1, 8;\n add.u32 a2, %1, 16;\n add.u32 a3, %1, 24;\n add.u32 a4, %1, 32;\n"
                     " add.u32 a5, %1, 40;\n add.u32 a6, %1, 48;\n add.u32 a7, %1, 56;\n"
                     " add.u64 b1, %2, 2;\n add.u64 b2, %2, 4;\n add.u64 b3, %2, 6;\n add.u64 b4, %2, %6;\n"
                     " add.u64 b5, b4, 2;\n add.u64 b6, b4, 4;\n add.u64 b7, b4, 6;\n"
                     SQNN_MMA("%0", "%1", "%2", "p") SQNN_MMA("%0", "a1", "b1", "t") SQNN_MMA("%0", "a2", "b2", "t")
                     SQNN_MMA("%0", "a3", "b3", "t") SQNN_MMA("%0", "a4", "b4", "t") SQNN_MMA("%0", "a5", "b5", "t")
                     SQNN_MMA("%0", "a6", "b6", "t") SQNN_MMA("%0", "a7", "b7", "t")
                     " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n}\n"
                     :: "r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(free_a), "l"(bdesc_hi) : "memory");
    } else {
        asm volatile("{\n .reg .pred e, p, t;\n .reg .b32 a1, a2, a3;\n .reg .b64 b1, b2, b3;\n"
                     " elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 t, %4, %4;\n"
                     " add.u32 a1, %1, 8;\n add.u32 a2, %1, 16;\n add.u32 a3, %1, 24;\n"
                     " add.u64 b1, %2, 2;\n add.u64 b2, %2, 4;\n add.u64 b3, %2, 6;\n"
                     SQNN_MMA("%0", "%1", "%2", "p") SQNN_MMA("%0", "a1", "b1", "t") SQNN_MMA("%0", "a2", "b2", "t")
                     SQNN_MMA("%0", "a3", "b3", "t")
                     " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n}\n"
                     :: "r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(free_a) : "memory");
    }
}
#undef SQNN_MMA
// Makes the mbarrier track completion of all MMAs the elected lane issued so far (converged warp).
SQNN_DEV void mma_commit(uint32_t bar)
{
    asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
                 " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n"
                 :: "r"(bar) : "memory");
}
// 16 consecutive accumulator columns of this thread's lane (one wait for the whole load).
SQNN_DEV void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
SQNN_DEV void tmem_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
// 16 consecutive columns of this thread's lane; tmem_st_wait() completes all stores of the warp.
SQNN_DEV void tmem_st16(uint32_t taddr, const uint32_t *v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};\n"
                 :: "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                    "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
                    "r"(taddr) : "memory");
}
SQNN_DEV void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major bf16 tile with 128-byte rows and 128-byte
// swizzle: rows 128 B apart, groups of 8 rows 1024 B apart (stride byte offset), descriptor
// version 1, layout type 2.  `addr` is the shared address of the first row, advanced by 32 B
// per K = 16 step inside the swizzled row.
SQNN_DEV uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3fffu);
    d |= (uint64_t)1u << 16;                       // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024u >> 4) << 32;             // stride byte offset
    d |= (uint64_t)1u << 46;                       // version
    d |= (uint64_t)2u << 61;                       // 128-byte swizzle
    return d;
}
// Instruction descriptor: D fp32, A and B bf16, both K-major, M = 128, N = n.
SQNN_DEV uint32_t instr_desc_bf16(uint32_t n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// Expands 32 columns (mask word m, plane word b, bit j = column j) into 16 registers of two bf16 each.
SQNN_DEV void expand32(uint32_t m, uint32_t b, uint32_t *v)
{
    const uint32_t s = ~b;                                                    // bit set: minus
    const uint32_t even = (m & 0x55555555u) | ((s << 1) & 0xaaaaaaaau);       // fields of columns 0, 2, .. 30
    const uint32_t odd = ((m >> 1) & 0x55555555u) | (s & 0xaaaaaaaau);        // fields of columns 1, 3, .. 31
    const uint32_t z0 = __byte_perm(even, odd, 0x5410), z1 = __byte_perm(even, odd, 0x7632);
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) {
        v[j] = (z0 << (14 - 2 * j)) & 0xc000c000u;
        v[8 + j] = (z1 << (14 - 2 * j)) & 0xc000c000u;
    }
}

}  // namespace sqnn
