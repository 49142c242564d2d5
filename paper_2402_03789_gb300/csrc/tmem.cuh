// tcgen05 pieces: tensor-memory allocation, the BF16 MMA with A in tensor memory and
// B in 128-byte-swizzled K-major shared memory, stores of A and reads of the accumulator.
#pragma once

#include <cstdint>

#include "async_copy.cuh"

namespace sn {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// one whole warp; ncols a power of two >= 32; the address is written to *dst (shared)
__device__ __forceinline__ void tmem_alloc(unsigned* dst, unsigned ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                 "tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned addr, unsigned ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(addr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// K-major operand tile of 128-byte rows (64 BF16), 128-byte swizzle, groups of
// eight rows 1,024 bytes apart; the tile starts on a 1,024-byte boundary.
__device__ __forceinline__ uint64_t umma_desc(unsigned saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// instruction descriptor: BF16 operands, FP32 accumulator, both K-major
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// One lane of a converged warp, the same each time.  MMA and commit instructions
// take their operands from uniform registers: under an elected lane they issue
// directly (under `lane == 0` each took about 310 cycles of operand shuffling).
__device__ __forceinline__ bool elect_one() {
    unsigned p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}
// D[tmem] (+)= A B^T, one thread; A in TMEM: a lane per row, two BF16 of K per column
__device__ __forceinline__ void umma_bf16_ts(unsigned d, unsigned a, uint64_t b, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d), "r"(a), "l"(b), "r"(idesc),
        "r"((unsigned)accumulate)
        : "memory");
}
// 32 columns of this lane's TMEM row
__device__ __forceinline__ void tmem_st32(unsigned addr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n" ::"r"(addr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
// arrive on the barrier when the MMAs issued so far by this thread are done
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}
// four columns of this lane's TMEM row; read only after tmem_wait
__device__ __forceinline__ void tmem_ld4(unsigned addr, float (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n"); }
// ties registers that a tmem_ld4 filled to the wait before it
__device__ __forceinline__ void tmem_tie(float (&v)[4]) {
    asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// expected bytes of the current phase, without an arrival
__device__ __forceinline__ void mbar_add_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// Bounded wait of a whole warp on a pipeline's barrier: false when `limit` clock cycles
// (at most about two seconds; 0: the phase is not over yet) ran out here or another thread
// of the CTA gave up (*abort).  The verdict is a vote: lanes that read the barrier and the
// flag at different times must not part, since full-warp shuffles and votes follow.
__device__ __forceinline__ bool pipe_wait(uint64_t* bar, unsigned parity, volatile int* abort, unsigned limit) {
    const unsigned a = smem_u32(bar);
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (__all_sync(0xffffffffu, done)) return true;
    const long long t0 = clock64();
    while (true) {
        if (__any_sync(0xffffffffu, *abort || clock64() - t0 >= (long long)limit)) {
            *abort = 1;
            return false;
        }
        // the last operand lets the hardware suspend the warp for up to that many ns
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(a), "r"(parity), "r"(20000u) : "memory");
        if (__all_sync(0xffffffffu, done)) return true;
    }
}

}  // namespace sn
