// tc_device.cuh -- the fifth-generation tensor-core instructions the library
// uses (tcgen05, sm_103a): FP16 MMA of a CTA pair with FP32 accumulators in
// tensor memory, both operands in shared memory, completion through mbarriers.
//
// A pair (a cluster of two CTAs on neighbouring SMs) multiplies as one unit:
// each CTA holds 128 rows of A, the same rows of D in its own tensor memory,
// and half the columns of B; one thread of the first CTA issues.
//
// Operand layout (both operands, no swizzle, M/N-contiguous): core matrices of
// 8 k x 8 m, 128 bytes each, row k holding 8 consecutive m as 16 bytes; the
// core matrices of the next 8 k follow at `lbo` bytes, those of the next 8 m at
// `sbo` bytes.  A thread that owns one sample (one k) so writes 8 rows of an
// operand with one 16-byte store, and 8 threads with consecutive samples fill
// a core matrix without bank conflicts.  128 rows x 256 columns x 16 k on one SM
// run in 130 cycles from this layout (128 is the peak rate).
#pragma once

#include <cstdint>

namespace lsp {
namespace tc {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t pair_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// True in one lane of a converged warp: code around it stays warp-uniform, so
// that descriptors are formed in uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p;
}
// Every thread of the pair; memory before it is visible after it to both CTAs.
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_done() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// One arrival at the first CTA's barrier of this name, from either CTA.  What it
// reports never leaves the CTA (operands and accumulators are read by the SM
// that wrote them, past the proxy fence or the tcgen05 fence before it), so it
// does not release at cluster scope, which costs a warp with stores in flight
// over 1,000 cycles.
__device__ __forceinline__ void mbar_arrive_first(uint64_t* b) {
    asm volatile(
        "{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %0, 0;\n"
        " mbarrier.arrive.shared::cluster.b64 _, [a];\n}" ::"r"(smem_addr(b))
        : "memory");
}

// Waits for the phase of the given parity, at most kWaitClocks (about a
// second); false when it ran out.
constexpr long long kWaitClocks = 2000000000ll;
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity) {
    const uint32_t a = smem_addr(b);
    long long t0 = 0;
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
        const long long now = clock64();
        if (t0 == 0) t0 = now;
        else if (now - t0 > kWaitClocks) return false;
    }
}
// Whether the phase is complete now.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(b)), "r"(parity)
        : "memory");
    return ok;
}

// Tensor memory: columns of 128 lanes x 32 bits; one warp of each CTA of the
// pair allocates and frees.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}

// D[256][N] (+)= A[16][256]^T B[16][N] over the pair, FP16 operands by
// descriptor (the same shared-memory offsets in both CTAs), FP32 D.
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Both CTAs' barriers of this name are arrived at once every MMA issued so far
// by this thread is done.
__device__ __forceinline__ void mma_commit(uint64_t* b) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_addr(b)),
        "h"((uint16_t)3)
        : "memory");
}

// Shared-memory stores of this thread become visible to the tensor cores.
__device__ __forceinline__ void fence_operands() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive columns of the calling warp's 32 lanes (a lane's row); the
// wait is part of the statement, so no use of r can move before it.
__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr)
        : "memory");
}

__device__ __forceinline__ uint64_t operand_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// FP16 operands, both M/N-contiguous, FP32 accumulators, M = 256 over the pair.
__device__ __forceinline__ uint32_t instr_desc(int N) {
    return (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | (16u << 24);
}

}  // namespace tc
}  // namespace lsp
