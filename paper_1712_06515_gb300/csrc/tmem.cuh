// Tensor memory as per-thread state: allocation by one warp, columns of a thread's lane to and
// from registers.  Every call is warp-collective.
#pragma once

#include "common.cuh"
#include "tma.cuh"

namespace cc {

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

#define CC_R8(v, o) "+f"(v[o]), "+f"(v[o + 1]), "+f"(v[o + 2]), "+f"(v[o + 3]), "+f"(v[o + 4]), "+f"(v[o + 5]), "+f"(v[o + 6]), "+f"(v[o + 7])
#define CC_W8(v, o) "=f"(v[o]), "=f"(v[o + 1]), "=f"(v[o + 2]), "=f"(v[o + 3]), "=f"(v[o + 4]), "=f"(v[o + 5]), "=f"(v[o + 6]), "=f"(v[o + 7])
#define CC_I8(v, o) "f"(v[o]), "f"(v[o + 1]), "f"(v[o + 2]), "f"(v[o + 3]), "f"(v[o + 4]), "f"(v[o + 5]), "f"(v[o + 6]), "f"(v[o + 7])

// 32 (16, 8) columns of this thread's lane into registers, complete on return, and back.  The
// wait takes the loaded values as operands, so that no use of them moves above it.
__device__ __forceinline__ void tmem_ld(float (&v)[32], uint32_t a) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : CC_W8(v, 0), CC_W8(v, 8), CC_W8(v, 16), CC_W8(v, 24) : "r"(a) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : CC_R8(v, 0), CC_R8(v, 8), CC_R8(v, 16) :: "memory");
    asm volatile("" : CC_R8(v, 24) :: "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&v)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
                 "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 :: "r"(a), CC_I8(v, 0), CC_I8(v, 8), CC_I8(v, 16), CC_I8(v, 24) : "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&v)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 :: "r"(a), CC_I8(v, 0), CC_I8(v, 8) : "memory");
}
__device__ __forceinline__ void tmem_ld(float (&v)[8], uint32_t a) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];" : CC_W8(v, 0) : "r"(a) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : CC_R8(v, 0) :: "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" :: "r"(a), CC_I8(v, 0) : "memory");
}

#undef CC_R8
#undef CC_W8
#undef CC_I8

}  // namespace cc
