// async.cuh -- thin inline-PTX wrappers for asynchronous global -> shared copies
// and for addresses in a cluster peer's shared memory.
#pragma once
#include <stdint.h>

namespace miugks {

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;\n" : "=l"(t));
    return t;
}

constexpr int kWaitRounds = 1 << 26;         // a bounded wait gives up after this many looks, too

// address of the same shared-memory location in cluster CTA `rank`
__device__ __forceinline__ unsigned peer_addr(const void* p, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}

// asynchronous 16-byte global -> shared copy (LDGSTS, cached in L2 only; both
// addresses 16-byte aligned), completed per commit group of the issuing thread
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's most recent commit groups are pending
template <int N>
__device__ __forceinline__ void cp_async_wait_n()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

}  // namespace miugks
