// st_common.cuh -- device helpers shared by the kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "st_kernels.cuh"

namespace st {

typedef unsigned long long ull;

static __host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// Programmatic dependent launch (PTX griddepcontrol): let the next kernel of
// the stream be scheduled once every CTA of this grid has signalled or ended,
// and wait for the completion and memory of the grids this one depends on.
__device__ __forceinline__ void pdl_signal() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bulk copies (the TMA's untiled form, cp.async.bulk) into shared memory,
// completing on an mbarrier: one thread initialises the barrier, one thread
// issues each copy with the byte count it expects, every thread waits for the
// phase.  Both addresses 16-byte aligned, the size a multiple of 16 bytes.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(ull* b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bulk_to_smem(void* dst, const void* src, unsigned bytes, ull* b) {
    // the CTA's earlier reads of dst (ordered by a barrier) before the copy's writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(b))
                 : "memory");
}
// Polls the barrier's phase `parity`; false after max_polls unsuccessful polls.
__device__ __forceinline__ bool mbar_wait(ull* b, unsigned parity, int max_polls) {
    const uint32_t a = smem_addr(b);
    for (int i = 0; i < max_polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// A staging copy that has not landed after this many polls (each of which
// may suspend the thread for a while) is given up: the launch is marked
// faulty and the item reads its hits from global memory.
constexpr int kStagePolls = 1 << 22;

// First container index of event e: events are laid out back to back with
// three spare entries each, rounded up to a multiple of four floats so that
// every event starts 16-byte aligned.
__device__ __forceinline__ int64_t cont_base(const int64_t* ev_off, int64_t e) {
    int64_t b = (ev_off[e] - ev_off[0]) + 3 * e;
    return (b + 3) & ~int64_t(3);
}

}  // namespace st
