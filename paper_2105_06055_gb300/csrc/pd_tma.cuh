// Bulk asynchronous copies and mbarrier helpers for sm_103a (private).
//
// Rows move between global and shared memory with cp.async.bulk (loads complete
// on an mbarrier, stores drain through a bulk group). Every wait on an mbarrier
// is bounded by the global timer: on time-out the block sets a bit in the plan's
// device status word, gives its copies as long again to land (they write to shared
// memory that the SM hands to another block) and leaves without touching the tile.
#pragma once

#include "pd_common.cuh"

namespace pd {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s
constexpr int kErrTmaTimeout = 1;

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(unsigned long long *mbar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long *mbar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned mbar, unsigned phase)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(mbar), "r"(phase)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `phase` of the barrier. Returns false on time-out
// (after recording it in *err).
__device__ __forceinline__ bool mbar_wait(unsigned long long *mbar, unsigned phase, int *err)
{
    const unsigned m = smem_u32(mbar);
    if (mbar_try_wait(m, phase)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(m, phase)) {
        if (global_ns() - t0 > kWaitLimitNs) {
            if (err) atomicOr(err, kErrTmaTimeout);
            return false;
        }
    }
    return true;
}

// The wait after one that ran out, bounded alike. Out of line: inlined it cost the row
// passes up to 2% in registers and code (128^3 solve 0.6 to 2%, so 0.1 to 0.4%).
static __device__ __noinline__ void mbar_drain(unsigned mbar, unsigned phase)
{
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(mbar, phase) && global_ns() - t0 <= kWaitLimitNs) {
    }
}

// A block's wait for the copies that its first thread has issued: wait() is one bounded
// wait (false on time-out), vote(x) whether x holds in any thread of the block (a block
// barrier). False when the wait of any thread ran out; the first thread has then
// drained the copies, and the block leaves behind its second vote, together.
template <class Wait, class Vote, class Drain>
__host__ __device__ __forceinline__ bool wait_for_copies(bool first, Wait wait, Vote vote, Drain drain)
{
    const bool out = vote(!wait());
    if (out) {
        if (first) drain();
        vote(false);
    }
    return !out;
}

// 1D bulk copy global -> shared (16-byte aligned addresses, size multiple of 16)
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, unsigned long long *mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(mbar))
                 : "memory");
}

// Bulk prefetch of [src, src + bytes) into L2 (16-byte aligned address, size a
// multiple of 16; no shared memory, no completion to wait for)
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// 1D bulk copy shared -> global
__device__ __forceinline__ void bulk_store(void *dst, const void *src, unsigned bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Programmatic dependent launch: wait for the preceding grid of the stream to
// complete (its memory visible); a no-op when the grid was launched without
// the programmatic-serialization attribute. The trigger lets the next grid's
// blocks start their prologue once every block of this grid has issued it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Early start of the dependent kernel. The FFT passes do not call it (their
// dependents start as they end): with the trigger at the head of a pass that does
// not fill the chip, all blocks of the next pass moved in at once, most of them on
// the SMs that the pass had left empty, and ran there one after the other. Without
// it: 64^3 FP64 224 -> 126 us, 1024 x 512 FP32 31 -> 23, 128 x 128 x 64 FP32 41 -> 33,
// state-based 77 -> 63. Kernels of one block (final reductions) call it, and the body
// sums (pd_affine.cuh), whose dependent is such a kernel.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// make this thread's generic-proxy shared-memory writes visible to the async proxy
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

}  // namespace pd
