// Grid-wide barrier for kernels launched cooperatively (all blocks co-resident): an arrival
// counter in global memory, release on arrival, acquire on the poll.  The wait is bounded all
// the same: a block that has polled `spin_limit` times without seeing `target` arrivals raises
// QP_DEV_STREAM_TIMEOUT in the status word and reports failure, so the kernel can leave and
// the context stays usable.  The counter must be zero when the launch starts and the kernel
// resets it when its last block leaves; after a time-out too where blocks leave through count_out,
// by qp_get_status where they do not (the small-tensor sender).
#pragma once

#include <cuda_runtime.h>

#include "quantpipe.h"                                        // QP_DEV_STREAM_TIMEOUT

namespace qp_grid {

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void arrive_release(unsigned* p)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Arrivals that a launch's barrier number `nr` (from 1 on) waits for.  extra: 0, or the number of the first barrier that a test makes
// wait for one arrival more than there are blocks.
__device__ __forceinline__ unsigned target(unsigned nr, unsigned blocks, unsigned extra) { return nr * blocks + (extra - 1u < nr ? 1u : 0u); }

// One thread polls until `target` arrivals; false when the wait ran out.
__device__ __forceinline__ bool poll(const unsigned* bar, unsigned target, unsigned spin_limit, unsigned* status)
{
    unsigned spins = 0;
    while (ld_acquire(bar) < target) {
        if (++spins > spin_limit) {
            atomicOr(status, QP_DEV_STREAM_TIMEOUT);
            return false;
        }
        if (spins > 64) __nanosleep(64);
    }
    return true;
}

// All blocks arrive, then all leave.  The block's writes are ordered before the arrival by the
// block barrier and the release; the acquire load orders the other blocks' writes before what
// follows.  Returns false (for the whole block) when the wait ran out.  s_ok: one int of
// shared memory.
__device__ __forceinline__ bool barrier(unsigned* bar, unsigned target, unsigned spin_limit, unsigned* status, int* s_ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        arrive_release(bar);
        *s_ok = poll(bar, target, spin_limit, status);
    }
    __syncthreads();
    return *s_ok != 0;
}

// The same for what warp 0 has written (and what the block had written before its last block barrier), and for what warp 0 reads
// next; the other warps do not stop here.  By warp 0; the block learns from s_ok, behind its next barrier, whether the wait ran out.
__device__ __forceinline__ void barrier_warp0(unsigned* bar, unsigned target, unsigned spin_limit, unsigned* status, int* s_ok)
{
    __syncwarp();
    if (threadIdx.x == 0) arrive_release(bar);
    unsigned spins = 0;
    while (__any_sync(0xFFFFFFFFu, ld_acquire(bar) < target)) {
        if (++spins > spin_limit) {
            if (threadIdx.x == 0) atomicOr(status, QP_DEV_STREAM_TIMEOUT);
            break;
        }
        if (spins > 64) __nanosleep(64);
    }
    if (threadIdx.x == 0) *s_ok = spins <= spin_limit;
    __syncwarp();
}

// A block's way out, by one of its threads, when the block will neither arrive nor poll again.  bar[1] counts the blocks out
// in its low half and those whose wait ran out in its high half, so that the last one learns both from one atomic (a flag of
// its own cost the launches 1.9 us at their ends).  The block's own arrivals must have been performed: it has polled since, or
// fences first.
constexpr unsigned GAVE_UP = 0x10000u;
__device__ __forceinline__ unsigned count_out(unsigned* bar, unsigned gave_up = 0u)
{
    return atomicAdd(bar + 1, 1u + gave_up);
}
// With what count_out returned: whether this was the last block (blocks are below 2^16) ...
__device__ __forceinline__ bool last_out(unsigned before, unsigned blocks) { return (before & 0xFFFFu) == blocks - 1; }
// ... which puts the words back to zero.
__device__ __forceinline__ void reset(unsigned* bar) { bar[0] = bar[1] = 0u; }

// A grid that is one thread-block cluster has the hardware's barrier instead (about 0.4 us against 1.2): all threads
// arrive, then all wait; it orders global memory like the counter does, and its blocks are resident together by definition.
// It has no limit and needs none: it waits for threads of the cluster that have not exited, every one of which is running
// and reaches the same barriers, for no block of a cluster waits for anything else.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

}  // namespace qp_grid
