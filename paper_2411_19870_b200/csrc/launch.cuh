// Launching: the resident-CTA count and the shared-memory limit of a kernel are asked for once per demo_ctx, and consecutive
// kernels of this library overlap one kernel's launch with the end of the one before (programmatic dependent launch).
//
// Device side.  A kernel launched with demo_launch_kernel may be resident before the previous work of its stream has
// finished.  A StreamOrder, the first object of the kernel, keeps the order; its begin(), which every thread calls, is the line:
//   wait_first = 1: nothing behind begin() happens before everything queued earlier has finished;
//   wait_first = 0: the kernel before it belongs to the same call, works on other data and itself waited for everything
//     earlier; the two run side by side, and this one finishes last, so that whatever follows sees both complete.  It reads
//     what earlier kernels wrote (momentum, records) before any wait of its own.  The wait instruction promises such writes to the
//     grid that executes it, here the kernel before; that this one sees them too rests on two things: its CTAs start after every CTA of that
//     kernel is past its wait, when those writes have reached the L2; and the fence below, without which an SM might still hold older
//     lines of its own L1.
// A CTA lets the next kernel be launched once it is itself past its wait, and the next kernel's CTAs come only when every
// CTA of this one has come so far: they take registers and shared memory that nothing of this kernel still needs.  Tensor
// memory is allocated behind the wait, so no CTA holds any while it waits for another kernel.
//
// In front of begin() a CTA looks up its first chunk and acquires its tensor maps, so that these chains of dependent reads run while
// the kernel before it drains.  It reads only what no kernel writes: the context's tables, written by demo_init, and the tables of
// pointers and maps, written by copies of the same stream that were complete before the kernel in front of this one could start (a copy
// between two kernels orders them in full).  The first chunk's data, which that kernel may still be writing, is brought to L2 by
// prefetches, which read nothing into the SM: L2 is where both kernels' accesses meet.  Counters, records, momenta, a caller-supplied
// basis and tensor memory come behind begin().  (Look-up and maps in front, one compress call, s = 64, 16 / 1184 chunks 8.4 / 22.5 -> 7.8 /
// 18.9 us, s = 128, 16 / 296 13.4 / 23.2 -> 12.8 / 21.7; decode of 16 chunks 4.7 -> 4.4 and 7.6 -> 7.2.  Where the first tiles are also
// prefetched was measured kernel by kernel: s = 64 compress and s = 32 / 64 decode are faster without.)
#pragma once

#include <cuda_runtime.h>

#include <mutex>

struct StreamOrder {
    const int wait_first;
    __device__ __forceinline__ explicit StreamOrder(int w) : wait_first(w)
    {
        if (!wait_first) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    __device__ __forceinline__ void begin() const
    {
        if (wait_first) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        } else {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        }
    }
    __device__ __forceinline__ ~StreamOrder()
    {
        if (!wait_first) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
};

// Chunks of a persistent grid are handed out on demand: a CTA starts with chunk blockIdx.x and draws every further one from
// a counter, so that a CTA that falls behind (another part of the memory system, a chunk with ties) gets fewer of them, and
// the launch does not depend on which SM the CTAs came to.  The counter is zero between launches: the last CTA that is done
// with it clears it.  One pair of words per kernel that may be in flight beside others of its context: two that drew from one counter
// would leave chunks out.  A grid with a CTA for
// every chunk has nothing to hand out and makes do without (NULL): an atomic operation and a wait for it less at either end
// (256 x 256, s = 64: compress 9.1 -> 8.3 us, decode 6.6 -> 5.6).
struct DemoTickets {
    unsigned next, done;
};
constexpr unsigned NO_TICKET = 0x80000000u;  // beyond every list
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ unsigned ticket_draw(DemoTickets *t) { return t ? atomicAdd(&t->next, 1u) : NO_TICKET; }
// A CTA that knows its chunks two ahead draws the second one when it starts: one that starts early would draw its third, too, before one
// that starts late has its second.  So in launches of up to three rounds the second is fixed, chunk gridDim.x behind the first, and tickets
// count from there (s = 64, decode of 1500 / 2368 chunks 17.1 / 20.3 -> 15.1 / 17.8 us); in longer ones the draw evens out the SMs' start
// (s = 128, 2368 chunks: fixed 86.6 us, drawn 85.3).  second_ticket: of the second chunk; tickets_from: what is added to the tickets of those
// behind it, where they are written down, not where they are drawn, which would be a wait for the draw (2 % of decode).
__device__ __forceinline__ bool second_fixed(unsigned n_chunks) { return n_chunks / 3u < gridDim.x; }
__device__ __forceinline__ unsigned second_ticket(DemoTickets *t, unsigned n_chunks)
{
    return t == nullptr ? NO_TICKET : second_fixed(n_chunks) ? blockIdx.x : ticket_draw(t);
}
__device__ __forceinline__ unsigned tickets_from(unsigned n_chunks) { return second_fixed(n_chunks) ? gridDim.x : 0u; }
// (one thread of each of the CTA's `parties` that draw, after its last draw has returned)
__device__ __forceinline__ void ticket_finish(DemoTickets *t, unsigned parties = 1)
{
    const unsigned last = gridDim.x * parties - 1u;
    if (t && atomicInc(&t->done, last) == last) atomicExch(&t->next, 0u);
}

// Host side.  What launches on a device need: its SM count, and what is known about kernels launched before.  One per demo_ctx: the
// limits set on a kernel belong to the CUDA context, so they must not outlive it or serve another one.  Calls of several threads may
// share it.
struct DemoLaunch {
    struct Known {
        const void *kernel;
        int threads;  // 0: the kernel's shared-memory limit is set
        size_t smem;
        int per_sm;
    };
    int sm_count = 0;
    std::mutex mutex;
    Known known[64];  // kernels x sizes; a full table only means asking again
    int n_known = 0;
};
// Raises the kernel's dynamic shared-memory limit to what the device has and returns how many CTAs of `threads` threads fit an SM (at least 1).
cudaError_t demo_resident_ctas(DemoLaunch &dev, const void *kernel, int threads, size_t smem, int *per_sm);
// The limit alone, for kernels whose residency is computed by hand.
cudaError_t demo_allow_smem(DemoLaunch &dev, const void *kernel);
// Launch of a kernel with a StreamOrder.
cudaError_t demo_launch_kernel(const void *kernel, long long grid, int threads, size_t smem, cudaStream_t stream, void **params);
