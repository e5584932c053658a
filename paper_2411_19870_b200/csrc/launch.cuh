// Launching: the resident-CTA count and the shared-memory limit of a kernel are asked for once per demo_ctx, and consecutive
// kernels of this library overlap one kernel's launch with the end of the one before (programmatic dependent launch).
//
// Device side.  A kernel launched with demo_launch_kernel may be resident before the previous work of its stream has
// finished.  A StreamOrder, the first object of the kernel, keeps the order:
//   wait_first = 1: it touches nothing before everything queued earlier has finished;
//   wait_first = 0: the kernel before it belongs to the same call, works on other data and itself waited for everything
//     earlier; the two run side by side, and this one finishes last, so that whatever follows sees both complete.  It reads
//     what earlier kernels wrote (momentum, records) before any wait of its own.  The wait instruction promises such writes to the
//     grid that executes it, here the kernel before; that this one sees them too rests on two things: its CTAs start after every CTA of that
//     kernel is past its wait, when those writes have reached the L2; and the fence below, without which an SM might still hold older
//     lines of its own L1.
// A CTA lets the next kernel be launched once it is itself past its wait, and the next kernel's CTAs come only when every
// CTA of this one has come so far: they take registers and shared memory that nothing of this kernel still needs.  Tensor
// memory is allocated behind the wait, so no CTA holds any while it waits for another kernel.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

struct StreamOrder {
    const int wait_first;
    __device__ __forceinline__ explicit StreamOrder(int w) : wait_first(w)
    {
        if (wait_first)
            asm volatile("griddepcontrol.wait;" ::: "memory");
        else
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
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
__device__ __forceinline__ unsigned ticket_draw(DemoTickets *t) { return t ? atomicAdd(&t->next, 1u) : NO_TICKET; }
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
