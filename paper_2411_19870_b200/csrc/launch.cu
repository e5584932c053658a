// Host side of launch.cuh.
#include "launch.cuh"

#include <mutex>
#include <new>
#include <vector>

namespace {

struct Known {
    int device;
    const void *kernel;
    int threads;  // 0: the entry holds the shared-memory limit set so far
    size_t smem;
    int per_sm;
};
std::mutex g_mutex;
std::vector<Known> g_known;  // a few dozen entries: kernels x devices x sizes

Known *find(int device, const void *kernel, int threads, size_t smem)
{
    for (Known &k : g_known)
        if (k.kernel == kernel && k.device == device && k.threads == threads && (threads == 0 || k.smem == smem)) return &k;
    return nullptr;
}
cudaError_t allow_locked(int device, const void *kernel, size_t smem)
{
    Known *k = find(device, kernel, 0, 0);
    if (k && k->smem >= smem) return cudaSuccess;
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    if (k)
        k->smem = smem;  // (only ever raised: another thread's larger launch stays valid)
    else
        g_known.push_back(Known{device, kernel, 0, smem, 0});
    return cudaSuccess;
}

}  // namespace

cudaError_t demo_allow_smem(const void *kernel, size_t smem)
{
    int device = 0;
    const cudaError_t err = cudaGetDevice(&device);
    if (err != cudaSuccess) return err;
    std::lock_guard<std::mutex> lock(g_mutex);
    try {
        return allow_locked(device, kernel, smem);
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

cudaError_t demo_resident_ctas(const void *kernel, int threads, size_t smem, int *per_sm)
{
    int device = 0;
    cudaError_t err = cudaGetDevice(&device);
    if (err != cudaSuccess) return err;
    std::lock_guard<std::mutex> lock(g_mutex);
    if (const Known *k = find(device, kernel, threads, smem)) {
        *per_sm = k->per_sm;
        return cudaSuccess;
    }
    try {
        err = allow_locked(device, kernel, smem);
        if (err != cudaSuccess) return err;
        int n = 0;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem);
        if (err != cudaSuccess) return err;
        if (n < 1) n = 1;
        g_known.push_back(Known{device, kernel, threads, smem, n});
        *per_sm = n;
        return cudaSuccess;
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

cudaError_t demo_launch_kernel(const void *kernel, long long grid, int threads, size_t smem, cudaStream_t stream, void **params)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, kernel, params);
}
