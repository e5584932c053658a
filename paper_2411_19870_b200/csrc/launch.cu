// Host side of launch.cuh.
#include "launch.cuh"

namespace {

DemoLaunch::Known *find(DemoLaunch &dev, const void *kernel, int threads, size_t smem)
{
    for (int i = 0; i < dev.n_known; ++i) {
        DemoLaunch::Known &k = dev.known[i];
        if (k.kernel == kernel && k.threads == threads && (threads == 0 || k.smem == smem)) return &k;
    }
    return nullptr;
}
void note(DemoLaunch &dev, const DemoLaunch::Known &k)
{
    if (dev.n_known < (int)(sizeof(dev.known) / sizeof(dev.known[0]))) dev.known[dev.n_known++] = k;
}
// The limit is set to all that the device has, so that contexts with other sizes do not lower it for one another.
cudaError_t allow_locked(DemoLaunch &dev, const void *kernel)
{
    if (find(dev, kernel, 0, 0)) return cudaSuccess;
    int device = 0, most = 0;
    cudaFuncAttributes attr;
    cudaError_t err = cudaGetDevice(&device);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (err == cudaSuccess) err = cudaFuncGetAttributes(&attr, kernel);
    if (err == cudaSuccess) err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)attr.sharedSizeBytes);
    if (err == cudaSuccess) note(dev, DemoLaunch::Known{kernel, 0, 0, 0});
    return err;
}

}  // namespace

cudaError_t demo_allow_smem(DemoLaunch &dev, const void *kernel)
{
    std::lock_guard<std::mutex> lock(dev.mutex);
    return allow_locked(dev, kernel);
}

cudaError_t demo_resident_ctas(DemoLaunch &dev, const void *kernel, int threads, size_t smem, int *per_sm)
{
    std::lock_guard<std::mutex> lock(dev.mutex);
    if (const DemoLaunch::Known *k = find(dev, kernel, threads, smem)) {
        *per_sm = k->per_sm;
        return cudaSuccess;
    }
    cudaError_t err = allow_locked(dev, kernel);
    if (err != cudaSuccess) return err;
    int n = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem);
    if (err != cudaSuccess) return err;
    if (n < 1) n = 1;
    note(dev, DemoLaunch::Known{kernel, threads, smem, n});
    *per_sm = n;
    return cudaSuccess;
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
