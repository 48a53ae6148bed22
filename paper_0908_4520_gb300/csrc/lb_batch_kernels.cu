// Instantiation and launch of the persistent multi-instance kernel for one
// storage type (compiled once per type with LB_BATCH_STORAGE / LB_BATCH_ENTRY).
#include "lb_batch.cuh"

namespace lbk {

namespace {
cudaLaunchConfig_t config(int grid, int cluster, int threads, int smem, cudaStream_t st, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cluster;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <class S>
cudaError_t launch_s(const void* args, int grid, int cluster, int threads, int smem, cudaStream_t st) {
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config(grid, cluster, threads, smem, st, &at);
    return cudaLaunchKernelEx(&cfg, lb_batch_kernel<S>, *static_cast<const BatchArgs*>(args));
}

template <class S>
cudaError_t setup_s(int threads, int cluster, int* smem, int* grid) {
    // the attribute belongs to the kernel, not to a batch: raise it to the device limit once,
    // so batches with different on-chip budgets can coexist
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // (the dynamic limit leaves room for the kernel's own static shared memory)
    cudaFuncAttributes attr{};
    cudaError_t e = cudaFuncGetAttributes(&attr, lb_batch_kernel<S>);
    if (e != cudaSuccess) return e;
    const int room = optin - (int)attr.sharedSizeBytes;
    // budgets up to 1156 bytes below the device's limit are taken (what a kernel with 1156 bytes of its
    // own would leave) and brought down to what this kernel leaves; larger ones are refused
    if (*smem > optin - 1156) return cudaErrorInvalidValue;
    if (*smem > room) *smem = room;
    e = cudaFuncSetAttribute(lb_batch_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config(cluster, cluster, threads, *smem, nullptr, &at);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, lb_batch_kernel<S>, &cfg);
    *grid = n * cluster;
    return e;
}
}  // namespace

#ifndef LB_BATCH_STORAGE
#error "LB_BATCH_STORAGE must name the storage type of this unit"
#endif

cudaError_t LB_BATCH_ENTRY(launch)(const void* args, int grid, int cluster, int threads, int smem, cudaStream_t st) {
    return launch_s<LB_BATCH_STORAGE>(args, grid, cluster, threads, smem, st);
}

cudaError_t LB_BATCH_ENTRY(setup)(int threads, int cluster, int* smem, int* grid) {
    return setup_s<LB_BATCH_STORAGE>(threads, cluster, smem, grid);
}

}  // namespace lbk
