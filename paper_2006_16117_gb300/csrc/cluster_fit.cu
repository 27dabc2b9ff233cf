// The occupancy queries behind cluster_fit.h.
#include "cluster_fit.h"

#include <map>
#include <mutex>
#include <set>
#include <tuple>

#include "common.cuh"

namespace sim {

namespace {

int device_attribute(cudaDeviceAttr attr) {
    int dev = 0, v = 0;
    SIM_CUDA(cudaGetDevice(&dev));
    SIM_CUDA(cudaDeviceGetAttribute(&v, attr, dev));
    return v;
}

}  // namespace

int sm_count() {
    static const int n = device_attribute(cudaDevAttrMultiProcessorCount);
    return n;
}

int clusters_that_fit(const void* kernel, int size, int threads, size_t smem) {
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> prepared;
    static std::map<std::tuple<int, const void*, int, int, size_t>, int> known;
    int dev = 0;
    SIM_CUDA(cudaGetDevice(&dev));
    const auto key = std::make_tuple(dev, kernel, size, threads, smem);
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    if (!prepared.count({dev, kernel})) {
        cudaFuncAttributes fa{};
        SIM_CUDA(cudaFuncGetAttributes(&fa, kernel));
        const int most = device_attribute(cudaDevAttrMaxSharedMemoryPerBlockOptin) - (int)fa.sharedSizeBytes;
        SIM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        // (where that is refused, the query below has no room for more than 8)
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            (void)cudaGetLastError();
        prepared.insert({dev, kernel});
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    known[key] = n;
    return n;
}

}  // namespace sim
