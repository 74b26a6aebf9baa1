// What the kernels of a file need once per device: shared-memory opt-ins, and whether the device grants their clusters.
#pragma once
#include <atomic>
#include <mutex>

#include "common.cuh"

namespace tpcg {

int cluster_limit();   // TPCG_OPT_CLUSTER

class PerDevice {
    std::mutex mu_;
    std::atomic<int> state_[64] = {};   // 0: not prepared; else 1, and 2 more where clusters of 16 are granted
    static int slot() {
        int dev = 0;
        return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 63 ? dev : 63;
    }

public:
    // f(&wide) once on the current device; takes driver locks, so it stays off the launch path
    template <typename F>
    int prepare(F f) {
        std::lock_guard<std::mutex> lock(mu_);
        std::atomic<int>& s = state_[slot()];
        if (s.load()) return TPCG_OK;
        bool wide = true;
        TPCG_TRY(f(&wide));
        s.store(wide ? 3 : 1);
        return TPCG_OK;
    }
    // whether launches may use the file's clusters of 16 CTAs
    bool wide() { return cluster_limit() >= 16 && (state_[slot()].load(std::memory_order_relaxed) & 2); }
};

// Allows a kernel clusters above the portable 8 CTAs and clears *wide where the device cannot hold one of them (a partition
// with smaller GPCs).
template <typename K>
int allow_cluster(K* kernel, int ctas, int threads, size_t smem, bool* wide) {
    if (ctas <= 8) return TPCG_OK;
    TPCG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    if (n < 1) *wide = false;
    return TPCG_OK;
}

}  // namespace tpcg
