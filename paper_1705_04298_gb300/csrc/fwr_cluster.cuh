// What the kernels that share a frame between the CTAs of a thread-block
// cluster have in common (fwr_cluster128.cu, fwr_cluster64.cu). Included inside
// namespace fwr.
#pragma once

namespace {

// every thread of the cluster: arrive orders this thread's earlier shared and
// remote-shared accesses before the accesses after the matching waits
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return int(r);
}
// the address of this CTA's shared-memory address a in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t a, int rank) {
    uint32_t o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(o) : "r"(a), "r"(rank));
    return o;
}
__device__ __forceinline__ void st_rank(uint32_t a, int rank, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(map_rank(a, rank)), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_rank(uint32_t a, int rank, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};\n" ::"r"(map_rank(a, rank)), "d"(v.x), "d"(v.y) : "memory");
}

// Columns are owned in pairs kx, -kx: of CTA `rank`, line j < SC is column SC
// rank + j, line SC + j its partner, with the self-paired N / 2 in place of the
// second column 0.
template <int N, int SC> __device__ __forceinline__ int owned_column(int rank, int line) {
    const int j = line - SC;
    if (line < SC) return SC * rank + line;
    return rank == 0 && j == 0 ? N / 2 : (N - SC * rank - j) & (N - 1);
}
template <int N, int SC> __device__ __forceinline__ void column_owner(int kx, int& rank, int& line) {
    const int k = kx < N / 2 ? kx : N - kx;
    rank = kx == N / 2 ? 0 : k / SC;
    line = kx == N / 2 ? SC : k % SC + (kx < N / 2 ? 0 : SC);
}

// Launch `kern` on as many clusters of cl CTAs as run at once, at most one per
// frame; `cache`: their number per device.
template <typename P>
cudaError_t launch_clusters(void (*kern)(P, int), const P& p, int cl, int threads, size_t smem, std::mutex& mu,
                            std::vector<std::pair<int, int>>& cache, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(cl);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(unsigned(cl));
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int dev = 0, clusters = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(mu);
        for (const auto& r : cache)
            if (r.first == dev) clusters = r.second;
        if (clusters == 0) {
            if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) != cudaSuccess)
                return e;
            if (cl > 8 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
                return e;
            if ((e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg)) != cudaSuccess) return e;
            if (clusters < 1) return cudaErrorInvalidConfiguration;
            cache.push_back({dev, clusters});
        }
    }
    if (p.F < clusters) clusters = p.F;
    cfg.gridDim = dim3(unsigned(cl * clusters));
    return cudaLaunchKernelEx(&cfg, kern, p, clusters);
}

}  // namespace
