// The CTAs of one (batch, head) unit as a thread-block cluster: barriers, stores to and loads from the other CTAs' shared
// memory, the merge of softmax states over the cluster, and how many clusters a device holds.
#pragma once
#include <atomic>

#include "psattn_common.cuh"
#include "psattn_launch.h"
#include "psattn_sm100.cuh"

namespace psattn {

constexpr int kMaxSplit = 8;           // CTAs per cluster at most (the portable limit)

__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ float peer_load(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
// Column c of row r over all CTAs of the unit: the states (m, l, acc) that every CTA left at `states` in its shared
// memory (66 floats per row) merged in rank order; returns acc / l.
template <int MOST>
__device__ __forceinline__ float merge_states_n(int split, uint32_t states, int r, int c) {
    float m[MOST], l[MOST], a[MOST];
#pragma unroll
    for (int x = 0; x < MOST; ++x) {                          // all loads in flight together
        m[x] = -INFINITY; l[x] = 0.f; a[x] = 0.f;
        if (x >= split) continue;
        const uint32_t p = peer_addr(states + (uint32_t)r * 264u, x);
        m[x] = peer_load(p); l[x] = peer_load(p + 4u); a[x] = peer_load(p + 8u + 4u * (uint32_t)c);
    }
    float mw = -INFINITY, lw = 0.f, aw = 0.f;
#pragma unroll
    for (int x = 0; x < MOST; ++x) mw = fmaxf(mw, m[x]);
#pragma unroll
    for (int x = 0; x < MOST; ++x) {
        const float f = l[x] > 0.f ? sm100::fast_exp2(m[x] - mw) : 0.f;
        lw += l[x] * f; aw += a[x] * f;
    }
    return lw > 0.f ? aw / lw : 0.f;
}
__device__ __forceinline__ float merge_states(int split, uint32_t states, int r, int c) {
    return split > 4 ? merge_states_n<kMaxSplit>(split, states, r, c) : split > 2 ? merge_states_n<4>(split, states, r, c) : merge_states_n<2>(split, states, r, c);
}

// Clusters of `split` CTAs of `kernel` (at the given shared memory) that the current device holds at once; asked once per
// device and kernel (`cached`: one record per kernel).
struct ClusterRecord {
    std::atomic<int> n[kMaxDevices][kMaxSplit + 1];
};
template <typename... KArgs>
inline int max_clusters(void (*kernel)(KArgs...), ClusterRecord &cached, int split, int threads, size_t smem) {
    const int k = split;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return 0; }
    int n = cached.n[dev][k].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)split);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        if (n <= 0) n = -1;
        cached.n[dev][k].store(n, std::memory_order_relaxed);
    }
    return n < 0 ? 0 : n;
}

// Launch with programmatic stream serialization, as clusters of `split` CTAs where split > 1.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_split(void (*kernel)(KArgs...), unsigned units, int split, int threads, size_t smem, cudaStream_t st,
                                Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(units * (unsigned)split);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = split > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace psattn
