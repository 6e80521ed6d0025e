// phase_barrier.cuh -- the barrier between the phases of one launch.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

namespace lbmd {

// Barrier of all blocks of a launch whose blocks are resident together.  Up to
// 16 blocks form one thread-block cluster and use its hardware barrier (0.25 us;
// 1.1 us with a load and an atomic of each thread in flight).  More blocks are a
// cooperative launch and count their arrivals in one word, which only grows
// during the launch (1.2 us / 1.8 us at 128 blocks of 256 threads; a count that
// the last block clears beside a generation word took 2.2 / 2.9 us).  The last
// block to finish clears the word for the next launch.  The wait is bounded
// (the blocks arrive within microseconds; the default limit is seconds): a
// block that gives up sets the error flags and ends, and so does every block
// that finds the flag set.  The words then keep counts that no launch can use,
// so while the flag is set no wait is passed, in this launch or a later one,
// until the owner clears the flag and the words.  What a kernel that ends there
// has not written keeps its former values: the owner's buffers must be safe to
// read in that state.
struct GridBarrier {
    uint32_t *word;       // arrivals, finished blocks
    int32_t *error;       // device memory
    int32_t *host_error;  // the same in host memory the GPU writes, or null
    int polls;            // limit of a wait
};
__device__ __forceinline__ int32_t load_flag(const int32_t *p) {
    int32_t v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
template <bool CLUSTER>
struct PhaseBarrier {
    GridBarrier g;
    uint32_t target = 0;
    // (The cluster instructions without .aligned: lanes that took different
    // branches just before need not have met again.)
    // The block's accesses so far are done, as far as the blocks that pass the
    // wait can see.  Work between the two hides a part of the barrier: two cycles
    // of 2,560 beads with Lennard-Jones forces 280 -> 275 us, a gradient of 200 MD
    // steps with 64 particles 1853 -> 1788 us.
    __device__ __forceinline__ void arrive() {
        if (gridDim.x == 1) {
            __syncthreads();
        } else if (CLUSTER) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        } else {
            target += gridDim.x;
            __syncthreads();
            if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(g.word) : "memory");
        }
    }
    __device__ __forceinline__ bool wait() {
        if (gridDim.x == 1) return true;
        if (CLUSTER) {
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
            return true;
        }
        bool ok = true;
        if (threadIdx.x == 0) {
            // At the first wait: a flag that an earlier launch set, or a limit of 0.
            // (A block of this launch that sets it arrives no more; tests inside the
            // loop cost 0.5 % of a cycle of 4,096 bonded particles.)
            int32_t failed = target == gridDim.x ? (load_flag(g.error) | (g.polls == 0)) : 0;
            for (int polls = 0;; ++polls) {
                uint32_t v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(g.word) : "memory");
                if ((int32_t)(v - target) >= 0) break;
                if (polls > g.polls) {
                    failed = 1;
                    break;
                }
            }
            if (failed) {
                atomicExch(g.error, 1);
                if (g.host_error) *(volatile int32_t *)g.host_error = 1;
                ok = false;
            }
        }
        return __syncthreads_and(ok) != 0;
    }
    __device__ __forceinline__ bool meet() {
        arrive();
        return wait();
    }
    // the block's last act
    __device__ __forceinline__ void finish() {
        if (CLUSTER || gridDim.x == 1) return;
        __syncthreads();
        if (threadIdx.x == 0 && atomicAdd(g.word + 1, 1u) == gridDim.x - 1) {
            g.word[0] = 0u;
            g.word[1] = 0u;
        }
    }
};

// Launch `kernel` (its CLUSTER form up to max_cluster blocks, its grid form
// above) with all blocks resident together.  Blocks of a cluster are rounded up
// to a power of two: the kernel ignores threads beyond its work.
inline cudaError_t launch_phase(const void *cluster_kernel, const void *grid_kernel, unsigned blocks, int threads,
                                int max_cluster, void **args, cudaStream_t stream) {
    const bool cluster = blocks <= (unsigned)max_cluster;
    while (cluster && (blocks & (blocks - 1))) ++blocks;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    cudaLaunchAttribute at = {};
    if (cluster) {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = blocks;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
    } else {
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
    }
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, cluster ? cluster_kernel : grid_kernel, args);
}

// Lowers max_cluster to the largest power of two the kernel can run as.
inline cudaError_t limit_cluster(const void *cluster_kernel, int threads, int &max_cluster) {
    cudaError_t e = cudaFuncSetAttribute(cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (; e == cudaSuccess && max_cluster > 1; max_cluster /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)max_cluster);
        cfg.blockDim = dim3((unsigned)threads);
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)max_cluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, cluster_kernel, &cfg);
        if (n > 0) break;
    }
    return e;
}

}  // namespace lbmd
