// Block shapes of the persistent time step.  Each shape (threads per block, blocks per SM) is an instantiation of
// k_persistent compiled in a translation unit of its own (persist_<precision>_s<n>.cu, built in parallel); the
// host picks one per handle, fixed (sim_options.block_shape >= 0) or by timing one time step in each
// (block_shape = -1, the block-shape autotuner).
#pragma once

#include "persistent.cuh"

namespace pncg {

constexpr int N_PSHAPES = 5;
// shape s: PSHAPE_PB[s] threads per block, at most PSHAPE_MINB[s] blocks per SM (the launch bound the compiler
// fits the registers to: 128 per thread at 2 x 256, 85 at 3 x 256, 255 at 1 x 256; 128 at 1 x 512, 168 at 1 x 384)
constexpr int PSHAPE_PB[N_PSHAPES] = {256, 512, 256, 256, 384};
constexpr int PSHAPE_MINB[N_PSHAPES] = {2, 1, 3, 1, 1};

// The cluster form of small meshes: CLUSTER_PB threads per block, all blocks of the launch in one cluster.
constexpr int CLUSTER_PB = 256;

// Launch of shape S (cooperative, grid blocks, PSHAPE_PB[S] threads) and its occupancy (blocks per SM).  The corotated
// densities (FCR, ARAP; CO) run instantiations of their own, so that the kernels of the others carry none of their
// code and registers; the FP32 form has them in the default shape only.
template <typename R, int S, bool CO> cudaError_t persist_launch(const Dev<R> &D, const BPDev &B, const PersistArgs &A,
                                                                 int grid, cudaStream_t s);
template <typename R, int S, bool CO> cudaError_t persist_occupancy(int *per_sm);
// The same of the cluster form; *blocks receives the blocks of the largest cluster (16 or 8) the device can hold, 0 = none.
template <typename R, bool CO> cudaError_t cluster_launch(const Dev<R> &D, const BPDev &B, const PersistArgs &A, int grid,
                                                          cudaStream_t s);
template <typename R, bool CO> cudaError_t cluster_blocks(int *blocks);

#define PNCG_PERSIST_DECL(R, S, CO)                                                                             \
    template <> cudaError_t persist_launch<R, S, CO>(const Dev<R> &, const BPDev &, const PersistArgs &, int,   \
                                                     cudaStream_t);                                            \
    template <> cudaError_t persist_occupancy<R, S, CO>(int *);
PNCG_PERSIST_DECL(float, 0, false) PNCG_PERSIST_DECL(float, 1, false) PNCG_PERSIST_DECL(float, 2, false)
PNCG_PERSIST_DECL(float, 3, false) PNCG_PERSIST_DECL(float, 4, false) PNCG_PERSIST_DECL(float, 0, true)
PNCG_PERSIST_DECL(double, 0, false) PNCG_PERSIST_DECL(double, 1, false) PNCG_PERSIST_DECL(double, 2, false)
PNCG_PERSIST_DECL(double, 3, false) PNCG_PERSIST_DECL(double, 4, false)
PNCG_PERSIST_DECL(double, 0, true) PNCG_PERSIST_DECL(double, 1, true) PNCG_PERSIST_DECL(double, 2, true)
PNCG_PERSIST_DECL(double, 3, true) PNCG_PERSIST_DECL(double, 4, true)
#undef PNCG_PERSIST_DECL
#define PNCG_CLUSTER_DECL(R, CO)                                                                                \
    template <> cudaError_t cluster_launch<R, CO>(const Dev<R> &, const BPDev &, const PersistArgs &, int,      \
                                                  cudaStream_t);                                               \
    template <> cudaError_t cluster_blocks<R, CO>(int *);
PNCG_CLUSTER_DECL(float, false) PNCG_CLUSTER_DECL(float, true) PNCG_CLUSTER_DECL(double, false) PNCG_CLUSTER_DECL(double, true)
#undef PNCG_CLUSTER_DECL

// the definitions, one shape per translation unit
#define PNCG_PERSIST_DEF(R, S, CO)                                                                              \
    template <> cudaError_t persist_launch<R, S, CO>(const Dev<R> &D, const BPDev &B, const PersistArgs &A,     \
                                                     int grid, cudaStream_t s)                                 \
    {                                                                                                          \
        Dev<R> d = D;                                                                                          \
        BPDev b = B;                                                                                           \
        PersistArgs a = A;                                                                                     \
        void *args[] = {(void *)&d, (void *)&b, (void *)&a};                                                   \
        return cudaLaunchCooperativeKernel((const void *)k_persistent<R, PSHAPE_PB[S], PSHAPE_MINB[S], CO>,     \
                                           dim3(grid), dim3(PSHAPE_PB[S]), args, 0, s);                        \
    }                                                                                                          \
    template <> cudaError_t persist_occupancy<R, S, CO>(int *per_sm)                                           \
    {                                                                                                          \
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(                                                  \
            per_sm, k_persistent<R, PSHAPE_PB[S], PSHAPE_MINB[S], CO>, PSHAPE_PB[S], 0);                        \
    }
#define PNCG_CLUSTER_DEF(R, CO)                                                                                 \
    template <> cudaError_t cluster_launch<R, CO>(const Dev<R> &D, const BPDev &B, const PersistArgs &A,        \
                                                  int grid, cudaStream_t s)                                    \
    {                                                                                                          \
        cudaLaunchAttribute at;                                                                                \
        const cudaLaunchConfig_t cfg = cluster_config(grid, at, s);                                            \
        return cudaLaunchKernelEx(&cfg, k_persistent<R, CLUSTER_PB, 1, CO, true>, D, B, A);                     \
    }                                                                                                          \
    template <> cudaError_t cluster_blocks<R, CO>(int *blocks)                                                 \
    {                                                                                                          \
        return largest_cluster((const void *)k_persistent<R, CLUSTER_PB, 1, CO, true>, blocks);                 \
    }

// one cluster of `blocks` blocks (the attribute must outlive the configuration)
inline cudaLaunchConfig_t cluster_config(int blocks, cudaLaunchAttribute &at, cudaStream_t s)
{
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(CLUSTER_PB);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cfg;
}
inline cudaError_t largest_cluster(const void *kernel, int *blocks)
{
    *blocks = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return cudaSuccess;
    }
    for (int c = CLUSTER_MAX; c >= 8 && *blocks == 0; c /= 2) {
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = cluster_config(c, at, nullptr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) cudaGetLastError();
        else if (n > 0) *blocks = c;
    }
    return cudaSuccess;
}

// run-time dispatch over the shapes
template <typename R, bool CO>
inline cudaError_t persist_launch_shape(int shape, const Dev<R> &D, const BPDev &B, const PersistArgs &A, int grid,
                                        cudaStream_t s)
{
    if constexpr (sizeof(R) == 8 || !CO) {
        switch (shape) {
        case 1: return persist_launch<R, 1, CO>(D, B, A, grid, s);
        case 2: return persist_launch<R, 2, CO>(D, B, A, grid, s);
        case 3: return persist_launch<R, 3, CO>(D, B, A, grid, s);
        case 4: return persist_launch<R, 4, CO>(D, B, A, grid, s);
        }
    }
    return persist_launch<R, 0, CO>(D, B, A, grid, s);
}
template <typename R, bool CO> inline cudaError_t persist_occupancy_shape(int shape, int *per_sm)
{
    if constexpr (sizeof(R) == 8 || !CO) {
        switch (shape) {
        case 1: return persist_occupancy<R, 1, CO>(per_sm);
        case 2: return persist_occupancy<R, 2, CO>(per_sm);
        case 3: return persist_occupancy<R, 3, CO>(per_sm);
        case 4: return persist_occupancy<R, 4, CO>(per_sm);
        }
    }
    return persist_occupancy<R, 0, CO>(per_sm);
}

} // namespace pncg
