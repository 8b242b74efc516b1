// glbe_resident_common.cuh -- many time steps of a small grid in one launch:
// what the 3D and the 2D march share (barriers, launch plans).
//
// The blocks stay on their SMs: each keeps a table of its nodes' gather slots in
// shared memory (filled once: no geometry, no wall choice and no divergence in
// the loop), updates its tiles from one population buffer into the other, and
// meets the others at a barrier.  What a step costs this way and launched, and
// where the line between the two lies, stands with the kernels
// (glbe_resident.cuh, glbe2d.cu).
//
// Two forms of the barrier:
//   - CLUSTER (up to 16 blocks): the grid is one thread-block cluster and the
//     hardware's cluster barrier orders the levels; the blocks are spread so
//     that even the smallest grids use 16 SMs.  Residual sums travel through
//     distributed shared memory.
//   - otherwise a cooperative launch (all blocks resident) and a counting
//     barrier in the workspace.  Every wait is bounded: a block that gives up
//     raises an error flag, every block returns, later marches end at their
//     first barrier (the count is stale) until a new state clears the words,
//     and the host reports GLBE_ERR_TIMEOUT at its next synchronising call.
//
// Populations written earlier in the launch are gathered with ld.global.ca:
// the barrier's release and acquire order them, and no buffer is written in
// the level that reads it.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "glbe_residual.cuh"

namespace glbe {

constexpr int RES_THREADS = 256;        // nodes per tile, at most
constexpr int RES_MAX_TILES = 8;        // tiles of a block, at most
constexpr uint32_t RES_MAX_NODES = 1u << 20;   // more than any SM's shared memory holds tables for
constexpr unsigned RES_SKIP = 0xffffffffu;   // flag word of a node that is not updated
constexpr int RES_CLUSTER = 16;         // blocks of the cluster form

// Bounded counting barrier over the grid; gen is the caller's copy of the
// barrier's generation (thread 0).  False once any block gave up.  A block that
// gives up also makes the count one that no arrivals complete: a later launch
// over the words as they are ends in its first barrier, at its first look at the
// flag.  (A look at the flag on entry or ahead of the count instead cost 64 x 64
// x 8 F32C coupled 0.06 to 0.36 us a level.)
constexpr unsigned RES_NEVER = 1u << 31;
__device__ __forceinline__ bool resident_barrier(unsigned* bar, unsigned& gen, unsigned spin_limit)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned arrived;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(arrived) : "l"(bar) : "memory");
        int good = 1;
        if (arrived == gridDim.x - 1) {
            asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(bar) : "memory");
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(bar + 1), "r"(gen + 1u) : "memory");
        } else {
            unsigned v, spins = 0;
            while (true) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar + 1) : "memory");
                if (v != gen) break;
                if ((++spins & 4095u) == 0 && (spins >= spin_limit || *(volatile unsigned*)(bar + 2))) {
                    atomicExch(bar + 2, 1u);
                    atomicExch(bar, RES_NEVER);
                    good = 0;
                    break;
                }
            }
        }
        ++gen;
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// Whether a solve stops at these sums.
__device__ __forceinline__ bool resident_stops(double tol, const double* tot)
{
    const double r = residual_of(tot[0], tot[1]);
    return (tol > 0.0 && r <= tol) || tot[6] > 0.0 || !isfinite(r);
}

__device__ __forceinline__ void cluster_level_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Blocks per SM of a cooperative form at `per` tiles a block (each of
// tile_bytes of tables), asked of the runtime once per kernel.
struct ResidentOcc {
    int n[RES_MAX_TILES + 1];
};
template <class K>
ResidentOcc resident_occupancy(K kernel, size_t tile_bytes)
{
    ResidentOcc r{};
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(RES_MAX_TILES * tile_bytes));
    for (int k = 1; k <= RES_MAX_TILES; ++k)
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.n[k], kernel, RES_THREADS, k * tile_bytes) != cudaSuccess)
            r.n[k] = 0;
    cudaGetLastError();
    return r;
}

inline cudaLaunchAttribute resident_attribute(bool cluster)
{
    cudaLaunchAttribute at{};
    if (cluster) {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = RES_CLUSTER;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
    } else {
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
    }
    return at;
}

// Whether the device places a cluster of RES_CLUSTER blocks of this kernel.
template <class K>
bool resident_cluster_fits(K kernel, size_t tile_bytes)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at = resident_attribute(true);
    cfg.gridDim = dim3(RES_CLUSTER);
    cfg.blockDim = dim3(RES_THREADS);
    cfg.dynamicSmemBytes = tile_bytes;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    const bool ok = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1;
    cudaGetLastError();
    return ok;
}

// One cluster: N nodes spread over its blocks in whole warps.
inline ResidentPlan resident_cluster_plan(uint32_t N, int rows)
{
    const int threads = 32 * (int)((N + RES_CLUSTER * 32 - 1) / (RES_CLUSTER * 32));
    return {1, 0, RES_CLUSTER, threads, (unsigned)(rows * threads * sizeof(uint32_t)), RES_LEAST_CLUSTER, 1};
}

// A cooperative form for `units` updates: the fewest tiles per block (at most
// max_per) at which all blocks are resident, while the tables leave the SM its
// full number of blocks and no more than `table_bytes` are theirs (the rest of
// the SM's 256 KB is the gathers' L1).
inline bool resident_grid_plan(const ResidentOcc& occ, uint32_t units, int sms, int max_per, size_t tile_bytes,
                               size_t table_bytes, int form, ResidentPlan* out)
{
    const uint32_t tiles = (units + RES_THREADS - 1) / RES_THREADS;
    if (occ.n[1] < 1) return false;
    for (int per = 1; per <= max_per && occ.n[per] == occ.n[1] && occ.n[1] * per * tile_bytes <= table_bytes; ++per) {
        const long long room = (long long)occ.n[1] * sms;
        if (room * per < tiles) continue;
        *out = {form, 0, (int)(room < tiles ? room : tiles), RES_THREADS, (unsigned)(per * tile_bytes), RES_LEAST_COOP, 1};
        return true;
    }
    return false;
}

// Plan of a march by three kernels: one cluster (up to 4096 nodes), one tile a
// block (registers unbounded), several tiles a block (held to the register
// budget of the launched steps).  units_dense: updates of the dense form.
// The attributes set are the device's: the same values whoever sets them.
// A form with a null kernel and no occupancy is left out.
template <class C, class K>
cudaError_t resident_plan_of(C cluster, K free_form, K dense, uint32_t N, uint32_t units_dense, int rows,
                             size_t table_bytes, const ResidentOcc& occ_free, const ResidentOcc& occ_dense, bool cluster_fits,
                             ResidentPlan* out)
{
    const size_t tile_bytes = (size_t)rows * RES_THREADS * sizeof(uint32_t);
    int dev = 0, sms = 0, coop = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (N <= (uint32_t)RES_CLUSTER * RES_THREADS && cluster_fits) {
        *out = resident_cluster_plan(N, rows);
        return cudaFuncSetAttribute(cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    if (!coop) return cudaSuccess;
    if (!resident_grid_plan(occ_free, N, sms, 1, tile_bytes, table_bytes, 2, out) &&
        !resident_grid_plan(occ_dense, units_dense, sms, RES_MAX_TILES, tile_bytes, table_bytes, 3, out))
        return cudaSuccess;
    return cudaFuncSetAttribute(out->form == 2 ? free_form : dense, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(RES_MAX_TILES * tile_bytes));
}

template <class K, class... A>
cudaError_t resident_launch(K kernel, const ResidentPlan& pl, cudaStream_t st, const A&... args)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at = resident_attribute(pl.form == 1);
    cfg.gridDim = dim3(pl.blocks);
    cfg.blockDim = dim3(pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) cudaGetLastError();   // returned, so not left for the next check to find
    return e;
}

}  // namespace glbe
