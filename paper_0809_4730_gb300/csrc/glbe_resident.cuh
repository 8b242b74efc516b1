// glbe_resident.cuh -- many time steps of a small grid in one launch.
//
// A grid of at most a few nodes per resident thread is not bound by memory: a
// launched step takes 8.5 us on every grid of up to 48^3 nodes (F32, flow),
// most of it the launch itself, kernel prologue, geometry and the latency of
// one gather.  Resident, a step takes (us, launched before -> resident):
//                 F32 flow      F32 coupled   F32C flow     F32C coupled
//   4 x 32 x 4    8.5 -> 2.2    8.5 -> 2.5    8.5 -> 2.4    10.0 -> 4.0
//   64 x 64 x 8   8.7 -> 3.9    8.7 -> 4.4    8.5 -> 4.1    10.5 -> 5.7
//   40^3          8.8 -> 4.6   10.8 -> 6.7   10.6 -> 5.9    14.6 -> 9.0
//   64^3         14.4 -> 9.5   24.4 -> 17.9  20.6 -> 15.4   41.0 -> 30.6
// Past about 70^3 the tables no longer leave the SM its full number of blocks
// (72^3 coupled, F32, with a block less: 34.0 us, launched 32.6), and single
// launches go on.  Here the blocks stay on their SMs
// and march: each keeps a table of its nodes' gather slots in shared memory
// (filled once: no geometry, no wall choice and no divergence in the loop),
// updates its tiles from one population buffer into the other, and meets the
// others at a barrier.  The node update is the step kernels' (node_from_sources),
// so the states are theirs bit for bit.
//
// Two forms of the barrier:
//   - CLUSTER (up to 16 blocks): the grid is one thread-block cluster and the
//     hardware's cluster barrier orders the levels; the blocks are spread so
//     that even the smallest grids use 16 SMs.  Residual sums travel through
//     distributed shared memory.
//   - otherwise a cooperative launch (all blocks resident) and a counting
//     barrier in the workspace.  Every wait is bounded: a block that gives up
//     raises an error flag, every block returns, and the host reports
//     GLBE_ERR_TIMEOUT at its next synchronising call.
//
// Populations written earlier in the launch are gathered with ld.global.ca
// (see ldp): the barrier's release and acquire order them.
#pragma once
#include <cooperative_groups.h>

#include "glbe_residual.cuh"

namespace glbe {

constexpr int RES_THREADS = 256;        // nodes per tile, at most
constexpr int RES_ROWS = 20;            // table rows: 19 slots and a flag word
constexpr int RES_MAX_TILES = 8;        // tiles of a block, at most (its tables: 160 KB)
constexpr size_t RES_TILE_BYTES = (size_t)RES_ROWS * RES_THREADS * sizeof(uint32_t);
constexpr unsigned RES_SKIP = 0xffffffffu;   // flag word of a node that is not updated
constexpr int RES_CLUSTER = 16;         // blocks of the cluster form
constexpr unsigned RES_SPIN_LIMIT = 1u << 24;   // polls of a barrier wait, several seconds

// Bounded counting barrier over the grid; gen is the caller's copy of the
// barrier's generation (thread 0).  False once any block gave up.
__device__ __forceinline__ bool resident_barrier(unsigned* bar, unsigned& gen)
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
                if (++spins > RES_SPIN_LIMIT || ((spins & 4095u) == 0 && *(volatile unsigned*)(bar + 2))) {
                    atomicExch(bar + 2, 1u);
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

__device__ __forceinline__ void cluster_level_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Slots of node i's gather in column tid of the table: row a holds the index
// of direction a's source in a population buffer (its own opposite slot where
// the link is bounced), row 19 the bounced-link bits.
__device__ __forceinline__ void resident_slots(const StepParams& p, uint32_t i, uint32_t* tab, int stride)
{
    if (i >= p.N) {
        tab[19 * stride] = RES_SKIP;
        return;
    }
    const Geo g = make_geo(p, i);
    if (g.solid) {
        tab[19 * stride] = RES_SKIP;
        return;
    }
    unsigned bounced = 0;
    tab[0] = g.n;
#define GLBE_SLOT(a, o, src, sol)                                                                     \
    {                                                                                                 \
        const bool s_ = (sol);                                                                        \
        tab[(a) * stride] = s_ ? (uint32_t)(o) * p.N + g.n : (uint32_t)(a) * p.N + (uint32_t)(src);   \
        bounced |= s_ ? 1u << (a) : 0u;                                                               \
    }
    GLBE_DIRS(GLBE_SLOT)
#undef GLBE_SLOT
    tab[19 * stride] = bounced;
}

// The same for the node pair (n0, n0 + 1), x0 even, of an x-periodic grid with
// an even nx: both nodes bounce alike, so row a holds the index of the
// source of an unshifted pair (e_x = 0), of the pair's own row at x0 (e_x =
// +-1) or of the pair's own opposite slots; the flag word also says whether
// x0 - 1 and x0 + 2 lie across the x seam.
constexpr unsigned RES_SEAM_L = 1u << 20, RES_SEAM_R = 1u << 21;
__device__ __forceinline__ void resident_slots_pair(const StepParams& p, uint32_t i, uint32_t* tab, int stride)
{
    if (i >= p.N >> 1) {
        tab[19 * stride] = RES_SKIP;
        return;
    }
    const GeoP q = make_geo_pair(p, 2u * i);
    const Geo& g = q.g;
    if (g.solid) {
        tab[19 * stride] = RES_SKIP;
        return;
    }
    unsigned bounced = (g.x == 0 ? RES_SEAM_L : 0u) | (g.x + 2 == p.nx ? RES_SEAM_R : 0u);
    tab[0] = g.n;
#define GLBE_SLOT(a, o, row, sol, ex)                                                                       \
    {                                                                                                       \
        const bool s_ = (sol);                                                                              \
        tab[(a) * stride] = s_ ? (uint32_t)(o) * p.N + g.n : (uint32_t)(a) * p.N + (row) + (uint32_t)g.x;   \
        bounced |= s_ ? 1u << (a) : 0u;                                                                     \
    }
    GLBE_PDIRS(GLBE_SLOT)
#undef GLBE_SLOT
    tab[19 * stride] = bounced;
}

// Pair loads of populations written earlier in the launch (see ldp).
template <int ST>
__device__ __forceinline__ F2 ldp2(const typename Store<ST>::T* q)
{
    if constexpr (base_storage(ST) == ST_BF16) {
        const uint32_t u = __ldca(reinterpret_cast<const unsigned*>(q));
        return F2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
    } else if constexpr (base_storage(ST) == ST_F16) {
        const unsigned u = __ldca(reinterpret_cast<const unsigned*>(q));
        __half2 h;
        memcpy(&h, &u, 4);
        return F2(__half22float2(h));
    } else {
        return F2(__ldca(reinterpret_cast<const float2*>(q)));
    }
}

template <int ST>
__device__ __forceinline__ void resident_load_f_pair(const StepParams& p, const typename Store<ST>::T* fs,
                                                     const uint32_t* tab, int stride, unsigned bounced, F2 (&d)[19])
{
    const int dl = bounced & RES_SEAM_L ? p.nx - 1 : -1, dr = bounced & RES_SEAM_R ? 2 - p.nx : 2;
#pragma unroll
    for (int a = 0; a < 19; ++a) {
        const typename Store<ST>::T* s = fs + tab[a * stride];
        const int ex = dir_ex(a);
        if (ex == 0) {
            d[a] = unscale<ST>(p, ldp2<ST>(s));
        } else {
            const bool back = (bounced >> a) & 1u;
            const int i0 = back ? 0 : (ex > 0 ? dl : 1), i1 = back ? 1 : (ex > 0 ? 0 : dr);
            d[a] = unscale<ST>(p, F2(ldp<ST, true>(s + i0), ldp<ST, true>(s + i1)));
        }
    }
}

template <int ST>
__device__ __forceinline__ void resident_load_f(const StepParams& p, const typename Store<ST>::T* fs,
                                                const uint32_t* tab, int stride, float (&d)[19], float (&l)[19])
{
#pragma unroll
    for (int a = 0; a < 19; ++a) {
        const uint32_t s = tab[a * stride];
        d[a] = unscale<ST>(p, ldp<ST, true>(fs + s));
        if constexpr (Store<ST>::COMP) l[a] = ldlo<true>(reinterpret_cast<const __half*>(fs + 19 * (size_t)p.N) + s);
    }
}

template <int ST>
__device__ __forceinline__ void resident_load_g(const StepParams& p, const typename Store<ST>::T* gs,
                                                const uint32_t* tab, int stride, unsigned bounced, float (&q)[21],
                                                float (&ql)[21])
{
    const size_t N = p.N;
#pragma unroll
    for (int a = 0; a < 7; ++a) {
        const uint32_t s = tab[a * stride];
        const bool back = (bounced >> a) & 1u;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float wall = 0.25f * p.bwall_dev[j];   // as load_g
            const float v = unscale<ST>(p, ldp<ST, true>(gs + (size_t)(j * 7) * N + s));
            q[j * 7 + a] = back ? wall - v : v;
            if constexpr (Store<ST>::COMP) {
                const float w = ldlo<true>(reinterpret_cast<const __half*>(gs + 21 * N) + (size_t)(j * 7) * N + s);
                ql[j * 7 + a] = back ? -w : w;
            }
        }
    }
}

// What a thread updates: a pair of nodes, as step_pair_kernel (flow, where
// pair_eligible says so), else one node, as step_kernel; a coupled node in one
// pass or (RES_NODE2) in two (see coupled_induction_pass).  Each is that
// kernel's arithmetic, so a march gives the same bits whichever launches it.
// RES_NODE1 is one node in the pair's arithmetic: on grids of no more than a
// tile per block a step is a chain of latencies, and a thread that gathers two
// nodes has the longer one (F32, 4 x 32 x 4: 2.41 us a step in pairs, 2.17 one
// node a thread; 64 x 64 x 8: 4.30 and 3.87 us); above, pairs issue fewer
// instructions (64^3: 9.45 us, 10.78 one node a thread).
enum ResidentUnit { RES_NODE = 0, RES_NODE2 = 1, RES_PAIR = 2, RES_NODE1 = 3 };

template <int ST, bool MHD, int MODE, int UNIT>
__device__ __forceinline__ void resident_update(const StepParams& p, const StepBuffers& b, uint32_t i,
                                                const uint32_t* tab, int stride, unsigned bounced, float (&acc)[7])
{
    using T = typename Store<ST>::T;
    const T* fs = static_cast<const T*>(b.fsrc);
    if constexpr (UNIT == RES_PAIR) {
        F2 d[19], dl[19], q[21], ql[21];
        resident_load_f_pair<ST>(p, fs, tab, stride, bounced, d);
        pair_from_sources<ST, false, MODE>(p, b, 2u * i, d, dl, q, ql, pair_inputs<false, MODE>(p, b, 2u * i), acc);
    } else {
        const FieldOut fo{nullptr, nullptr, nullptr};
        float d[19], dl[19], q[21], ql[21];
        resident_load_f<ST>(p, fs, tab, stride, d, dl);
        if constexpr (UNIT == RES_NODE1) {
            F1 v[19], vl[19], w[21], wl[21];
#pragma unroll
            for (int a = 0; a < 19; ++a) v[a] = F1(d[a]);
            pair_from_sources<ST, false, MODE, false, F1>(p, b, i, v, vl, w, wl, pair_inputs<false, MODE, F1>(p, b, i),
                                                          acc);
            return;
        }
        if constexpr (MHD) resident_load_g<ST>(p, static_cast<const T*>(b.gsrc), tab, stride, bounced, q, ql);
        if constexpr (UNIT == RES_NODE2) {
            induction_from_sources<ST>(p, b, i, d, dl, q, ql);
            resident_load_f<ST>(p, fs, tab, stride, d, dl);
            node_from_sources<ST, false, MODE, false, 0>(p, b, fo, i, d, dl, q, ql,
                                                         node_inputs<false, MODE, true>(p, b, i), acc);
        } else {
            node_from_sources<ST, MHD, MODE, false, 0>(p, b, fo, i, d, dl, q, ql, node_inputs<MHD, MODE>(p, b, i), acc);
        }
    }
}

// Blocks of RES_THREADS per SM that the dense form is held to: the register
// budgets of the step kernels (see step_dense_blocks, pair_dense_blocks,
// step_kernel_coupled2).
template <int ST, bool MHD, bool PAIR>
constexpr int resident_dense_blocks()
{
    if (PAIR) return ST == ST_F32 ? 2 : 3;
    if (MHD) return ST == ST_F32C || ST == ST_F32 ? 2 : 3;
    return ST == ST_F32 || ST == ST_F32C ? 3 : 5;
}

template <int ST, bool MHD, bool PAIR, bool DENSE, bool CLUSTER>
__global__ void __launch_bounds__(RES_THREADS, DENSE ? resident_dense_blocks<ST, MHD, PAIR>() : 1)
    resident_kernel(const StepParams p, const ResidentMarch m)
{
    static_assert(!PAIR || (!MHD && !Store<ST>::COMP), "pairs: the flow step of the plain storage types");
    // the F32C coupled update needs over 128 registers in one pass
    constexpr int UNIT = PAIR ? (DENSE ? RES_PAIR : RES_NODE1) : DENSE && MHD && ST == ST_F32C ? RES_NODE2 : RES_NODE;
    extern __shared__ uint32_t slots[];          // [tile][RES_ROWS][blockDim.x]
    __shared__ float wsum[RES_THREADS / 32][RES_SUMS];
    __shared__ double bsum[RES_SUMS];
    __shared__ double part[CLUSTER ? RES_SUMS * RES_CLUSTER : 1];
    __shared__ double tot[RES_SUMS];
    __shared__ int verdict;
    const int BT = blockDim.x, G = gridDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (m.solve && *(volatile int*)m.out.stop) return;   // converged in an earlier launch
    const uint32_t units = UNIT == RES_PAIR ? p.N >> 1 : p.N, ntiles = (units + BT - 1) / BT;
    int mine = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += G, ++mine) {
        uint32_t* tab = slots + (size_t)mine * RES_ROWS * BT + threadIdx.x;
        if constexpr (UNIT == RES_PAIR) resident_slots_pair(p, tile * BT + threadIdx.x, tab, BT);
        else resident_slots(p, tile * BT + threadIdx.x, tab, BT);
    }
    unsigned gen = 0;
    if constexpr (CLUSTER) cluster_level_barrier();      // every block's shared memory is there to write to
    else if (threadIdx.x == 0) gen = *(volatile unsigned*)(m.bar + 1);
    const bool writer = blockIdx.x == G - 1;    // the last block has no more tiles than any other
    StepBuffers b{};
    b.FL = m.FL;
    b.Ffield = m.Ffield;
    b.usnap = m.usnap;
    b.snap_lo = m.snap_lo;
    bool snap = m.have_snap != 0;               // the snapshot is of the previous residual level
    for (long long s = 0; s < m.nsteps; ++s) {
        const long long t = m.t0 + s;
        const int par = (int)(t & 1);
        const bool resid = t % 10 == 0;
        b.fsrc = m.f[par];
        b.fdst = m.f[par ^ 1];
        b.gsrc = m.g[par];
        b.gdst = m.g[par ^ 1];
        b.have_snap = snap ? 1 : 0;
        if (resid && threadIdx.x < RES_SUMS) bsum[threadIdx.x] = 0.0;
        for (int k = 0; k < mine; ++k) {
            const uint32_t i = (blockIdx.x + (uint32_t)k * G) * BT + threadIdx.x;
            const uint32_t* tab = slots + (size_t)k * RES_ROWS * BT + threadIdx.x;
            const unsigned bounced = tab[19 * BT];
            float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (!resid) {
                if (bounced != RES_SKIP) resident_update<ST, MHD, MODE_STEP, UNIT>(p, b, i, tab, BT, bounced, acc);
            } else {
                if (bounced != RES_SKIP)
                    resident_update<ST, MHD, MODE_STEP_RESID, UNIT>(p, b, i, tab, BT, bounced, acc);
                // the tile's sums: FP32 within it as block_partials forms them, FP64 over the tiles
#pragma unroll
                for (int r = 0; r < RES_SUMS; ++r) {
                    const float v = warp_sum(acc[r]);
                    if (lane == 0) wsum[warp][r] = v;
                }
                __syncthreads();
                if (threadIdx.x < RES_SUMS) {
                    float v = 0.f;
                    for (int w = 0; w < BT / 32; ++w) v += wsum[w][threadIdx.x];
                    bsum[threadIdx.x] += (double)v;
                }
                __syncthreads();
            }
        }
        if (resid && snap) {
            __syncthreads();
            if constexpr (CLUSTER) {
                // every block's sums into every block's shared memory
                auto cl = cooperative_groups::this_cluster();
                for (int i = threadIdx.x; i < RES_SUMS * G; i += BT) {
                    double* to = cl.map_shared_rank(part, (unsigned)(i / RES_SUMS));
                    to[(i % RES_SUMS) * RES_CLUSTER + blockIdx.x] = bsum[i % RES_SUMS];
                }
            } else if (threadIdx.x < RES_SUMS) {
                m.partials[(size_t)threadIdx.x * G + blockIdx.x] = bsum[threadIdx.x];
            }
        }
        if constexpr (CLUSTER) cluster_level_barrier();
        else if (!resident_barrier(m.bar, gen)) return;
        if (resid) {
            if (snap && (m.solve || writer)) {
                // a solve's blocks all take the decision, from the same sums in the same order
                for (int k = warp; k < RES_SUMS; k += BT / 32) {
                    if (!(writer || k < 2 || k == 6)) continue;
                    const double v = CLUSTER ? partial_row_sum_shared(part + k * RES_CLUSTER, G)
                                             : partial_row_sum(m.partials + (size_t)k * G, 0, (unsigned)G);
                    if (lane == 0) tot[k] = v;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    verdict = 0;
                    if (m.solve) {
                        const double r = residual_of(tot[0], tot[1]);
                        verdict = (m.tol > 0.0 && r <= m.tol) || tot[6] > 0.0 || !isfinite(r);
                    }
                    if (writer && !*m.out.stop) write_record(m.out, tot, *m.out.t_dev);
                }
                __syncthreads();
                if (verdict) return;            // the state is the one after level t, in every block
            } else if (!snap && writer && threadIdx.x == 0) {
                *m.out.t_dev = t + 10;
            }
            snap = true;
        }
    }
}

// Blocks per SM at `per` tiles a block, asked of the runtime once per kernel.
template <int ST, bool MHD, bool PAIR, bool DENSE>
int resident_blocks_per_sm(int per)
{
    static const auto occ = [] {
        struct { int n[RES_MAX_TILES + 1]; } r{};
        auto* kernel = resident_kernel<ST, MHD, PAIR, DENSE, false>;
        for (int k = 1; k <= RES_MAX_TILES; ++k)
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.n[k], kernel, RES_THREADS, k * RES_TILE_BYTES) !=
                cudaSuccess)
                r.n[k] = 0;
        cudaGetLastError();
        return r;
    }();
    return per <= RES_MAX_TILES ? occ.n[per] : 0;
}

template <int ST, bool MHD, bool PAIR>
bool resident_cluster_fits()
{
    static const bool fits = [] {
        auto* kernel = resident_kernel<ST, MHD, PAIR, false, true>;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = RES_CLUSTER;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(RES_CLUSTER);
        cfg.blockDim = dim3(RES_THREADS);
        cfg.dynamicSmemBytes = RES_TILE_BYTES;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        const bool ok = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1;
        cudaGetLastError();
        return ok;
    }();
    return fits;
}

template <int ST, bool MHD, bool PAIR, bool DENSE>
bool resident_grid_plan(uint32_t N, int sms, int max_per, ResidentPlan* out)
{
    // the fewest tiles per block at which all blocks are resident, while the
    // tables leave the SM its full number of blocks
    const int full = resident_blocks_per_sm<ST, MHD, PAIR, DENSE>(1);
    for (int per = 1; per <= max_per && resident_blocks_per_sm<ST, MHD, PAIR, DENSE>(per) == full; ++per) {
        const long long room = (long long)full * sms;
        const uint32_t tiles = ((PAIR && DENSE ? N >> 1 : N) + RES_THREADS - 1) / RES_THREADS;
        if (room * per < tiles) continue;
        *out = {DENSE ? 3 : 2, PAIR ? 1 : 0, (int)(room < tiles ? room : tiles), RES_THREADS,
                (unsigned)(per * RES_TILE_BYTES)};
        return true;
    }
    return false;
}

template <int ST, bool MHD, bool PAIR>
cudaError_t resident_plan_t(uint32_t N, ResidentPlan* out)
{
    int dev = 0, sms = 0, coop = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if ((long long)N > (long long)RES_MAX_TILES * sms * 4 * RES_THREADS) return cudaSuccess;   // more tables than shared memory
    // the limits are function attributes of the device: the same values whoever sets them
    const int most = RES_MAX_TILES * (int)RES_TILE_BYTES;
    e = cudaFuncSetAttribute(resident_kernel<ST, MHD, PAIR, false, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(resident_kernel<ST, MHD, PAIR, false, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(resident_kernel<ST, MHD, PAIR, true, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    if (N <= (uint32_t)RES_CLUSTER * RES_THREADS && resident_cluster_fits<ST, MHD, PAIR>()) {
        const int threads = 32 * (int)((N + RES_CLUSTER * 32 - 1) / (RES_CLUSTER * 32));
        *out = {1, PAIR ? 1 : 0, RES_CLUSTER, threads, (unsigned)(RES_ROWS * threads * sizeof(uint32_t))};
        return cudaSuccess;
    }
    if (!coop) return cudaSuccess;
    if (resident_grid_plan<ST, MHD, PAIR, false>(N, sms, 1, out)) return cudaSuccess;
    resident_grid_plan<ST, MHD, PAIR, true>(N, sms, RES_MAX_TILES, out);
    return cudaSuccess;
}

template <int ST, bool MHD, bool PAIR, bool DENSE, bool CLUSTER>
cudaError_t resident_launch(const StepParams& p, const ResidentMarch& m, const ResidentPlan& pl, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    if (CLUSTER) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = RES_CLUSTER;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.gridDim = dim3(pl.blocks);
    cfg.blockDim = dim3(pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident_kernel<ST, MHD, PAIR, DENSE, CLUSTER>, p, m);
}

template <int ST, bool MHD, bool PAIR>
cudaError_t resident_march_t(const StepParams& p, const ResidentMarch& m, const ResidentPlan& pl, cudaStream_t st)
{
    if (pl.form == 1) return resident_launch<ST, MHD, PAIR, false, true>(p, m, pl, st);
    if (pl.form == 2) return resident_launch<ST, MHD, PAIR, false, false>(p, m, pl, st);
    return resident_launch<ST, MHD, PAIR, true, false>(p, m, pl, st);
}

template <int ST>
cudaError_t resident_plan(bool mhd, const StepParams& p, ResidentPlan* out)
{
    *out = ResidentPlan{0, 0, 0, 0, 0};
    if (mhd) return resident_plan_t<ST, true, false>(p.N, out);
    if constexpr (!Store<ST>::COMP) {
        if (pair_eligible(p, mhd, MODE_STEP)) return resident_plan_t<ST, false, true>(p.N, out);
    }
    return resident_plan_t<ST, false, false>(p.N, out);
}

template <int ST>
cudaError_t resident_march(bool mhd, const StepParams& p, const ResidentMarch& m, const ResidentPlan& pl, cudaStream_t st)
{
    if (mhd) return resident_march_t<ST, true, false>(p, m, pl, st);
    if constexpr (!Store<ST>::COMP) {
        if (pl.pair) return resident_march_t<ST, false, true>(p, m, pl, st);
    }
    return resident_march_t<ST, false, false>(p, m, pl, st);
}

}  // namespace glbe
