// glbe_resident.cuh -- many time steps of a small 3D grid in one launch
// (glbe_resident_common.cuh): the gather tables, node updates and launch forms.
//
// A grid of at most a few nodes per resident thread is not bound by memory: a
// launched step takes 4 to 6 us on every grid of up to 40^3 nodes (F32, flow),
// most of it the launch itself, kernel prologue, geometry and the latency of
// one gather.  A step of long marches takes (us, launched with overlap ->
// resident):
//            F32 flow       F32 coupled    F32C flow      F32C coupled   BF16 flow
//   16^3     4.1 -> 2.1     4.5 -> 2.9     4.6 -> 1.95    5.7 -> 3.9     4.2 -> 1.8
//   32^3     5.0 -> 3.6     6.0 -> 4.1     6.3 -> 3.8     6.2 -> 5.2     4.5 -> 3.4
//   40^3     5.7 -> 4.4     7.2 -> 6.2     7.3 -> 5.5    10.1 -> 8.8     5.9 -> 3.7
//   64^3     9.2 -> 8.8    17.8 -> 16.4   13.9 -> 12.65  31.9 -> 27.8    6.95 -> 6.9
//   80^3    15.9 -> 13.6        -              -              -         11.45 -> 9.8
//   84^3    18.8 -> 16.3        -              -              -         12.3 -> 10.7
// The line lies where the tables crowd out the gathers' L1 (RES_TABLES_FLOW,
// RES_TABLES_MHD) or the SM is full: pairs (flow, even nx, x periodic) march to
// 622,592 nodes in F32 and 700,416 in the 16-bit forms, one node a thread to
// 350,208 (F32, F32C; 16 bits 194,560), coupled ones to 311,296 (16 bits
// 233,472) on 152 SMs.  72^3 coupled marched 32.7 us a step with 205 KB of
// tables on an SM, 27.1 launched (F32C 56.3 and 44.8).  The node update is the step kernels'
// (node_from_sources, pair_from_sources), so the states are theirs bit for bit.
#pragma once
#include <type_traits>

#include "glbe_resident_common.cuh"

namespace glbe {

constexpr int RES_ROWS = 20;            // table rows: 19 slots and a flag word
// Table bytes of an SM, at most: 9 tiles (70^3 F32C flow: 16.3 us a step with
// them, 17.2 launched), 8 where a coupled node gathers f twice (64^3 F32C: 27.8
// and 31.9 us; with 10 tiles the launched step is faster).
constexpr size_t RES_TABLES_FLOW = (size_t)9 * RES_ROWS * 256 * 4, RES_TABLES_MHD = (size_t)8 * RES_ROWS * 256 * 4;

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
// pass or (RES_NODE2) in two (see coupled_node2).  Each is that
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
        if constexpr (UNIT == RES_NODE2) {
            float rho_inv, mx, my, mz;
            const NodeIn<float> in = node_inputs<true, MODE_STEP>(p, b, i);
            resident_load_g<ST>(p, static_cast<const T*>(b.gsrc), tab, stride, bounced, q, ql);
            node_momentum<ST, false>(p, d, dl, rho_inv, mx, my, mz);
            induction_from_sources<ST, false>(p, b, i, in, rho_inv, mx, my, mz, q, ql);
            resident_load_f<ST>(p, fs, tab, stride, d, dl);
            node_from_sources<ST, false, MODE, false, 0, false>(p, b, fo, i, d, dl, q, ql,
                                                         node_inputs<false, MODE, true>(p, b, i), acc);
            return;
        }
        if constexpr (UNIT == RES_NODE1) {
            F1 v[19], vl[19], w[21], wl[21];
#pragma unroll
            for (int a = 0; a < 19; ++a) v[a] = F1(d[a]);
            pair_from_sources<ST, false, MODE, false, F1>(p, b, i, v, vl, w, wl, pair_inputs<false, MODE, F1>(p, b, i),
                                                          acc);
            return;
        }
        if constexpr (MHD) resident_load_g<ST>(p, static_cast<const T*>(b.gsrc), tab, stride, bounced, q, ql);
        node_from_sources<ST, MHD, MODE, false, 0, false>(p, b, fo, i, d, dl, q, ql, node_inputs<MHD, MODE>(p, b, i), acc);
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
    static_assert(RES_THREADS == 2 * PAIR_THREADS, "a tile of pairs is two launched blocks");
    extern __shared__ uint32_t slots[];          // [tile][RES_ROWS][blockDim.x]
    __shared__ float wsum[RES_THREADS / 32][RES_SUMS];
    __shared__ double bsum[RES_SUMS];
    __shared__ double part[CLUSTER ? RES_SUMS * RES_CLUSTER : 1];
    __shared__ double tot[RES_SUMS];
    __shared__ int verdict;
    const int BT = blockDim.x, G = gridDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (m.solve && *(volatile int*)m.out.stop) return;   // converged in an earlier launch
    if (!CLUSTER && (int)blockIdx.x == m.absent) return;
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
    b.FLsrc = m.FL;
    b.FL = m.FL;
    b.Ffield = m.Ffield;
    b.usnap = m.usnap;
    b.snap_lo = m.snap_lo;
    bool snap = m.have_snap != 0;               // the snapshot is of the previous residual level
    int par = m.phase & 1;                      // t0 and t0 mod 10 have the same parity
    for (int s = 0, phase = m.phase; s < m.nsteps; ++s, par ^= 1, phase = phase == 9 ? 0 : phase + 1) {
        const bool resid = phase == 0;
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
                // the tile's sums: FP32 over the nodes of a launched block (see block_partials), FP64 from there on
#pragma unroll
                for (int r = 0; r < RES_SUMS; ++r) {
                    const float v = warp_sum(acc[r]);
                    if (lane == 0) wsum[warp][r] = v;
                }
                __syncthreads();
                if (threadIdx.x < RES_SUMS) {
                    float v = 0.f;
                    if constexpr (UNIT == RES_PAIR) {
                        // a tile is two launched blocks of pairs
                        constexpr int GROUP = PAIR_THREADS / 32;
                        float u = 0.f;
#pragma unroll
                        for (int w = 0; w < GROUP; ++w) {
                            v += wsum[w][threadIdx.x];
                            u += wsum[GROUP + w][threadIdx.x];
                        }
                        bsum[threadIdx.x] += (double)u;
                    } else {
                        for (int w = 0; w < BT / 32; ++w) v += wsum[w][threadIdx.x];
                    }
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
        else if (!resident_barrier(m.bar, gen, m.spin_limit)) return;
        if (resid) {
            if (snap && (m.solve || writer)) {
                // a solve's blocks all take the decision, from the same sums in the same order
                for (int k = warp; k < RES_SUMS; k += BT / 32) {
                    if (!(writer || k < 2 || k == 6)) continue;
                    const double v = CLUSTER ? warp_sum_all(lane < G ? part[k * RES_CLUSTER + lane] : 0.0)
                                             : partial_row_sum(m.partials + (size_t)k * G, 0, (unsigned)G);
                    if (lane == 0) tot[k] = v;
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    verdict = 0;
                    if (m.solve) verdict = resident_stops(m.tol, tot);
                    if (writer && !*m.out.stop) write_record(m.out, tot, *m.out.t_dev);
                }
                __syncthreads();
                if (verdict) return;            // the state is the one after level t, in every block
            } else if (!snap && writer && threadIdx.x == 0) {
                *m.out.t_dev = m.t0 + s + 10;
            }
            snap = true;
        }
    }
}

// The cluster form of the flow lattice (up to 16 x 256 nodes): it lives in the
// shared memory of 16 blocks, both population buffers, forces and snapshot, and
// a gather is a load from distributed shared memory: the tables hold the
// sources' addresses in the cluster's window.  A level then costs two
// shared-memory latencies and a cluster barrier instead of two trips to L2
// (4 x 32 x 4: F32 2.16 us a step through L2, 1.89 here; F32C 2.4 and 1.6).  The state is read
// from the workspace at the start and left there at the end.
template <class T>
__device__ __forceinline__ float ld_cluster(uint32_t addr)
{
    if constexpr (sizeof(T) == 4) {
        float v;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
        return v;
    } else {
        unsigned short u;
        asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(u) : "r"(addr));
        if constexpr (std::is_same<T, __half>::value) return __half2float(__ushort_as_half(u));
        else return __uint_as_float((unsigned)u << 16);
    }
}
__device__ __forceinline__ uint32_t cluster_address(uint32_t local, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}

// Inputs of the node in column tid (see node_inputs): b's force field, lagged
// force and snapshot are columns of shared memory here.  Volatile loads, like
// the gathers': with plain ones the compiler forms what the two kinds of levels
// have in common ahead of the branch between them (the product of the half
// force, say) and then cannot contract it with what follows, as the launched
// steps do: a unit in the last place, rarely, but not the same bits.
template <class V, int MODE>
__device__ __forceinline__ NodeIn<V> cluster_inputs(const StepParams& p, const StepBuffers& b, int tid)
{
    const int N = (int)p.N;
    const volatile float *F = b.Ffield, *us = b.usnap;
    NodeIn<V> in;
    in.FLx = in.FLy = in.FLz = V(0.f);
    in.Fx = V(p.F[0]);
    in.Fy = V(p.F[1]);
    in.Fz = V(p.F[2]);
    if (p.force_ncomp >= 1) in.Fx += V(F[tid]);
    if (p.force_ncomp == 3) {
        in.Fy += V(F[N + tid]);
        in.Fz += V(F[2 * N + tid]);
    }
    in.us0 = in.us1 = in.us2 = V(0.f);
    in.ul0 = in.ul1 = in.ul2 = V(0.f);
    if (MODE == MODE_STEP_RESID && b.have_snap) {
        in.us0 = V(us[tid]);
        in.us1 = V(us[N + tid]);
        in.us2 = V(us[2 * N + tid]);
        if (b.snap_lo) {
            in.ul0 = V(us[3 * N + tid]);
            in.ul1 = V(us[4 * N + tid]);
            in.ul2 = V(us[5 * N + tid]);
        }
    }
    return in;
}

// Bytes of a block's shared memory and where its parts lie.
struct ClusterLayout {
    unsigned f, flo, fstep, F, snap, tab, tablo, total;
};
__host__ __device__ inline ClusterLayout cluster_layout(int T, bool comp, int BT)
{
    ClusterLayout L{};
    unsigned off = 0;
    const unsigned lo = comp ? 2u : 0u, b = (unsigned)BT;
    L.f = off;
    L.flo = off + 19u * b * T;
    L.fstep = 19u * b * (T + lo);
    off += 2 * L.fstep;
    L.F = off;
    off += 3u * b * 4u;
    L.snap = off;
    off += 6u * b * 4u;
    L.tab = off;
    off += RES_ROWS * b * 4u;
    L.tablo = off;
    if (comp) off += 19u * b * 4u;
    L.total = off;
    return L;
}

template <int ST, bool PAIR>
__global__ void __launch_bounds__(RES_THREADS, 1) resident_cluster_kernel(const StepParams p, const ResidentMarch m)
{
    using S = Store<ST>;
    using T = typename S::T;
    constexpr bool COMP = S::COMP;
    extern __shared__ __align__(16) char sm[];
    __shared__ float wsum[RES_THREADS / 32][RES_SUMS];
    __shared__ double bsum[RES_SUMS];
    __shared__ double part[RES_SUMS * RES_CLUSTER];
    __shared__ double tot[RES_SUMS];
    __shared__ int verdict;
    const int BT = blockDim.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (m.solve && *(volatile int*)m.out.stop) return;   // converged in an earlier launch
    const ClusterLayout L = cluster_layout(sizeof(T), COMP, BT);
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
    const uint32_t n = blockIdx.x * BT + tid;
    const bool inb = n < p.N;
    const size_t N = p.N;
    uint32_t* tab = reinterpret_cast<uint32_t*>(sm + L.tab) + tid;
    uint32_t* tablo = reinterpret_cast<uint32_t*>(sm + L.tablo) + tid;
    resident_slots(p, n, tab, BT);
    const unsigned flags = tab[19 * BT];
    if (flags != RES_SKIP) {
        for (int a = 0; a < 19; ++a) {
            const uint32_t s = tab[a * BT], row = s / p.N, src = s - row * p.N, rank = src / BT;
            const uint32_t k = row * BT + (src - rank * BT);
            tab[a * BT] = cluster_address(base + L.f + k * (uint32_t)sizeof(T), rank);
            if constexpr (COMP) tablo[a * BT] = cluster_address(base + L.flo + k * 2u, rank);
        }
    }
    // the state of level t0; of a node that is not updated both buffers, since a
    // ghost plane's is gathered from (a solid node's never)
    const int par0 = m.phase & 1;
    float* const F = reinterpret_cast<float*>(sm + L.F);
    float* const snapc = reinterpret_cast<float*>(sm + L.snap);
    auto rows = [&](int h, bool load) {
        T* g = static_cast<T*>(m.f[h]);
        T* c = reinterpret_cast<T*>(sm + L.f + h * L.fstep);
        for (int a = 0; a < 19; ++a) {
            if (load) c[a * BT + tid] = g[a * N + n];
            else g[a * N + n] = c[a * BT + tid];
        }
        if constexpr (COMP) {
            __half* gl = reinterpret_cast<__half*>(g + 19 * N);
            __half* cl = reinterpret_cast<__half*>(sm + L.flo + h * L.fstep);
            for (int a = 0; a < 19; ++a) {
                if (load) cl[a * BT + tid] = gl[a * N + n];
                else gl[a * N + n] = cl[a * BT + tid];
            }
        }
    };
    if (inb) {
        for (int k = 0; k < (flags == RES_SKIP ? 2 : 1); ++k) rows(par0 ^ k, true);
        for (int k = 0; k < p.force_ncomp; ++k) F[k * BT + tid] = m.Ffield[k * N + n];
        for (int k = 0; k < (m.snap_lo ? 6 : 3); ++k) snapc[k * BT + tid] = m.usnap[k * N + n];
    }
    cluster_level_barrier();
    StepParams q = p;
    q.N = (uint32_t)BT;                         // the columns' stride in shared memory
    StepBuffers b{};
    b.Ffield = F;
    b.usnap = snapc;
    b.snap_lo = m.snap_lo;
    const FieldOut fo{nullptr, nullptr, nullptr};
    const bool writer = blockIdx.x == G - 1;
    bool snap = m.have_snap != 0;               // the snapshot is of the previous residual level
    int par = par0;
    for (int s = 0, phase = m.phase; s < m.nsteps; ++s, phase = phase == 9 ? 0 : phase + 1) {
        const bool resid = phase == 0;
        b.fdst = sm + L.f + (par ^ 1) * L.fstep;
        b.have_snap = snap ? 1 : 0;
        float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (flags != RES_SKIP) {
            auto update = [&](auto mode) {
                constexpr int MODE = decltype(mode)::value;
                float d[19], dl[19], v[21], vl[21];
                const uint32_t df = par * L.fstep;
#pragma unroll
                for (int a = 0; a < 19; ++a) {
                    d[a] = unscale<ST>(p, ld_cluster<T>(tab[a * BT] + df));
                    if constexpr (COMP) dl[a] = ld_cluster<__half>(tablo[a * BT] + df) * LO_INV;
                }
                if constexpr (PAIR) {
                    F1 w[19], wl[19], z[21], zl[21];
#pragma unroll
                    for (int a = 0; a < 19; ++a) w[a] = F1(d[a]);
                    pair_from_sources<ST, false, MODE, false, F1>(q, b, tid, w, wl, z, zl,
                                                                  cluster_inputs<F1, MODE>(q, b, tid), acc);
                } else {
                    node_from_sources<ST, false, MODE, false, 0, false>(q, b, fo, tid, d, dl, v, vl,
                                                                      cluster_inputs<float, MODE>(q, b, tid), acc);
                }
            };
            if (resid) update(std::integral_constant<int, MODE_STEP_RESID>{});
            else update(std::integral_constant<int, MODE_STEP>{});
        }
        if (resid && snap) {
#pragma unroll
            for (int r = 0; r < RES_SUMS; ++r) {
                const float x = warp_sum(acc[r]);
                if (lane == 0) wsum[warp][r] = x;
            }
            __syncthreads();
            if (tid < RES_SUMS) {
                float x = 0.f;
                for (int w = 0; w < BT / 32; ++w) x += wsum[w][tid];
                bsum[tid] = (double)x;
            }
            __syncthreads();
            // every block's sums into every block's shared memory
            auto cl = cooperative_groups::this_cluster();
            for (int i = tid; i < RES_SUMS * G; i += BT)
                cl.map_shared_rank(part, (unsigned)(i / RES_SUMS))[(i % RES_SUMS) * RES_CLUSTER + blockIdx.x] =
                    bsum[i % RES_SUMS];
        }
        cluster_level_barrier();
        par ^= 1;
        if (!resid) continue;
        if (snap && (m.solve || writer)) {
            // a solve's blocks all take the decision, from the same sums in the same order
            for (int k = warp; k < RES_SUMS; k += BT / 32) {
                const double x = warp_sum_all(lane < G ? part[k * RES_CLUSTER + lane] : 0.0);
                if (lane == 0) tot[k] = x;
            }
            __syncthreads();
            if (tid == 0) {
                verdict = m.solve && resident_stops(m.tol, tot);
                if (writer && !*m.out.stop) write_record(m.out, tot, *m.out.t_dev);
            }
            __syncthreads();
            if (verdict) break;                 // the state is the one after this level, in every block
        } else if (!snap && writer && tid == 0) {
            *m.out.t_dev = m.t0 + s + 10;
        }
        snap = true;
    }
    if (inb && flags != RES_SKIP) {
        rows(par, false);
        for (int k = 0; k < (m.snap_lo ? 6 : 3); ++k) m.usnap[k * N + n] = snapc[k * BT + tid];
    }
}

// The kernel of the cluster form.  A coupled lattice goes through L2: from
// shared memory its update came out a unit in the last place off now and then
// (the compiler contracted it differently there).
template <int ST, bool MHD, bool PAIR>
constexpr auto resident_cluster_form()
{
    if constexpr (MHD) return resident_kernel<ST, true, false, false, true>;
    else return resident_cluster_kernel<ST, PAIR>;
}
template <int ST, bool MHD>
unsigned resident_cluster_bytes(int threads)
{
    return MHD ? (unsigned)(RES_ROWS * threads * sizeof(uint32_t))
               : cluster_layout(sizeof(typename Store<ST>::T), Store<ST>::COMP, threads).total;
}

template <int ST, bool MHD, bool PAIR>
cudaError_t resident_plan_t(uint32_t N, ResidentPlan* out)
{
    constexpr size_t tile = (size_t)RES_ROWS * RES_THREADS * sizeof(uint32_t);
    constexpr auto cluster = resident_cluster_form<ST, MHD, PAIR>();
    auto* free_form = resident_kernel<ST, MHD, PAIR, false, false>;
    auto* dense = resident_kernel<ST, MHD, PAIR, true, false>;
    const unsigned most = resident_cluster_bytes<ST, MHD>(RES_THREADS);
    static const ResidentOcc of = resident_occupancy(free_form, tile), od = resident_occupancy(dense, tile);
    static const bool fits = [&] {
        cudaFuncSetAttribute(cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaFuncSetAttribute(cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        return resident_cluster_fits(cluster, most);
    }();
    cudaError_t e = resident_plan_of(cluster, free_form, dense, N, PAIR ? N >> 1 : N, RES_ROWS,
                                     MHD ? RES_TABLES_MHD : RES_TABLES_FLOW, of, od, fits, out);
    out->pair = PAIR ? 1 : 0;
    if (e == cudaSuccess && out->form == 1) {
        out->smem = resident_cluster_bytes<ST, MHD>(out->threads);
        e = cudaFuncSetAttribute(cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    }
    return e;
}

template <int ST, bool MHD, bool PAIR>
cudaError_t resident_march_t(const StepParams& p, const ResidentMarch& m, const ResidentPlan& pl, cudaStream_t st)
{
    if (pl.form == 1) return resident_launch(resident_cluster_form<ST, MHD, PAIR>(), pl, st, p, m);
    if (pl.form == 2) return resident_launch(resident_kernel<ST, MHD, PAIR, false, false>, pl, st, p, m);
    return resident_launch(resident_kernel<ST, MHD, PAIR, true, false>, pl, st, p, m);
}

template <int ST>
cudaError_t resident_plan(bool mhd, const StepParams& p, ResidentPlan* out)
{
    *out = ResidentPlan{0, 0, 0, 0, 0};
    if (p.N > RES_MAX_NODES) return cudaSuccess;
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
