// glbe_cavity.cuh -- the step of grids with a fluid box and / or a moving
// lid: the 3D lid-driven cavity of Sec. 5 and its MHD case on an extended
// magnetic domain.  One node per thread.
//
// Wall planes of the grid (wall_lo / wall_hi) bound both lattices: the flow
// lattice bounces back there and the vector lattice anti-bounces to B0 (a
// zero induced field).  The flow lattice is fluid only inside the box
// [blo, bhi]; a link whose source lies outside it is bounced back half-way,
// and when the source lies above the highest fluid z plane (the lid) it
// returns with the lid's momentum 6 w_a rho0 (e_a . U) added (Ladd's
// moving-wall rule; the preconditioned equilibrium keeps the unscaled linear
// term 3 e.j, so the term is the plain scheme's).  Outside the box, up to the
// wall planes, the vector lattice continues at rest: its collision relaxes
// g to W_a B (u = 0, Eq. mcollision), no Lorentz force is formed there, and
// the magnetic field diffuses out to the zero induced field at the walls.
#pragma once

namespace glbe {

__device__ __forceinline__ bool in_box(const StepParams& p, int x, int y, int z)
{
    return x >= p.blo[0] && x <= p.bhi[0] && y >= p.blo[1] && y <= p.bhi[1] && z >= p.blo[2] && z <= p.bhi[2];
}

// What the gathers of one node need, per axis d and shift s = -1, 0, +1 of the
// coordinate (index s + 1): the linear offset of the wrapped coordinate, and
// whether it is solid for the flow lattice (a wall plane or outside the box:
// fout) or for the vector lattice (a wall plane: wout).  A direction then
// combines three entries, the same way for every node, so the gathers, the
// induction part and the flow part are each in the kernel once.  (A form with
// separate gathers for nodes inside the box and one induction part for each
// side of its boundary was bound by instruction fetch: 2.6 stalled cycles per
// issued instruction; the F32C step of the 98^3 MHD cavity took 152 us.  Now 98
// us: bound by the latency of its gathers, hence 24 warps an SM in spite of
// 216 B spilled (two blocks, no spill: 109 us) and the L2 prefetch.)
struct CavGeo {
    uint32_t n;
    uint32_t off[3][3];
    bool fout[3][3], wout[3][3];
    bool solid;      // a wall plane: neither lattice is updated
    bool flow;       // a node of the flow lattice
    bool under_lid;  // ... on its highest plane
};

__device__ __forceinline__ CavGeo cavity_geo(const StepParams& p, uint32_t n)
{
    CavGeo g;
    g.n = n;
    const uint32_t zy = fdiv(n, p.div_nx), zi = fdiv(n, p.div_nxy);
    const int c[3] = {(int)(n - zy * (uint32_t)p.nx), (int)(zy - zi * (uint32_t)p.ny), (int)zi};
    const int dim[3] = {p.nx, p.ny, p.nz};
    const uint32_t stride[3] = {1u, (uint32_t)p.nx, (uint32_t)p.nx * (uint32_t)p.ny};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            int v = c[d] + s - 1;
            v = v < 0 ? v + dim[d] : (v >= dim[d] ? v - dim[d] : v);
            g.off[d][s] = (uint32_t)v * stride[d];
            g.wout[d][s] = plane_solid(v, dim[d], p.wlo[d], p.whi[d]);
            g.fout[d][s] = g.wout[d][s] || v < p.blo[d] || v > p.bhi[d];
        }
    }
    g.solid = g.wout[0][1] || g.wout[1][1] || g.wout[2][1];
    g.flow = !(g.fout[0][1] || g.fout[1][1] || g.fout[2][1]);
    g.under_lid = g.flow && c[2] == p.top_z;
    return g;
}

// Gather of f for a node of the flow lattice: source x - e_a (periodic wrap
// on axes without walls); a source on a wall plane or outside the box is
// bounced back (own slot of the opposite direction), plus the lid term when
// it lies above top_z.
template <int ST>
__device__ __forceinline__ void load_f_box(const StepParams& p, const typename Store<ST>::T* __restrict__ fs,
                                           const CavGeo& g, float (&d)[19], float (&l)[19])
{
    const size_t N = p.N;
    const __half* __restrict__ fl = Store<ST>::COMP ? reinterpret_cast<const __half*>(fs + 19 * N) : nullptr;
#pragma unroll
    for (int a = 0; a < 19; ++a) {
        const int sx = 1 - dir_ex(a), sy = 1 - dir_ey(a), sz = 1 - dir_ez(a);
        const bool out = g.fout[0][sx] || g.fout[1][sy] || g.fout[2][sz];
        const size_t slot = out ? (size_t)dir_opp(a) * N + g.n
                                : (size_t)a * N + (g.off[0][sx] + g.off[1][sy] + g.off[2][sz]);
        d[a] = unscale<ST>(p, Store<ST>::ld(fs + slot));
        if constexpr (Store<ST>::COMP) l[a] = Store<ST_F32C>::ld_lo(fl + slot);
    }
    if (g.under_lid) {
        // only the directions that come down have their source above top_z
#pragma unroll
        for (int a = 0; a < 19; ++a) {
            if (dir_ez(a) != -1) continue;
            if (!(g.fout[0][1 - dir_ex(a)] || g.fout[1][1 - dir_ey(a)] || g.fout[2][2])) continue;
            const float c = p.lid_corr[a];
            if constexpr (Store<ST>::COMP) {
                // exact: the rounding of high part + lid term goes to the low part, so the
                // compensated form keeps its resolution at the lid (a rounded add there
                // floored the cavity's residual near 1.7e-7)
                const float s = vadd_rn(d[a], c);
                const float bp = vsub_rn(s, d[a]);
                const float e = vadd_rn(vsub_rn(d[a], vsub_rn(s, bp)), vsub_rn(c, bp));
                d[a] = s;
                l[a] = vadd_rn(l[a], e);
            } else {
                d[a] += c;
            }
        }
    }
}

// Gather of g (see load_g): anti-bounce-back at the wall planes only.
template <int ST>
__device__ __forceinline__ void load_g_box(const StepParams& p, const typename Store<ST>::T* __restrict__ gs,
                                           const CavGeo& g, float (&q)[21], float (&ql)[21])
{
    const size_t N = p.N;
    const __half* __restrict__ gl = Store<ST>::COMP ? reinterpret_cast<const __half*>(gs + 21 * N) : nullptr;
#pragma unroll
    for (int a = 0; a < 7; ++a) {
        const int sx = 1 - dir_ex(a), sy = 1 - dir_ey(a), sz = 1 - dir_ez(a);
        const bool out = g.wout[0][sx] || g.wout[1][sy] || g.wout[2][sz];
        const size_t slot = out ? (size_t)dir_opp(a) * N + g.n
                                : (size_t)a * N + (g.off[0][sx] + g.off[1][sy] + g.off[2][sz]);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float wall = 0.25f * p.bwall_dev[j];   // 2 W_a (B_wall - B0), W_a = 1/8
            const float v = unscale<ST>(p, Store<ST>::ld(gs + (size_t)(j * 7) * N + slot));
            q[j * 7 + a] = out ? wall - v : v;
            if constexpr (Store<ST>::COMP) {
                const float w = Store<ST_F32C>::ld_lo(gl + (size_t)(j * 7) * N + slot);
                ql[j * 7 + a] = out ? -w : w;
            }
        }
    }
}

// The outputs of a node that no lattice (or only the vector lattice) covers.
template <bool MHD>
__device__ __forceinline__ void cavity_zero_fields(const StepParams& p, const FieldOut& fo, uint32_t n, bool with_B)
{
    const size_t N = p.N;
    if (fo.rho) fo.rho[n] = 0.f;
    if (fo.u) { fo.u[n] = 0.f; fo.u[N + n] = 0.f; fo.u[2 * N + n] = 0.f; }
    if (MHD && with_B && fo.B) { fo.B[n] = 0.f; fo.B[N + n] = 0.f; fo.B[2 * N + n] = 0.f; }
}

// Vector lattice alone at a node outside the box (u = 0, no Lorentz force).
template <int ST, int MODE>
__device__ __forceinline__ void induction_at_rest(const StepParams& p, const StepBuffers& b, const FieldOut& fo,
                                                  uint32_t n, const float (&q)[21], const float (&ql)[21])
{
    constexpr bool PRECISE = (ST == ST_F32 || ST == ST_F32C);
    const size_t N = p.N;
    float og[21];
    NodeMacro<float> mac;
    const float zero = 0.f;
    induction_collide<float, PRECISE, Store<ST>::COMP>(p, q, ql, og, 1.f, zero, zero, zero, zero, zero, zero, zero,
                                                      zero, zero, mac);
    if (MODE == MODE_FIELDS) {
        cavity_zero_fields<false>(p, fo, n, false);
        if (fo.B) { fo.B[n] = mac.Bx; fo.B[N + n] = mac.By; fo.B[2 * N + n] = mac.Bz; }
        return;
    }
    store_induction<ST>(p, b, n, q, ql, og, zero, zero, zero);
}

template <int ST, bool MHD, int MODE, int COLL>
__global__ void __launch_bounds__(STEP_THREADS) cavity_kernel(const StepParams p, const StepBuffers b,
                                                              const FieldOut fo)
{
    using T = typename Store<ST>::T;
    grid_dependency_release();
    grid_dependency_wait();
    if (b.stop != nullptr && *b.stop) return;
    const uint32_t i = blockIdx.x * STEP_THREADS + threadIdx.x;
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < p.N) {
        const CavGeo g = cavity_geo(p, i);
        if (g.solid) {
            if (MODE == MODE_FIELDS) cavity_zero_fields<MHD>(p, fo, i, true);
        } else {
            float q[21], ql[21];
            if (MHD) load_g_box<ST>(p, static_cast<const T*>(b.gsrc), g, q, ql);
            if (g.flow) {
                float d[19], dl[19];
                load_f_box<ST>(p, static_cast<const T*>(b.fsrc), g, d, dl);
                node_from_sources<ST, MHD, MODE, false, COLL>(p, b, fo, i, d, dl, q, ql,
                                                              node_inputs<MHD, MODE>(p, b, i), acc);
            } else if (MHD) {
                induction_at_rest<ST, MODE>(p, b, fo, i, q, ql);
            } else if (MODE == MODE_FIELDS) {
                cavity_zero_fields<false>(p, fo, i, false);
            }
        }
    }
    if (MODE == MODE_STEP_RESID) block_partials<STEP_THREADS>(acc, b.partials);
}

// Whether the block that this one prefetches for may hold nodes of the flow
// lattice: its rows meet the box's in z and, when it lies within one z plane,
// in y.
__device__ __forceinline__ bool box_ahead(const StepParams& p, const StepBuffers& b)
{
    const long long first = ((long long)blockIdx.x + b.pf_ahead) * STEP_THREADS;
    if (first >= (long long)p.N) return false;
    const uint32_t n0 = (uint32_t)first, n1 = n0 + STEP_THREADS - 1 < p.N ? n0 + STEP_THREADS - 1 : p.N - 1;
    const int z0 = (int)fdiv(n0, p.div_nxy), z1 = (int)fdiv(n1, p.div_nxy);
    if (z1 < p.blo[2] || z0 > p.bhi[2]) return false;
    if (z0 != z1) return true;
    const int y0 = (int)fdiv(n0, p.div_nx) - z0 * p.ny, y1 = (int)fdiv(n1, p.div_nx) - z1 * p.ny;
    return y1 >= p.blo[1] && y0 <= p.bhi[1];
}

// The coupled cavity step in two passes per thread (the FP32 forms; the
// one-pass coupled F32C update needs 172 registers, one block per SM): pass 1
// gathers g, and f at a node of the flow lattice, for rho and m (at rest
// elsewhere: m = 0), and runs the induction part (g~ and this step's Lorentz
// force, zero outside the box); pass 2 gathers f again and runs the flow
// update with F = F_ext + F_L.  The one-pass arithmetic in the same order, bit
// for bit.
template <int ST, int MODE>
__global__ void __launch_bounds__(STEP_THREADS, 3) cavity_kernel_coupled2(const StepParams p, const StepBuffers b,
                                                                           const FieldOut fo)
{
    using T = typename Store<ST>::T;
    constexpr bool PRECISE = (ST == ST_F32 || ST == ST_F32C);
    grid_dependency_release();
    grid_dependency_wait();
    if (b.stop != nullptr && *b.stop) return;
    prefetch_ahead<ST, STEP_THREADS, true, MODE == MODE_STEP_RESID>(p, b, box_ahead(p, b));
    const uint32_t i = blockIdx.x * STEP_THREADS + threadIdx.x;
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < p.N) {
        const CavGeo g = cavity_geo(p, i);
        if (!g.solid) {
            float rho_inv = 1.f, mx = 0.f, my = 0.f, mz = 0.f;
            NodeIn<float> in{};
            if (g.flow) {
                float d[19], dl[19];
                in = node_inputs<true, MODE_STEP>(p, b, i);
                load_f_box<ST>(p, static_cast<const T*>(b.fsrc), g, d, dl);
                node_momentum<ST>(p, d, dl, rho_inv, mx, my, mz);
            }
            f_before_g();
            float q[21], ql[21], og[21];
            load_g_box<ST>(p, static_cast<const T*>(b.gsrc), g, q, ql);
            NodeMacro<float> mac;
            induction_collide<float, PRECISE, Store<ST>::COMP>(p, q, ql, og, rho_inv, mx, my, mz, in.Fx, in.Fy, in.Fz,
                                                              in.FLx, in.FLy, in.FLz, mac);
            store_induction<ST>(p, b, i, q, ql, og, g.flow ? mac.FLx : 0.f, g.flow ? mac.FLy : 0.f,
                                g.flow ? mac.FLz : 0.f);
        }
        if (g.flow) {
            float d[19], dl[19], q[21], ql[21];
            load_f_box<ST>(p, static_cast<const T*>(b.fsrc), g, d, dl);
            node_from_sources<ST, false, MODE, false, 0>(p, b, fo, i, d, dl, q, ql,
                                                         node_inputs<false, MODE, true>(p, b, i), acc);
        }
    }
    if (MODE == MODE_STEP_RESID) block_partials<STEP_THREADS>(acc, b.partials);
}

// Initial state under a moving lid.  A pull gathers from the other buffer as
// from the post-collision values of the previous step, so a link bounced off
// the lid returns with the lid term added.  For the first step to gather the
// rest state, the slot of every such link of buffer fbuf holds -lid_corr of
// the direction it returns as (the slot is read by that bounce only).
template <int ST>
__global__ void lid_init_kernel(const StepParams p, void* fbuf)
{
    using S = Store<ST>;
    using T = typename S::T;
    const uint32_t i = blockIdx.x * STEP_THREADS + threadIdx.x;
    if (i >= p.N) return;
    const Geo g = make_geo(p, i);
    if (g.solid || !in_box(p, g.x, g.y, g.z) || g.z != p.top_z) return;
    T* fs = static_cast<T*>(fbuf);
    const size_t N = p.N;
#pragma unroll
    for (int a = 0; a < 19; ++a) {
        if (dir_ez(a) != -1) continue;     // returns from above the top fluid plane
        const int ex = dir_ex(a), ey = dir_ey(a);
        int sx = g.x - ex, sy = g.y - ey;
        sx = sx < 0 ? sx + p.nx : (sx >= p.nx ? sx - p.nx : sx);
        sy = sy < 0 ? sy + p.ny : (sy >= p.ny ? sy - p.ny : sy);
        const int sz = g.z + 1 >= p.nz ? g.z + 1 - p.nz : g.z + 1;
        const bool solid = plane_solid(sx, p.nx, p.wlo[0], p.whi[0]) || plane_solid(sy, p.ny, p.wlo[1], p.whi[1]) ||
                           plane_solid(sz, p.nz, p.wlo[2], p.whi[2]) || !in_box(p, sx, sy, sz);
        if (!solid) continue;
        const size_t slot = (size_t)dir_opp(a) * N + g.n;
        fs[slot] = S::cv(toscale<ST>(p, -p.lid_corr[a]));
        if constexpr (S::COMP) reinterpret_cast<__half*>(fs + 19 * N)[slot] = __float2half_rn(0.f);
    }
}

template <int ST>
cudaError_t launch_lid_init_t(const StepParams& p, void* fbuf, cudaStream_t st)
{
    const unsigned grid = (unsigned)(((size_t)p.N + STEP_THREADS - 1) / STEP_THREADS);
    lid_init_kernel<ST><<<grid, STEP_THREADS, 0, st>>>(p, fbuf);
    return cudaGetLastError();
}

}  // namespace glbe
