// glbe_residual.cuh -- the reduction of a residual step's per-block partials
// (FP64, fixed order) and the record it leaves: shared by the stand-alone
// reduction kernel (glbe_api.cu) and the resident marches of small grids,
// which reduce inside their own launch.
//
// What bounds it: latency and the FP64 pipe.  An SM of this GPU issues two
// FP64 operations a clock, so a warp's addition occupies the pipe for 16
// clocks; what matters is how few additions lie behind one another and on one
// SM.  Each of the seven sums is therefore one warp's: its lanes read
// consecutive partials into four independent accumulators, and five shuffles
// combine them.  (A form in which thread 0 added 7 x 32 warp sums one after
// another took 22 us for 2 blocks' partials, and its first stage, with seven
// block-wide sums one after the other, another 16 us.)
#pragma once
#include "glbe_internal.h"

namespace glbe {

template <typename V>
__device__ __forceinline__ V warp_sum(V v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

constexpr int RES_SUMS = 7;   // num, den, sum drho, Mx, My, Mz, non-finite count

constexpr unsigned FIN_CHUNK = 256;   // partials that one block (or pass) sums

__device__ __forceinline__ double warp_sum_all(double t)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Sum of row[b0, b1) by one warp, in every lane: a fixed order.  Reads through
// L2 (the partials may have been written earlier in the same launch).
__device__ __forceinline__ double partial_row_sum(const double* row, unsigned b0, unsigned b1)
{
    const unsigned lane = threadIdx.x & 31u;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned b = b0 + lane;
#pragma unroll 2
    for (; b + 96u < b1; b += 128u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] += __ldcg(row + b + 32u * k);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (b + 32u * k < b1) s[k] += __ldcg(row + b + 32u * k);
    return warp_sum_all((s[0] + s[1]) + (s[2] + s[3]));
}

// r(t) of the sums (Sec. 5): ||u(t) - u(t-10)|| / ||u(t)||.
__device__ __forceinline__ double residual_of(double num, double den)
{
    return den > 0.0 ? sqrt(num / den) : (num > 0.0 ? INFINITY : 0.0);
}

// Writes the record of level t from the sums tot[RES_SUMS] (one thread).
// Returns whether the march stops there.
__device__ __forceinline__ bool write_record(const RecordOut& o, const double* tot, long long t)
{
    const double r = residual_of(tot[0], tot[1]);
    double rec[RECORD_STRIDE] = {(double)t, r, tot[0], tot[1], o.mass0 + tot[2], tot[3], tot[4], tot[5], tot[6]};
    const unsigned long long c = *o.hist_count;
    double* h = o.hist + (size_t)(c % o.hist_cap) * RECORD_STRIDE;
#pragma unroll
    for (int k = 0; k < RECORD_STRIDE; ++k) {
        o.record[k] = rec[k];
        h[k] = rec[k];
    }
    *o.hist_count = c + 1;
    *o.t_dev = t + 10;
    const bool stops = (*o.tol > 0.0 && r <= *o.tol) || rec[8] > 0.0 || !isfinite(r);
    if (stops) *o.stop = 1;
    return stops;
}

}  // namespace glbe
