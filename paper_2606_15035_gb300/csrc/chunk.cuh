// A chunk of THREADS cell-sorted particles in the closed-form particle kernels: their hand-over to the
// threads in order of orbit-piece count, and the local-solve gates on cell coordinates.
#pragma once

#include "orbit_cell.cuh"
#include "particle_common.cuh"
#include "scatter_warp.cuh"

namespace pic {

// Shared-memory hand-over of a chunk's particles to the threads in order of orbit-piece count:
// what the ranking computed (cell, coordinate, v^{p} + v^n) travels with the particle.
struct ChunkOrder {
    int order[THREADS];
    int wcount[THREADS / 32][PIECE_CLASSES];
    double f[3][THREADS], vs[3][THREADS];
    int c[3][THREADS];
};

// Dynamic shared memory of the kernels that also deposit: the hand-over and one tile per warp.
constexpr size_t CHUNK_SMEM = sizeof(ChunkOrder) + sizeof(long long) * DEPOSIT_TILE * (THREADS / 32);

// Knots crossed by an axis whose orbit ends at te (relative to its start cell).
__device__ __forceinline__ unsigned crossings(double te) {
    return (at_least_one(te) || below_zero(te)) ? min((unsigned)abs(__double2int_rd(te)), 3u) : 0u;
}

// Rank the chunk's particles by piece count and hand them over; ends with a barrier.  Returns the
// index of this thread's particle (>= np: none).
__device__ __forceinline__ int64_t chunk_exchange(const StepParams& p, ChunkOrder& co, int64_t base, bool valid,
                                                  const double x0[3], const double v2[3], CellStart<double>& st,
                                                  double vs[3]) {
    int cls = PIECE_CLASSES - 1;
    if (valid) {
        cell_start(x0, p.m, st);
        unsigned pieces = 1;
#pragma unroll
        for (int a = 0; a < 3; ++a) pieces += crossings(st.f[a] + p.cb[a] * v2[a]);
        cls = (int)min(pieces, (unsigned)(PIECE_CLASSES - 1)) - 1;
    }
    const int r = stable_class_rank(cls, co.wcount);
    co.order[r] = threadIdx.x;
    if (valid) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            co.f[a][r] = st.f[a];
            co.vs[a][r] = v2[a];
            co.c[a][r] = st.c[a];
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        st.f[a] = co.f[a][threadIdx.x];
        vs[a] = co.vs[a][threadIdx.x];
        st.c[a] = co.c[a][threadIdx.x];
    }
    return base + co.order[threadIdx.x];
}

// is_creeping from the start's cell coordinate: on an axis with |beta| < BETA_CREEP, does twice
// the orbit reach a knot, or does it start within D_KNOT of one?  Integer comparisons throughout.
__device__ __forceinline__ bool is_creeping_cell(const double f[3], const double beta[3]) {
    bool r = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double u = f[a] + 2.0 * beta[a];
        const bool reach = at_least_one(u) || below_zero(u);
        const bool near = less_pos(f[a], D_KNOT) || less_pos(1.0 - D_KNOT, f[a]);
        r |= less_pos(fabs(beta[a]), BETA_CREEP) && (reach || near);
    }
    return r;
}

__device__ __forceinline__ double max_pos(double a, double b) { return less_pos(a, b) ? b : a; }

}  // namespace pic
