// A chunk of cell-sorted particles in the closed-form particle kernels: their hand-over to the threads
// in order of orbit-piece count, and the local-solve gates on cell coordinates.
#pragma once

#include "orbit_cell.cuh"
#include "particle_common.cuh"
#include "scatter_warp.cuh"

namespace pic {

// Shared-memory hand-over of a chunk's particles to the threads in order of orbit-piece count, so that
// the lanes of a warp run the same number of pieces: what the ranking computed (cell, coordinate, v^{p}
// + v^n) travels with the particle.  A block of WARPS warps takes chunks of 32 WARPS ITEMS particles;
// with two items a warp takes one group from each end of the order, so that the block's warps have
// about equal work and wait little at the chunk's barriers (with one group of 32 per warp, eight warps
// a block, barriers were the first stall reason).
template <int WARPS, int ITEMS>
struct ChunkOrder {
    static constexpr int THREADS_ = 32 * WARPS, GROUPS = WARPS * ITEMS, SIZE = THREADS_ * ITEMS;
    int order[SIZE];
    int wcount[GROUPS][PIECE_CLASSES];
    double f[3][SIZE], vs[3][SIZE];
    int c[3][SIZE];

    // Dynamic shared memory of a kernel that also deposits: the hand-over and one tile per warp.
    static constexpr size_t smem() { return sizeof(ChunkOrder) + sizeof(long long) * DEPOSIT_TILE * WARPS; }
    static __device__ __forceinline__ ChunkOrder& in(unsigned char* dyn) { return *reinterpret_cast<ChunkOrder*>(dyn); }
    static __device__ __forceinline__ long long* tile(unsigned char* dyn) {
        return reinterpret_cast<long long*>(dyn + sizeof(ChunkOrder)) + (threadIdx.x >> 5) * DEPOSIT_TILE;
    }

    // The place of this thread's item `it` in the order; its particle's data and index (>= np: none).
    __device__ __forceinline__ int64_t take(int it, int64_t base, CellStart<double>& st, double v[3]) const {
        const int w = threadIdx.x >> 5, s = 32 * (it == 0 ? w : GROUPS - 1 - w) + (threadIdx.x & 31);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            st.f[a] = f[a][s];
            v[a] = vs[a][s];
            st.c[a] = c[a][s];
        }
        return base + order[s];
    }
};

// The chunk sizes: four warps with two groups each, or, for runs too small to fill the SMs that way,
// one group per block.  The pushes, whose instruction stream passes the caches of an SM's schedulers (the
// first stall reason with four warps a block: the blocks' warps are at different places of it), take eight
// warps a block where each resident block gets two chunks or more: at 32^3 with 2,097,152 particles 1.03 ->
// 0.96 ms (iterate) and 0.68 -> 0.65 (final sweep), in pairs 0.88 -> 0.81; at 128^3 with 134M 59.0 -> 53.9
// and 82.8 -> 70.9; sixteen warps 1.04, 0.75, 0.87, 59.8 and 70.6.  With 131,072 particles four warps take
// 63 us, eight 69.  The deposits by themselves prefer four (354 against 385 us).
typedef ChunkOrder<4, 2> ChunkLarge;
typedef ChunkOrder<8, 2> ChunkPush;
typedef ChunkOrder<1, 1> ChunkSmall;

// Knots crossed by an axis whose orbit ends at te (relative to its start cell).
__device__ __forceinline__ unsigned crossings(double te) {
    return (at_least_one(te) || below_zero(te)) ? min((unsigned)abs(__double2int_rd(te)), 3u) : 0u;
}

// Rank the chunk's particles by piece count (a stable order) and hand them over; ends with a barrier.
// load(j, x0, v2) gives particle j's position and v^{p} + v^n.
template <int WARPS, int ITEMS, typename L>
__device__ __forceinline__ void chunk_exchange(const StepParams& p, ChunkOrder<WARPS, ITEMS>& co, int64_t base,
                                               L&& load) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    CellStart<double> st[ITEMS];
    double v2[ITEMS][3];
    int cls[ITEMS];
    unsigned mine[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int64_t j = base + it * 32 * WARPS + threadIdx.x;
        cls[it] = PIECE_CLASSES - 1;
        mine[it] = 0;
        if (j < p.np) {
            double x0[3];
            load(j, x0, v2[it]);
            cell_start(x0, p.m, st[it]);
            unsigned pieces = 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) pieces += crossings(st[it].f[a] + p.cb[a] * v2[it][a]);
            cls[it] = (int)min(pieces, (unsigned)(PIECE_CLASSES - 1)) - 1;
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < PIECE_CLASSES; ++c) {
            const unsigned m = __ballot_sync(0xffffffffu, cls[it] == c);
            if (lane == 0) co.wcount[it * WARPS + w][c] = __popc(m);
            if (cls[it] == c) mine[it] = m;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        int r = __popc(mine[it] & ((1u << lane) - 1u));
        for (int c = 0; c < cls[it]; ++c)
#pragma unroll
            for (int v = 0; v < WARPS * ITEMS; ++v) r += co.wcount[v][c];
        for (int v = 0; v < it * WARPS + w; ++v) r += co.wcount[v][cls[it]];
        co.order[r] = it * 32 * WARPS + threadIdx.x;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            co.f[a][r] = st[it].f[a];
            co.vs[a][r] = v2[it][a];
            co.c[a][r] = st[it].c[a];
        }
    }
    __syncthreads();
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
