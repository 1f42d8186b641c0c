// The orbit current of a warp's particles, summed per cell on the integer pipe (sm_103a).
//
// Depositing a piece in FP64 takes 46 FP64 instructions and 24 L2 reductions per particle, on a
// pipe with 1/64 of the issue rate and with one L2 request per lane and reduction (equal addresses
// of a warp are not merged): both bound the scatters.  Every factor of a deposit is bounded (the
// moments of orbit_cell.cuh lie in [0, 1], the weights below the largest of the cell's particles), so the
// products and sums run in 64-bit fixed point instead: moments to 2^-62, each component's weights to
// 2^-57 of the largest that the warp adds to the same cell, and exact sums.  A cell's sum so has an error of
// a few 2^-57 of its largest deposit, where FP64 rounds each product at 2^-53 and J at every addition; a
// slow particle in a cell of its own keeps all its bits beside fast ones in others.  The warp's particles
// hold few distinct cells (the store is cell-sorted), so each cell's 24 sums (8 moments, 3 components) are
// taken by 24 lanes from a transposed shared tile, turned into node weights by three exchanges, and added to J once.
#pragma once

#include "fixed.cuh"
#include "orbit_cell.cuh"

namespace pic {

constexpr int DEPOSIT_ROWS = 24;
constexpr int DEPOSIT_STRIDE = 33;   // 33 x 8 B: a row's lanes and a column's rows miss each other's banks
constexpr int DEPOSIT_TILE = DEPOSIT_ROWS * DEPOSIT_STRIDE;   // 64-bit words per warp

// The lanes with `has` by cell: lanes of one row (its cell, -1 without) get adjacent columns of the tile.
struct TileOrder {
    unsigned group;   // lanes of this lane's cell
    int col;          // this lane's column

    // top_k: the largest e_k of the lanes of this lane's cell.
    template <int E>
    __device__ __forceinline__ TileOrder(bool has, int row, const int (&e)[E], int (&top)[E]) : group(0), col(0) {
        const unsigned full = 0xffffffffu, below = (1u << (threadIdx.x & 31)) - 1u;
        int base = 0;
        for (unsigned rest = __ballot_sync(full, has); rest;) {
            const int r = __shfl_sync(full, row, __ffs(rest) - 1);
            const bool mine = row == r;
            const unsigned g = __ballot_sync(full, mine);
            int t[E];
#pragma unroll
            for (int k = 0; k < E; ++k) t[k] = (int)__reduce_max_sync(full, mine ? (unsigned)e[k] : 0u);
            if (mine) {
                group = g;
                col = base + __popc(g & below);
#pragma unroll
                for (int k = 0; k < E; ++k) top[k] = t[k];
            }
            base += __popc(g);
            rest &= ~g;
        }
    }

    // The tile's sums over the columns of each cell (coordinates pc of its lanes): add(sum, cell, one of
    // its lanes) on every lane, lane r < DEPOSIT_ROWS with the sum of row r.
    template <typename F>
    __device__ __forceinline__ void sums(bool has, const int pc[3], const long long* tile, F&& add) const {
        const unsigned full = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        int base = 0;
        for (unsigned rest = __ballot_sync(full, has); rest;) {
            const int lead = __ffs(rest) - 1;
            const unsigned g = __shfl_sync(full, group, lead);
            rest &= ~g;
            int c[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) c[a] = __shfl_sync(full, pc[a], lead);
            const int end = base + __popc(g);
            long long s = 0;
            if (lane < DEPOSIT_ROWS) {
                const long long* rowp = tile + lane * DEPOSIT_STRIDE;
                for (int j = base; j < end; j += 4) {   // four loads in flight; the zero column pads the last ones
                    long long v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] = rowp[j + k < end ? j + k : 32];
                    s += (v[0] + v[1]) + (v[2] + v[3]);
                }
            }
            base = end;
            add(s, c, lead);
        }
    }
};

// Row of the node of a cell that the lowest three bits of k name.
__device__ __forceinline__ int64_t subset_node(const int c0[3], int k, const MeshDims& m) {
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) c[a] = ((k >> a) & 1) ? next_cell(c0[a], m.n[a]) : c0[a];
    return cell_row(c, m);
}

// Measured at 32^3 with 2,097,152 particles (1.31 pieces each): the first scatter 0.82 -> 0.49 ms with
// 4.5M L2 reduction requests where there were 67M; at 128^3 with 134M (2.2 pieces) 96 -> 44 ms;
// 0.34 and 29.8 ms with balanced chunks, the one-crossing walk and columns by cell, 0.35 and 31.5 with each
// cell's own unit (one a warp lost what separates slow particles from fast ones in other cells).
// In the push it takes 46 FP64 instructions a piece off the pipe that bounds it (1.59 -> 1.43 ms).
//
// Add the orbit currents q v_bar S_bar / dV (weights w, orbits st.f + s beta) of the lanes with `act`
// to J.  Every lane of the warp calls it; `tile` is the warp's DEPOSIT_TILE words.  Returns the lane's number of breakpoint intervals (-1: too many; 0: not active).
__device__ __forceinline__ int scatter_warp(const MeshDims& m, bool act, const CellStart<double>& st,
                                            const double beta[3], const double w[3], long long* tile, int det,
                                            const ExactAcc& acc, double* __restrict__ J) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t N = m.ncell;
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) finite = finite && exponent_of(w[a]) < 0x7ff && exponent_of(st.f[a]) < 0x7ff;
    if (det || __any_sync(full, act && !finite)) {
        // Deterministic mode: each deposit goes to the exact accumulators by itself (the warp's unit
        // would depend on which particles share it, and with that on the order a state was restored
        // in).  A weight or a coordinate that is not finite: the plain deposit hands it on to J.
        if (!act) return 0;
        CellStart<double> s = st;
        return for_each_piece(s, beta, m, [&](double h, double, const double mid[3], const int c[3]) {
            double W[8];
            int64_t g[8];
            node_weights(piece_moments(h, mid, beta), W);
            cell_nodes8(c, m, g);
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (det) exact_add(acc, a * N + g[k], h * w[a] * W[k]);
                    else atomicAdd(J + a * N + g[k], h * w[a] * W[k]);
                }
        });
    }
    if (lane < DEPOSIT_ROWS) tile[lane * DEPOSIT_STRIDE + 32] = 0;
    const int comp = min(lane >> 3, 2);   // this lane's component (lanes 24..31 sum nothing)
    const Fx c12 = fx_split(FX_ONE / 12);
    PieceWalk<double> wk(st, beta, m);
    bool last = !act;
    while (__any_sync(full, !last)) {
        bool has = false;
        int row = -1, pc[3] = {0, 0, 0};
        double h = 0.0, sm, mid[3] = {0.0, 0.0, 0.0};
        if (!last) {
            has = wk.next(beta, m, h, sm, mid, pc, last);
            if (has) row = (int)cell_row(pc, m);
        }
        double hw[3];
        int e[3], top[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            hw[a] = h * w[a];
            e[a] = max(exponent_of(hw[a]), 64);   // (the unit 2^(top - 1079) stays a normal number)
            top[a] = 64;
        }
        const TileOrder order(has, row, e, top);
        if (has) {
            long long M[8];
            Fx q[3], d[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                M[1 << a] = fixed_of(mid[a], 1023, 10);
                q[a] = fx_split(M[1 << a]);
                d[a] = fx_split(fixed_of(h * beta[a], 1023, 10));
            }
            const Fx dy = fx_split(fx_mul(d[1], c12)), dz = fx_split(fx_mul(d[2], c12));
            const long long kxy = fx_mul(d[0], dy), kxz = fx_mul(d[0], dz), kyz = fx_mul(d[1], dz);
            M[3] = fx_mul(q[0], q[1]) + kxy;
            M[5] = fx_mul(q[0], q[2]) + kxz;
            M[6] = fx_mul(q[1], q[2]) + kyz;
            M[7] = fx_mul(q[0], fx_split(M[6])) + fx_mul(q[1], fx_split(kxz)) + fx_mul(q[2], fx_split(kxy));
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const long long wf = fixed_of(hw[a], top[a], 4);
                const Fx ws = fx_split(wf);
                tile[(8 * a) * DEPOSIT_STRIDE + order.col] = wf;
#pragma unroll
                for (int k = 1; k < 8; ++k) tile[(8 * a + k) * DEPOSIT_STRIDE + order.col] = fx_mul(ws, fx_split(M[k]));
            }
        }
        __syncwarp();
        order.sums(has, pc, tile, [&](long long sum, const int c0[3], int lead) {
            const int t01 = __shfl_sync(full, top[0] | top[1] << 16, lead), t2 = __shfl_sync(full, top[2], lead);
            const double unit = __hiloint2double(((comp == 0 ? t01 & 0xffff : (comp == 1 ? t01 >> 16 : t2)) - 56) << 20, 0);
            // moments of the subsets -> weights of the nodes (inclusion--exclusion, axis by axis)
#pragma unroll
            for (int bit = 1; bit < 8; bit <<= 1) {
                const long long o = __shfl_xor_sync(full, sum, bit);
                if (!(lane & bit)) sum -= o;
            }
            if (lane < DEPOSIT_ROWS && sum != 0)
                atomicAdd(J + comp * N + subset_node(c0, lane, m), (double)sum * unit);
        });
        __syncwarp();   // the tile is rewritten by the next pieces
    }
    return act ? wk.count : 0;
}

}  // namespace pic
