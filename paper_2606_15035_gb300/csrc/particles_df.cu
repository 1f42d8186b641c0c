// FP32-pair refinement push of the mixed-precision path (sm_103a).
//
// After the FP32 Picard iterations have brought the iterate to the FP32 floor (~1e-9), the
// mixed path refines it with Algorithm 1 iterations whose particle half (orbit breakpoints,
// Appendix A/B orbit integrals, gather, canonical-momentum push, point interpolant, next-orbit
// current) runs in FP32-pair arithmetic (dfloat.cuh: 48-bit significands on the FP32 pipes)
// instead of FP64.  The iterates stay FP64 arrays, so the FP64 particle-local solves, the
// residual sums and the FP64 iterations that close the step use them unchanged.  The pair
// map differs from the FP64 map G by ~1e-15 of the velocity (positions are carried as the
// cell index plus a pair offset in the cell, so their resolution is 2^-48 cells at any mesh
// size), so its fixed point is the FP64 fixed point to that level.  What checks the iterate
// is FP64: the FP64 final sweep, which measures ||G(v*) - v*|| of the pair iterate itself
// before committing it (the mixed path's default with mixed_tol64 > 0), or the FP64
// iterations that follow.
//
// The orbit integrals are those of the FP64 kernels (orbit_cell.cuh) on pairs, from a cell table of
// pairs; the hand-over by piece count, the gates and the next orbit's current (fixed point,
// scatter_warp.cuh) are theirs too.
#include <algorithm>
#include <climits>
#include <cmath>

#include "pic_internal.h"
#include "dfloat.cuh"
#include "chunk.cuh"

namespace pic {
namespace {

// Warps per SM: 16 (128 registers) measured 88.5 ms at 128^3 with 134M particles, 24 (85) 100.4.
constexpr int DF_WARPS = 16;

struct ParamsDF {
    StepParams p;       // the FP64 parameters (creeping tests, residual sums, iterate I/O)
    DF cb[3], ihs[3];   // dt / (2 H), 1 / (2 H): factors of v^p + v^n
    DF dtq, q;          // dt q, q
};

DF pair_of(double d) {
    const float h = (float)d;
    return DF(h, (float)(d - (double)h));
}

// Loader of a cell's pair entries, as FieldLoad: from the pair cell table, or from the pairs of the
// gather table (5 float4 per node: A^n, A^{n+1}, grad phi), taking the nodes' differences.
template <bool CELLS>
struct PairLoad {
    const float4* t;
    __device__ __forceinline__ PairLoad(const float4* table, const int c[3], const MeshDims& m)
        : t(table + (CELL_VALUES / 2) * cell_row(c, m)) {}
    __device__ __forceinline__ void operator()(int p, int col, DF& a, DF& b) const {
        const float4 q = __ldg(t + p * CELL_COLS + col);
        a = DF(q.x, q.y);
        b = DF(q.z, q.w);
    }
};

constexpr int DF_NODE = 10;   // pairs per node of the pair gather table (9 and a pad)

template <>
struct PairLoad<false> {
    const float2* t;
    int64_t g[8];
    __device__ __forceinline__ PairLoad(const float4* table, const int c[3], const MeshDims& m)
        : t(reinterpret_cast<const float2*>(table)) {
        cell_nodes8(c, m, g);
    }
    __device__ __forceinline__ DF get(int k, int col) const {
        const float2 q = __ldg(t + DF_NODE * g[k] + col);
        return DF(q.x, q.y);
    }
    __device__ __forceinline__ DF node(int k, int col) const {
        return col < 3 ? get(k, 3 + col) : (col < 6 ? get(k, col) - get(k, col - 3) : -get(k, col));
    }
    __device__ __forceinline__ void operator()(int p, int col, DF& a, DF& b) const {
        a = node(0, col);
        b = node(1, col) - a;
        if (p == 0) return;
        if (p == 3) {
            DF lo = node(2, col), hi = node(3, col) - lo;
            a = lo - a;
            b = hi - b;
            lo = node(4, col);
            hi = node(5, col) - lo;
            const DF l6 = node(6, col);
            a = (l6 - lo) - a;
            b = ((node(7, col) - l6) - hi) - b;
        } else {
            const DF lo = node(2 * p, col);
            a = lo - a;
            b = (node(2 * p + 1, col) - lo) - b;
        }
    }
};

// The FP32-pair iteration (239 -> 88.5 ms at 128^3 with 134M particles, from start-based integrals, a
// node table and shared 64-bit atomics before; 70.9 with the one-crossing walk, deposit columns by cell and
// blocks of eight warps, 73.0 with the deposits' units by cell): G(v^p) for every particle, creeping ones
// listed for k_local (as in k_push_cell), the e_v partial sums, and the orbit current of v^{p+1} = G(v^p) into Jnext.
template <bool CELLS, typename Chunk>
__global__ void __launch_bounds__(Chunk::THREADS_, 32 * DF_WARPS / Chunk::THREADS_) k_push_df(ParamsDF pd, const double* __restrict__ xi,
                                                               const double* __restrict__ v,
                                                               const double* __restrict__ P,
                                                               const double* __restrict__ vit,
                                                               const float4* __restrict__ table,
                                                               double* __restrict__ vnew, double* __restrict__ Jnext,
                                                               int32_t* __restrict__ creep_list,
                                                               int* __restrict__ creep_count,
                                                               const uint8_t* __restrict__ slide,
                                                               double* __restrict__ partials,
                                                               int* __restrict__ status) {
    __shared__ double sm[32];
    extern __shared__ __align__(16) unsigned char dyn[];
    Chunk& co = Chunk::in(dyn);
    long long* tile = Chunk::tile(dyn);
    const StepParams& p = pd.p;
    const int64_t np = p.np, nchunks = (np + Chunk::SIZE - 1) / Chunk::SIZE;
    double ev_num = 0.0, ev_den = 0.0;
    long long pieces_push = 0, pieces_scatter = 0;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * Chunk::SIZE;
        chunk_exchange(p, co, base, [&](int64_t j, double x0[3], double v2[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + j];
                v2[a] = vit[a * np + j] + v[a * np + j];
            }
        });
#pragma unroll 1
        for (int it = 0; it < 2; ++it) {
            CellStart<double> st;
            double vs[3];
            const int64_t i = co.take(it, base, st, vs);
            bool scat = false;               // this lane's next orbit is scattered here
            double bn[3] = {0.0, 0.0, 0.0}, w[3] = {0.0, 0.0, 0.0};
            if (i < np) {
                DF kick[3];
                {
                    CellStart<DF> sd;
                    DF vd[3], beta[3], acc[3], Ae[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        sd.f[a] = df_bits(st.f[a]);
                        sd.c[a] = st.c[a];
                        vd[a] = df_bits(vs[a]);
                        beta[a] = pd.cb[a] * vd[a];
                    }
                    const int nseg = for_each_piece(sd, beta, p.m, [&](DF h, DF sc, const DF mid[3], const int c[3]) {
                        piece_impulse(h, sc, mid, beta, vd, pd.ihs, PairLoad<CELLS>(table, c, p.m), acc);
                    });
                    if (nseg < 0) atomicOr(status, DEV_ERR_SEGMENTS);
                    pieces_push += nseg;
                    cell_A1(sd.f, PairLoad<CELLS>(table, sd.c, p.m), Ae);
                    // P^{n+1} - P^n - q A_h^{n+1}(x^{n+1}) (Eqs. (orbit-P-update), (orbit-v-update))
#pragma unroll
                    for (int a = 0; a < 3; ++a) kick[a] = mad(pd.dtq, acc[a], -(pd.q * Ae[a]));
                }
                double vw[3], d[3], vn[3], vi[3], beta[3];
                bool finite = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    vw[a] = (P[a * np + i] + dbl_of(kick[a])) * p.inv_mass;
                    finite = finite && isfinite(vw[a]);
                    vi[a] = vit[a * np + i];
                    vn[a] = v[a * np + i];
                    d[a] = vw[a] - vi[a];
                    beta[a] = p.cb[a] * vs[a];
                }
                if (!finite) atomicOr(status, DEV_ERR_NONFINITE);
                // the local-solve gate of k_push_cell, in FP64
                bool slow = false;
                if (p.hist) {
                    double dold = 0.0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) dold = max_pos(dold, ::fabs(vi[a] - vnew[a * np + i]));
                    const double dn = max_pos(max_pos(::fabs(d[0]), ::fabs(d[1])), ::fabs(d[2]));
                    if (less_pos(SLOW_RATIO * dold, dn))
                        slow = dn > p.slow_floor * sqrt(vi[0] * vi[0] + vi[1] * vi[1] + vi[2] * vi[2]);
                }
                const bool creep = p.accel && (is_creeping_cell(st.f, beta) || (slide[i] & SLIDE_CREPT) || slow);
#pragma unroll
                for (int a = 0; a < 3; ++a) vnew[a * np + i] = vw[a];
                if (creep) {
                    const int k = atomicAdd(creep_count, 1);
                    creep_list[k] = (int32_t)i;
                } else {
                    scat = true;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        ev_num += d[a] * d[a];
                        ev_den += vw[a] * vw[a];
                        const double v2n = vw[a] + vn[a];
                        bn[a] = p.cb[a] * v2n;
                        w[a] = p.q_dV_half * v2n;
                    }
                }
            }
            const int ns = scatter_warp(p.m, scat, st, bn, w, tile, 0, p.acc, Jnext);
            if (ns < 0) atomicOr(status, DEV_ERR_SEGMENTS);
            pieces_scatter += ns;
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
    write_partial<double>(partials, S_EV_NUM, ev_num, sm, false);
    write_partial<double>(partials, S_EV_DEN, ev_den, sm, false);
    write_partial<double>(partials, S_PIECES_PUSH, (double)pieces_push, sm, false);
    write_partial<double>(partials, S_PIECES_SCATTER, (double)pieces_scatter, sm, false);
}

__device__ __forceinline__ float4 pairs_of(double a, double b) {
    const float ah = (float)a, bh = (float)b;
    return make_float4(ah, (float)(a - (double)ah), bh, (float)(b - (double)bh));
}

// FP64 cell table -> pair cell table, entry by entry.
__global__ void k_cells_df(int64_t n, const double2* __restrict__ t64, float4* __restrict__ tdf) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const double2 q = t64[k];
        tdf[k] = pairs_of(q.x, q.y);
    }
}

// FP64 gather table (12 doubles per node) -> pair table (A^n, A^{n+1}, grad phi as pairs).
__global__ void k_table_df(int64_t N, const double* __restrict__ t64, float4* __restrict__ tdf) {
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x) {
        const double* t = t64 + 12 * g;
#pragma unroll
        for (int q = 0; q < DF_NODE / 2; ++q) tdf[(DF_NODE / 2) * g + q] = pairs_of(t[2 * q], q < 4 ? t[2 * q + 1] : 0.0);
    }
}

ParamsDF make_params_df(const Ctx& c) {
    ParamsDF pd;
    pd.p = make_params(c);
    pd.p.hist = c.cfg.picard_accel && c.run.hist;
    for (int a = 0; a < 3; ++a) {
        pd.cb[a] = pair_of(pd.p.cb[a]);
        pd.ihs[a] = pair_of(pd.p.ihs[a]);
    }
    pd.dtq = pair_of(pd.p.dtq);
    pd.q = pair_of(c.q);
    return pd;
}

}  // namespace

bool setup_pair_kernels() {
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_push_df<true, ChunkLarge>, at, (int)ChunkLarge::smem()) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_df<false, ChunkLarge>, at, (int)ChunkLarge::smem()) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_df<true, ChunkPush>, at, (int)ChunkPush::smem()) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_df<false, ChunkPush>, at, (int)ChunkPush::smem()) == cudaSuccess;
}

void launch_table_df(Ctx& c) {
    float4* t = reinterpret_cast<float4*>(c.pair_ctab ? c.pair_ctab : c.table_pair);
    if (c.pair_ctab) {
        const int64_t n = CELL_VALUES / 2 * c.m.ncell;
        const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((n + THREADS - 1) / THREADS, (int64_t)c.sms * 16));
        k_cells_df<<<nb, THREADS, 0, c.stream>>>(n, reinterpret_cast<const double2*>(c.ctab), t);
    } else {
        k_table_df<<<mesh_blocks(c), THREADS, 0, c.stream>>>(c.m.ncell, c.table, t);
    }
    ++c.launches;
}

void launch_push_df(Ctx& c, const double* vit, double* vnew, double* Jnext) {
    cudaMemsetAsync(c.creep_count, 0, 2 * sizeof(int), c.stream);   // count, k_local queue head
    const int nb = chunk_blocks(c);
    const float4* t = reinterpret_cast<const float4*>(c.pair_ctab ? c.pair_ctab : c.table_pair);
#define PIC_PUSH_DF(T, K)                                                                                           \
    k_push_df<T, K><<<nb, K::THREADS_, K::smem(), c.stream>>>(make_params_df(c), c.xi, c.v, c.P, vit, t, vnew, Jnext, \
                                                              c.creep_list, c.creep_count, c.slide, c.partials,    \
                                                              c.dev_status)
    const bool wide = wide_chunks(c);
    if (c.pair_ctab && wide) PIC_PUSH_DF(true, ChunkPush);
    else if (c.pair_ctab) PIC_PUSH_DF(true, ChunkLarge);
    else if (wide) PIC_PUSH_DF(false, ChunkPush);
    else PIC_PUSH_DF(false, ChunkLarge);
#undef PIC_PUSH_DF
    ++c.launches;
}

}  // namespace pic
