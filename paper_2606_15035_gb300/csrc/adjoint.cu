// Adjoint (reverse mode) of the implicit step and of the initial data (sm_103a, FP64).
//
// One step maps the level-n state s = (x, v, P, phi, psi, A, U, rho) to level n+1 through the
// accepted iterate v*, a fixed point of Algorithm 1's map, v* = G(v*; s), and the final sweep
// s' = F(v*, s) (§5.4), whose velocity output is G itself.  For a scalar L(s') with adjoint
// lambda' = dL/ds', the implicit-function theorem gives dL/ds = F_s^T (lambda' + mu e_v) with
// mu (the adjoint of v*) the solution of the transposed fixed point
//     mu = F_v*^T (lambda' + mu e_v),
// e_v placing mu on the velocity output.  Each application of F^T (a "sweep") is:
//   1. the particles' value pass: lambda_P' + lambda_v / m becomes the adjoint of the impulse,
//      which scatters onto the mesh adjoints of the gather table (grad phi^{n+1/2}, and A^n,
//      A^{n+1} through the transposed contraction of D_i A with vbar) and of A^{n+1} at the end
//      point (the point interpolant's transpose);
//   2. the mesh phase transposed: grad^T = -div, the Crank--Nicolson Helmholtz operator
//      I - a Delta_h is symmetric (one Chebyshev solve of the same schedule), continuity's
//      div^T = -grad; this gives the adjoints of phi^n, psi^n, A^n, U^n, rho^n and of J;
//   3. the particles' derivative pass: each particle's scalar
//         Phi = lam_gphibar . gphibar + lam_F . (D A)^T vbar + lam_Aend . A_h^{n+1}(x + beta)
//             + lam_x' . (x + beta) + sum_g lam_J[g] . J_g(particle)
//      is differentiated with respect to its start position and displacement beta in reverse
//      through the closed-form orbit integrals, with the mesh adjoints and fields held fixed.
//      beta = dt (v* + v^n) / (2 H) gives the adjoints of v* and v^n.
// The transposed fixed point (I - K) mu = b0, g(mu) = K mu + b0 being step 3's adjoint of v*,
// is solved by restarted GMRES with right preconditioning.  The preconditioner is the transpose
// of the forward iteration's own splitting: a particle that the step solved locally (its
// slide byte's SLIDE_CREPT bit) gets its 3 x 3 block (I - B^T)^{-1}, B = dG_i / dv*_i with the
// fields fixed (dual numbers, dual.cuh); every other particle gets the identity, as the plain
// Picard update treats it.  The stationary iteration with this splitting is the transposed
// linearisation of the forward solve, so its spectral radius is that of the forward iteration
// at the accepted step (below one, since the step converged), and the preconditioned operator's
// spectrum lies in a disc around 1 of that radius.  Within a restart cycle GMRES's residual is
// never above the stationary iteration's, and it is far below it where the forward iteration
// itself converged slowly.
//
// Sliding components (the step committed them by the sliding equations, §9 of the notes on the
// local solve): their iterate is the explicit landing velocity v*_a = 2 d_a H_a / dt - v^n_a,
// d_a the start's signed distance to its knot, their velocity output is v*_a itself and their
// momentum m v*_a + q A_h,a(x^{n+1}).  So they have no fixed-point equation (mu_a = 0, their
// rows and columns of B are dropped), their push impulse is unused (the adjoint of P^n_a is
// zero), the adjoint of their momentum reaches A_h at the end point and m v*_a, and the total
// adjoint nu_a of v*_a (direct, plus the orbit's g_a) goes to the start through d_a
// (d v*_a / d xi_a = -2 H_a / dt) and to v^n_a (-1).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "pic_internal.h"
#include "chunk.cuh"
#include "dual.cuh"

namespace pic {
namespace {

struct AdjParams {
    StepParams p;
    double a, c_rho, c_J;     // CN constants: a = kappa^2 dt^2 / 4, dt^2 kappa^2 sigma_i / 2
    double sigma1, sigma2;
};

AdjParams adj_params(const Ctx& c) {
    AdjParams ap;
    ap.p = make_params(c);
    const double k2 = c.cfg.kappa * c.cfg.kappa, dt = c.cfg.dt;
    ap.a = 0.25 * k2 * dt * dt;
    ap.c_rho = 0.5 * dt * dt * k2 * c.cfg.sigma1;
    ap.c_J = 0.5 * dt * dt * k2 * c.cfg.sigma2;
    ap.sigma1 = c.cfg.sigma1;
    ap.sigma2 = c.cfg.sigma2;
    return ap;
}

__device__ __forceinline__ int64_t nshift(int64_t g, int dx, int dy, int dz, const MeshDims& m) {
    const int ix = (int)(g % m.n[0]);
    const int64_t t = g / m.n[0];
    const int iy = (int)(t % m.n[1]), iz = (int)(t / m.n[1]);
    return node_index(wrapi(ix + dx, m.n[0]), wrapi(iy + dy, m.n[1]), wrapi(iz + dz, m.n[2]), m);
}

// D_a f at node g (stride: distance between a field's consecutive node values in memory)
__device__ __forceinline__ double dcen_s(const double* __restrict__ f, int64_t stride, int64_t g, int a,
                                         const MeshDims& m, const double* invH) {
    const int64_t p = a == 0 ? nshift(g, 1, 0, 0, m) : (a == 1 ? nshift(g, 0, 1, 0, m) : nshift(g, 0, 0, 1, m));
    const int64_t q = a == 0 ? nshift(g, -1, 0, 0, m) : (a == 1 ? nshift(g, 0, -1, 0, m) : nshift(g, 0, 0, -1, m));
    return 0.5 * invH[a] * (f[stride * p] - f[stride * q]);
}

__device__ __forceinline__ double lap_s(const double* __restrict__ f, int64_t g, const MeshDims& m, const double* invH) {
    const double c = f[g];
    double s = 0.25 * invH[0] * invH[0] * (f[nshift(g, 2, 0, 0, m)] - 2.0 * c + f[nshift(g, -2, 0, 0, m)]);
    s += 0.25 * invH[1] * invH[1] * (f[nshift(g, 0, 2, 0, m)] - 2.0 * c + f[nshift(g, 0, -2, 0, m)]);
    s += 0.25 * invH[2] * invH[2] * (f[nshift(g, 0, 0, 2, m)] - 2.0 * c + f[nshift(g, 0, 0, -2, m)]);
    return s;
}

#define ADJ_LOOP(i, n) for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// ---- the particles' push, templated on the scalar type (double, or Dual for derivatives) -----
//
// The formulas of the FP64 push from a piece's start (k_adj_blocks differentiates them by dual numbers): the
// orbit gather of grad phi, (D_i A)^T vbar contracted with vbar first, the end point's
// A_h^{n+1}, and the orbit weights of the current.  Positions are in cell units.

template <typename T>
__device__ __forceinline__ void push_piece_t(const StepParams& p, const Segment<T>& sg, const T beta[3], const T vb[3],
                                             const double* __restrict__ table, T gphi[3], T F[3]) {
    const PieceInts<T> I = piece_integrals(sg, beta, true);
    T W[8];
    weights_from_ints(I, W);
    int64_t g[8];
    Segment<double> sd;
    sd.cell[0] = sg.cell[0];
    sd.cell[1] = sg.cell[1];
    sd.cell[2] = sg.cell[2];
    segment_nodes8(sd, p.m, g);
    const T s = sg.s0, oms = T(1) - sg.s0, h = sg.h, hh2 = T(0.5) * sg.h * sg.h;
    T am[8], cc[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const double* t = table + 12 * g[k];
        const T an = vb[0] * t[0] + vb[1] * t[1] + vb[2] * t[2];
        const T a1 = vb[0] * t[3] + vb[1] * t[4] + vb[2] * t[5];
        am[k] = oms * an + s * a1;
        cc[k] = a1 - an;
        gphi[0] += W[k] * t[6];
        gphi[1] += W[k] * t[7];
        gphi[2] += W[k] * t[8];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int pa = j == 0 ? 1 : 0, qa = j == 2 ? 1 : 2;
        const int sp = j == 0 ? 2 : 1, sq = j == 2 ? 2 : 4;
        const int sj = j == 0 ? 1 : (j == 1 ? 2 : 4);
        const T D00 = am[sj] - am[0], D10 = am[sp + sj] - am[sp];
        const T D01 = am[sq + sj] - am[sq], D11 = am[sp + sq + sj] - am[sp + sq];
        const T C00 = cc[sj] - cc[0], C10 = cc[sp + sj] - cc[sp];
        const T C01 = cc[sq + sj] - cc[sq], C11 = cc[sp + sq + sj] - cc[sp + sq];
        const T t0 = D00 * h + (D10 - D00) * I.S1[pa] + (D01 - D00) * I.S1[qa] + (D11 - D10 - D01 + D00) * I.S2[j];
        const T t1 = C00 * hh2 + (C10 - C00) * I.E1[pa] + (C01 - C00) * I.E1[qa] + (C11 - C10 - C01 + C00) * I.E2[j];
        F[j] += T(p.invH[j]) * (t0 + t1);
    }
}

// Wrap onto [0, n) as the forward push does (derivative 1).
template <typename T>
__device__ __forceinline__ T wrap_t(T x, double n) {
    T w = x < T(0) ? x + T(n) : (x >= T(n) ? x - T(n) : x);
    return w >= T(n) ? w - T(n) : w;
}

// A_h^{n+1} at a wrapped position (8 linear B-splines), table column block 3..5.
template <typename T>
__device__ __forceinline__ void point_A1_t(const StepParams& p, const T xq[3], const double* __restrict__ table, T out[3]) {
    int c[3];
    T r[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const T f = floor(xq[a]);
        c[a] = (int)f;
        r[a] = xq[a] - f;
    }
    Segment<double> sd;
    sd.cell[0] = c[0];
    sd.cell[1] = c[1];
    sd.cell[2] = c[2];
    int64_t g[8];
    segment_nodes8(sd, p.m, g);
    out[0] = out[1] = out[2] = T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const T wx = (k & 1) ? r[0] : T(1) - r[0];
        const T wy = (k & 2) ? r[1] : T(1) - r[1];
        const T wz = (k & 4) ? r[2] : T(1) - r[2];
        const T w = wx * wy * wz;
        const double* t = table + 12 * g[k] + 3;
        out[0] += w * t[0];
        out[1] += w * t[1];
        out[2] += w * t[2];
    }
}

// ---- step 1: the particles' value pass (mesh adjoints of the gather table) ---------------------

// lam_tab per node: [A^n (3) | A^{n+1} (3) | grad phi^{n+1/2} (3)], 9 doubles, accumulated.
// The output adjoints of one particle component: lP1 (of P^{n+1}), lAe (of A_h^{n+1} at the end
// point), lg and lF (of the orbit gathers grad phi-bar and (D A)^T vbar).
__device__ __forceinline__ void out_adjoints(const StepParams& p, bool sl, double lv, double lP, double mu_c,
                                             double& lP1, double& lAe, double& lg, double& lF) {
    if (sl) {             // v1 = v*, P1 = m v* + q A_end: no impulse
        lP1 = lP;
        lAe = p.q * lP;
        lg = lF = 0.0;
    } else {              // v1 = (P1 - q A_end) / m, P1 = P + dt q (-gphibar + F)
        const double lv1 = lv + mu_c;
        lP1 = lP + lv1 * p.inv_mass;
        lAe = -p.q * p.inv_mass * lv1;
        lg = -p.dt * p.q * lP1;
        lF = p.dt * p.q * lP1;
    }
}

// Per orbit piece the transposes of piece_impulse (orbit_cell.cuh) on the mixed differences of A^{n+1},
// A^n and grad phi, 8 subsets of the axes and 3 components each, and of the interpolant of A^{n+1} at the
// end point.  Every particle's 72 terms a piece went to the mesh by atomics, 96 L2 reductions a particle
// and more, which bounded the kernel (0.80 ms at 32^3 with 524,288 particles).  As in scatter_warp the
// warp's particles are summed per cell first, in 64-bit fixed point (each component's values to 2^-57 of the
// largest product that the warp adds to the cell), three tiles a piece, and turned into node values once
// per cell: 0.43 ms, 0.46 with the units by cell (one a warp lost the bits of small cotangents beside large ones).
__device__ __forceinline__ void plain_rows(double* __restrict__ col, const int c[3], const MeshDims& m, const double M[8],
                                           const double w[3]) {
    double W[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) W[k] = M[k];
#pragma unroll
    for (int bit = 1; bit < 8; bit <<= 1)
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (!(k & bit)) W[k] -= W[k | bit];
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a) atomicAdd(col + 9 * subset_node(c, k, m) + a, w[a] * W[k]);
}

__global__ void __launch_bounds__(ChunkLarge::THREADS_, 4) k_adj_scatter(
    AdjParams ap, const double* __restrict__ xi, const double* __restrict__ v, const double* __restrict__ vstar,
    const double* __restrict__ lam_P, const double* __restrict__ lam_v, const double* __restrict__ mu,
    const uint8_t* __restrict__ slide, double* __restrict__ lam_tab) {
    extern __shared__ __align__(16) unsigned char dyn[];
    ChunkLarge& co = ChunkLarge::in(dyn);
    long long* tile = ChunkLarge::tile(dyn);
    const StepParams& p = ap.p;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, comp = min(lane >> 3, 2);
    const int64_t np = p.np, nchunks = (np + ChunkLarge::SIZE - 1) / ChunkLarge::SIZE;
    if (lane < DEPOSIT_ROWS) tile[lane * DEPOSIT_STRIDE + 32] = 0;
    // the tile's sums per cell into column `col` of lam_tab, component a's unit 2^(unit_a - 2046)
    auto flush = [&](const TileOrder& order, bool has, const int c[3], int col, const int unit[3]) {
        __syncwarp();
        order.sums(has, c, tile, [&](long long sum, const int c0[3], int lead) {
            const int u01 = __shfl_sync(full, unit[0] | unit[1] << 16, lead), u2 = __shfl_sync(full, unit[2], lead);
            const int u = comp == 0 ? u01 & 0xffff : (comp == 1 ? u01 >> 16 : u2);
            double x = (double)sum;
#pragma unroll
            for (int bit = 1; bit < 8; bit <<= 1) {
                const double o = __shfl_xor_sync(full, x, bit);
                if (!(lane & bit)) x -= o;
            }
            if (lane < DEPOSIT_ROWS)
                atomicAdd(lam_tab + 9 * subset_node(c0, lane, p.m) + col + comp,
                          x * pow2_biased(u >> 1) * pow2_biased(u - (u >> 1)));
        });
        __syncwarp();
    };
    // rows (a, k) = w_a M_k, w given at 2^(-top - 56 + 1023), M at 2^-62
    auto rows = [&](int col, const long long w[3], const long long M[8]) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const Fx ws = fx_split(w[a]);
            tile[8 * a * DEPOSIT_STRIDE + col] = w[a];
#pragma unroll
            for (int k = 1; k < 8; ++k) tile[(8 * a + k) * DEPOSIT_STRIDE + col] = fx_mul(ws, fx_split(M[k]));
        }
    };
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * ChunkLarge::SIZE;
        chunk_exchange(p, co, base, [&](int64_t j, double x0[3], double v2[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + j];
                v2[a] = vstar[a * np + j] + v[a * np + j];
            }
        });
#pragma unroll 1
        for (int item = 0; item < 2; ++item) {
            CellStart<double> st;
            double vs[3], beta[3], f[3] = {0.0, 0.0, 0.0}, lg[3] = {0.0, 0.0, 0.0}, lA[3] = {0.0, 0.0, 0.0};
            const int64_t i = co.take(item, base, st, vs);
            const bool act = i < np;
            double fs = 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (act) {
                    double lP1, lF;
                    out_adjoints(p, (slide[i] >> a) & 1u, lam_v[a * np + i], lam_P[a * np + i], mu[a * np + i], lP1, lA[a],
                                 lg[a], lF);
                    f[a] = lF * p.ihs[a];
                } else {
                    vs[a] = 0.0;
                }
                beta[a] = p.cb[a] * vs[a];
                fs += fabs(f[a]);
            }
            // a value that is not finite goes on as it is
            bool finite = exponent_of(fs) < 0x7fe;
#pragma unroll
            for (int a = 0; a < 3; ++a)
                finite = finite && max(exponent_of(vs[a]), max(exponent_of(lg[a]), exponent_of(lA[a]))) < 0x7ff;
            const bool plain = __any_sync(full, !finite);
            PieceWalk<double> wk(st, beta, p.m);
            bool last = !act;
            while (__any_sync(full, !last)) {
                bool has = false;
                int c[3] = {0, 0, 0};
                double h = 0.0, sm = 0.0, m[3] = {0.0, 0.0, 0.0};
                if (!last) has = wk.next(beta, p.m, h, sm, m, c, last);
                double ab[8], x1[8];   // adjoints of A_k . vs at the piece's middle: all, and A^{n+1}'s share
                double M[8];
                if (has) {
                    const PieceMoments<double> q = piece_moments(h, m, beta);
                    const double hf[3] = {h * f[0], h * f[1], h * f[2]};
                    ab[0] = x1[0] = 0.0;
                    ab[1] = hf[0];
                    ab[2] = hf[1];
                    ab[4] = hf[2];
                    ab[3] = hf[0] * m[1] + hf[1] * m[0];
                    ab[5] = hf[0] * m[2] + hf[2] * m[0];
                    ab[6] = hf[1] * m[2] + hf[2] * m[1];
                    ab[7] = hf[0] * q.Pyz + hf[1] * q.Pxz + hf[2] * q.Pxy;
                    x1[1] = sm * ab[1];
                    x1[2] = sm * ab[2];
                    x1[4] = sm * ab[4];
                    x1[3] = sm * ab[3] + (hf[0] * q.e[1] + hf[1] * q.e[0]);
                    x1[5] = sm * ab[5] + (hf[0] * q.e[2] + hf[2] * q.e[0]);
                    x1[6] = sm * ab[6] + (hf[1] * q.e[2] + hf[2] * q.e[1]);
                    x1[7] = sm * ab[7] + (hf[0] * (m[1] * q.e[2] + m[2] * q.e[1]) + hf[1] * (m[0] * q.e[2] + m[2] * q.e[0]) +
                                          hf[2] * (m[0] * q.e[1] + m[1] * q.e[0]));
                    M[0] = 1.0;
                    M[1] = m[0];
                    M[2] = m[1];
                    M[3] = q.Pxy;
                    M[4] = m[2];
                    M[5] = q.Pxz;
                    M[6] = q.Pyz;
                    M[7] = q.S;
                }
                if (plain) {
                    if (has) {
                        double x0[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) x0[k] = ab[k] - x1[k];
                        plain_rows(lam_tab, c, p.m, x0, vs);
                        plain_rows(lam_tab + 3, c, p.m, x1, vs);
                        const double hl[3] = {h * lg[0], h * lg[1], h * lg[2]};
                        plain_rows(lam_tab + 6, c, p.m, M, hl);
                    }
                    continue;
                }
                // exponents of the factors: |a piece's sums| < 1.2 h fs, so one above that of h fs
                const int tf = max(exponent_of(h * fs), 64) + 1;
                double hl[3];
                int e[6], top[6];   // of the products v (a piece's sum), and of h lg
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    hl[a] = h * lg[a];
                    e[a] = max(exponent_of(vs[a]), 64) + tf;
                    e[3 + a] = max(exponent_of(hl[a]), 64);
                    top[a] = top[3 + a] = 129;
                }
                const TileOrder order(has, has ? (int)cell_row(c, p.m) : -1, e, top);
                // the velocities' shift brings every lane's products to the cell's unit
                Fx vf[3];
                int unit[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    vf[a] = fx_split(fixed_of(vs[a], top[a] - tf, 9));
                    unit[a] = top[a] - 55;
                }
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (has) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const Fx x = fx_split(fixed_of(half == 0 ? ab[k] - x1[k] : x1[k], tf, 4));
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                tile[(8 * a + k) * DEPOSIT_STRIDE + order.col] = k == 0 ? 0 : fx_mul(vf[a], x);
                        }
                    }
                    flush(order, has, c, 3 * half, unit);
                }
                if (has) {
                    long long w[3], Mf[8];
#pragma unroll
                    for (int a = 0; a < 3; ++a) w[a] = fixed_of(hl[a], top[3 + a], 4);
#pragma unroll
                    for (int k = 1; k < 8; ++k) Mf[k] = fixed_of(M[k], 1023, 10);
                    rows(order.col, w, Mf);
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) unit[a] = top[3 + a] + 967;
                flush(order, has, c, 6, unit);
            }
            // the end point's interpolant of A^{n+1}, transposed
            const double M[8] = {1.0, wk.te[0], wk.te[1], wk.te[0] * wk.te[1], wk.te[2], wk.te[0] * wk.te[2],
                                 wk.te[1] * wk.te[2], wk.te[0] * wk.te[1] * wk.te[2]};
            if (plain) {
                if (act) plain_rows(lam_tab + 3, wk.c, p.m, M, lA);
                continue;
            }
            int e[3], top[3], unit[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                e[a] = max(exponent_of(lA[a]), 64);
                top[a] = 64;
            }
            const TileOrder order(act, act ? (int)cell_row(wk.c, p.m) : -1, e, top);
            if (act) {
                long long w[3], Mf[8];
#pragma unroll
                for (int a = 0; a < 3; ++a) w[a] = fixed_of(lA[a], top[a], 4);
#pragma unroll
                for (int k = 1; k < 8; ++k) Mf[k] = fixed_of(M[k], 1023, 10);
                rows(order.col, w, Mf);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) unit[a] = top[a] + 967;
            flush(order, act, wk.c, 3, unit);
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
}

// ---- step 2: the mesh phase transposed -----------------------------------------------------------
//
// Inputs: lam_tab, and the level-(n+1) adjoints lF1 = [phi | A] (4 N), lW1 = [psi | U] (4 N),
// lrho1 (N).  t_f = lF1_f + (particles' adjoint of F^{n+1}_f) + (2/dt) lW1_f is the right-hand
// side of the adjoint Helmholtz solve (psi^{n+1} = 2 (phi^{n+1} - phi^n)/dt - psi^n);
// pn_f collects the particles' adjoint of F^n_f.  grad phi^{n+1/2} = grad (phi^n + phi^{n+1})/2
// gives -div(lam_gphi)/2 to both levels of phi.
__global__ void k_adj_mesh_rhs(AdjParams ap, const double* __restrict__ lam_tab, const double* __restrict__ lF1,
                               const double* __restrict__ lW1, double* __restrict__ t, double* __restrict__ pn) {
    const StepParams& p = ap.p;
    const int64_t N = p.m.ncell;
    ADJ_LOOP(g, N) {
        double ldiv = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) ldiv += dcen_s(lam_tab + 6 + a, 9, g, a, p.m, p.invH);
        const double lphi_half = -0.5 * ldiv;
        t[g] = lF1[g] + lphi_half + 2.0 / p.dt * lW1[g];
        pn[g] = lphi_half;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int64_t o = (1 + c) * N + g;
            t[o] = lF1[o] + lam_tab[9 * g + 3 + c] + 2.0 / p.dt * lW1[o];
            pn[o] = lam_tab[9 * g + c];
        }
    }
}

// After y = (I - a Delta_h)^{-1} t: the level-n adjoints and the adjoint of J.
__global__ void k_adj_mesh_out(AdjParams ap, const double* __restrict__ y, const double* __restrict__ pn,
                               const double* __restrict__ lW1, const double* __restrict__ lrho1,
                               double* __restrict__ lF0, double* __restrict__ lW0, double* __restrict__ lrho0,
                               double* __restrict__ lJ) {
    const StepParams& p = ap.p;
    const int64_t N = p.m.ncell;
    ADJ_LOOP(g, N) {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const double* yf = y + f * N;
            lF0[f * N + g] = yf[g] + ap.a * lap_s(yf, g, p.m, p.invH) - 2.0 / p.dt * lW1[f * N + g] + pn[f * N + g];
            lW0[f * N + g] = p.dt * yf[g] - lW1[f * N + g];
        }
        // rho^{n+1/2} = (rho^n + rho^{n+1}) / 2 feeds phi's source with c_rho; rho^{n+1} = rho^n - dt div J
        lrho0[g] = lrho1[g] + ap.c_rho * y[g];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // lam_rho^{n+1} (total) = lrho1 + c_rho y_phi / 2 at the neighbours, then J's dt grad
            const int64_t pp = c == 0 ? nshift(g, 1, 0, 0, p.m) : (c == 1 ? nshift(g, 0, 1, 0, p.m) : nshift(g, 0, 0, 1, p.m));
            const int64_t qq = c == 0 ? nshift(g, -1, 0, 0, p.m) : (c == 1 ? nshift(g, 0, -1, 0, p.m) : nshift(g, 0, 0, -1, p.m));
            const double lr_p = lrho1[pp] + 0.5 * ap.c_rho * y[pp], lr_q = lrho1[qq] + 0.5 * ap.c_rho * y[qq];
            lJ[c * N + g] = ap.c_J * y[(1 + c) * N + g] + p.dt * 0.5 * p.invH[c] * (lr_p - lr_q);
        }
    }
}

// ---- step 3: the particles' derivative pass --------------------------------------------------------
//
// Each particle's scalar Phi (file comment) is differentiated with respect to its start coordinate
// and displacement in reverse, by hand, piece by piece in the centred form of orbit_cell.cuh.  With
// f_j = lam_F,j / (2 H_j), a piece contributes h X,
//     X = sum_k a_k abar_k + cc_k cbar_k + sum_T K_T M_T,
// where a_k and cc_k are the table's A columns contracted with v (k = subsets of the axes), M_T the
// moments, abar_k and cbar_k the moments that multiply them in sum_j f_j F_j, and K_T the adjoint-
// weighted coefficients of -grad phi and of J's adjoint.  X is multilinear in the midpoint m, in
// kappa = h^2 / 12 (through e = kappa beta and k_pq = kappa beta_p beta_q) and in v, so every partial
// is one more contraction of the same loaded values; the limits s0, s1 = (knot - x) / beta of the
// piece pass theirs on to the axis that crosses.  About 300 FP64 operations a piece, where the same
// derivatives by six dual-number evaluations of the push took 13.6 ms a sweep at 32^3 with 524,288
// particles.

template <int FROM>
__global__ void __launch_bounds__(ChunkLarge::THREADS_, 4) k_adj_derivs(AdjParams ap, const double* __restrict__ xi,
                                                           const double* __restrict__ v,
                                                           const double* __restrict__ vstar,
                                                           const double* __restrict__ table,
                                                           const double* __restrict__ ctab,
                                                           const double* __restrict__ lJ,
                                                           const double* __restrict__ lam_P,
                                                           const double* __restrict__ lam_v,
                                                           const double* __restrict__ lam_xe,
                                                           const double* __restrict__ mu,
                                                           const uint8_t* __restrict__ slide,
                                                           double* __restrict__ lam_xi, double* __restrict__ gout,
                                                           double* __restrict__ lvn, double* __restrict__ lPn,
                                                           int* __restrict__ status) {
    __shared__ ChunkLarge co;
    const StepParams& p = ap.p;
    const int64_t np = p.np, N = p.m.ncell, nchunks = (np + ChunkLarge::SIZE - 1) / ChunkLarge::SIZE;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * ChunkLarge::SIZE;
        chunk_exchange(p, co, base, [&](int64_t j, double x0[3], double v2[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + j];
                v2[a] = vstar[a * np + j] + v[a * np + j];
            }
        });
#pragma unroll 1
        for (int item = 0; item < 2; ++item) {
            CellStart<double> st;
            double vs[3];
            const int64_t i = co.take(item, base, st, vs);
            if (i >= np) continue;
            const uint8_t sb = slide[i];
            double beta[3], f[3], ng[3], xbar[3], bbar[3], vbar[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double lP1, lAe, lg, lF;
                out_adjoints(p, (sb >> a) & 1u, lam_v[a * np + i], lam_P[a * np + i], mu[a * np + i], lP1, lAe, lg, lF);
                beta[a] = p.cb[a] * vs[a];
                f[a] = lF * p.ihs[a];
                ng[a] = -lg;              // the table holds -grad phi
                xbar[a] = bbar[a] = vbar[a] = 0.0;
            }
            PieceWalk<double> wk(st, beta, p.m);
            int axis = -1;                // the axis of the crossing that opened the piece
            double pend = 0.0;            // what the piece before it passed on to that crossing's s
            for (int it = 0; it < MAX_SEGMENTS; ++it) {
                const double s0 = wk.s0, s1 = wk.upcoming();
                double s1bar = 0.0;
                if (less_pos(s0, s1)) {
                    const double h = s1 - s0, sm = 0.5 * (s0 + s1), nms = sm - 1.0;
                    double m[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) m[a] = wk.fd[a] + sm * beta[a];
                    const PieceMoments<double> q = piece_moments(h, m, beta);
                    // abar_k and cbar_k
                    double ab[8], cb[8];
                    ab[1] = f[0];
                    ab[2] = f[1];
                    ab[4] = f[2];
                    ab[3] = f[0] * m[1] + f[1] * m[0];
                    ab[5] = f[0] * m[2] + f[2] * m[0];
                    ab[6] = f[1] * m[2] + f[2] * m[1];
                    ab[7] = f[0] * q.Pyz + f[1] * q.Pxz + f[2] * q.Pxy;
                    cb[1] = cb[2] = cb[4] = 0.0;
                    cb[3] = f[0] * q.e[1] + f[1] * q.e[0];
                    cb[5] = f[0] * q.e[2] + f[2] * q.e[0];
                    cb[6] = f[1] * q.e[2] + f[2] * q.e[1];
                    cb[7] = f[0] * (m[1] * q.e[2] + m[2] * q.e[1]) + f[1] * (m[0] * q.e[2] + m[2] * q.e[0]) +
                            f[2] * (m[0] * q.e[1] + m[1] * q.e[0]);
                    double K[8], vb[3], X = 0.0, smx = 0.0, eb[3];
                    // the adjoint of J: contracted with q v / dV per node, then to mixed differences
                    {
                        double W[8];
                        int64_t g[8];
                        node_weights(q, W);
                        cell_nodes8(wk.c, p.m, g);
                        double w[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            w[a] = p.q_dV_half * vs[a];
                            vb[a] = 0.0;
                        }
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const double l0 = lJ[g[k]], l1 = lJ[N + g[k]], l2 = lJ[2 * N + g[k]];
                            K[k] = w[0] * l0 + w[1] * l1 + w[2] * l2;
                            vb[0] += W[k] * l0;
                            vb[1] += W[k] * l1;
                            vb[2] += W[k] * l2;
                        }
#pragma unroll
                        for (int a = 0; a < 3; ++a) vb[a] *= p.q_dV_half;
#pragma unroll
                        for (int bit = 1; bit < 8; bit <<= 1)
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                if (k & bit) K[k] -= K[k ^ bit];
                    }
                    const FieldLoad<FROM> ld({table, ctab}, wk.c, p.m);
                    double a3 = 0.0, a5 = 0.0, a6 = 0.0, a7 = 0.0, c3 = 0.0, c5 = 0.0, c6 = 0.0, c7 = 0.0;
#pragma unroll
                    for (int pr = 0; pr < 4; ++pr) {
                        double C[3][2], A[3][2], G[3][2];
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            ld(pr, c, A[c][0], A[c][1]);
                            ld(pr, 3 + c, C[c][0], C[c][1]);
                            ld(pr, 6 + c, G[c][0], G[c][1]);
                        }
#pragma unroll
                        for (int o = 0; o < 2; ++o) {
                            const int k = 2 * pr + o;
                            K[k] += ng[0] * G[0][o] + ng[1] * G[1][o] + ng[2] * G[2][o];
                            if (k == 0) continue;
                            const double cc = C[0][o] * vs[0] + C[1][o] * vs[1] + C[2][o] * vs[2];
                            const double aa = A[0][o] * vs[0] + A[1][o] * vs[1] + A[2][o] * vs[2] + nms * cc;
                            const double t = nms * ab[k] + cb[k];
#pragma unroll
                            for (int c = 0; c < 3; ++c) vb[c] += ab[k] * A[c][o] + t * C[c][o];
                            smx += ab[k] * cc;
                            X += aa * ab[k] + cc * cb[k];
                            if (k == 3) a3 = aa, c3 = cc;
                            if (k == 5) a5 = aa, c5 = cc;
                            if (k == 6) a6 = aa, c6 = cc;
                            if (k == 7) a7 = aa, c7 = cc;
                        }
                    }
                    X += K[0] + K[1] * m[0] + K[2] * m[1] + K[3] * q.Pxy + K[4] * m[2] + K[5] * q.Pxz + K[6] * q.Pyz +
                         K[7] * q.S;
                    // what F adds to the coefficients of the moments
                    K[1] += f[1] * a3 + f[2] * a5;
                    K[2] += f[0] * a3 + f[2] * a6;
                    K[4] += f[0] * a5 + f[1] * a6;
                    K[3] += f[2] * a7;
                    K[5] += f[1] * a7;
                    K[6] += f[0] * a7;
                    const double mb[3] = {K[1] + K[3] * m[1] + K[5] * m[2] + K[7] * q.Pyz + c7 * cb[6],
                                          K[2] + K[3] * m[0] + K[6] * m[2] + K[7] * q.Pxz + c7 * cb[5],
                                          K[4] + K[5] * m[0] + K[6] * m[1] + K[7] * q.Pxy + c7 * cb[3]};
                    eb[0] = c3 * f[1] + c5 * f[2] + c7 * ab[6];
                    eb[1] = c3 * f[0] + c6 * f[2] + c7 * ab[5];
                    eb[2] = c5 * f[0] + c6 * f[1] + c7 * ab[3];
                    const double kxy = K[3] + K[7] * m[2], kxz = K[5] + K[7] * m[1], kyz = K[6] + K[7] * m[0];
                    const double t[3] = {eb[0] + kxy * beta[1] + kxz * beta[2], eb[1] + kxy * beta[0] + kyz * beta[2],
                                         eb[2] + kxz * beta[0] + kyz * beta[1]};
                    const double h2 = h * h, kap = h2 * (1.0 / 12.0);
                    double kb = 0.0, mbb = 0.0;   // adjoint of kappa; mb . beta
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        kb += 0.5 * beta[a] * (eb[a] + t[a]);
                        mbb += mb[a] * beta[a];
                        xbar[a] += h * mb[a];
                        bbar[a] += h * (sm * mb[a] + kap * t[a]);
                        vbar[a] += h * vb[a];
                    }
                    const double hbar = X + h2 * (1.0 / 6.0) * kb, half = 0.5 * h * (smx + mbb);
                    s1bar = half + hbar;
                    const double sbar = pend + (half - hbar);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a == axis) {
                            const double r = sbar / beta[a];
                            xbar[a] -= r;
                            bbar[a] -= r * s0;
                        }
                } else {
                    s1bar = pend;   // a second axis at the same breakpoint
                }
                if (same_bits(s1, 1.0)) break;
                pend = s1bar;
#pragma unroll
                for (int a = 2; a >= 0; --a)
                    if (same_bits(wk.sn[a], s1)) axis = a;
                wk.cross(s1, beta, p.m);
            }
            // the end point: A_h^{n+1}(x + beta) and x + beta themselves
            double g[3], lP1[3];
            {
                double lAe[3], KA[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    double lg, lF;
                    out_adjoints(p, (sb >> a) & 1u, lam_v[a * np + i], lam_P[a * np + i], mu[a * np + i], lP1[a],
                                 lAe[a], lg, lF);
                }
                const FieldLoad<FROM> ld({table, ctab}, wk.c, p.m);
#pragma unroll
                for (int pr = 0; pr < 4; ++pr)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        double e0, e1;
                        ld(pr, c, e0, e1);
                        KA[2 * pr] += lAe[c] * e0;
                        KA[2 * pr + 1] += lAe[c] * e1;
                    }
                const double x = wk.te[0], y = wk.te[1], z = wk.te[2];
                const double r[3] = {KA[1] + KA[3] * y + z * (KA[5] + KA[7] * y),
                                     KA[2] + KA[3] * x + z * (KA[6] + KA[7] * x),
                                     KA[4] + KA[5] * x + y * (KA[6] + KA[7] * x)};
                bool ok = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double e = r[a] + lam_xe[a * np + i];
                    xbar[a] += e;
                    g[a] = p.cb[a] * (bbar[a] + e) + vbar[a];   // the orbit's adjoint of v*_a, also of v^n_a
                    ok = ok && isfinite(xbar[a]) && isfinite(g[a]);
                }
                if (!ok) atomicOr(status, DEV_ERR_NONFINITE);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if ((sb >> a) & 1u) {
                    // nu_a: the direct adjoint of v*_a (its velocity and momentum outputs) plus the
                    // orbit's; v*_a = 2 d_a H_a / dt - v^n_a with d_a = knot - xi_a
                    const double nu = lam_v[a * np + i] + p.mass * lam_P[a * np + i] + g[a];
                    lam_xi[a * np + i] = xbar[a] - nu * 2.0 * p.H[a] / p.dt;
                    lvn[a * np + i] = g[a] - nu;
                    lPn[a * np + i] = 0.0;
                    gout[a * np + i] = 0.0;                  // no fixed-point equation: mu_a = 0
                } else {
                    lam_xi[a * np + i] = xbar[a];
                    lvn[a * np + i] = g[a];
                    lPn[a * np + i] = lP1[a];
                    gout[a * np + i] = g[a];
                }
            }
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
}

// The blocks B = dG_i/dv*_i (9, row-major) of the transposed solve's preconditioner for the particles
// that the step solved locally, by dual numbers along the three displacements; the caller zeroes the
// others'.  They depend on the step alone, so once per solve.  Each block lists its share's few such
// particles first, so that its warps work on full ones.
constexpr int BLOCKS_SPAN = 4096;

__global__ void __launch_bounds__(THREADS) k_adj_blocks(AdjParams ap, const double* __restrict__ xi,
                                                        const double* __restrict__ v, const double* __restrict__ vstar,
                                                        const double* __restrict__ table,
                                                        const uint8_t* __restrict__ slide, double* __restrict__ Bout) {
    __shared__ int list[BLOCKS_SPAN];
    __shared__ int count;
    const StepParams& p = ap.p;
    const int64_t np = p.np, nspans = (np + BLOCKS_SPAN - 1) / BLOCKS_SPAN;
    for (int64_t sp = blockIdx.x; sp < nspans; sp += gridDim.x) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        for (int k = threadIdx.x; k < BLOCKS_SPAN && sp * BLOCKS_SPAN + k < np; k += blockDim.x)
            if (slide[sp * BLOCKS_SPAN + k] & SLIDE_CREPT) list[atomicAdd(&count, 1)] = k;
        __syncthreads();
        for (int t = threadIdx.x; t < 3 * count; t += blockDim.x) {
            const int64_t i = sp * BLOCKS_SPAN + list[t / 3];
            const int d = t % 3;
            const uint8_t sb = slide[i];
            Dual x0[3], beta[3], vb[3], gphi[3], F[3], xe[3], Ae[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = Dual(xi[a * np + i], 0.0);
                beta[a] = Dual(p.dt * 0.5 * (vstar[a * np + i] + v[a * np + i]) * p.invH[a], a == d ? 1.0 : 0.0);
                vb[a] = beta[a] * Dual(p.H[a] / p.dt);
            }
            for_each_segment(x0, beta, true,
                             [&](const Segment<Dual>& sg) { push_piece_t(p, sg, beta, vb, table, gphi, F); });
#pragma unroll
            for (int a = 0; a < 3; ++a) xe[a] = wrap_t(x0[a] + beta[a], (double)p.m.n[a]);
            point_A1_t(p, xe, table, Ae);
            const double c = d == 0 ? p.cb[0] : (d == 1 ? p.cb[1] : p.cb[2]);   // d beta_d / d v*_d
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                // v1 = (P + dt q (-gphibar + F) - q A_end) / m; sliding components have no equation
                const double dv1 = (p.dtq * (F[a].d - gphi[a].d) - p.q * Ae[a].d) * p.inv_mass;
                const bool drop = ((sb >> a) & 1u) || ((sb >> d) & 1u);
                Bout[(3 * a + d) * np + i] = drop ? 0.0 : c * dv1;
            }
        }
        __syncthreads();   // the list is rewritten by the next span
    }
}

// x = (I - B^T)^{-1} r for particle i's 3 x 3 block (Cramer's rule); false if singular.
__device__ __forceinline__ bool solve_block(const double* __restrict__ B, int64_t np, int64_t i, const double r[3],
                                            double x[3]) {
    double M[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int d = 0; d < 3; ++d) M[a][d] = (a == d ? 1.0 : 0.0) - B[(3 * d + a) * np + i];   // (B^T)[a][d] = B[d][a]
    const double det = M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) -
                       M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
                       M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
    if (!(fabs(det) > 1e-300)) {
        x[0] = x[1] = x[2] = 0.0;
        return false;
    }
#pragma unroll
    for (int col = 0; col < 3; ++col) {
        double Mc[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int d = 0; d < 3; ++d) Mc[a][d] = d == col ? r[a] : M[a][d];
        const double dc = Mc[0][0] * (Mc[1][1] * Mc[2][2] - Mc[1][2] * Mc[2][1]) -
                          Mc[0][1] * (Mc[1][0] * Mc[2][2] - Mc[1][2] * Mc[2][0]) +
                          Mc[0][2] * (Mc[1][0] * Mc[2][1] - Mc[1][1] * Mc[2][0]);
        x[col] = dc / det;
    }
    return true;
}

// The preconditioner of the transposed solve, z = P r: per particle (I - B^T)^{-1} r, with B
// zero outside the particles the step solved locally (there P = I).
__global__ void k_adj_precond(int64_t np, const double* __restrict__ B, const double* __restrict__ r,
                              double* __restrict__ z, int* __restrict__ status) {
    ADJ_LOOP(i, np) {
        double ri[3], x[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) ri[a] = r[a * np + i];
        if (!solve_block(B, np, i, ri, x)) atomicOr(status, DEV_ERR_NONFINITE);
#pragma unroll
        for (int a = 0; a < 3; ++a) z[a * np + i] = x[a];
    }
}

// w = z - (g - b0): the transposed fixed point's operator (I - K) applied to z, g = K z + b0
// being the sweep's output at mu = z.
__global__ void k_adj_apply(int64_t n, const double* __restrict__ z, const double* __restrict__ g,
                            const double* __restrict__ b0, double* __restrict__ w) {
    ADJ_LOOP(i, n) w[i] = z[i] - g[i] + b0[i];
}

// part[k * gridDim.x + b] = block b's share of w . V_k, k < nv (V_k at V + k ldv).
__global__ void k_adj_mdot(int64_t n, const double* __restrict__ w, const double* __restrict__ V, int64_t ldv, int nv,
                           double* __restrict__ part) {
    __shared__ double sm[32];
    for (int k = 0; k < nv; ++k) {
        double s = 0.0;
        const double* vk = V + k * ldv;
        ADJ_LOOP(i, n) s += w[i] * vk[i];
        s = block_sum(s, sm);
        if (threadIdx.x == 0) part[k * gridDim.x + blockIdx.x] = s;
    }
}

// out[k] = sum over the nb block shares of dot k, in a fixed order (one block per dot).
__global__ void k_adj_mdot_final(const double* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ double sm[32];
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += part[blockIdx.x * nb + b];
    s = block_sum(s, sm);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// w += sign * sum_k h[k] V_k, k < nv (h on the device).
__global__ void k_adj_combine(int64_t n, double* __restrict__ w, const double* __restrict__ V, int64_t ldv, int nv,
                              const double* __restrict__ h, double sign) {
    ADJ_LOOP(i, n) {
        double s = 0.0;
        for (int k = 0; k < nv; ++k) s += h[k] * V[k * ldv + i];
        w[i] += sign * s;
    }
}

// Elementwise helpers.
__global__ void k_adj_axpy(int64_t n, double* __restrict__ y, const double* __restrict__ x, double s) {
    ADJ_LOOP(i, n) y[i] += s * x[i];
}

// ---- the initial data: rho^0 = sum q S(x)/dV, phi^0 from Poisson, P^0 = m v^0 ------------------
//
// lam_xi_i += (q/dV) sum_g dS_g/dxi (x_i) lam_dep[g] (the point deposit transposed).
__global__ void k_adj_deposit(AdjParams ap, const double* __restrict__ xi, const double* __restrict__ lam_dep,
                              double* __restrict__ lam_xi) {
    const StepParams& p = ap.p;
    const int64_t np = p.np;
    ADJ_LOOP(i, np) {
        double x[3], r[3];
        int c[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            x[a] = xi[a * np + i];
            const double f = ::floor(x[a]);
            c[a] = (int)f;
            r[a] = x[a] - f;
        }
        Segment<double> sd;
        sd.cell[0] = c[0];
        sd.cell[1] = c[1];
        sd.cell[2] = c[2];
        int64_t g[8];
        segment_nodes8(sd, p.m, g);
        double out[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double wx = (k & 1) ? r[0] : 1.0 - r[0], sx = (k & 1) ? 1.0 : -1.0;
            const double wy = (k & 2) ? r[1] : 1.0 - r[1], sy = (k & 2) ? 1.0 : -1.0;
            const double wz = (k & 4) ? r[2] : 1.0 - r[2], sz = (k & 4) ? 1.0 : -1.0;
            const double l = p.q_dV * lam_dep[g[k]];
            out[0] += sx * wy * wz * l;
            out[1] += wx * sy * wz * l;
            out[2] += wx * wy * sz * l;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) lam_xi[a * np + i] += out[a];
    }
}

// The adjoint of W (field energy) with respect to phi, U and A of the current state:
// W = sum (|E|^2 / (2 sigma1) + |B|^2 / (2 sigma2)) dV with E = -grad phi - U, B = curl A.
__global__ void k_energy_grad(AdjParams ap, const double* __restrict__ F, const double* __restrict__ Wf,
                              double* __restrict__ lF, double* __restrict__ lW) {
    const StepParams& p = ap.p;
    const int64_t N = p.m.ncell;
    const double dV = p.H[0] * p.H[1] * p.H[2];
    ADJ_LOOP(g, N) {
        // E at a node and B at a node, as in the energy sum
        auto E = [&](int64_t n, int a) { return -dcen_s(F, 1, n, a, p.m, p.invH) - Wf[(1 + a) * N + n]; };
        auto Bc = [&](int64_t n, int c) {
            const double* Ax = F + N;
            const double* Ay = F + 2 * N;
            const double* Az = F + 3 * N;
            if (c == 0) return dcen_s(Az, 1, n, 1, p.m, p.invH) - dcen_s(Ay, 1, n, 2, p.m, p.invH);
            if (c == 1) return dcen_s(Ax, 1, n, 2, p.m, p.invH) - dcen_s(Az, 1, n, 0, p.m, p.invH);
            return dcen_s(Ay, 1, n, 0, p.m, p.invH) - dcen_s(Ax, 1, n, 1, p.m, p.invH);
        };
        // dW/dphi = -(D^T E) dV / sigma1 = (div E) dV / sigma1 (D_a^T = -D_a), dW/dU = -E dV / sigma1
        double divE = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int64_t pp = a == 0 ? nshift(g, 1, 0, 0, p.m) : (a == 1 ? nshift(g, 0, 1, 0, p.m) : nshift(g, 0, 0, 1, p.m));
            const int64_t qq = a == 0 ? nshift(g, -1, 0, 0, p.m) : (a == 1 ? nshift(g, 0, -1, 0, p.m) : nshift(g, 0, 0, -1, p.m));
            divE += 0.5 * p.invH[a] * (E(pp, a) - E(qq, a));
            lW[(1 + a) * N + g] = -E(g, a) * dV / ap.sigma1;
        }
        lF[g] = divE * dV / ap.sigma1;
        lW[g] = 0.0;
        // dW/dA = curl^T (B) dV / sigma2 = curl(B) dV / sigma2 (curl is symmetric for skew D)
        auto dB = [&](int c, int a) {
            const int64_t pp = a == 0 ? nshift(g, 1, 0, 0, p.m) : (a == 1 ? nshift(g, 0, 1, 0, p.m) : nshift(g, 0, 0, 1, p.m));
            const int64_t qq = a == 0 ? nshift(g, -1, 0, 0, p.m) : (a == 1 ? nshift(g, 0, -1, 0, p.m) : nshift(g, 0, 0, -1, p.m));
            return 0.5 * p.invH[a] * (Bc(pp, c) - Bc(qq, c));
        };
        lF[N + g] = (dB(2, 1) - dB(1, 2)) * dV / ap.sigma2;
        lF[2 * N + g] = (dB(0, 2) - dB(2, 0)) * dV / ap.sigma2;
        lF[3 * N + g] = (dB(1, 0) - dB(0, 1)) * dV / ap.sigma2;
    }
}

}  // namespace

// ---- launchers ---------------------------------------------------------------------------------

int adj_blocks(const Ctx& c, int64_t n) {
    int64_t b = (n + THREADS - 1) / THREADS;
    b = std::min<int64_t>(std::max<int64_t>(b, 1), (int64_t)c.sms * 8);
    return (int)std::min<int64_t>(b, MAX_BLOCKS);
}

bool setup_adjoint_kernels() {
    return cudaFuncSetAttribute(k_adj_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)ChunkLarge::smem()) == cudaSuccess;
}

void launch_adj_scatter(Ctx& c, const double* xi, const double* v, const double* vstar, const double* lam_P,
                        const double* lam_v, const double* mu, double* lam_tab) {
    const int64_t chunks = (c.np + ChunkLarge::SIZE - 1) / ChunkLarge::SIZE;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(chunks, (int64_t)c.sms * 4));
    k_adj_scatter<<<nb, ChunkLarge::THREADS_, ChunkLarge::smem(), c.stream>>>(adj_params(c), xi, v, vstar, lam_P, lam_v,
                                                                           mu, c.slide, lam_tab);
    ++c.launches;
}

void launch_adj_mesh_rhs(Ctx& c, const double* lam_tab, const double* lF1, const double* lW1, double* t, double* pn) {
    k_adj_mesh_rhs<<<adj_blocks(c, c.m.ncell), THREADS, 0, c.stream>>>(adj_params(c), lam_tab, lF1, lW1, t, pn);
    ++c.launches;
}

void launch_adj_mesh_out(Ctx& c, const double* y, const double* pn, const double* lW1, const double* lrho1,
                         double* lF0, double* lW0, double* lrho0, double* lJ) {
    k_adj_mesh_out<<<adj_blocks(c, c.m.ncell), THREADS, 0, c.stream>>>(adj_params(c), y, pn, lW1, lrho1, lF0, lW0,
                                                                        lrho0, lJ);
    ++c.launches;
}

void launch_adj_derivs(Ctx& c, const double* xi, const double* v, const double* vstar, const double* lJ,
                       const double* lam_P, const double* lam_v, const double* lam_xe, const double* mu,
                       double* lam_xi, double* g, double* lvn, double* lPn) {
    const int nb = adj_blocks(c, c.np);
#define PIC_DERIVS(T)                                                                                            \
    k_adj_derivs<T><<<nb, ChunkLarge::THREADS_, 0, c.stream>>>(adj_params(c), xi, v, vstar, c.table, c.ctab, lJ, lam_P, \
                                                               lam_v, lam_xe, mu, c.slide, lam_xi, g, lvn, lPn,    \
                                                               c.dev_status)
    if (c.ctab) PIC_DERIVS(FROM_CELLS);
    else PIC_DERIVS(FROM_NODES);
#undef PIC_DERIVS
    ++c.launches;
}

void launch_adj_block_rows(Ctx& c, const double* xi, const double* v, const double* vstar, double* B) {
    cudaMemsetAsync(B, 0, sizeof(double) * 9 * c.np, c.stream);
    const int64_t spans = (c.np + BLOCKS_SPAN - 1) / BLOCKS_SPAN;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(spans, (int64_t)c.sms * 2));
    k_adj_blocks<<<nb, THREADS, 0, c.stream>>>(adj_params(c), xi, v, vstar, c.table, c.slide, B);
    ++c.launches;
}

void launch_adj_precond(Ctx& c, const double* B, const double* r, double* z) {
    k_adj_precond<<<adj_blocks(c, c.np), THREADS, 0, c.stream>>>(c.np, B, r, z, c.dev_status);
    ++c.launches;
}

void launch_adj_apply(Ctx& c, int64_t n, const double* z, const double* g, const double* b0, double* w) {
    k_adj_apply<<<adj_blocks(c, n), THREADS, 0, c.stream>>>(n, z, g, b0, w);
    ++c.launches;
}

void launch_adj_mdot(Ctx& c, int64_t n, const double* w, const double* V, int64_t ldv, int nv, double* part,
                     double* out) {
    const int nb = adj_blocks(c, n);
    k_adj_mdot<<<nb, THREADS, 0, c.stream>>>(n, w, V, ldv, nv, part);
    k_adj_mdot_final<<<nv, THREADS, 0, c.stream>>>(part, nb, out);
    c.launches += 2;
}

void launch_adj_combine(Ctx& c, int64_t n, double* w, const double* V, int64_t ldv, int nv, const double* h,
                        double sign) {
    k_adj_combine<<<adj_blocks(c, n), THREADS, 0, c.stream>>>(n, w, V, ldv, nv, h, sign);
    ++c.launches;
}

void launch_adj_axpy(Ctx& c, int64_t n, double* y, const double* x, double s) {
    k_adj_axpy<<<adj_blocks(c, n), THREADS, 0, c.stream>>>(n, y, x, s);
    ++c.launches;
}

void launch_adj_deposit(Ctx& c, const double* xi, const double* lam_dep, double* lam_xi) {
    k_adj_deposit<<<adj_blocks(c, c.np), THREADS, 0, c.stream>>>(adj_params(c), xi, lam_dep, lam_xi);
    ++c.launches;
}

void launch_energy_grad(Ctx& c, double* lF, double* lW) {
    k_energy_grad<<<adj_blocks(c, c.m.ncell), THREADS, 0, c.stream>>>(adj_params(c), c.F0, c.W0, lF, lW);
    ++c.launches;
}

}  // namespace pic
