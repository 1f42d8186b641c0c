// Particle kernels of the orbit-averaged PIC step (FP64, sm_103a).
//
// Particles in structure-of-arrays layout (component c of particle i at c * np + i), cell-sorted
// so that neighbouring threads gather the same mesh nodes.  The closed forms take one particle per thread
// from chunks ordered by piece count (chunk.cuh) and the mesh fields from the cell tables (orbit_cell.cuh);
// the Gauss rules, and the closed forms without cell tables, take them from a per-node table of 12 doubles:
// A^n (3), A^{n+1,p} (3), grad_h phi^{n+1/2,p} (3), U^{n+1/2,p} (3).
#include <algorithm>
#include <cmath>

#include "pic_internal.h"
#include "particle_common.cuh"
#include "orbit_cell.cuh"
#include "chunk.cuh"
#include "orbit_fixed.cuh"

namespace pic {

// The Gauss--Legendre rules of 1 .. 16 points on [0, 1], rule nq at nq (nq - 1) / 2 (a place for each,
// so that contexts of different rules do not share one).
constexpr int GAUSS_MAX = 16;
__constant__ double c_gauss_t[GAUSS_MAX * (GAUSS_MAX + 1) / 2];
__constant__ double c_gauss_w[GAUSS_MAX * (GAUSS_MAX + 1) / 2];

// Nodes by Newton's method on the Legendre polynomial P_nq (three-term recurrence), weights
// 1 / ((1 - x^2) P'(x)^2) mapped from [-1, 1].
void set_gauss_rule(int nq) {
    double t[GAUSS_MAX] = {0}, w[GAUSS_MAX] = {0};
    for (int k = 0; k < nq; ++k) {
        double x = std::cos(M_PI * (k + 0.75) / (nq + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int j = 2; j <= nq; ++j) {
                double p2 = ((2.0 * j - 1.0) * x * p1 - (j - 1.0) * p0) / j;
                p0 = p1;
                p1 = p2;
            }
            double pn = nq == 0 ? 1.0 : (nq == 1 ? x : p1);
            double pm = nq == 1 ? 1.0 : p0;
            dp = nq * (x * pn - pm) / (x * x - 1.0);
            double dx = pn / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-17) break;
        }
        t[k] = 0.5 * (1.0 - x);
        w[k] = 1.0 / ((1.0 - x * x) * dp * dp);  // = 0.5 * 2 / ((1 - x^2) P'^2)
    }
    const size_t at = sizeof(double) * (size_t)(nq * (nq - 1) / 2);
    cudaMemcpyToSymbol(c_gauss_t, t, sizeof(double) * nq, at);
    cudaMemcpyToSymbol(c_gauss_w, w, sizeof(double) * nq, at);
}

namespace {


// ---- orbit current scatter (Eq. (orbit-current)) -------------------------------------

// Same with an n_q-point Gauss rule on the whole path (unsplit).
__device__ __forceinline__ int scatter_gauss(const StepParams& p, const double x0[3], const double beta[3],
                                             const double w[3], double* __restrict__ J) {
    const int64_t N = p.m.ncell;
    return for_each_segment(x0, beta, false, [&](const Segment<double>& sg) {
        for (int qd = 0; qd < p.nq; ++qd) {
            double s = sg.s0 + sg.h * c_gauss_t[p.rule + qd];
            double wq = sg.h * c_gauss_w[p.rule + qd];
            double xq[3] = {x0[0] + s * beta[0], x0[1] + s * beta[1], x0[2] + s * beta[2]};
            int64_t g[8];
            double S[8];
            point_weights8(xq, p.m, g, S);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                double f = wq * S[k];
                if (p.det) {
                    exact_add(p.acc, g[k], w[0] * f);
                    exact_add(p.acc, N + g[k], w[1] * f);
                    exact_add(p.acc, 2 * N + g[k], w[2] * f);
                } else {
                    atomicAdd(J + g[k], w[0] * f);
                    atomicAdd(J + N + g[k], w[1] * f);
                    atomicAdd(J + 2 * N + g[k], w[2] * f);
                }
            }
        }
    });
}

// ---- shapes of degree R = 2, 3 (§4.7) ---------------------------------------------------
//
// One axis of the tensor-product B-spline of degree R at x (cell units): the R + 1 non-zero
// values, their x-derivatives and the first node.  The nodes sit at the integers, the knots
// at the integers (odd R) or the half-integers (even R); on the knot interval holding x, in
// its local coordinate t in [0, 1), the centred cardinal B-spline's pieces are
//   R = 2:  (1 - t)^2 / 2,  1/2 + t (1 - t),  t^2 / 2;
//   R = 3:  (1 - t)^3 / 6,  (3 t^3 - 6 t^2 + 4) / 6,  (-3 t^3 + 3 t^2 + 3 t + 1) / 6,  t^3 / 6.
template <int R>
struct Basis1 {
    double w[R + 1], dw[R + 1];
    int first;
};

template <int R>
__device__ __forceinline__ void basis1(double x, double invH, Basis1<R>& b) {
    const double xs = (R % 2 == 0) ? x - 0.5 : x;
    const double f = floor(xs), t = xs - f, u = 1.0 - t;
    b.first = (int)f - (R - 1) / 2;
    if constexpr (R == 2) {
        b.w[0] = 0.5 * u * u;
        b.w[1] = 0.5 + t * u;
        b.w[2] = 0.5 * t * t;
        b.dw[0] = -u * invH;
        b.dw[1] = (u - t) * invH;
        b.dw[2] = t * invH;
    } else {
        const double t2 = t * t, t3 = t2 * t;
        b.w[0] = u * u * u * (1.0 / 6.0);
        b.w[1] = (3.0 * t3 - 6.0 * t2 + 4.0) * (1.0 / 6.0);
        b.w[2] = (-3.0 * t3 + 3.0 * t2 + 3.0 * t + 1.0) * (1.0 / 6.0);
        b.w[3] = t3 * (1.0 / 6.0);
        b.dw[0] = -0.5 * u * u * invH;
        b.dw[1] = (1.5 * t2 - 2.0 * t) * invH;
        b.dw[2] = (-1.5 * t2 + t + 0.5) * invH;
        b.dw[3] = 0.5 * t2 * invH;
    }
}

template <int R>
__device__ __forceinline__ void basis3(const StepParams& p, const double x[3], Basis1<R> b[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) basis1<R>(x[a], p.invH[a], b[a]);
}

// Visit the (R + 1)^3 nodes of the shape at a point: f(node row, S_g, grad S_g).
template <int R, typename F>
__device__ __forceinline__ void for_each_node(const StepParams& p, const Basis1<R> b[3], F&& f) {
    for (int iz = 0; iz <= R; ++iz) {
        const int gz = wrapi(b[2].first + iz, p.m.n[2]);
        for (int iy = 0; iy <= R; ++iy) {
            const int gy = wrapi(b[1].first + iy, p.m.n[1]);
            const double wyz = b[1].w[iy] * b[2].w[iz];
            const double dy = b[1].dw[iy] * b[2].w[iz], dz = b[1].w[iy] * b[2].dw[iz];
#pragma unroll
            for (int ix = 0; ix <= R; ++ix) {
                const int gx = wrapi(b[0].first + ix, p.m.n[0]);
                const double wx = b[0].w[ix];
                const double dS[3] = {b[0].dw[ix] * wyz, wx * dy, wx * dz};
                f(node_index(gx, gy, gz, p.m), wx * wyz, dS);
            }
        }
    }
}

// The orbit current of the degree-R shape with an n_q-point Gauss rule on the whole path (unsplit).
template <int R>
__device__ __forceinline__ int scatter_gauss_r(const StepParams& p, const double x0[3], const double beta[3],
                                               const double w[3], double* __restrict__ J) {
    const int64_t N = p.m.ncell;
    return for_each_segment(x0, beta, false, [&](const Segment<double>& sg) {
        for (int qd = 0; qd < p.nq; ++qd) {
            const double s = sg.s0 + sg.h * c_gauss_t[p.rule + qd];
            const double wq = sg.h * c_gauss_w[p.rule + qd];
            const double xq[3] = {x0[0] + s * beta[0], x0[1] + s * beta[1], x0[2] + s * beta[2]};
            Basis1<R> b[3];
            basis3<R>(p, xq, b);
            for_each_node<R>(p, b, [&](int64_t g, double S, const double*) {
                const double f = wq * S;
                if (p.det) {
                    exact_add(p.acc, g, w[0] * f);
                    exact_add(p.acc, N + g, w[1] * f);
                    exact_add(p.acc, 2 * N + g, w[2] * f);
                } else {
                    atomicAdd(J + g, w[0] * f);
                    atomicAdd(J + N + g, w[1] * f);
                    atomicAdd(J + 2 * N + g, w[2] * f);
                }
            });
        }
    });
}

// ---- pieces of split orbits with a Gauss rule, any degree ----------------------------------
//
// On a piece between the knots of the degree-R shape the stencil does not change, so the rule's nq
// points share its (R + 1)^3 nodes: each node is loaded and contracted with v once per piece, and
// the points are summed in the tensor product's order (rows of R + 1 nodes along x, then y and z),
// which takes 18 operations per row and point at R = 2 where the pointwise form took 20 per node
// and point.  Bound by the FP64 pipe; measured at R = 2, nq = 4 with 442,368 particles (36 x 32 x 24):
// iterate 4.91 -> 2.32 ms, first scatter 1.35 -> 0.55 ms (a quarter of the L2 reductions).

// The start on the knot lattice of the shape (knots at the integers or half-integers).
__device__ __forceinline__ void knot_start(const StepParams& p, const double x0[3], CellStart<double>& st) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double xs = x0[a] - p.koff, fl = floor(xs);
        st.f[a] = xs - fl;
        const int c = (int)fl;
        st.c[a] = c < 0 ? p.m.n[a] - 1 : min(c, p.m.n[a] - 1);
    }
}

// Values and derivatives (per cell) of the R + 1 splines at coordinate t of their knot interval.
template <int R>
__device__ __forceinline__ void splines(double t, double w[R + 1], double d[R + 1]) {
    const double u = 1.0 - t;
    if constexpr (R == 1) {
        w[0] = u;
        w[1] = t;
        d[0] = -1.0;
        d[1] = 1.0;
    } else if constexpr (R == 2) {
        w[0] = 0.5 * u * u;
        w[1] = 0.5 + t * u;
        w[2] = 0.5 * t * t;
        d[0] = -u;
        d[1] = u - t;
        d[2] = t;
    } else {
        const double t2 = t * t, u2 = u * u;
        w[0] = u2 * u * (1.0 / 6.0);
        w[1] = (3.0 * t - 6.0) * t2 * (1.0 / 6.0) + 4.0 / 6.0;
        w[2] = (3.0 * u - 6.0) * u2 * (1.0 / 6.0) + 4.0 / 6.0;
        w[3] = t2 * t * (1.0 / 6.0);
        d[0] = -0.5 * u2;
        d[1] = 1.5 * t2 - 2.0 * t;
        d[2] = 2.0 * u - 1.5 * u2;
        d[3] = 0.5 * t2;
    }
}

// A piece's splines at its points: per point and axis the values and derivatives, those of z times
// the point's weight (points in local memory, read back through L1).  A split orbit's rule has at
// most the points that integrate the degree exactly (setup_geometry).
template <int R>
struct PiecePoints {
    static constexpr int MAX = (3 * R + 2) / 2;
    double w[MAX][3][R + 1], d[MAX][3][R + 1];

    __device__ __forceinline__ PiecePoints(const StepParams& p, double h, const double mid[3], const double beta[3],
                                           bool derivs) {
        for (int q = 0; q < p.nq; ++q) {
            const double hu = h * (c_gauss_t[p.rule + q] - 0.5), wq = c_gauss_w[p.rule + q];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double v[R + 1], e[R + 1];
                splines<R>(mid[a] + hu * beta[a], v, e);
#pragma unroll
                for (int k = 0; k <= R; ++k) {
                    w[q][a][k] = a == 2 ? wq * v[k] : v[k];
                    if (derivs) d[q][a][k] = a == 2 ? wq * e[k] : e[k];
                }
            }
        }
    }
};

// The stencil's first node per axis, and node rows along x.
template <int R>
struct Stencil {
    int x[R + 1], first[3];
    __device__ __forceinline__ Stencil(const int c[3], const MeshDims& m) {
#pragma unroll
        for (int a = 0; a < 3; ++a) first[a] = wrapi(c[a] - (R - 1) / 2, m.n[a]);
        x[0] = first[0];
#pragma unroll
        for (int k = 1; k <= R; ++k) x[k] = next_cell(x[k - 1], m.n[0]);
    }
    // Index of the row of nodes (., ky, kz).
    __device__ __forceinline__ int64_t row(int ky, int kz, const MeshDims& m) const {
        return (int64_t)m.n[0] * ((int64_t)wrapi(first[1] + ky, m.n[1]) + (int64_t)m.n[1] * wrapi(first[2] + kz, m.n[2]));
    }
};

// J_c[g] += w_c Sbar of the orbit's pieces.
// Rows part, part + parts, ... of the stencil only (k_local shares a particle among lanes).
template <int R>
__device__ __forceinline__ int scatter_pieces(const StepParams& p, const double x0[3], const double beta[3],
                                              const double w[3], double* __restrict__ J, int part = 0, int parts = 1) {
    const int64_t N = p.m.ncell;
    CellStart<double> st;
    knot_start(p, x0, st);
    return for_each_piece(st, beta, p.m, [&](double h, double, const double mid[3], const int c[3]) {
        const PiecePoints<R> pt(p, h, mid, beta, false);
        const Stencil<R> sl(c, p.m);
        const double wh[3] = {h * w[0], h * w[1], h * w[2]};
        for (int r = part; r < (R + 1) * (R + 1); r += parts) {
            const int kz = r / (R + 1), ky = r - kz * (R + 1);
            const int64_t row = sl.row(ky, kz, p.m);
            double M[R + 1];
#pragma unroll
            for (int k = 0; k <= R; ++k) M[k] = 0.0;
            for (int q = 0; q < p.nq; ++q) {
                const double wyz = pt.w[q][1][ky] * pt.w[q][2][kz];
#pragma unroll
                for (int k = 0; k <= R; ++k) M[k] += wyz * pt.w[q][0][k];
            }
#pragma unroll
            for (int k = 0; k <= R; ++k) {
                const int64_t g = row + sl.x[k];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (p.det) exact_add(p.acc, a * N + g, wh[a] * M[k]);
                    else atomicAdd(J + a * N + g, wh[a] * M[k]);
                }
            }
        }
    });
}

__device__ __forceinline__ int scatter_orbit(const StepParams& p, const double x0[3], const double beta[3],
                                             const double w[3], double* J) {
    if (p.split) {
        if (p.order == 2) return scatter_pieces<2>(p, x0, beta, w, J);
        if (p.order == 3) return scatter_pieces<3>(p, x0, beta, w, J);
        return scatter_pieces<1>(p, x0, beta, w, J);
    }
    if (p.order == 2) return scatter_gauss_r<2>(p, x0, beta, w, J);
    if (p.order == 3) return scatter_gauss_r<3>(p, x0, beta, w, J);
    return scatter_gauss(p, x0, beta, w, J);
}

// ---- push (Eq. (orbit-push)) -------------------------------------------------------

struct PushAcc {
    double gphi[3];   // orbit gather of grad_h phi^{n+1/2} (Eq. (gphibar-definition))
    double F[3];      // (D_i A)^T vbar (Eq. (DA-def), Appendix B)
    double Ubar[3];   // orbit gather of U^{n+1/2} (Eq. (Ubar-def)), diagnostics only
    double DAv[3];    // (D_i A) vbar, diagnostics only
    double pu;        // sum_g Sbar_ig, diagnostics only
};

template <bool DIAG>
__device__ __forceinline__ void push_piece_gauss(const StepParams& p, const Segment<double>& sg, const double x0[3],
                                                 const double beta[3], const double vb[3],
                                                 const double* __restrict__ table, PushAcc& acc) {
    for (int qd = 0; qd < p.nq; ++qd) {
        const double s = sg.s0 + sg.h * c_gauss_t[p.rule + qd];
        const double wq = sg.h * c_gauss_w[p.rule + qd];
        double xq[3] = {x0[0] + s * beta[0], x0[1] + s * beta[1], x0[2] + s * beta[2]};
        int c[3];
        double r[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double f = floor(xq[a]);
            c[a] = (int)f;
            r[a] = xq[a] - f;
        }
        Segment<double> cs;
        cs.cell[0] = c[0];
        cs.cell[1] = c[1];
        cs.cell[2] = c[2];
        int64_t g[8];
        segment_nodes8(cs, p.m, g);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int nx = k & 1, ny = (k >> 1) & 1, nz = (k >> 2) & 1;
            const double wx = nx ? r[0] : 1.0 - r[0], wy = ny ? r[1] : 1.0 - r[1], wz = nz ? r[2] : 1.0 - r[2];
            const double W = wq * wx * wy * wz;
            const double dW[3] = {wq * (nx ? p.invH[0] : -p.invH[0]) * wy * wz,
                                  wq * (ny ? p.invH[1] : -p.invH[1]) * wx * wz,
                                  wq * (nz ? p.invH[2] : -p.invH[2]) * wx * wy};
            const double* t = table + 12 * g[k];
            const double an = t[0] * vb[0] + t[1] * vb[1] + t[2] * vb[2];
            const double a1 = t[3] * vb[0] + t[4] * vb[1] + t[5] * vb[2];
            const double as = (1.0 - s) * an + s * a1;           // A_g(s) . vbar
            acc.gphi[0] += W * t[6];
            acc.gphi[1] += W * t[7];
            acc.gphi[2] += W * t[8];
            acc.F[0] += as * dW[0];
            acc.F[1] += as * dW[1];
            acc.F[2] += as * dW[2];
            if constexpr (DIAG) {
                acc.Ubar[0] += W * t[9];
                acc.Ubar[1] += W * t[10];
                acc.Ubar[2] += W * t[11];
                acc.pu += W;
                const double vdW = vb[0] * dW[0] + vb[1] * dW[1] + vb[2] * dW[2];
#pragma unroll
                for (int l = 0; l < 3; ++l) acc.DAv[l] += ((1.0 - s) * t[l] + s * t[3 + l]) * vdW;
            }
        }
    }
}

// The Gauss-rule piece of push_piece_gauss for the degree-R shape.
template <int R, bool DIAG>
__device__ __forceinline__ void push_piece_gauss_r(const StepParams& p, const Segment<double>& sg, const double x0[3],
                                                   const double beta[3], const double vb[3],
                                                   const double* __restrict__ table, PushAcc& acc) {
    for (int qd = 0; qd < p.nq; ++qd) {
        const double s = sg.s0 + sg.h * c_gauss_t[p.rule + qd];
        const double wq = sg.h * c_gauss_w[p.rule + qd];
        const double xq[3] = {x0[0] + s * beta[0], x0[1] + s * beta[1], x0[2] + s * beta[2]};
        Basis1<R> b[3];
        basis3<R>(p, xq, b);
        for_each_node<R>(p, b, [&](int64_t g, double S, const double* dS) {
            const double W = wq * S;
            const double dW[3] = {wq * dS[0], wq * dS[1], wq * dS[2]};
            const double* t = table + 12 * g;
            const double an = t[0] * vb[0] + t[1] * vb[1] + t[2] * vb[2];
            const double a1 = t[3] * vb[0] + t[4] * vb[1] + t[5] * vb[2];
            const double as = (1.0 - s) * an + s * a1;           // A_g(s) . vbar
            acc.gphi[0] += W * t[6];
            acc.gphi[1] += W * t[7];
            acc.gphi[2] += W * t[8];
            acc.F[0] += as * dW[0];
            acc.F[1] += as * dW[1];
            acc.F[2] += as * dW[2];
            if constexpr (DIAG) {
                acc.Ubar[0] += W * t[9];
                acc.Ubar[1] += W * t[10];
                acc.Ubar[2] += W * t[11];
                acc.pu += W;
                const double vdW = vb[0] * dW[0] + vb[1] * dW[1] + vb[2] * dW[2];
#pragma unroll
                for (int l = 0; l < 3; ++l) acc.DAv[l] += ((1.0 - s) * t[l] + s * t[3 + l]) * vdW;
            }
        });
    }
}

// One piece of a split orbit (see scatter_pieces): the impulse's two integrals and, with DIAG, the
// orbit gathers of the chain-rule and power tests.
template <int R, bool DIAG>
__device__ __forceinline__ void push_piece_points(const StepParams& p, double h, double sm, const double mid[3],
                                                  const int c[3], const double beta[3], const double vb[3],
                                                  const double* __restrict__ table, PushAcc& acc, int part = 0,
                                                  int parts = 1) {
    const PiecePoints<R> pt(p, h, mid, beta, true);
    const Stencil<R> sl(c, p.m);
    double F[3] = {0.0, 0.0, 0.0}, g3[3] = {0.0, 0.0, 0.0}, U3[3] = {0.0, 0.0, 0.0}, D3[3] = {0.0, 0.0, 0.0}, pu = 0.0;
    const double vh[3] = {vb[0] * p.invH[0], vb[1] * p.invH[1], vb[2] * p.invH[2]};
    for (int r = part; r < (R + 1) * (R + 1); r += parts) {
        const int kz = r / (R + 1), ky = r - kz * (R + 1);
        const double* row = table + 12 * sl.row(ky, kz, p.m);
        double a1[R + 1], cc[R + 1], M[R + 1];
#pragma unroll
        for (int k = 0; k <= R; ++k) {
            const double* t = row + 12 * sl.x[k];
            a1[k] = t[3] * vb[0] + t[4] * vb[1] + t[5] * vb[2];                  // A^{n+1}_g . vbar
            cc[k] = a1[k] - (t[0] * vb[0] + t[1] * vb[1] + t[2] * vb[2]);        // its change over the step
            M[k] = 0.0;
        }
        for (int q = 0; q < p.nq; ++q) {
            const double wz = pt.w[q][2][kz], wy = pt.w[q][1][ky];
            const double wyz = wy * wz, dyz = pt.d[q][1][ky] * wz, ydz = wy * pt.d[q][2][kz];
            const double nms = sm + h * (c_gauss_t[p.rule + q] - 0.5) - 1.0;    // s - 1
            double tw = 0.0, td = 0.0;
#pragma unroll
            for (int k = 0; k <= R; ++k) {
                const double as = a1[k] + nms * cc[k];                          // A_g(s) . vbar
                tw += as * pt.w[q][0][k];
                td += as * pt.d[q][0][k];
                M[k] += wyz * pt.w[q][0][k];
            }
            F[0] += td * wyz;
            F[1] += tw * dyz;
            F[2] += tw * ydz;
            if constexpr (DIAG) {
                const double vx = vh[0] * wyz, vyz = vh[1] * dyz + vh[2] * ydz;
#pragma unroll
                for (int k = 0; k <= R; ++k) {
                    const double* t = row + 12 * sl.x[k];
                    const double vdW = vx * pt.d[q][0][k] + vyz * pt.w[q][0][k];
#pragma unroll
                    for (int l = 0; l < 3; ++l) D3[l] += (t[3 + l] + nms * (t[3 + l] - t[l])) * vdW;
                }
            }
        }
#pragma unroll
        for (int k = 0; k <= R; ++k) {
            const double* t = row + 12 * sl.x[k];
#pragma unroll
            for (int l = 0; l < 3; ++l) g3[l] += M[k] * t[6 + l];
            if constexpr (DIAG) {
#pragma unroll
                for (int l = 0; l < 3; ++l) U3[l] += M[k] * t[9 + l];
                pu += M[k];
            }
        }
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        acc.F[l] += h * p.invH[l] * F[l];
        acc.gphi[l] += h * g3[l];
        if constexpr (DIAG) {
            acc.Ubar[l] += h * U3[l];
            acc.DAv[l] += h * D3[l];
        }
    }
    if constexpr (DIAG) acc.pu += h * pu;
}

// Point interpolant of columns [col, col+3) of the table at a wrapped position.
__device__ __forceinline__ void point_gather3(const StepParams& p, const double xq[3], const double* __restrict__ table,
                                              int col, double out[3]) {
    out[0] = out[1] = out[2] = 0.0;
    auto add = [&](int64_t g, double S, const double*) {
        const double* t = table + 12 * g + col;
        out[0] += S * t[0];
        out[1] += S * t[1];
        out[2] += S * t[2];
    };
    if (p.order == 2) {
        Basis1<2> b[3];
        basis3<2>(p, xq, b);
        for_each_node<2>(p, b, add);
        return;
    }
    if (p.order == 3) {
        Basis1<3> b[3];
        basis3<3>(p, xq, b);
        for_each_node<3>(p, b, add);
        return;
    }
    int64_t g[8];
    double w[8];
    point_weights8(xq, p.m, g, w);
#pragma unroll
    for (int k = 0; k < 8; ++k) add(g[k], w[k], nullptr);
}

// ---- kernels ----------------------------------------------------------------------

__global__ void k_init_positions(StepParams p, const double* __restrict__ x, double* __restrict__ xi,
                                 int64_t* __restrict__ id) {
    const int64_t np = p.np;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) xi[a * np + i] = wrap_pos_any(x[a * np + i] * p.invH[a], (double)p.m.n[a]);
        id[i] = i;
    }
}

// Cell-unit positions in caller order -> device order, wrapped to [0, n_a) (the identity on
// values already in range).
__global__ void k_set_positions(StepParams p, const int64_t* __restrict__ id, const double* __restrict__ src,
                                double* __restrict__ xi) {
    const int64_t np = p.np;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) xi[a * np + i] = wrap_pos_any(src[a * np + id[i]], (double)p.m.n[a]);
    }
}

__global__ void k_point_deposit(StepParams p, const double* __restrict__ xi, double* __restrict__ rho) {
    const int64_t np = p.np;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        double x[3] = {xi[i], xi[np + i], xi[2 * np + i]};
        auto dep = [&](int64_t g, double S, const double*) {
            if (p.det) exact_add(p.acc, g, p.q_dV * S);
            else atomicAdd(rho + g, p.q_dV * S);
        };
        if (p.order == 2) {
            Basis1<2> b[3];
            basis3<2>(p, x, b);
            for_each_node<2>(p, b, dep);
        } else if (p.order == 3) {
            Basis1<3> b[3];
            basis3<3>(p, x, b);
            for_each_node<3>(p, b, dep);
        } else {
            int64_t g[8];
            double w[8];
            point_weights8(x, p.m, g, w);
#pragma unroll
            for (int k = 0; k < 8; ++k) dep(g[k], w[k], nullptr);
        }
    }
}

// v^{n+1,0} = 2 v^n - v^{n-1} (Algorithm 1, extrapolated start) unless an iterate is given;
// then the orbit current of that iterate, and sum_i |v^n_i| for the e_J floor.
__global__ void k_first_scatter(StepParams p, const double* __restrict__ xi, const double* __restrict__ v,
                                const double* __restrict__ vprev, const double* __restrict__ vgiven,
                                double* __restrict__ vit, double* __restrict__ J, double* __restrict__ partials,
                                int* __restrict__ status) {
    __shared__ double sm[32];
    __shared__ int order[THREADS];
    __shared__ int wcount[THREADS / 32][PIECE_CLASSES];
    const int64_t np = p.np, nchunks = (np + THREADS - 1) / THREADS;
    double jsc = 0.0;
    // chunks of THREADS particles handed to the threads by orbit-piece count (as in k_push)
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * THREADS;
        double x0[3], vn[3], vi[3], beta[3], w[3];
        int cls = PIECE_CLASSES - 1;
        if (base + threadIdx.x < np) {
            const int64_t j = base + threadIdx.x;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + j];
                vn[a] = v[a * np + j];
                vi[a] = vgiven ? vgiven[a * np + j] : 2.0 * vn[a] - vprev[a * np + j];
                vit[a * np + j] = vi[a];
                beta[a] = p.dt * 0.5 * (vi[a] + vn[a]) * p.invH[a];
            }
            jsc += sqrt(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
            cls = piece_class_of(p, x0, beta);
        }
        order[stable_class_rank(cls, wcount)] = threadIdx.x;
        __syncthreads();
        const int64_t i = base + order[threadIdx.x];
        if (i < np) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + i];
                vn[a] = v[a * np + i];
                vi[a] = vgiven ? vgiven[a * np + i] : 2.0 * vn[a] - vprev[a * np + i];
                const double vb = 0.5 * (vi[a] + vn[a]);
                beta[a] = p.dt * vb * p.invH[a];
                w[a] = p.q_dV * vb;
            }
            if (scatter_orbit(p, x0, beta, w, J) < 0) atomicOr(status, DEV_ERR_SEGMENTS);
        }
        __syncthreads();   // order[] is rewritten by the next chunk
    }
    write_partial<double>(partials, S_JSCALE, jsc, sm, false);
}

// Constants of the particle-local solve for "creeping" particles (see k_local); the
// classifier is_creeping and its BETA_CREEP / D_KNOT live in pic_device.cuh.
constexpr int LOCAL_STEPS = 32;      // push evaluations per creeping particle
constexpr double LOCAL_TOL = 1e-15;  // relative to the particle's speed
constexpr double OMEGA_MAX = 8.0;    // bound on the secant step factor
constexpr double SLIDE_PROBE = 1e-12; // cells: the sliding test probes SLIDE_PROBE short of the knot
constexpr double SLIDE_FAR = 64.0;    // ... and max(SLIDE_PROBE, SLIDE_FAR |d|) past it
constexpr double D_FALLBACK = 1e-6;   // cells: a failed solve slides the components that start
                                      // this near a knot
constexpr double FAIL_RES = 1e-10;    // failed: best residual above FAIL_RES x the speed
constexpr double BETA_TRIAL = 1.0;    // cells: trial orbits stay within this beyond the iterate's
                                      // own orbit, per axis

struct PushOut {
    double Pw[3], xe[3], Ae[3], vw[3];
    int nseg;
};

// G(u): the Algorithm 1 push of one particle for the end-of-step iterate u with the
// current mesh table: orbit vbar = (u + v^n)/2, P^{n+1} (Eq. (orbit-P-update)),
// x^{n+1} (Eq. (orbit-x-update)) and v^{n+1} = (P^{n+1} - q A_h^{n+1}(x^{n+1})) / m.
template <bool DIAG>
__device__ __forceinline__ void push_eval(const StepParams& p, const double x0[3], const double vn[3],
                                          const double Pn[3], const double u[3], const double* __restrict__ table,
                                          PushAcc& acc, PushOut& o) {
    double vb[3], beta[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        vb[a] = 0.5 * (u[a] + vn[a]);
        beta[a] = p.dt * vb[a] * p.invH[a];
    }
    acc = PushAcc{};
    if (p.split) {
        CellStart<double> st;
        knot_start(p, x0, st);
        o.nseg = for_each_piece(st, beta, p.m, [&](double h, double sm, const double mid[3], const int c[3]) {
            if (p.order == 2) push_piece_points<2, DIAG>(p, h, sm, mid, c, beta, vb, table, acc);
            else if (p.order == 3) push_piece_points<3, DIAG>(p, h, sm, mid, c, beta, vb, table, acc);
            else push_piece_points<1, DIAG>(p, h, sm, mid, c, beta, vb, table, acc);
        });
    } else {
        o.nseg = for_each_segment(x0, beta, false, [&](const Segment<double>& sg) {
            if (p.order == 2) push_piece_gauss_r<2, DIAG>(p, sg, x0, beta, vb, table, acc);
            else if (p.order == 3) push_piece_gauss_r<3, DIAG>(p, sg, x0, beta, vb, table, acc);
            else push_piece_gauss<DIAG>(p, sg, x0, beta, vb, table, acc);
        });
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o.Pw[a] = Pn[a] + p.dt * (-p.q * acc.gphi[a] + p.q * acc.F[a]);
        o.xe[a] = wrap_pos(x0[a] + beta[a], (double)p.m.n[a]);
    }
    point_gather3(p, o.xe, table, 3, o.Ae);
#pragma unroll
    for (int a = 0; a < 3; ++a) o.vw[a] = (o.Pw[a] - p.q * o.Ae[a]) * p.inv_mass;
}

// G(u) of the closed forms, from the start (cell, coordinate) and vs = u + v^n =
// 2 vbar: in fixed point from the cell tables, or (FROM_NODES) in FP64 from the gather table.
struct CellOut {
    double Pw[3], Ae[3], vw[3];
    int nseg;
};

template <int FROM>
__device__ __forceinline__ void push_eval_cell(const StepParams& p, CellStart<double> st, const double vs[3],
                                               const double Pn[3], FixedTables ft, CellOut& o) {
    double beta[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) beta[a] = p.cb[a] * vs[a];
    if constexpr (FROM != FROM_NODES) {
        const int ev = max(max(exponent_of(vs[0]), exponent_of(vs[1])), max(exponent_of(vs[2]), 64));
        Fs v[3];
        double accF[3] = {0.0, 0.0, 0.0}, accG[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fs_of(fixed_of(vs[a], ev, FX_V_UP));
        o.nseg = for_each_piece(st, beta, p.m, [&](double h, double sm, const double mid[3], const int c[3]) {
            const double d[3] = {h * beta[0], h * beta[1], h * beta[2]};
            if (FROM == FROM_CELLS || ft.cells) {
                piece_impulse_fixed(h, sm, mid, d, v, ev, FixedLoad(ft, c, p.m), accF, accG);
            } else {
                const PieceOrbit o = {h, sm, {mid[0], mid[1], mid[2]}, {d[0], d[1], d[2]}, {v[0], v[1], v[2]},
                                      ev, {c[0], c[1], c[2]}, {p.m.n[0], p.m.n[1], p.m.n[2]}};
                const PieceSums s = piece_impulse_of_nodes(
                    ft.nodes, o, PieceSums{{accF[0], accF[1], accF[2]}, {accG[0], accG[1], accG[2]}});
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    accF[a] = s.F[a];
                    accG[a] = s.G[a];
                }
            }
        });
        CellA1 A1;
        if (FROM == FROM_CELLS || ft.cells) {
            const FixedLoad ld(ft, st.c, p.m);
            cell_A1_fixed(st.f, ld, A1.a);
            A1.top = ld.top_A();
        } else {
            A1 = cell_A1_of_nodes(ft.nodes, st.c[0], st.c[1], st.c[2], p.m.n[0], p.m.n[1], p.m.n[2], st.f[0], st.f[1],
                                  st.f[2]);
        }
        // values that are not finite stay so (the start's coordinate: the end's is its sum with beta)
        const int ef = max(max(exponent_of(st.f[0]), exponent_of(st.f[1])), exponent_of(st.f[2]));
        const double dtq = max(ev, ef) < 0x7ff ? p.dtq : NAN;
        const double uA = pow2_biased(A1.top - 57);
        const double* low = ft.nodes + 12 * cell_row(st.c, p.m) + 3;   // A^{n+1} at the cell's lowest node
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            o.Ae[a] = __ldg(low + a) + uA * (double)A1.a[a];
            o.Pw[a] = Pn[a] + dtq * (accG[a] + p.ihs[a] * accF[a]);
        }
    } else {
        double acc[3] = {0.0, 0.0, 0.0};
        o.nseg = for_each_piece(st, beta, p.m, [&](double h, double sm, const double mid[3], const int c[3]) {
            piece_impulse(h, sm, mid, beta, vs, p.ihs, FieldLoad<FROM_NODES>({ft.nodes, nullptr}, c, p.m), acc);
        });
        cell_A1(st.f, FieldLoad<FROM_NODES>({ft.nodes, nullptr}, st.c, p.m), o.Ae);
#pragma unroll
        for (int a = 0; a < 3; ++a) o.Pw[a] = Pn[a] + p.dtq * acc[a];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) o.vw[a] = (o.Pw[a] - p.q * o.Ae[a]) * p.inv_mass;
}

// Warps per SM that the kernels are compiled for.  First scatter: 16 (128 registers) measured 37.2 ms at
// 128^3 with 134M particles, 20 38.7, 24 42.3.  Push: 16 measured 1.13 ms (iterate, 32^3, 2,097,152
// particles), 20 (102 registers, more spills) 1.26, 12 1.29.
constexpr int SCATTER_WARPS = 16;
constexpr int PUSH_WARPS = 16;

// k_first_scatter for the closed forms.
template <int WARPS, int ITEMS>
__global__ void __launch_bounds__(32 * WARPS, SCATTER_WARPS / WARPS) k_first_scatter_cell(
    StepParams p, const double* __restrict__ xi, const double* __restrict__ v, const double* __restrict__ vprev,
    const double* __restrict__ vgiven, double* __restrict__ vit, double* __restrict__ J, double* __restrict__ partials,
    int* __restrict__ status) {
    typedef ChunkOrder<WARPS, ITEMS> Chunk;
    __shared__ double sm[32];
    extern __shared__ __align__(16) unsigned char dyn[];
    Chunk& co = Chunk::in(dyn);
    long long* tile = Chunk::tile(dyn);
    const int64_t np = p.np, nchunks = (np + Chunk::SIZE - 1) / Chunk::SIZE;
    double jsc = 0.0;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * Chunk::SIZE;
        chunk_exchange(p, co, base, [&](int64_t j, double x0[3], double v2[3]) {
            double vn[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + j];
                vn[a] = v[a * np + j];
                const double vi = vgiven ? vgiven[a * np + j] : 2.0 * vn[a] - vprev[a * np + j];
                vit[a * np + j] = vi;
                v2[a] = vi + vn[a];
            }
            jsc += sqrt(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
        });
#pragma unroll 1
        for (int it = 0; it < ITEMS; ++it) {
            CellStart<double> st;
            double vs[3], beta[3], w[3];
            const int64_t i = co.take(it, base, st, vs);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                beta[a] = p.cb[a] * vs[a];
                w[a] = p.q_dV_half * vs[a];
            }
            if (scatter_warp(p.m, i < np, st, beta, w, tile, p.det, p.acc, J) < 0) atomicOr(status, DEV_ERR_SEGMENTS);
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
    write_partial<double>(partials, S_JSCALE, jsc, sm, false);
}

// The Algorithm 1 push for the closed forms without diagnostics: as k_push (below), in fixed point
// from the cell tables or (FROM_NODES) in FP64 from the gather table.
//
// It was bound by the FP64 pipe (one warp instruction in 16 clocks per SM), so the steps that made it
// faster take instructions off that pipe.  Measured at 32^3 with 2,097,152 particles (1.31 pieces
// each), iterate and final sweep: 3.52 and 2.40 ms from start-based integrals and node weights (58.2M
// FP64 warp instructions in the iterate); 1.59 and 1.11 with centred moments and the cell's mixed
// differences (25.6M); 1.43 with the fixed-point deposit; 1.22 and 0.77 with the fixed-point pieces
// (11.4M and 9.0M, the pipe 52% and 62% busy); 1.13 and 0.73 with chunks whose warps have equal work and
// sums of products shifted once; 1.03 and 0.68 with the one-crossing walk (10.3M and 7.5M); 0.96 and 0.65 with
// eight warps a block (chunk.cuh); 1.00 and 0.66 (10.7M and 7.7M) with each cell's own exponents and units, which
// keep the bits of fields and particles far smaller than others elsewhere.  At 128^3 with 134M particles the final
// sweep took 225, 102, 64, 54, now 56 ms.
// What is left is latency (36% issue-active): fixed-latency waits, shared memory, the instruction cache.
template <bool COMMIT, int FROM, int WARPS, int ITEMS>
__global__ void __launch_bounds__(32 * WARPS, PUSH_WARPS / WARPS) k_push_cell(StepParams p, const double* __restrict__ xi,
                                                          const double* __restrict__ v, const double* __restrict__ P,
                                                          const double* __restrict__ vit,
                                                          FixedTables ft, double* __restrict__ vnew,
                                                          double* __restrict__ Jnext, double* __restrict__ xi_out,
                                                          double* __restrict__ P_out,
                                                          int32_t* __restrict__ creep_list,
                                                          int* __restrict__ creep_count,
                                                          uint8_t* __restrict__ creep_flag,
                                                          const uint8_t* __restrict__ slide,
                                                          double* __restrict__ partials, int* __restrict__ status) {
    __shared__ double sm[32];
    extern __shared__ __align__(16) unsigned char dyn[];
    typedef ChunkOrder<WARPS, ITEMS> Chunk;
    Chunk& co = Chunk::in(dyn);
    long long* tile = Chunk::tile(dyn);
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
        for (int it = 0; it < ITEMS; ++it) {
            CellStart<double> st;
            double vs[3];
            const int64_t i = co.take(it, base, st, vs);
            bool scat = false;               // this lane's next orbit is scattered here
            double bn[3] = {0.0, 0.0, 0.0}, w[3] = {0.0, 0.0, 0.0};
            if (i < np) {
                double vi[3], vn[3], Pn[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) Pn[a] = P[a * np + i];
                CellOut o;
                push_eval_cell<FROM>(p, st, vs, Pn, ft, o);
                if (o.nseg < 0) atomicOr(status, DEV_ERR_SEGMENTS);
                pieces_push += o.nseg;
                if (!(isfinite(o.vw[0]) && isfinite(o.vw[1]) && isfinite(o.vw[2]))) atomicOr(status, DEV_ERR_NONFINITE);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    vi[a] = vit[a * np + i];
                    vn[a] = v[a * np + i];
                }
                if constexpr (!COMMIT) {
                    // a particle solved locally earlier in this step keeps the local solve, so that
                    // none alternates between it and the plain update.  So does one whose change did
                    // not shrink below SLOW_RATIO of the previous one: its own feedback is too strong
                    // for the outer iteration (orbits crossing a knot just past the creeping range,
                    // once the force jumps at knots grow).  A contracting outer loop shrinks
                    // field-driven changes far faster, so it flags almost none.
                    double d[3], beta[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        d[a] = o.vw[a] - vi[a];   // change of the iterate, v^{p+1} - v^p
                        beta[a] = p.cb[a] * vs[a];
                    }
                    bool slow = false;
                    if (p.hist) {
                        double dold = 0.0;
#pragma unroll
                        for (int a = 0; a < 3; ++a) dold = max_pos(dold, fabs(vi[a] - vnew[a * np + i]));
                        const double dn = max_pos(max_pos(fabs(d[0]), fabs(d[1])), fabs(d[2]));
                        if (less_pos(SLOW_RATIO * dold, dn))
                            slow = dn > p.slow_floor * sqrt(vi[0] * vi[0] + vi[1] * vi[1] + vi[2] * vi[2]);
                    }
                    const bool creep = p.accel && (is_creeping_cell(st.f, beta) || (slide[i] & SLIDE_CREPT) || slow);
                    if (creep_flag) creep_flag[i] = creep ? 1 : 0;   // deterministic mode: k_local walks the flags
#pragma unroll
                    for (int a = 0; a < 3; ++a) vnew[a * np + i] = o.vw[a];   // G(v^p)
                    if (creep) {
                        if (!creep_flag) {
                            const int k = atomicAdd(creep_count, 1);   // k_local solves it and adds its e_v terms
                            creep_list[k] = (int32_t)i;
                        }
                    } else {
                        scat = true;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            ev_num += d[a] * d[a];
                            ev_den += o.vw[a] * o.vw[a];
                            const double v2n = o.vw[a] + vn[a];
                            bn[a] = p.cb[a] * v2n;
                            w[a] = p.q_dV_half * v2n;
                        }
                    }
                } else {
                    // components sliding onto a knot (set by k_local): the orbit lands on the knot,
                    // v^{n+1}_a is the iterate itself and P_a follows from v = (P - q A_h(x)) / m
                    const uint8_t sb = slide ? slide[i] : 0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        if (sb & (1u << a)) {
                            o.vw[a] = vi[a];
                            o.Pw[a] = p.mass * o.vw[a] + p.q * o.Ae[a];
                        }
                        vnew[a * np + i] = o.vw[a];
                        xi_out[a * np + i] = wrap_pos(xi[a * np + i] + p.cb[a] * vs[a], (double)p.m.n[a]);
                        P_out[a * np + i] = o.Pw[a];
                        // the residual of the accepted iterate itself, ||G(v*) - v*||
                        const double d = o.vw[a] - vi[a];
                        ev_num += d * d;
                        ev_den += o.vw[a] * o.vw[a];
                    }
                }
            }
            if constexpr (!COMMIT) {
                const int ns = scatter_warp(p.m, scat, st, bn, w, tile, p.det, p.acc, Jnext);
                if (ns < 0) atomicOr(status, DEV_ERR_SEGMENTS);
                pieces_scatter += ns;
            }
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
    write_partial<double>(partials, S_EV_NUM, ev_num, sm, false);
    write_partial<double>(partials, S_EV_DEN, ev_den, sm, false);
    if constexpr (!COMMIT) {
        write_partial<double>(partials, S_PIECES_PUSH, (double)pieces_push, sm, false);
        write_partial<double>(partials, S_PIECES_SCATTER, (double)pieces_scatter, sm, false);
    }
}

// One piece of an orbit for the final sweep with diagnostics: piece_impulse's two integrals apart, and
// those of the identities, (D A) vbar and the gather of U, per particle.
struct DiagAcc {
    double F[3], g[3];        // (D_j A)^T vbar and -grad phi
    double DAv[3], U[3], pu;  // (D A) vbar, U^{n+1/2}, sum of the weights
};

// vh_j = vbar_j / H_j; `ld` as for piece_impulse; U from the gather table's rows g (columns 9 to 11).
template <typename L>
__device__ __forceinline__ void piece_diag(double h, double sm, const double mid[3], const double beta[3],
                                           const double vs[3], const double ihs[3], const double vh[3], L&& ld,
                                           const double* __restrict__ table, const int64_t g[8], DiagAcc& acc) {
    const PieceMoments<double> q = piece_moments(h, mid, beta);
    const double nms = sm - 1.0;
    {
        double W[8], u[3] = {0.0, 0.0, 0.0}, sum = 0.0;
        node_weights(q, W);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double* t = table + 12 * g[k] + 9;
            sum += W[k];
#pragma unroll
            for (int j = 0; j < 3; ++j) u[j] += W[k] * __ldg(t + j);
        }
        acc.pu += h * sum;
#pragma unroll
        for (int j = 0; j < 3; ++j) acc.U[j] += h * u[j];
    }
    const double M[8] = {1.0, mid[0], mid[1], q.Pxy, mid[2], q.Pxz, q.Pyz, q.S};
    const double E[8] = {0.0, q.e[0], q.e[1], mid[0] * q.e[1] + mid[1] * q.e[0],
                         q.e[2], mid[0] * q.e[2] + mid[2] * q.e[0], mid[1] * q.e[2] + mid[2] * q.e[1], 0.0};
    double F[3] = {0.0, 0.0, 0.0}, gg[3] = {0.0, 0.0, 0.0}, D[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        double x[3][2], d[3][2], y[3][2];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            ld(p, j, x[j][0], x[j][1]);
            ld(p, 3 + j, d[j][0], d[j][1]);
            ld(p, 6 + j, y[j][0], y[j][1]);
        }
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            const int k = 2 * p + o;
#pragma unroll
            for (int j = 0; j < 3; ++j) gg[j] += y[j][o] * M[k];
            if (k == 0) continue;
            double am[3], a = 0.0, cc = 0.0, dk = 0.0, ek = 0.0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                am[j] = x[j][o] + nms * d[j][o];   // A_k at s_mid
                a += am[j] * vs[j];
                cc += d[j][o] * vs[j];
                if ((k >> j) & 1) {
                    dk += vh[j] * M[k ^ (1 << j)];
                    if ((k ^ (1 << j)) != 0) ek += vh[j] * E[k ^ (1 << j)];
                }
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if ((k >> j) & 1) F[j] += a * M[k ^ (1 << j)] + cc * E[k ^ (1 << j)];
                D[j] += am[j] * dk + d[j][o] * ek;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        acc.F[j] += h * ihs[j] * F[j];
        acc.g[j] += h * gg[j];
        acc.DAv[j] += h * D[j];
    }
}

// The closed forms' final sweep with the particle diagnostics, in the centred form of k_push_cell
// (FP64).  Bound by the FP64 pipe like that: some 240 operations a piece where
// the integrals from the piece's start took some 700: 1.62 ms at 50 x 35 x 22 with 539,000 particles, now
// 0.68.
constexpr int DIAG_WARPS = 16;   // 12 (168 registers): two steps at 16^3 2.77 ms, 16 2.69
template <int FROM, int WARPS, int ITEMS>
__global__ void __launch_bounds__(32 * WARPS, DIAG_WARPS / WARPS) k_commit_diag(
    StepParams p, const double* __restrict__ xi, const double* __restrict__ v, const double* __restrict__ P,
    const double* __restrict__ vit, const double* __restrict__ table, const double* __restrict__ ctab,
    double* __restrict__ vnew, double* __restrict__ xi_out, double* __restrict__ P_out,
    const uint8_t* __restrict__ slide, double* __restrict__ partials, int* __restrict__ status) {
    __shared__ double sm[32];
    extern __shared__ __align__(16) unsigned char dyn[];
    typedef ChunkOrder<WARPS, ITEMS> Chunk;
    Chunk& co = Chunk::in(dyn);
    const int64_t np = p.np, nchunks = (np + Chunk::SIZE - 1) / Chunk::SIZE;
    double ev_num = 0.0, ev_den = 0.0, k1 = 0.0, pwork = 0.0, ra_sq = 0.0, ra_max = 0.0, pu_max = 0.0;
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
        for (int it = 0; it < ITEMS; ++it) {
            CellStart<double> st;
            double vs[3];
            const int64_t i = co.take(it, base, st, vs);
            if (i >= np) continue;
            double beta[3], vh[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                beta[a] = p.cb[a] * vs[a];
                vh[a] = vs[a] * p.ihs[a];
            }
            DiagAcc acc{};
            const int nseg = for_each_piece(st, beta, p.m, [&](double h, double s, const double mid[3], const int c[3]) {
                int64_t g[8];
                cell_nodes8(c, p.m, g);
                piece_diag(h, s, mid, beta, vs, p.ihs, vh, FieldLoad<FROM>({table, ctab}, c, p.m), table, g, acc);
            });
            if (nseg < 0) atomicOr(status, DEV_ERR_SEGMENTS);
            double Ae[3], As[3], x0[3], ra2 = 0.0;
            cell_A1(st.f, FieldLoad<FROM>({table, ctab}, st.c, p.m), Ae);
#pragma unroll
            for (int a = 0; a < 3; ++a) x0[a] = xi[a * np + i];
            {   // A_h^n(x^n)
                double w[8];
                int64_t g[8];
                point_weights8(x0, p.m, g, w);
                As[0] = As[1] = As[2] = 0.0;
#pragma unroll
                for (int k = 0; k < 8; ++k)
#pragma unroll
                    for (int a = 0; a < 3; ++a) As[a] += w[k] * __ldg(table + 12 * g[k] + a);
            }
            const uint8_t sb = slide ? slide[i] : 0;
            bool finite = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double vi = vit[a * np + i];
                double Pw = P[a * np + i] + p.dt * (p.q * acc.g[a] + p.q * acc.F[a]);
                double vw = (Pw - p.q * Ae[a]) * p.inv_mass;
                finite = finite && isfinite(vw);
                // components sliding onto a knot, as in k_push_cell
                if (sb & (1u << a)) {
                    vw = vi;
                    Pw = p.mass * vw + p.q * Ae[a];
                }
                vnew[a * np + i] = vw;
                xi_out[a * np + i] = wrap_pos(x0[a] + beta[a], (double)p.m.n[a]);
                P_out[a * np + i] = Pw;
                const double d = vw - vi;
                ev_num += d * d;
                ev_den += vw * vw;
                const double ra = Ae[a] - As[a] - p.dt * (acc.U[a] + acc.DAv[a]);        // Eq. (RA-test)
                ra2 += ra * ra;
                ra_max = fmax(ra_max, fabs(ra));
                pwork += p.q * (0.5 * vs[a]) * (acc.g[a] - acc.U[a]);                     // q vbar . Ebar
                k1 += 0.5 * p.mass * vw * vw;
            }
            if (!finite) atomicOr(status, DEV_ERR_NONFINITE);
            ra_sq += ra2;
            pu_max = fmax(pu_max, fabs(acc.pu - 1.0));
        }
        __syncthreads();   // the hand-over buffers are rewritten by the next chunk
    }
    write_partial<double>(partials, S_EV_NUM, ev_num, sm, false);
    write_partial<double>(partials, S_EV_DEN, ev_den, sm, false);
    write_partial<double>(partials, S_K1, k1, sm, false);
    write_partial<double>(partials, S_PWORK, pwork, sm, false);
    write_partial<double>(partials, S_RA_SQ, ra_sq, sm, false);
    write_partial<double>(partials, S_RA_MAX, ra_max, sm, true);
    write_partial<double>(partials, S_PU_MAX, pu_max, sm, true);
}

// The Algorithm 1 push for iterate vit, then either
//   (iterate)  the next iterate and its orbit current into Jnext, plus the e_v partial sums.
//              The next iterate is G(v^p); with p.accel, creeping particles are instead
//              appended to a list and solved locally by k_local (which also scatters them);
//   (commit)   x^{n+1}, P^{n+1}, v^{n+1} and (optionally) the particle diagnostics.
// For the Gauss rules; the closed forms run k_push_cell and k_commit_diag.  Two resident blocks per SM (128
// registers, some spills): quadratic shapes at 36^3 2.26 ms, one block (255 registers) 2.40; the diagnostics
// variant keeps one block, its larger state would spill far more.
template <bool COMMIT, bool DIAG>
__global__ void __launch_bounds__(THREADS, DIAG ? 1 : 2) k_push(StepParams p, const double* __restrict__ xi,
                                                  const double* __restrict__ v, const double* __restrict__ P,
                                                  const double* __restrict__ vit, const double* __restrict__ table,
                                                  double* __restrict__ vnew, double* __restrict__ Jnext,
                                                  double* __restrict__ xi_out, double* __restrict__ P_out,
                                                  int32_t* __restrict__ creep_list, int* __restrict__ creep_count,
                                                  uint8_t* __restrict__ creep_flag,
                                                  const uint8_t* __restrict__ slide, double* __restrict__ partials,
                                                  int* __restrict__ status) {
    __shared__ double sm[32];
    const int64_t np = p.np;
    double ev_num = 0.0, ev_den = 0.0, pieces_push = 0.0, pieces_scatter = 0.0;
    double k1 = 0.0, pwork = 0.0, ra_sq = 0.0, ra_max = 0.0, pu_max = 0.0;
    __shared__ int order[THREADS];
    __shared__ int wcount[THREADS / 32][PIECE_CLASSES];
    const int64_t nchunks = (np + THREADS - 1) / THREADS;
    // Chunks of THREADS consecutive particles; inside a chunk the particles are handed to the
    // threads in order of their (estimated) number of orbit pieces, so that the lanes of a
    // warp run the same number of piece iterations (a stable ordering: deterministic).
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch * THREADS;
        {
            const int64_t j = base + threadIdx.x;
            const int cls = j < np ? piece_class(p, xi, v, vit, j) : PIECE_CLASSES - 1;
            order[stable_class_rank(cls, wcount)] = threadIdx.x;
        }
        __syncthreads();
        const int64_t i = base + order[threadIdx.x];
        if (i < np) {
            double x0[3], vn[3], vi[3], Pn[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                x0[a] = xi[a * np + i];
                vn[a] = v[a * np + i];
                vi[a] = vit[a * np + i];
                Pn[a] = P[a * np + i];
            }
            PushAcc acc;
            PushOut o;
            push_eval<DIAG>(p, x0, vn, Pn, vi, table, acc, o);
            if (o.nseg < 0) atomicOr(status, DEV_ERR_SEGMENTS);
            pieces_push += (double)o.nseg;
            if (!(isfinite(o.vw[0]) && isfinite(o.vw[1]) && isfinite(o.vw[2]))) atomicOr(status, DEV_ERR_NONFINITE);
            if constexpr (COMMIT) {
#pragma unroll
                for (int a = 0; a < 3; ++a) vnew[a * np + i] = o.vw[a];
            }
            if constexpr (!COMMIT) {
                double beta_it[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) beta_it[a] = p.dt * 0.5 * (vi[a] + vn[a]) * p.invH[a];
                const double xk[3] = {x0[0] - p.koff, x0[1] - p.koff, x0[2] - p.koff};   // knot lattice
                // a particle solved locally earlier in this step keeps the local solve, so that
                // none alternates between it and the plain update
                // So does one whose change did not shrink below SLOW_RATIO of the previous one: its
                // own feedback is too strong for the outer iteration (orbits crossing a knot just
                // past the creeping range, once the force jumps at knots grow).  A contracting
                // outer loop shrinks field-driven changes far faster, so it flags almost none.
                bool slow = false;
                if (p.hist) {
                    double dn = 0.0, dold = 0.0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        dn = fmax(dn, fabs(o.vw[a] - vi[a]));
                        dold = fmax(dold, fabs(vi[a] - vnew[a * np + i]));   // v^p - v^{p-1}
                    }
                    const double spd = sqrt(vi[0] * vi[0] + vi[1] * vi[1] + vi[2] * vi[2]);
                    slow = dn > SLOW_RATIO * dold && dn > p.slow_floor * spd;
                }
                const bool creep = p.accel && (is_creeping(xk, beta_it) || (slide[i] & SLIDE_CREPT) || slow);
                if (creep_flag) creep_flag[i] = creep ? 1 : 0;   // deterministic mode: k_local walks the flags
                if (creep) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) vnew[a * np + i] = o.vw[a];   // G(v^p): the local solve starts there
                    if (!creep_flag) {
                        int k = atomicAdd(creep_count, 1);   // k_local solves it and adds its e_v terms
                        creep_list[k] = (int32_t)i;
                    }
                } else {
                    double wv[3], bet2[3], dnum = 0.0, dden = 0.0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        vnew[a * np + i] = o.vw[a];
                        const double d = o.vw[a] - vi[a];   // change of the iterate, v^{p+1} - v^p
                        dnum += d * d;
                        dden += o.vw[a] * o.vw[a];
                        const double vb2 = 0.5 * (o.vw[a] + vn[a]);
                        bet2[a] = p.dt * vb2 * p.invH[a];
                        wv[a] = p.q_dV * vb2;
                    }
                    ev_num += dnum;
                    ev_den += dden;
                    int ns = scatter_orbit(p, x0, bet2, wv, Jnext);
                    if (ns < 0) atomicOr(status, DEV_ERR_SEGMENTS);
                    pieces_scatter += (double)ns;
                }
            } else {
                // components sliding onto a knot (set by k_local): the orbit lands on the knot,
                // v^{n+1}_a is the iterate itself and P_a follows from v = (P - q A_h(x)) / m
                const uint8_t sb = slide ? slide[i] : 0;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (sb & (1u << a)) {
                        o.vw[a] = vi[a];
                        o.Pw[a] = p.mass * o.vw[a] + p.q * o.Ae[a];
                        vnew[a * np + i] = o.vw[a];
                    }
                    xi_out[a * np + i] = o.xe[a];
                    P_out[a * np + i] = o.Pw[a];
                    // the residual of the accepted iterate itself, ||G(v*) - v*||
                    const double d = o.vw[a] - vi[a];
                    ev_num += d * d;
                    ev_den += o.vw[a] * o.vw[a];
                }
                if constexpr (DIAG) {
                    double As[3], vb[3];
                    point_gather3(p, x0, table, 0, As);                       // A_h^n(x^n)
                    double ra2 = 0.0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        vb[a] = 0.5 * (vi[a] + vn[a]);
                        double ra = o.Ae[a] - As[a] - p.dt * (acc.Ubar[a] + acc.DAv[a]);   // Eq. (RA-test)
                        ra2 += ra * ra;
                        ra_max = fmax(ra_max, fabs(ra));
                        pwork += p.q * vb[a] * (-acc.gphi[a] - acc.Ubar[a]);                // q vbar . Ebar
                        k1 += 0.5 * p.mass * o.vw[a] * o.vw[a];
                    }
                    ra_sq += ra2;
                    pu_max = fmax(pu_max, fabs(acc.pu - 1.0));
                }
            }
        }
        __syncthreads();   // order[] is rewritten by the next chunk
    }
    write_partial<double>(partials, S_EV_NUM, ev_num, sm, false);
    write_partial<double>(partials, S_EV_DEN, ev_den, sm, false);
    if constexpr (!COMMIT) {
        write_partial<double>(partials, S_PIECES_PUSH, pieces_push, sm, false);
        write_partial<double>(partials, S_PIECES_SCATTER, pieces_scatter, sm, false);
    } else if constexpr (DIAG) {
        write_partial<double>(partials, S_K1, k1, sm, false);
        write_partial<double>(partials, S_PWORK, pwork, sm, false);
        write_partial<double>(partials, S_RA_SQ, ra_sq, sm, false);
        write_partial<double>(partials, S_RA_MAX, ra_max, sm, true);
        write_partial<double>(partials, S_PU_MAX, pu_max, sm, true);
    }
}

// Particle-local solve of v = G_i(v) with the iteration's fields fixed, for the creeping
// particles listed by k_push (§4.8 allows any converged solver).  Per component of
// g(u) = G_i(u) - u, starting from (v^p, G(v^p)): clamped secant steps while each one at
// least halves |g| (a nearby root is found first); otherwise steps u + f g with f = 2, 4,
// 8, ... (g is continuous and G bounded, so g changes sign that way: a particle that barely
// crosses a knot can have no root near its iterate).  Inside a bracket the new point replaces
// the end of its sign:
//  - a bracket holding the velocity that lands the orbit exactly on a knot is first split
//    there: the force weight of the path beyond a knot makes G steep just past it, so g is
//    smooth only between landings;
//  - inside one knot-free piece past a crossing (landing beta_L), G in cells is close to
//    A + B beta_L / beta; the step solves beta = A + B beta_L / beta exactly for the line
//    through the two ends (a quadratic), elsewhere it is the regula falsi point;
//  - the components share each evaluation, so another component's move can leave a bracket
//    stale, and regula falsi can stagnate: a bracket whose same end is replaced twice running
//    is released for a secant step.
// At most LOCAL_STEPS push evaluations, stopping once one evaluation has every component's
// residual below LOCAL_TOL times the particle's speed; the evaluation with the smallest
// largest-component residual is kept whole (the components are coupled).  A particle solved
// here keeps the local solve for the rest of the step (SLIDE_CREPT), so that none alternates
// between it and the plain update.  Sliding (sticky for the rest of the step once detected,
// so that the outer iteration cannot cycle between pinned and free): a component starting
// within D_KNOT of a knot (signed distance d) whose two sides, probed SLIDE_PROBE short of
// the landing and max(SLIDE_PROBE, SLIDE_FAR |d|) past it, both push onto the knot has no
// root that double precision resolves; it lands exactly on the knot (the Filippov solution)
// and the commit push sets v^{n+1}_a to it with P_a from the canonical relation.  The energy
// identities hold to the size of vbar_a = d H / dt < D_KNOT H / dt.  The plain image G(v^p)
// is saved in gsave (diagnostics), then the orbit current of the result is scattered.
//
// Four lanes share a particle (eight with a Gauss rule).  A solve is a serial chain of evaluations (up
// to 34, two on average), and on the FP64 pipe a warp instruction takes 64 clocks of its scheduler
// whether one lane is active or 32, so what bounds the launch is the length of that chain, or, with
// many particles, the instructions a warp spends on each.  Lanes 0 .. 2 hold one component each (state
// and step logic), lane k evaluates table entries k and k + 4 of a piece (subsets of the axes; rows k,
// k + 8 of a Gauss piece's nodes) and the sums meet in two exchanges per evaluation, and only the step
// that is taken is computed.  Groups take particles from a queue, a warp's groups together
// (deterministic mode: in index order from the warp's own share of the flags, so that every partial
// sum is reproducible), the first warps of all blocks first.
// With one particle per lane (13 of 32 lanes active on average, the particles on the blocks that came
// first) the mean launch of two steps at 32^3 with 2,097,152 particles took 377 us, now 113; two
// diagnosed steps at 50 x 35 x 22 with 539,000 particles, one in ten of them solved here, 454, now 247;
// quadratic shapes 800, now 294.  With eight lanes the closed forms measured 110, 327, and 5.3 ms
// where four take 3.5 at 128^3 with 134M particles; quadratic shapes with four 348.
template <int QUAD>
constexpr int local_lanes() {
    return QUAD == 0 ? 4 : 8;
}
constexpr int LOCAL_MINB = 1;   // blocks per SM: 2 (128 registers, 480 bytes of spills) measured 114 us

// v[k] of an 8-array held in registers.
__device__ __forceinline__ double pick8(const double v[8], int k) {
    const double a0 = (k & 1) ? v[1] : v[0], a1 = (k & 1) ? v[3] : v[2];
    const double a2 = (k & 1) ? v[5] : v[4], a3 = (k & 1) ? v[7] : v[6];
    const double b0 = (k & 2) ? a1 : a0, b1 = (k & 2) ? a3 : a2;
    return (k & 4) ? b1 : b0;
}

// Lane r's share of piece_impulse: acc_j += its terms, those of the subsets r, r + LANES, ... (summed
// over the lanes they are the piece's).
template <int FROM, int LANES>
__device__ __forceinline__ void piece_impulse_share(const StepParams& p, int r, double h, double sm, const double mid[3],
                                                    const double beta[3], const double vs[3], const int c[3],
                                                    FieldTables ft, double acc[3]) {
    const PieceMoments<double> q = piece_moments(h, mid, beta);
    const double M[8] = {1.0, mid[0], mid[1], q.Pxy, mid[2], q.Pxz, q.Pyz, q.S};
    const double E[8] = {0.0, q.e[0], q.e[1], mid[0] * q.e[1] + mid[1] * q.e[0],
                         q.e[2], mid[0] * q.e[2] + mid[2] * q.e[0], mid[1] * q.e[2] + mid[2] * q.e[1], 0.0};
    const FieldLoad<FROM> ld(ft, c, p.m);
    const double hi[3] = {h * p.ihs[0], h * p.ihs[1], h * p.ihs[2]};
#pragma unroll
    for (int s = 0; s < 8 / LANES; ++s) {
        const int k = r + s * LANES;
        double col[CELL_COLS];
#pragma unroll
        for (int t = 0; t < CELL_COLS; ++t) {
            double e0, e1;
            ld(k >> 1, t, e0, e1);
            col[t] = (k & 1) ? e1 : e0;
        }
        const double cc = col[3] * vs[0] + col[4] * vs[1] + col[5] * vs[2];
        const double a = col[0] * vs[0] + col[1] * vs[1] + col[2] * vs[2] + (sm - 1.0) * cc;
        const double m = h * pick8(M, k);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const bool in = (k >> j) & 1;
            const double F = a * pick8(M, k ^ (1 << j)) + cc * pick8(E, k ^ (1 << j));
            acc[j] += col[6 + j] * m;
            acc[j] += in ? hi[j] * F : 0.0;
        }
    }
}

// A_h^{n+1} at a wrapped position, rows part, part + parts, ... of the stencil.
template <int R>
__device__ __forceinline__ void point_A1_rows(const StepParams& p, const double x[3], const double* __restrict__ table,
                                              int part, int parts, double out[3]) {
    Basis1<R> b[3];
    basis3<R>(p, x, b);
    for (int r = part; r < (R + 1) * (R + 1); r += parts) {
        const int kz = r / (R + 1), ky = r - kz * (R + 1);
        const int gy = wrapi(b[1].first + ky, p.m.n[1]), gz = wrapi(b[2].first + kz, p.m.n[2]);
        const double wyz = b[1].w[ky] * b[2].w[kz];
#pragma unroll
        for (int k = 0; k <= R; ++k) {
            const double* t = table + 12 * node_index(wrapi(b[0].first + k, p.m.n[0]), gy, gz, p.m) + 3;
            const double w = wyz * b[0].w[k];
#pragma unroll
            for (int a = 0; a < 3; ++a) out[a] += w * t[a];
        }
    }
}

// Basis1 of the linear shape (degrees 2 and 3: basis1).
template <>
__device__ __forceinline__ void basis1<1>(double x, double invH, Basis1<1>& b) {
    const double f = floor(x), t = x - f;
    b.first = (int)f;
    b.w[0] = 1.0 - t;
    b.w[1] = t;
    b.dw[0] = -invH;
    b.dw[1] = invH;
}

// G(u) of the particle that a group of lanes shares, u = vs - v^n: every lane gets the component `comp` of
// v^{n+1}.  Every lane of the warp calls it (inactive groups with any valid start).
template <int QUAD, int FROM>
__device__ __forceinline__ double push_eval_shared(const StepParams& p, int k, int comp, const double x0[3],
                                                   const CellStart<double>& start, const double vs[3], double Pn,
                                                   const double* __restrict__ table,
                                                   const double* __restrict__ ctab, int& nseg) {
    constexpr int LANES = local_lanes<QUAD>();
    double beta[3], acc[3] = {0.0, 0.0, 0.0}, Ae[3] = {0.0, 0.0, 0.0};
    CellStart<double> st = start;
#pragma unroll
    for (int a = 0; a < 3; ++a) beta[a] = p.cb[a] * vs[a];
    if constexpr (QUAD == 0) {
        nseg = for_each_piece(st, beta, p.m, [&](double h, double sm, const double mid[3], const int c[3]) {
            piece_impulse_share<FROM, LANES>(p, k, h, sm, mid, beta, vs, c, {table, ctab}, acc);
        });
        const FieldLoad<FROM> ld({table, ctab}, st.c, p.m);
#pragma unroll
        for (int s = 0; s < 8 / LANES; ++s) {
            const int kk = k + s * LANES;
            double e = (kk & 1) ? st.f[0] : 1.0;
            if (kk & 2) e *= st.f[1];
            if (kk & 4) e *= st.f[2];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double e0, e1;
                ld(kk >> 1, a, e0, e1);
                Ae[a] += e * ((kk & 1) ? e1 : e0);
            }
        }
    } else {
        PushAcc pa{};
        const double vb[3] = {0.5 * vs[0], 0.5 * vs[1], 0.5 * vs[2]};
        if (p.split) {
            nseg = for_each_piece(st, beta, p.m, [&](double h, double sm, const double mid[3], const int c[3]) {
                if (p.order == 2) push_piece_points<2, false>(p, h, sm, mid, c, beta, vb, table, pa, k, LANES);
                else if (p.order == 3) push_piece_points<3, false>(p, h, sm, mid, c, beta, vb, table, pa, k, LANES);
                else push_piece_points<1, false>(p, h, sm, mid, c, beta, vb, table, pa, k, LANES);
            });
        } else {
            nseg = for_each_segment(x0, beta, false, [&](const Segment<double>& sg) {
                if (p.order == 2) push_piece_gauss_r<2, false>(p, sg, x0, beta, vb, table, pa);
                else if (p.order == 3) push_piece_gauss_r<3, false>(p, sg, x0, beta, vb, table, pa);
                else push_piece_gauss<false>(p, sg, x0, beta, vb, table, pa);
            });
        }
        const bool mine = p.split || k == 0;   // the whole path's points are not shared out
        double xe[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc[a] = mine ? pa.F[a] - pa.gphi[a] : 0.0;
            xe[a] = wrap_pos(x0[a] + beta[a], (double)p.m.n[a]);
        }
        if (p.order == 2) point_A1_rows<2>(p, xe, table, k, LANES, Ae);
        else if (p.order == 3) point_A1_rows<3>(p, xe, table, k, LANES, Ae);
        else point_A1_rows<1>(p, xe, table, k, LANES, Ae);
    }
    __syncwarp();
    double kick = 0.0;   // P^{n+1} - P^n - q A_h^{n+1}(x^{n+1}) of this lane's component
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double t = p.dtq * acc[a] - p.q * Ae[a];
#pragma unroll
        for (int o = 1; o < LANES; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (a == comp) kick = t;
    }
    return (Pn + kick) * p.inv_mass;
}

template <int QUAD, int FROM>
__global__ void __launch_bounds__(THREADS, LOCAL_MINB) k_local(StepParams p, const double* __restrict__ xi,
                                                   const double* __restrict__ v, const double* __restrict__ P,
                                                   const double* __restrict__ vit, const double* __restrict__ table,
                                                   const double* __restrict__ ctab,
                                                   double* __restrict__ vnew, double* __restrict__ gsave,
                                                   double* __restrict__ Jnext, const int32_t* __restrict__ creep_list,
                                                   const int* __restrict__ creep_count,
                                                   const uint8_t* __restrict__ creep_flag, uint8_t* __restrict__ slide,
                                                   int* __restrict__ queue_head, double* __restrict__ partials,
                                                   int* __restrict__ status) {
    __shared__ double sm[32];
    constexpr int LANES = local_lanes<QUAD>();
    const unsigned full = 0xffffffffu;
    const int64_t np = p.np;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = lane & (LANES - 1), comp = min(k, 2), gbase = lane & ~(LANES - 1);
    // this warp's share of the flags (deterministic mode), or of the queue
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t share = (np + nwarps - 1) / nwarps, wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    int64_t pos = wid * share, word = 0;
    const int64_t end = min(pos + share, np);
    unsigned bits = 0;
    const int64_t count = creep_flag ? 0 : (int64_t)*creep_count;
    // few particles: the warps that the others' SMs can do without stay out
    const int64_t per = (int64_t)gridDim.x * (32 / LANES);
    bool active = false, exhausted = !creep_flag && count <= per * warp;
    double ev_num = 0.0, ev_den = 0.0;
    // One particle's solve is a sequence of push evaluations: sliding probes (phase 0: just
    // short of the knot, phase 1: just past it, per probed axis), the first evaluation
    // (phase 2), then up to LOCAL_STEPS - 1 iteration steps (phase 3).  Every round, each group
    // with a particle makes its next evaluation, and one whose particle is done takes a new one.
    int64_t i = 0;
    int phase = 2, paxis = 0, nstep = 0, probes = 0, nrep = 0;
    double x0[3] = {0.0, 0.0, 0.0}, xa = 0.0, vn = 0.0, Pn = 0.0, u0 = 0.0, r0 = 0.0, u1 = 0.0, r1 = 0.0, bu = 0.0;
    double ua = 0.0, ga = 0.0, ub = 0.0, gb = 0.0, side = 0.0, fac = 2.0, uland = 0.0, dk = 0.0, blim = 0.0;
    bool brk = false, secok = false, sl = false;
    CellStart<double> st{};
    double tol = 0.0, spd = 0.0, gm = 0.0, brs = 0.0;
    double nsolve = 0.0, neval = 0.0, nfail = 0.0, nfail_free = 0.0;
    const double Ha = comp == 0 ? p.H[0] : (comp == 1 ? p.H[1] : p.H[2]);
    const double cba = comp == 0 ? p.cb[0] : (comp == 1 ? p.cb[1] : p.cb[2]);   // beta = cba (u + v^n), in cells
    const double ha = 2.0 * Ha / p.dt;                                          // u + v^n = ha beta
    auto of = [&](double x, int a) { return __shfl_sync(full, x, gbase + a); };
    auto max3 = [&](double x) { return fmax(fmax(of(x, 0), of(x, 1)), of(x, 2)); };
    auto bits3 = [&](bool f) { return (int)(__ballot_sync(full, f) >> gbase) & 7; };
    while (true) {
        // groups without a particle take one
        const bool want = !active && !exhausted;
        const unsigned asking = __ballot_sync(full, want && k == 0);
        if (asking) {
            const int rank = __popc(asking & ((1u << gbase) - 1u));
            int64_t got = -1;
            if (!creep_flag) {
                int first = 0;
                if (lane == 0) first = atomicAdd(queue_head, __popc(asking));
                first = __shfl_sync(full, first, 0);
                if (want && first + rank < count) got = creep_list[first + rank];
            } else {
                int taken = 0;
                const int need = __popc(asking);
                while (taken < need) {
                    if (bits == 0) {
                        if (pos >= end) break;
                        const int64_t j = pos + lane;
                        bits = __ballot_sync(full, j < end && creep_flag[j]);
                        word = pos;
                        pos += 32;
                        continue;
                    }
                    if (want && rank == taken) got = word + __ffs(bits) - 1;
                    bits &= bits - 1;
                    ++taken;
                }
            }
            if (want) {
                if (got < 0) {
                    exhausted = true;
                } else {
                    i = got;
#pragma unroll
                    for (int a = 0; a < 3; ++a) x0[a] = xi[a * np + i];
                    if constexpr (QUAD == 0) cell_start(x0, p.m, st);
                    else knot_start(p, x0, st);
                    xa = (comp == 0 ? x0[0] : (comp == 1 ? x0[1] : x0[2])) - p.koff;   // start on the knot lattice
                    vn = v[comp * np + i];
                    Pn = P[comp * np + i];
                    u0 = vit[comp * np + i];
                    u1 = vnew[comp * np + i];          // G(v^p) from k_push
                    if (k < 3) gsave[comp * np + i] = u1;
                    r0 = u1 - u0;
                    blim = fabs(cba * (u0 + vn)) + BETA_TRIAL;   // trial-orbit bound
                    dk = rint(xa) - xa;                // signed distance to the nearest knot
                    uland = ha * dk - vn;
                    sl = (slide[i] >> comp) & 1u;      // pinned earlier in this step: stays pinned
                }
            }
            const double un = u0 * u0;
            const double nrm = sqrt(of(un, 0) + of(un, 1) + of(un, 2));
            const int pm = bits3(!sl && fabs(dk) < D_KNOT);
            if (want && got >= 0) {
                spd = fmax(nrm, 1e-300);
                tol = LOCAL_TOL * spd;
                probes = pm;
                paxis = 0;
                while (paxis < 3 && !((probes >> paxis) & 1)) ++paxis;
                phase = paxis < 3 ? 0 : 2;
                if (phase == 2 && sl) u1 = uland;
                nstep = 0;
                active = true;
            }
        }
        if (!__any_sync(full, active)) break;
        // the evaluation point of this round
        double ue = u1;
        if (active) {
            if (phase <= 1) {
                // Sliding probes: a component starting within D_KNOT of a knot (signed distance
                // d) is tested SLIDE_PROBE short of landing on it and max(SLIDE_PROBE,
                // SLIDE_FAR |d|) past it, where the path beyond the knot carries most of the
                // orbit average; if both sides push onto the knot, the root lies within that
                // hair, unresolved in double precision, and the component lands on the knot.
                if (comp == paxis) {
                    const double far = fmax(SLIDE_PROBE, SLIDE_FAR * fabs(dk));
                    ue = phase == 0 ? ha * (dk - (dk > 0.0 ? SLIDE_PROBE : far)) - vn
                                    : ha * (dk + (dk > 0.0 ? far : SLIDE_PROBE)) - vn;
                }
            } else if (phase == 3) {
                // the knot landing strictly inside the bracket (the highest one, if several)
                const double lo = fmin(ua, ub), hi = fmax(ua, ub);
                const double bland = (ceil(xa + cba * (hi + vn)) - 1.0) - xa;
                const double usplit = ha * bland - vn;
                double fp = NAN;
                if (sl) {
                    ue = uland;                          // pinned: lands on the knot
                } else if (brk && bland > cba * (lo + vn) && usplit > lo && usplit < hi) {
                    ue = usplit;                         // split the bracket where G kinks
                } else {
                    if (brk) {
                        fp = ub - gb * (ub - ua) / (gb - ga);
                        // Both ends past the same last knot (landing beta_L): on that knot-free
                        // piece the image G in cells is close to A + B w, w = beta_L / beta, steep
                        // near the knot and flat far past it; solve beta = A + B w exactly for the
                        // line through the two ends (D beta^2 - c1 beta - e = 0, root in bracket).
                        const double ba = cba * (ua + vn), bb = cba * (ub + vn);
                        const double la = ba > 0.0 ? floor(xa + ba) - xa : ceil(xa + ba) - xa;
                        const double lb = bb > 0.0 ? floor(xa + bb) - xa : ceil(xa + bb) - xa;
                        if (la == lb && la != 0.0 && la * ba > 0.0 && la * bb > 0.0) {
                            const double Ga = cba * ga + ba, Gb = cba * gb + bb;
                            const double wa = la / ba, wb = la / bb;
                            const double D = wb - wa;
                            const double c1 = Ga * D - (Gb - Ga) * wa;
                            const double e = (Gb - Ga) * la;
                            const double disc = c1 * c1 + 4.0 * D * e;
                            const double qq = 0.5 * (c1 + copysign(sqrt(fmax(disc, 0.0)), c1));
                            const double x1 = qq / D, x2 = -e / qq;
                            const double bl = fmin(ba, bb), bh = fmax(ba, bb);
                            const bool in1 = x1 > bl && x1 < bh, in2 = x2 > bl && x2 < bh;
                            const double fpm = ha * (in1 ? x1 : x2) - vn;
                            if (disc >= 0.0 && (in1 || in2) && isfinite(fpm)) fp = fpm;
                        }
                    }
                    if (brk && isfinite(fp)) {
                        ue = fp;                             // bracketed step
                    } else if (!brk && !secok) {
                        ue = u1 + fac * r1;                  // grow along g until g changes sign
                        fac *= 2.0;
                    } else {
                        double sec = -(u1 - u0) / (r1 - r0);
                        sec = isfinite(sec) ? fmin(fmax(sec, -OMEGA_MAX), OMEGA_MAX) : 1.0;
                        ue = u1 + sec * r1;                  // secant while it converges
                    }
                }
                // trial orbits stay within BETA_TRIAL cells beyond the iterate's own orbit, per
                // axis (the growing steps along g would otherwise run past any neighbourhood
                // of the root)
                ue = fmin(fmax(ue, -blim / cba - vn), blim / cba - vn);
            }
        }
        const double vsa = active ? ue + vn : 0.0;
        const double vs[3] = {of(vsa, 0), of(vsa, 1), of(vsa, 2)};
        int nseg = 0;
        const double vw = push_eval_shared<QUAD, FROM>(p, k, comp, x0, st, vs, Pn, table, ctab, nseg);
        const double res = vw - ue;                          // g of this lane's component
        const double gp = of(res, paxis < 3 ? paxis : 0);
        const double a0 = max3(sl ? 0.0 : fabs(r0)), a1 = max3(sl ? 0.0 : fabs(res));
        bool done = false;
        if (active) {
            if (phase >= 2 && nseg < 0) atomicOr(status, DEV_ERR_SEGMENTS);
            if (k == 0) neval += 1.0;
            if (phase == 0) {
                gm = gp;
                phase = 1;
            } else if (phase == 1) {
                if (comp == paxis) sl = gm > 0.0 && gp < 0.0;
                ++paxis;
                while (paxis < 3 && !((probes >> paxis) & 1)) ++paxis;
                if (paxis < 3) {
                    phase = 0;
                } else {
                    if (sl) u1 = uland;
                    phase = 2;
                }
            } else if (phase == 2) {
                r1 = sl ? 0.0 : res;
                if (sl) r0 = 0.0;
                brk = !sl && r0 * r1 < 0.0;
                ua = u0;
                ga = r0;
                ub = u1;
                gb = r1;
                side = 0.0;
                secok = fabs(r1) <= 0.5 * fabs(r0);
                fac = 2.0;
                nrep = 0;
                // the best evaluation so far, whole (the components are coupled): the smallest
                // largest-component |g|; pinned components land on their knot
                bu = sl ? uland : (a1 < a0 ? u1 : u0);
                brs = fmin(a0, a1);
                phase = 3;
                done = nstep >= LOCAL_STEPS - 1 || brs <= tol;
            } else {
                const double r2 = sl ? 0.0 : res;
                if (a1 < brs) {
                    brs = a1;
                    bu = ue;
                }
                secok = secok && fabs(r2) <= 0.5 * fabs(r1);
                if (brk) {
                    if (r2 * gb > 0.0) {               // replaces the b end
                        nrep = side > 0.0 ? nrep + 1 : 1;
                        ub = ue;
                        gb = r2;
                        side = 1.0;
                    } else {                           // replaces the a end
                        nrep = side < 0.0 ? nrep + 1 : 1;
                        ua = ue;
                        ga = r2;
                        side = -1.0;
                    }
                    // the same end replaced twice running: the kept end is stale (its g was
                    // taken before the other components moved) or regula falsi stagnates;
                    // released, the next step is a secant one from two fresh points
                    if (nrep >= 2) {
                        brk = false;
                        secok = true;
                        nrep = 0;
                        side = 0.0;
                    }
                } else if (!sl && r2 * r1 < 0.0) {
                    brk = true;
                    ua = u1;
                    ga = r1;
                    ub = ue;
                    gb = r2;
                }
                u0 = u1;
                r0 = r1;
                u1 = ue;
                r1 = r2;
                ++nstep;
                done = nstep >= LOCAL_STEPS - 1 || brs <= tol;
            }
        }
        if (!__any_sync(full, done)) continue;
        // the particle's solve is over: its best iterate, sliding marks, e_v terms and current.
        // A solve that ends above the tolerance on the landing of its nearest knot, or that
        // fails (best residual above FAIL_RES of the speed) with a component starting within
        // D_FALLBACK of a knot: that root lies in the hair past the knot that double precision
        // (or the steps) did not resolve, and the component slides onto the knot.  Its energy
        // defect is then bounded by vbar_a = d H / dt times its residual, where it would
        // otherwise be the whole velocity times that residual; below FAIL_RES the residual
        // itself costs less.
        const bool failed = brs > FAIL_RES * spd;
        const bool hair = failed && fabs(dk) < D_FALLBACK;
        if (done && ((brs > tol && bu == uland) || hair)) sl = true;
        const int pinned = bits3(hair), slides = bits3(sl);
        if (done && sl) bu = uland;
        const double v2 = bu + vn;
        const double v2n[3] = {of(v2, 0), of(v2, 1), of(v2, 2)};
        if (done) {
            if (!isfinite(bu)) atomicOr(status, DEV_ERR_NONFINITE);
            if (k < 3) {
                const double d = bu - vit[comp * np + i];
                ev_num += d * d;
                ev_den += bu * bu;
                vnew[comp * np + i] = bu;
            }
            if (k == 0) {
                slide[i] = (uint8_t)(slides | SLIDE_CREPT);
                nsolve += 1.0;
                nfail += failed ? 1.0 : 0.0;
                nfail_free += (failed && !pinned) ? 1.0 : 0.0;
            }
            double beta[3], w[3];
            int ns;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                beta[a] = p.cb[a] * v2n[a];
                w[a] = p.q_dV_half * v2n[a];
            }
            if constexpr (QUAD == 0) {
                const int64_t N = p.m.ncell;
                CellStart<double> s = st;
                ns = for_each_piece(s, beta, p.m, [&](double h, double, const double mid[3], const int c[3]) {
                    double W[8];
                    node_weights(piece_moments(h, mid, beta), W);
#pragma unroll
                    for (int t = 0; t < 8 / LANES; ++t) {
                        const int kk = k + t * LANES;
                        int cn[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) cn[a] = ((kk >> a) & 1) ? next_cell(c[a], p.m.n[a]) : c[a];
                        const int64_t g = cell_row(cn, p.m);
                        const double Wk = h * pick8(W, kk);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            if (p.det) exact_add(p.acc, a * N + g, w[a] * Wk);
                            else atomicAdd(Jnext + a * N + g, w[a] * Wk);
                        }
                    }
                });
            } else if (p.split) {
                if (p.order == 2) ns = scatter_pieces<2>(p, x0, beta, w, Jnext, k, LANES);
                else if (p.order == 3) ns = scatter_pieces<3>(p, x0, beta, w, Jnext, k, LANES);
                else ns = scatter_pieces<1>(p, x0, beta, w, Jnext, k, LANES);
            } else {
                ns = k == 0 ? scatter_orbit(p, x0, beta, w, Jnext) : 0;
            }
            if (ns < 0) atomicOr(status, DEV_ERR_SEGMENTS);
            active = false;
        }
        __syncwarp();
    }
    write_partial<double>(partials, S_EVL_NUM, ev_num, sm, false);
    write_partial<double>(partials, S_EVL_DEN, ev_den, sm, false);
    write_partial<double>(partials, S_LOCAL_SOLVES, nsolve, sm, false);
    write_partial<double>(partials, S_LOCAL_EVALS, neval, sm, false);
    write_partial<double>(partials, S_LOCAL_FAILED, nfail, sm, false);
    write_partial<double>(partials, S_LOCAL_FAILED_FREE, nfail_free, sm, false);
}

__global__ void k_kinetic(StepParams p, const double* __restrict__ v, double* __restrict__ partials) {
    __shared__ double sm[32];
    const int64_t np = p.np;
    double k = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        double a = v[i], b = v[np + i], c = v[2 * np + i];
        k += 0.5 * p.mass * (a * a + b * b + c * c);
    }
    write_partial<double>(partials, S_K, k, sm, false);
}

// ---- counting sort by cell of x^n -------------------------------------------------------

__global__ void k_sort_keys(StepParams p, const double* __restrict__ xi, int32_t* __restrict__ key,
                            int32_t* __restrict__ count) {
    const int64_t np = p.np;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        int c0 = min(max((int)floor(xi[i]), 0), p.m.n[0] - 1);
        int c1 = min(max((int)floor(xi[np + i]), 0), p.m.n[1] - 1);
        int c2 = min(max((int)floor(xi[2 * np + i]), 0), p.m.n[2] - 1);
        int32_t k = (int32_t)node_index(c0, c1, c2, p.m);
        key[i] = k;
        atomicAdd(count + k, 1);
    }
}

// Exclusive scan of n ints in blocks of 1024 (phase 1: local scan and block totals).
__global__ void k_scan_local(const int32_t* __restrict__ in, int32_t* __restrict__ out, int32_t* __restrict__ totals,
                             int64_t n) {
    __shared__ int32_t s[1024];
    int64_t i = blockIdx.x * 1024LL + threadIdx.x;
    int32_t v = i < n ? in[i] : 0;
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        int32_t t = threadIdx.x >= o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += t;
        __syncthreads();
    }
    if (i < n) out[i] = s[threadIdx.x] - v;
    if (threadIdx.x == 1023) totals[blockIdx.x] = s[1023];
}

// Phase 2: one block scans the block totals sequentially in chunks of 1024.
__global__ void k_scan_totals(int32_t* __restrict__ totals, int nb) {
    __shared__ int32_t s[1024];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += 1024) {
        int i = base + threadIdx.x;
        int32_t v = i < nb ? totals[i] : 0;
        s[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            int32_t t = threadIdx.x >= o ? s[threadIdx.x - o] : 0;
            __syncthreads();
            s[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) totals[i] = carry + s[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry += s[1023];
        __syncthreads();
    }
}

__global__ void k_scan_add(int32_t* __restrict__ out, const int32_t* __restrict__ totals, int64_t n) {
    int64_t i = blockIdx.x * 1024LL + threadIdx.x;
    if (i < n) out[i] += totals[blockIdx.x];
}

// Place particle i at offset[key] + (arrival order within its cell) in the destination arrays.
__global__ void k_sort_scatter(StepParams p, const int32_t* __restrict__ key, const int32_t* __restrict__ offset,
                               int32_t* __restrict__ cursor, const double* __restrict__ xi, const double* __restrict__ v,
                               const double* __restrict__ P, const double* __restrict__ vprev,
                               const int64_t* __restrict__ id, double* __restrict__ xi_d, double* __restrict__ v_d,
                               double* __restrict__ P_d, double* __restrict__ vprev_d, int64_t* __restrict__ id_d) {
    const int64_t np = p.np;
    const int lane = threadIdx.x & 31;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t k = key[i];
        // the lanes of a warp with the same cell take consecutive places with one atomic (the
        // particles are nearly sorted already, so a warp holds one or two cells)
        const unsigned act = __activemask();
        const unsigned peers = __match_any_sync(act, k);
        const int leader = __ffs(peers) - 1;
        int first = 0;
        if (lane == leader) first = atomicAdd(cursor + k, __popc(peers));
        first = __shfl_sync(peers, first, leader);
        const int64_t pos = (int64_t)offset[k] + first + __popc(peers & ((1u << lane) - 1u));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            xi_d[a * np + pos] = xi[a * np + i];
            v_d[a * np + pos] = v[a * np + i];
            P_d[a * np + pos] = P[a * np + i];
            vprev_d[a * np + pos] = vprev[a * np + i];
        }
        id_d[pos] = id[i];
    }
}

// ---- stable LSD radix sort of the cell keys (deterministic mode) ---------------------------
//
// 8-bit digits; each pass counts the digits of every tile of RS_TILE keys, scans the counts
// in digit-major order (so tile b's keys of digit d go after those of every earlier tile),
// and scatters each tile in index order, ranking equal digits within a warp by
// __match_any_sync.  Every pass is stable, so the result is ordered by key and, among equal
// keys, by the previous order: a deterministic permutation.

constexpr int RS_RADIX = 256, RS_ITEMS = 8, RS_TILE = THREADS * RS_ITEMS;
static_assert(THREADS == RS_RADIX, "one thread per digit in the scatter's bookkeeping");

__global__ void k_rs_hist(const int32_t* __restrict__ key, int64_t n, int shift, int ntiles,
                          int32_t* __restrict__ hist) {
    __shared__ int32_t cnt[RS_RADIX];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = base + r * THREADS + threadIdx.x;
        if (i < n) atomicAdd(&cnt[(key[i] >> shift) & (RS_RADIX - 1)], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

__global__ void k_rs_scatter(const int32_t* __restrict__ key_in, const int32_t* __restrict__ val_in, int64_t n,
                             int shift, int ntiles, const int32_t* __restrict__ offs, int32_t* __restrict__ key_out,
                             int32_t* __restrict__ val_out) {
    __shared__ int32_t run[RS_RADIX];
    __shared__ int32_t wc[THREADS / 32][RS_RADIX];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    run[tid] = offs[(int64_t)tid * ntiles + blockIdx.x];
#pragma unroll
    for (int v = 0; v < THREADS / 32; ++v) wc[v][tid] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = base + r * THREADS + tid;
        const bool valid = i < n;
        const int32_t k = valid ? key_in[i] : 0;
        const int d = valid ? (k >> shift) & (RS_RADIX - 1) : RS_RADIX + lane;   // invalid lanes: own groups
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && rank == 0) wc[w][d] = __popc(peers);
        __syncthreads();
        int pos = 0;
        if (valid) {
            pos = run[d] + rank;
            for (int v = 0; v < w; ++v) pos += wc[v][d];
        }
        __syncthreads();
        int add = 0;
#pragma unroll
        for (int v = 0; v < THREADS / 32; ++v) {
            add += wc[v][tid];
            wc[v][tid] = 0;
        }
        run[tid] += add;
        __syncthreads();
        if (valid) {
            key_out[pos] = k;
            val_out[pos] = val_in[i];
        }
    }
}

__global__ void k_iota(int64_t n, int32_t* __restrict__ a) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = (int32_t)i;
}

// Destination j takes particle perm[j].
__global__ void k_sort_gather(StepParams p, const int32_t* __restrict__ perm, const double* __restrict__ xi,
                              const double* __restrict__ v, const double* __restrict__ P,
                              const double* __restrict__ vprev, const int64_t* __restrict__ id,
                              double* __restrict__ xi_d, double* __restrict__ v_d, double* __restrict__ P_d,
                              double* __restrict__ vprev_d, int64_t* __restrict__ id_d) {
    const int64_t np = p.np;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < np; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = perm[j];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            xi_d[a * np + j] = xi[a * np + i];
            v_d[a * np + j] = v[a * np + i];
            P_d[a * np + j] = P[a * np + i];
            vprev_d[a * np + j] = vprev[a * np + i];
        }
        id_d[j] = id[i];
    }
}

// dst[c, id[i]] = scale_c * src[c, i]  (device order -> caller order)
__global__ void k_unpermute(int64_t np, const int64_t* __restrict__ id, const double* __restrict__ src,
                            double* __restrict__ dst, double s0, double s1, double s2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = id[i];
        dst[j] = s0 * src[i];
        dst[np + j] = s1 * src[np + i];
        dst[2 * np + j] = s2 * src[2 * np + i];
    }
}

// dst[c, i] = scale_c * src[c, id[i]]  (caller order -> device order)
__global__ void k_permute_in(int64_t np, const int64_t* __restrict__ id, const double* __restrict__ src,
                             double* __restrict__ dst, double s0, double s1, double s2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = id[i];
        dst[i] = s0 * src[j];
        dst[np + i] = s1 * src[np + j];
        dst[2 * np + i] = s2 * src[2 * np + j];
    }
}

}  // namespace

StepParams make_params(const Ctx& c) {
    StepParams p;
    p.m = c.m;
    for (int a = 0; a < 3; ++a) {
        p.H[a] = c.H[a];
        p.invH[a] = c.invH[a];
    }
    p.dt = c.cfg.dt;
    p.q = c.q;
    p.mass = c.mass;
    p.inv_mass = 1.0 / c.mass;
    p.q_dV = c.q / c.dV;
    for (int a = 0; a < 3; ++a) {
        p.cb[a] = 0.5 * c.cfg.dt / c.H[a];
        p.ihs[a] = 0.5 * c.invH[a];
    }
    p.dtq = c.cfg.dt * c.q;
    p.q_dV_half = 0.5 * p.q_dV;
    p.np = c.np;
    p.split = c.cfg.split_orbit_at_knots;
    p.nq = c.nq;
    p.rule = c.nq * (c.nq - 1) / 2;
    p.accel = c.cfg.picard_accel;
    p.hist = 0;
    p.slow_floor = c.run.after32 ? SLOW_FLOOR_AFTER32 : SLOW_FLOOR;
    p.order = c.cfg.shape_order;
    p.koff = (c.cfg.shape_order % 2 == 0) ? 0.5 : 0.0;
    p.det = c.cfg.deterministic;
    p.acc = ExactAcc{c.acc_hi, c.acc_lo, c.inv_u_J, c.dev_status};
    return p;
}

// Where the closed-form FP64 kernels take the fields from (see Fields).
static Fields fields_of(const Ctx& c) {
    if (c.cfg.deterministic) return c.cell_form ? FROM_EITHER : FROM_NODES;
    return c.ctab ? FROM_CELLS : FROM_NODES;
}

// Opt the depositing kernels in to their dynamic shared memory (above the 48 KB default where the chunk
// is large; once per context, on its device).
bool setup_particle_kernels() {
    const int bytes = (int)ChunkLarge::smem(), push = (int)ChunkPush::smem();
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_first_scatter_cell<4, 2>, at, bytes) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_CELLS, 4, 2>, at, bytes) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_NODES, 4, 2>, at, bytes) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_EITHER, 4, 2>, at, bytes) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_CELLS, 8, 2>, at, push) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_NODES, 8, 2>, at, push) == cudaSuccess &&
           cudaFuncSetAttribute(k_push_cell<false, FROM_EITHER, 8, 2>, at, push) == cudaSuccess;
}

// Chunks of one warp while they leave every scheduler at most two of them.
bool small_chunks(const Ctx& c) { return c.np <= (int64_t)c.sms * 8 * ChunkSmall::SIZE; }

// The pushes' larger chunks (two blocks an SM) while each block gets at least two.
bool wide_chunks(const Ctx& c) { return c.np >= 2 * (int64_t)c.sms * 2 * ChunkPush::SIZE; }

// Grid of the kernels that walk chunks, and of the push of this context's kind (partials per block).
int chunk_blocks(const Ctx& c) {
    const int size = small_chunks(c) ? ChunkSmall::SIZE : ChunkLarge::SIZE;
    const int64_t b = (c.np + size - 1) / size, cap = std::min<int64_t>((int64_t)c.sms * c.push_bps, MAX_BLOCKS);
    return (int)std::max<int64_t>(1, std::min(b, std::max<int64_t>(cap, small_chunks(c) ? b : 1)));
}

int push_blocks(const Ctx& c) { return c.closed ? chunk_blocks(c) : particle_blocks(c); }

int local_blocks(const Ctx& c) {
    const int64_t b = (c.np * 8 + THREADS - 1) / THREADS;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)c.sms * LOCAL_MINB));
}

int particle_blocks(const Ctx& c) {
    int64_t b = (c.np + THREADS - 1) / THREADS;
    int64_t cap = (int64_t)c.sms * c.push_bps;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

void launch_init_positions(Ctx& c, const double* x_dev) {
    StepParams p = make_params(c);
    k_init_positions<<<particle_blocks(c), THREADS, 0, c.stream>>>(p, x_dev, c.xi, c.id);
    ++c.launches;
}

void launch_set_positions(Ctx& c, const double* src_dev) {
    k_set_positions<<<particle_blocks(c), THREADS, 0, c.stream>>>(make_params(c), c.id, src_dev, c.xi);
    ++c.launches;
}

void launch_point_deposit(Ctx& c) {
    StepParams p = make_params(c);
    p.acc.inv_u = c.inv_u_rho;
    k_point_deposit<<<particle_blocks(c), THREADS, 0, c.stream>>>(p, c.xi, c.rho0);
    ++c.launches;
    if (c.cfg.deterministic) launch_exact_finish(c, c.rho0, c.m.ncell, c.inv_u_rho);
}

void launch_first_scatter(Ctx& c, double* J, const double* v_iter_or_null) {
    StepParams p = make_params(c);
    int nb = particle_blocks(c);
    if (c.closed && small_chunks(c))
        k_first_scatter_cell<1, 1><<<chunk_blocks(c), 32, ChunkSmall::smem(), c.stream>>>(
            p, c.xi, c.v, c.vprev, v_iter_or_null, c.vit, J, c.partials, c.dev_status);
    else if (c.closed)
        k_first_scatter_cell<4, 2><<<chunk_blocks(c), 128, ChunkLarge::smem(), c.stream>>>(
            p, c.xi, c.v, c.vprev, v_iter_or_null, c.vit, J, c.partials, c.dev_status);
    else
        k_first_scatter<<<nb, THREADS, 0, c.stream>>>(p, c.xi, c.v, c.vprev, v_iter_or_null, c.vit, J, c.partials,
                                                         c.dev_status);
    ++c.launches;
    if (c.cfg.deterministic) launch_exact_finish(c, J, 3 * c.m.ncell, c.inv_u_J);
}

void launch_push(Ctx& c, const double* vit, double* vnew, double* Jnext, bool commit, bool diag) {
    StepParams p = make_params(c);
    p.hist = !commit && c.cfg.picard_accel && c.run.hist;
    int nb = particle_blocks(c);
    const bool det = c.cfg.deterministic && !commit;
    const bool closed = c.closed;
    if (!commit) cudaMemsetAsync(c.creep_count, 0, 2 * sizeof(int), c.stream);   // count, k_local queue head
#define PIC_PUSH(C, D)                                                                                           \
    k_push<C, D><<<nb, THREADS, 0, c.stream>>>(p, c.xi, c.v, c.P, vit, c.table, vnew, Jnext, c.xi_new, c.P_new, \
                                                  c.creep_list, c.creep_count, det ? c.creep_flag : nullptr,  \
                                                  c.slide,                                                    \
                                                  c.partials, c.dev_status)
    const FixedTables ft{c.table, reinterpret_cast<const longlong2*>(c.fxtab)};
    const Fields from = fields_of(c);
    const bool small = small_chunks(c), wide = wide_chunks(c);
#define PIC_PUSH_CELL_AS(C, T, W, I)                                                                              \
    k_push_cell<C, T, W, I><<<chunk_blocks(c), 32 * W, C ? sizeof(ChunkOrder<W, I>) : ChunkOrder<W, I>::smem(),     \
                              c.stream>>>(p, c.xi, c.v, c.P, vit, ft, vnew, Jnext, c.xi_new, c.P_new, c.creep_list, \
                                          c.creep_count, det ? c.creep_flag : nullptr, c.slide, c.partials,        \
                                          c.dev_status)
#define PIC_PUSH_CELL(C, T)                \
    do {                                   \
        if (small) PIC_PUSH_CELL_AS(C, T, 1, 1); \
        else if (wide) PIC_PUSH_CELL_AS(C, T, 8, 2); \
        else PIC_PUSH_CELL_AS(C, T, 4, 2);       \
    } while (0)
#define PIC_COMMIT_DIAG(T, W, I)                                                                                  \
    k_commit_diag<T, W, I><<<chunk_blocks(c), 32 * W, sizeof(ChunkOrder<W, I>), c.stream>>>(                        \
        p, c.xi, c.v, c.P, vit, c.table, c.ctab, vnew, c.xi_new, c.P_new, c.slide, c.partials, c.dev_status)
#define PIC_COMMIT_DIAG_AS(T)                  \
    do {                                       \
        if (small) PIC_COMMIT_DIAG(T, 1, 1);   \
        else PIC_COMMIT_DIAG(T, 4, 2);         \
    } while (0)
    if (closed && diag) {   // (commit)
        if (from == FROM_CELLS) PIC_COMMIT_DIAG_AS(FROM_CELLS);
        else if (from == FROM_EITHER) PIC_COMMIT_DIAG_AS(FROM_EITHER);
        else PIC_COMMIT_DIAG_AS(FROM_NODES);
    } else if (closed && commit) {
        if (from == FROM_CELLS) PIC_PUSH_CELL(true, FROM_CELLS);
        else if (from == FROM_EITHER) PIC_PUSH_CELL(true, FROM_EITHER);
        else PIC_PUSH_CELL(true, FROM_NODES);
    } else if (closed) {
        if (from == FROM_CELLS) PIC_PUSH_CELL(false, FROM_CELLS);
        else if (from == FROM_EITHER) PIC_PUSH_CELL(false, FROM_EITHER);
        else PIC_PUSH_CELL(false, FROM_NODES);
    } else if (!commit) {
        PIC_PUSH(false, false);
    } else if (!diag) {
        PIC_PUSH(true, false);
    } else {
        PIC_PUSH(true, true);
    }
#undef PIC_COMMIT_DIAG
#undef PIC_COMMIT_DIAG_AS
#undef PIC_PUSH
#undef PIC_PUSH_CELL
#undef PIC_PUSH_CELL_AS
    ++c.launches;
    // in deterministic mode the exact current is rounded once all of its deposits are in
    if (det && Jnext && !c.cfg.picard_accel) launch_exact_finish(c, Jnext, 3 * c.m.ncell, c.inv_u_J);
}

void launch_local(Ctx& c, const double* vit, double* vnew, double* Jnext) {
    StepParams p = make_params(c);
    const bool det = c.cfg.deterministic != 0;
    const int lb = local_blocks(c);
#define PIC_LOCAL(Q, T)                                                                                             \
    k_local<Q, T><<<lb, THREADS, 0, c.stream>>>(p, c.xi, c.v, c.P, vit, c.table, c.ctab, vnew, c.gsave, Jnext,        \
                                                c.creep_list, c.creep_count, det ? c.creep_flag : nullptr, c.slide, \
                                                c.creep_count + 1, c.partials, c.dev_status)
    const Fields from = fields_of(c);
    if (!c.closed) PIC_LOCAL(1, FROM_NODES);
    else if (from == FROM_CELLS) PIC_LOCAL(0, FROM_CELLS);
    else if (from == FROM_EITHER) PIC_LOCAL(0, FROM_EITHER);
    else PIC_LOCAL(0, FROM_NODES);
#undef PIC_LOCAL
    ++c.launches;
    if (det && Jnext) launch_exact_finish(c, Jnext, 3 * c.m.ncell, c.inv_u_J);
}

void launch_kinetic(Ctx& c) {
    StepParams p = make_params(c);
    k_kinetic<<<particle_blocks(c), THREADS, 0, c.stream>>>(p, c.v, c.partials);
    ++c.launches;
}

// out[i] = (hi[i] 2^40 + lo[i]) u, then hi[i] = lo[i] = 0 for the next deposit (the
// deterministic mode's exact accumulators; see ExactAcc).
__global__ void k_exact_finish(int64_t n, long long* __restrict__ hi, long long* __restrict__ lo, double u,
                               double* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        out[i] = ((double)hi[i] * 0x1p40 + (double)lo[i]) * u;
        hi[i] = 0;
        lo[i] = 0;
    }
}

void launch_exact_finish(Ctx& c, double* out, int64_t n, double inv_u) {
    int64_t nb = (n + THREADS - 1) / THREADS;
    if (nb > (int64_t)c.sms * 8) nb = (int64_t)c.sms * 8;
    if (nb < 1) nb = 1;
    k_exact_finish<<<(int)nb, THREADS, 0, c.stream>>>(n, c.acc_hi, c.acc_lo, 1.0 / inv_u, out);
    ++c.launches;
}

int radix_tiles(int64_t np) { return (int)std::max<int64_t>(1, (np + RS_TILE - 1) / RS_TILE); }

// Stable radix sort of the cell keys; the particle arrays are then gathered in that order.
void launch_sort_stable(Ctx& c) {
    StepParams p = make_params(c);
    const int64_t N = c.m.ncell, np = c.np;
    const int nb = particle_blocks(c);
    cudaMemsetAsync(c.count, 0, sizeof(int32_t) * N, c.stream);
    k_sort_keys<<<nb, THREADS, 0, c.stream>>>(p, c.xi, c.rs_key[0], c.count);
    k_iota<<<nb, THREADS, 0, c.stream>>>(np, c.rs_val[0]);
    c.launches += 2;
    int bits = 0;
    while (bits < 31 && ((int64_t)1 << bits) < N) ++bits;
    const int passes = std::max(1, (bits + 7) / 8);
    const int ntiles = radix_tiles(np);
    const int64_t nh = (int64_t)RS_RADIX * ntiles;
    const int nsb = (int)((nh + 1023) / 1024);
    int cur = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        k_rs_hist<<<ntiles, THREADS, 0, c.stream>>>(c.rs_key[cur], np, shift, ntiles, c.rs_hist);
        k_scan_local<<<nsb, 1024, 0, c.stream>>>(c.rs_hist, c.rs_offs, c.rs_scan_tmp, nh);
        k_scan_totals<<<1, 1024, 0, c.stream>>>(c.rs_scan_tmp, nsb);
        k_scan_add<<<nsb, 1024, 0, c.stream>>>(c.rs_offs, c.rs_scan_tmp, nh);
        k_rs_scatter<<<ntiles, THREADS, 0, c.stream>>>(c.rs_key[cur], c.rs_val[cur], np, shift, ntiles, c.rs_offs,
                                                        c.rs_key[cur ^ 1], c.rs_val[cur ^ 1]);
        c.launches += 5;
        cur ^= 1;
    }
    k_sort_gather<<<nb, THREADS, 0, c.stream>>>(p, c.rs_val[cur], c.xi, c.v, c.P, c.vprev, c.id, c.xi_new, c.vnew,
                                                c.P_new, c.vit, c.id_tmp);
    ++c.launches;
    std::swap(c.xi, c.xi_new);
    std::swap(c.v, c.vnew);
    std::swap(c.P, c.P_new);
    std::swap(c.vprev, c.vit);
    std::swap(c.id, c.id_tmp);
}

void launch_sort(Ctx& c) {
    if (c.cfg.deterministic) {
        launch_sort_stable(c);
        return;
    }
    StepParams p = make_params(c);
    const int64_t N = c.m.ncell;
    int nb = particle_blocks(c);
    cudaMemsetAsync(c.count, 0, sizeof(int32_t) * N, c.stream);
    cudaMemsetAsync(c.cursor, 0, sizeof(int32_t) * N, c.stream);
    k_sort_keys<<<nb, THREADS, 0, c.stream>>>(p, c.xi, c.key, c.count);
    ++c.launches;
    int nsb = (int)((N + 1023) / 1024);
    k_scan_local<<<nsb, 1024, 0, c.stream>>>(c.count, c.offset, c.scan_tmp, N);
    ++c.launches;
    k_scan_totals<<<1, 1024, 0, c.stream>>>(c.scan_tmp, nsb);
    ++c.launches;
    k_scan_add<<<nsb, 1024, 0, c.stream>>>(c.offset, c.scan_tmp, N);
    ++c.launches;
    // destinations: the free iterate/commit buffers of the step
    k_sort_scatter<<<nb, THREADS, 0, c.stream>>>(p, c.key, c.offset, c.cursor, c.xi, c.v, c.P, c.vprev, c.id,
                                                 c.xi_new, c.vnew, c.P_new, c.vit, c.id_tmp);
    ++c.launches;
    std::swap(c.xi, c.xi_new);
    std::swap(c.v, c.vnew);
    std::swap(c.P, c.P_new);
    std::swap(c.vprev, c.vit);
    std::swap(c.id, c.id_tmp);
}

// g[c, list[k]] = gsave[c, list[k]] for the particles solved locally in the last iteration.
__global__ void k_patch_local(int64_t np, const int32_t* __restrict__ list, const int* __restrict__ count,
                              const double* __restrict__ gsave, double* __restrict__ g) {
    const int n = *count;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int64_t i = list[k];
        g[i] = gsave[i];
        g[np + i] = gsave[np + i];
        g[2 * np + i] = gsave[2 * np + i];
    }
}

void launch_patch_local(Ctx& c, double* g) {
    k_patch_local<<<std::max(1, c.sms), THREADS, 0, c.stream>>>(c.np, c.creep_list, c.creep_count, c.gsave, g);
    ++c.launches;
}

// dst[id[i]] = the sliding bits (components 0..2) of particle i (device order -> caller order).
__global__ void k_slide_out(int64_t np, const int64_t* __restrict__ id, const uint8_t* __restrict__ slide,
                            uint8_t* __restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x)
        dst[id[i]] = slide[i] & 7u;
}

void launch_slide_out(Ctx& c, uint8_t* dst) {
    k_slide_out<<<particle_blocks(c), THREADS, 0, c.stream>>>(c.np, c.id, c.slide, dst);
    ++c.launches;
}

void launch_unpermute(Ctx& c, const double* src, double* dst, double s0, double s1, double s2) {
    k_unpermute<<<particle_blocks(c), THREADS, 0, c.stream>>>(c.np, c.id, src, dst, s0, s1, s2);
    ++c.launches;
}

void launch_permute_in(Ctx& c, const double* src, double* dst, double s0, double s1, double s2) {
    k_permute_in<<<particle_blocks(c), THREADS, 0, c.stream>>>(c.np, c.id, src, dst, s0, s1, s2);
    ++c.launches;
}

}  // namespace pic
