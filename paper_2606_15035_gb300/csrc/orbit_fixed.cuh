// The closed-form push of one particle with its piece integrals in 64-bit fixed point (sm_103a).
//
// Same formulas as piece_impulse (orbit_cell.cuh).  Of a particle's ~330 FP64 instructions in the
// iterate about 230 were the contractions and moments of its pieces; on the integer pipe they leave the
// FP64 pipe the walk (9 a piece), the conversions at the end and the gates.
//
// Formats: coordinates, moments and piece lengths at 2^-62; v^p + v^n at 2^(ev - 1084), ev the largest
// biased exponent of its components; the table's mixed differences (A^{n+1} and its change together,
// and -grad phi) at 2^(e - 1080), e the largest exponent of that group in the cell: sums of up to eight of
// them stay in range.  A factor of a product is its upper 60 (velocities) or 56 bits (differences), so that a
// piece's integrals carry an error of a few 2^-55 of the cell's largest difference times the largest
// velocity component, where FP64 rounds each product at 2^-53 of itself: small components beside large ones
// of the same cell are held to that absolute bound.  Pieces are summed in FP64.  (With one exponent for the
// whole mesh, a field of 2^-20 of its peak elsewhere was left with 35 bits.)  The end point's A_h^{n+1} adds
// the differences to the cell's lowest node value in FP64.
#pragma once

#include "fixed.cuh"
#include "orbit_cell.cuh"

namespace pic {

constexpr int FX_FIELD_UP = 5;   // fixed_of's shift for the table: 58 bits
constexpr int FX_V_UP = 9;       // ... for velocities: 62 bits

struct FixedTables {
    const double* nodes;      // gather table
    const longlong2* cells;   // fixed-point cell table
};

// Loader of a cell's entries from the fixed-point table, or from a copy of the cell's part of it.  The
// entries k = 0 of the A columns are not used; two of them hold the exponents of the cell's groups.
struct FixedLoad {
    const longlong2* t;
    __device__ __forceinline__ FixedLoad(FixedTables ft, const int c[3], const MeshDims& m)
        : t(ft.cells + (CELL_VALUES / 2) * cell_row(c, m)) {}
    __device__ __forceinline__ void operator()(int p, int col, long long& a, long long& b) const {
        const longlong2 q = __ldg(t + p * CELL_COLS + col);
        a = q.x;
        b = q.y;
    }
    __device__ __forceinline__ int top_A() const { return (int)__ldg(&t[0].x); }
    __device__ __forceinline__ int top_g() const { return (int)__ldg(&t[1].x); }
};

// A cell's entries as the fixed-point table has them, made from the gather table.
struct FixedOfNodes {
    longlong2 t[CELL_VALUES / 2];
    __device__ __forceinline__ FixedOfNodes(const double* nodes, const int c[3], const int n[3]) {
        double2 q[CELL_VALUES / 2];
        entries_of_nodes(nodes, c[0], c[1], c[2], n[0], n[1], n[2], q);
        int top[2] = {64, 64};
        for (int k = 0; k < CELL_VALUES / 2; ++k) {
            const int col = k % CELL_COLS;
            const int e = max(k < 6 ? 0 : exponent_of(q[k].x), exponent_of(q[k].y));
            if (col < 6) top[0] = max(top[0], e);
            else top[1] = max(top[1], e);
        }
        for (int k = 0; k < CELL_VALUES / 2; ++k) {
            const int e = k % CELL_COLS < 6 ? top[0] : top[1];
            t[k].x = k < 2 ? top[k] : (k < 6 ? 0 : fixed_of(q[k].x, e, FX_FIELD_UP));
            t[k].y = fixed_of(q[k].y, e, FX_FIELD_UP);
        }
    }
    __device__ __forceinline__ void operator()(int p, int col, long long& a, long long& b) const {
        a = t[p * CELL_COLS + col].x;
        b = t[p * CELL_COLS + col].y;
    }
    __device__ __forceinline__ int top_A() const { return (int)t[0].x; }
    __device__ __forceinline__ int top_g() const { return (int)t[1].x; }
};

// The unit 2^e' of a sum, e' = e - 1023, of quantities whose largest biased exponent is `top`: NaN where that
// is not finite.
__device__ __forceinline__ double fixed_unit(int e, int top) { return top < 0x7ff ? pow2_biased(e) : NAN; }

// accF_j += int (D_j A)^T v, the difference along j per cell, and accG_j -= int d_j phi of one piece (h, s_mid,
// midpoint, displacement d = h beta), v in the format above.
template <typename L>
__device__ __forceinline__ void piece_impulse_fixed(double h, double sm, const double mid[3], const double d[3],
                                                    const Fs v[3], int ev, const L& ld, double accF[3], double accG[3]) {
    const Fs hf = fs_of(fixed_of(h, 1023, 10));
    const Fs nms = fs_of(fixed_of(sm, 1023, 10) - FX_ONE);   // s_mid - 1
    Fs m[3], e[3], Pxy, Pxz, Pyz, S, E3, E5, E6;
    {
        const Fs c12 = fs_of(FX_ONE / 12);
        Fs df[3], d12[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            m[a] = fs_of(fixed_of(mid[a], 1023, 10));
            df[a] = fs_of(fixed_of(d[a], 1023, 10));
            d12[a] = fx_sum(df[a], c12).factor();
            e[a] = fx_sum(hf, d12[a]).factor();
        }
        Pxy = fx_sum(m[0], m[1], df[0], d12[1]).factor();
        Pxz = fx_sum(m[0], m[2], df[0], d12[2]).factor();
        Pyz = fx_sum(m[1], m[2], df[1], d12[2]).factor();
        // <w_x w_y w_z> = m_x P_yz + d_x (m_y d_z + m_z d_y) / 12
        S = fx_sum(m[0], Pyz, df[0], fx_sum(m[1], d12[2], m[2], d12[1]).factor()).factor();
        E3 = fx_sum(m[0], e[1], m[1], e[0]).factor();
        E5 = fx_sum(m[0], e[2], m[2], e[0]).factor();
        E6 = fx_sum(m[1], e[2], m[2], e[1]).factor();
    }
    FxSum F[3], g[3];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        Fs a[2], cc[2];
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            if (p == 0 && o == 0) continue;
            FxSum sc, sa;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                long long q[2];
                ld(p, 3 + c, q[0], q[1]);
                sc.add(fs_of(q[o]), v[c]);
                ld(p, c, q[0], q[1]);
                sa.add(fs_of(q[o]), v[c]);
            }
            cc[o] = sc.factor();
            sa.add(nms, cc[o]);
            a[o] = sa.factor();
        }
        if (p == 0) {            // k = 1: x
            F[0].add_one(a[1]);
        } else if (p == 1) {     // k = 2: y, k = 3: xy
            F[1].add_one(a[0]);
            F[0].add(a[1], m[1]);
            F[0].add(cc[1], e[1]);
            F[1].add(a[1], m[0]);
            F[1].add(cc[1], e[0]);
        } else if (p == 2) {     // k = 4: z, k = 5: xz
            F[2].add_one(a[0]);
            F[0].add(a[1], m[2]);
            F[0].add(cc[1], e[2]);
            F[2].add(a[1], m[0]);
            F[2].add(cc[1], e[0]);
        } else {                 // k = 6: yz, k = 7: xyz
            F[1].add(a[0], m[2]);
            F[1].add(cc[0], e[2]);
            F[2].add(a[0], m[1]);
            F[2].add(cc[0], e[1]);
            F[0].add(a[1], Pyz);
            F[0].add(cc[1], E6);
            F[1].add(a[1], Pxz);
            F[1].add(cc[1], E5);
            F[2].add(a[1], Pxy);
            F[2].add(cc[1], E3);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long g0, g1;
            ld(p, 6 + j, g0, g1);
            if (p == 0) g[j].add_one(fs_of(g0));
            else g[j].add(fs_of(g0), p == 1 ? m[1] : (p == 2 ? m[2] : Pyz));
            g[j].add(fs_of(g1), p == 0 ? m[0] : (p == 1 ? Pxy : (p == 2 ? Pxz : S)));
        }
    }
    const int eA = ld.top_A(), eG = ld.top_g();
    const double uF = fixed_unit(eA + ev - 1079, max(eA, ev)), uG = fixed_unit(eG - 57, eG);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        accF[j] = fma(uF, (double)fx_sum(hf, F[j].factor()).value(), accF[j]);
        accG[j] = fma(uG, (double)fx_sum(hf, g[j].factor()).value(), accG[j]);
    }
}

// A^{n+1} at coordinate r of the cell less its lowest node's value, in the table's format.
template <typename L>
__device__ __forceinline__ void cell_A1_fixed(const double r[3], const L& ld, long long out[3]) {
    Fs q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] = fs_of(fixed_of(r[a], 1023, 10));
    const Fs xy = fx_sum(q[0], q[1]).factor(), xz = fx_sum(q[0], q[2]).factor(), yz = fx_sum(q[1], q[2]).factor();
    const Fs xyz = fx_sum(xy, q[2]).factor();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        long long k0, k1, k2, k3, k4, k5, k6, k7;
        ld(0, c, k0, k1);
        ld(1, c, k2, k3);
        ld(2, c, k4, k5);
        ld(3, c, k6, k7);
        FxSum s;
        s.add(fs_of(k1), q[0]);
        s.add(fs_of(k2), q[1]);
        s.add(fs_of(k3), xy);
        s.add(fs_of(k4), q[2]);
        s.add(fs_of(k5), xz);
        s.add(fs_of(k6), yz);
        s.add(fs_of(k7), xyz);
        out[c] = s.value();
    }
}

// The same two from the gather table, for deterministic runs whose cell tables were refused: integers and
// single FP64 multiply-adds throughout, so that the bits are those of the table's (values in and out, which keeps
// the callers' in registers).
struct PieceSums {
    double F[3], G[3];
};
struct PieceOrbit {
    double h, sm, mid[3], d[3];
    Fs v[3];
    int ev, c[3], n[3];
};
static __device__ __noinline__ PieceSums piece_impulse_of_nodes(const double* nodes, PieceOrbit o, PieceSums s) {
    const FixedOfNodes ld(nodes, o.c, o.n);
    piece_impulse_fixed(o.h, o.sm, o.mid, o.d, o.v, o.ev, ld, s.F, s.G);
    return s;
}

struct CellA1 {
    long long a[3];
    int top;
};
static __device__ __noinline__ CellA1 cell_A1_of_nodes(const double* nodes, int c0, int c1, int c2, int n0, int n1, int n2,
                                                       double r0, double r1, double r2) {
    const int c[3] = {c0, c1, c2}, n[3] = {n0, n1, n2};
    const double r[3] = {r0, r1, r2};
    const FixedOfNodes ld(nodes, c, n);
    CellA1 A;
    cell_A1_fixed(r, ld, A.a);
    A.top = ld.top_A();
    return A;
}

}  // namespace pic
