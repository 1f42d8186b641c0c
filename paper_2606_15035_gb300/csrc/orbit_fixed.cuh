// The closed-form push of one particle with its piece integrals in 64-bit fixed point (sm_103a).
//
// Same formulas as piece_impulse (orbit_cell.cuh).  Of a particle's ~330 FP64 instructions in the
// iterate about 230 were the contractions and moments of its pieces; on the integer pipe they leave the
// FP64 pipe the walk (9 a piece), the conversions at the end and the gates.
//
// Formats: coordinates, moments and piece lengths at 2^-62; v^p + v^n at 2^(ev - 1084), ev the largest
// biased exponent of its components; the table's mixed differences (A^{n+1} and its change together,
// and -grad phi) at 2^(e - 1079), e the largest exponent of that group over the mesh: 57 bits of the
// largest difference, and sums of up to eight of them stay in range.  The end point's A_h^{n+1} adds the
// differences to the cell's lowest node value in FP64.
#pragma once

#include "fixed.cuh"
#include "orbit_cell.cuh"

namespace pic {

constexpr int FX_FIELD_UP = 4;   // fixed_of's shift for the table: 57 bits
constexpr int FX_V_UP = 9;       // ... for velocities: 62 bits

struct FixedLoad {
    const longlong2* t;
    __device__ __forceinline__ FixedLoad(const longlong2* table, const int c[3], const MeshDims& m)
        : t(table + (CELL_VALUES / 2) * cell_row(c, m)) {}
    __device__ __forceinline__ void operator()(int p, int col, long long& a, long long& b) const {
        const longlong2 q = __ldg(t + p * CELL_COLS + col);
        a = q.x;
        b = q.y;
    }
};

// accF_j += int (D_j A)^T v and accG_j -= int d_j phi of one piece (h, s_mid, midpoint, displacement
// d = h beta), in the formats above.
__device__ __forceinline__ void piece_impulse_fixed(double h, double sm, const double mid[3], const double d[3],
                                                    const Fx v[3], const FixedLoad& ld, long long accF[3],
                                                    long long accG[3]) {
    const Fx hf = fx_split(fixed_of(h, 1023, 10));
    const Fx nms = fx_split(fixed_of(sm, 1023, 10) - FX_ONE);   // s_mid - 1
    Fx m[3], e[3];
    long long E3, E5, E6;
    Fx Pxy, Pxz, Pyz, S;
    {
        const Fx c12 = fx_split(FX_ONE / 12);
        Fx df[3], d12[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            m[a] = fx_split(fixed_of(mid[a], 1023, 10));
            df[a] = fx_split(fixed_of(d[a], 1023, 10));
            d12[a] = fx_split(fx_mul(df[a], c12));
            e[a] = fx_split(fx_mul(hf, d12[a]));
        }
        const Fx kxy = fx_split(fx_mul(df[0], d12[1])), kxz = fx_split(fx_mul(df[0], d12[2]));
        const long long kyz = fx_mul(df[1], d12[2]);
        const long long kxyl = fx_mul(df[0], d12[1]), kxzl = fx_mul(df[0], d12[2]);
        Pxy = fx_split(fx_mad(m[0], m[1], kxyl));
        Pxz = fx_split(fx_mad(m[0], m[2], kxzl));
        Pyz = fx_split(fx_mad(m[1], m[2], kyz));
        S = fx_split(fx_mad(m[0], Pyz, fx_mad(m[1], kxz, fx_mul(m[2], kxy))));
        E3 = fx_mad(m[0], e[1], fx_mul(m[1], e[0]));
        E5 = fx_mad(m[0], e[2], fx_mul(m[2], e[0]));
        E6 = fx_mad(m[1], e[2], fx_mul(m[2], e[1]));
    }
    long long F[3], g[3];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        Fx a[2], cc[2];
        {
            long long x0, x1, y0, y1, z0, z1;
            ld(p, 3, x0, x1);
            ld(p, 4, y0, y1);
            ld(p, 5, z0, z1);
            if (p > 0) cc[0] = fx_split(fx_mad(fx_split(z0), v[2], fx_mad(fx_split(y0), v[1], fx_mul(fx_split(x0), v[0]))));
            cc[1] = fx_split(fx_mad(fx_split(z1), v[2], fx_mad(fx_split(y1), v[1], fx_mul(fx_split(x1), v[0]))));
            ld(p, 0, x0, x1);
            ld(p, 1, y0, y1);
            ld(p, 2, z0, z1);
            if (p > 0)
                a[0] = fx_split(fx_mad(nms, cc[0], fx_mad(fx_split(z0), v[2],
                                                          fx_mad(fx_split(y0), v[1], fx_mul(fx_split(x0), v[0])))));
            a[1] = fx_split(fx_mad(nms, cc[1], fx_mad(fx_split(z1), v[2],
                                                      fx_mad(fx_split(y1), v[1], fx_mul(fx_split(x1), v[0])))));
        }
        auto whole = [](Fx q) { return ((long long)q.h << 32) | ((unsigned)q.l << 1); };
        if (p == 0) {            // k = 1: x
            F[0] = whole(a[1]);
        } else if (p == 1) {     // k = 2: y, k = 3: xy
            F[0] = fx_mad(cc[1], e[1], fx_mad(a[1], m[1], F[0]));
            F[1] = fx_mad(cc[1], e[0], fx_mad(a[1], m[0], whole(a[0])));
        } else if (p == 2) {     // k = 4: z, k = 5: xz
            F[0] = fx_mad(cc[1], e[2], fx_mad(a[1], m[2], F[0]));
            F[2] = fx_mad(cc[1], e[0], fx_mad(a[1], m[0], whole(a[0])));
        } else {                 // k = 6: yz, k = 7: xyz
            F[1] = fx_mad(cc[0], e[2], fx_mad(a[0], m[2], F[1]));
            F[2] = fx_mad(cc[0], e[1], fx_mad(a[0], m[1], F[2]));
            F[0] = fx_mad(cc[1], fx_split(E6), fx_mad(a[1], Pyz, F[0]));
            F[1] = fx_mad(cc[1], fx_split(E5), fx_mad(a[1], Pxz, F[1]));
            F[2] = fx_mad(cc[1], fx_split(E3), fx_mad(a[1], Pxy, F[2]));
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long g0, g1;
            ld(p, 6 + j, g0, g1);
            if (p == 0) g[j] = fx_mad(fx_split(g1), m[0], g0);
            else if (p == 1) g[j] = fx_mad(fx_split(g1), Pxy, fx_mad(fx_split(g0), m[1], g[j]));
            else if (p == 2) g[j] = fx_mad(fx_split(g1), Pxz, fx_mad(fx_split(g0), m[2], g[j]));
            else g[j] = fx_mad(fx_split(g1), S, fx_mad(fx_split(g0), Pyz, g[j]));
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        accF[j] = fx_mad(hf, fx_split(F[j]), accF[j]);
        accG[j] = fx_mad(hf, fx_split(g[j]), accG[j]);
    }
}

// A^{n+1} at coordinate r of the cell less its lowest node's value, in the table's format.
__device__ __forceinline__ void cell_A1_fixed(const double r[3], const FixedLoad& ld, long long out[3]) {
    Fx q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] = fx_split(fixed_of(r[a], 1023, 10));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        long long k0, k1, k2, k3, k4, k5, k6, k7;
        ld(0, c, k0, k1);
        ld(1, c, k2, k3);
        ld(2, c, k4, k5);
        ld(3, c, k6, k7);
        const long long lo = fx_mad(q[1], fx_split(fx_mad(fx_split(k3), q[0], k2)), fx_mul(fx_split(k1), q[0]));
        const long long hi = fx_mad(q[1], fx_split(fx_mad(fx_split(k7), q[0], k6)), fx_mad(fx_split(k5), q[0], k4));
        out[c] = fx_mad(q[2], fx_split(hi), lo);
    }
}

}  // namespace pic
