// Orbit integrals in centred form, and the cell table they contract with.
//
// The orbit of one particle over a step is cut at the knots it crosses (§4.7, Eq.
// (breakpoint-set)).  Inside one piece [s0, s0 + h] the orbit stays in one cell, where every
// mesh field of linear splines is the trilinear polynomial
//     f(w) = sum_k f_k prod_{a in k} w_a,   k = subsets of {x, y, z} (bit a = axis a),
// w_a in [0, 1] the coordinate in the cell and f_k the mixed differences of the cell's 8 node
// values.  With u = s - s_mid running over [-h/2, h/2] the orbit is w_a = m_a + beta_a u, m_a its
// midpoint, and odd powers of u integrate to zero, so the closed forms of Appendices A and B
// become, per unit of h and with e_a = beta_a h^2 / 12,
//     <w_a>         = m_a                         <u w_a>     = e_a
//     <w_p w_q>     = P_pq = m_p m_q + e_p beta_q  <u w_p w_q> = m_p e_q + m_q e_p
//     <w_x w_y w_z> = m_x P_yz + m_y e_x beta_z + m_z e_x beta_y          <u> = 0.
// That is 20 operations where the integrals from the piece's start took 74, and the 8 node
// weights with their 8-node differences (16 + 84) disappear into the table.
#pragma once

#include <cuda_runtime.h>

#include "pic_device.cuh"

namespace pic {

// Cell table: per cell and k the 9 columns A^{n+1} (3), A^{n+1} - A^n (3), -grad phi^{n+1/2} (3),
// k in pairs (2 p, 2 p + 1) that one 16-byte load brings: entry [p][column][k & 1].
constexpr int CELL_COLS = 9;
constexpr int CELL_VALUES = 8 * CELL_COLS;

// a b + c (FP32 pairs have an overload that rounds once).
template <typename T>
__device__ __forceinline__ T mad(T a, T b, T c) {
    return a * b + c;
}

// Order and range tests of the walk.  On doubles they run on the integer pipe (for values >= 0
// the bit patterns order like the values; the sign and exponent decide t < 0 and t >= 1): the
// FP64 pipe, which has 1/64 of the issue rate, is what bounds the particle kernels.
__device__ __forceinline__ bool less_pos(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
__device__ __forceinline__ bool same_bits(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
__device__ __forceinline__ bool at_least_one(double t) { return __double2hiint(t) >= 0x3ff00000; }
__device__ __forceinline__ bool below_zero(double t) { return __double2hiint(t) < 0; }
__device__ __forceinline__ bool less_pos(float a, float b) { return a < b; }
__device__ __forceinline__ bool same_bits(float a, float b) { return a == b; }
__device__ __forceinline__ bool at_least_one(float t) { return t >= 1.f; }
__device__ __forceinline__ bool below_zero(float t) { return t < 0.f; }
// 0 <= s < 1 (not a NaN of either sign)
__device__ __forceinline__ bool before_end(double s) { return in_box(s, 1.0); }
__device__ __forceinline__ bool before_end(float s) { return s < 1.f; }
__device__ __forceinline__ bool is_zero(float t) { return t == 0.f; }
__device__ __forceinline__ bool is_zero(double t) { return (__double_as_longlong(t) << 1) == 0; }

// A particle's start: cell and coordinate in it.
template <typename T>
struct CellStart {
    T f[3];
    int c[3];
};

// c + 1 and c - 1 on a periodic axis of n cells, c in [0, n)
__device__ __forceinline__ int next_cell(int c, int n) { return c + 1 >= n ? 0 : c + 1; }
__device__ __forceinline__ int prev_cell(int c, int n) { return c > 0 ? c - 1 : n - 1; }

// The knot-free pieces of the orbit f + s beta of a start, one per next().  c stays in [0, n)
// whatever the input.  After the last piece c is the end point's cell and te its coordinate in it
// (in [0, 1]; an end exactly on a knot keeps the cell it came from, where the fields have the same
// value), and count the number of breakpoint intervals, or -1 if MAX_SEGMENTS was exceeded.
template <typename T>
struct PieceWalk {
    T fd[3], te[3], sn[3], s0;   // start and end coordinate relative to cell c, next crossing per axis
    int c[3];
    int it, count;

    __device__ __forceinline__ PieceWalk(const CellStart<T>& st, const T beta[3], const MeshDims& m) {
        unsigned ahead = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            c[a] = st.c[a];
            fd[a] = st.f[a];
            te[a] = fd[a] + beta[a];
            const bool down = below_zero(te[a]);
            if (down && is_zero(fd[a])) {   // on a knot, moving down: the cell below
                c[a] = prev_cell(c[a], m.n[a]);
                fd[a] = T(1);
                te[a] = T(1) + beta[a];
            }
            sn[a] = T(2);                          // 2: no crossing ahead
            // (an end of one after a move down: 1 + beta rounds to one, the orbit stays below the knot)
            if (below_zero(te[a]) || (!down && at_least_one(te[a]))) ahead |= 1u << a;
        }
        for (; ahead; ahead &= ahead - 1) {
            const int a = __ffs(ahead) - 1;
            put(a, sn, crossing(pick(a, fd), pick(a, te), pick(a, beta)));
        }
        s0 = T(0);
        it = 0;
        count = 0;
    }

    // One axis by its number, without indexing registers.  The crossings go one axis a lane at a time, so
    // that a warp whose lanes cross one knot each, on different axes, runs their divisions and FP64
    // additions once; with the axes unrolled, and the two directions apart, a warp could run six.  At
    // 128^3 with 134M particles (1.2 crossings each) the first scatter went from 37.2 to 31.6 ms with this,
    // the final sweep from 64.2 to 59.1, the push in pairs from 90.8 to 84.7.
    static __device__ __forceinline__ T pick(int a, const T v[3]) { return a == 0 ? v[0] : (a == 1 ? v[1] : v[2]); }
    static __device__ __forceinline__ void put(int a, T v[3], T x) {
        v[0] = a == 0 ? x : v[0];
        v[1] = a == 1 ? x : v[1];
        v[2] = a == 2 ? x : v[2];
    }

    // Where an axis meets the next knot, its end t being outside the cell; 2: at or past the orbit's end.
    static __device__ __forceinline__ T crossing(T f, T t, T b) {
        const bool down = below_zero(t);
        const T s = (down ? f : T(1) - f) / (down ? -b : b);
        return before_end(s) ? s : T(2);
    }

    // The next breakpoint (1: the end of the orbit).
    __device__ __forceinline__ T upcoming() const {
        T s1 = T(1);
#pragma unroll
        for (int a = 0; a < 3; ++a) s1 = less_pos(sn[a], s1) ? sn[a] : s1;
        return s1;
    }

    // Cross the knots met at s1.
    __device__ __forceinline__ void cross(T s1, const T beta[3], const MeshDims& m) {
        unsigned met = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) met |= same_bits(sn[a], s1) ? 1u << a : 0u;
        for (; met; met &= met - 1) {
            const int a = __ffs(met) - 1;
            const T t0 = pick(a, te);
            const bool down = below_zero(t0);
            const T one = down ? T(1) : T(-1), f = pick(a, fd) + one, t = t0 + one;
            const int ca = a == 0 ? c[0] : (a == 1 ? c[1] : c[2]), n = a == 0 ? m.n[0] : (a == 1 ? m.n[1] : m.n[2]);
            const int cn = down ? prev_cell(ca, n) : next_cell(ca, n);
            c[0] = a == 0 ? cn : c[0];
            c[1] = a == 1 ? cn : c[1];
            c[2] = a == 2 ? cn : c[2];
            put(a, fd, f);
            put(a, te, t);
            put(a, sn, (down ? below_zero(t) : at_least_one(t)) ? crossing(f, t, pick(a, beta)) : T(2));
        }
        s0 = s1;
    }

    // The next piece [s_mid - h/2, s_mid + h/2], h > 0, in cell pc with the midpoint mid; false when
    // there is none.  `last` is set with the orbit's last interval.
    __device__ __forceinline__ bool next(const T beta[3], const MeshDims& m, T& h, T& sm, T mid[3], int pc[3], bool& last) {
        last = false;
        while (true) {
            const T s1 = upcoming();
            ++it;
            const bool piece = less_pos(s0, s1);
            if (piece) {
                h = s1 - s0;
                sm = T(0.5) * (s0 + s1);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    mid[a] = fd[a] + sm * beta[a];
                    pc[a] = c[a];
                }
            }
            if (same_bits(s1, T(1)) || it == MAX_SEGMENTS) {
                last = true;
                count = same_bits(s1, T(1)) ? it : -1;
                return piece;
            }
            cross(s1, beta, m);
            if (piece) return true;
        }
    }
};

// Visit the pieces of the orbit: visit(h, s_mid, mid, cell).  On return st is the end point's cell
// and coordinate.  Returns PieceWalk's count.  (The kernels that visit inside this loop measured 10%
// faster than through next(), which keeps the walk's state across calls.)
template <typename T, typename F>
__device__ __forceinline__ int for_each_piece(CellStart<T>& st, const T beta[3], const MeshDims& m, F&& visit) {
    PieceWalk<T> wk(st, beta, m);
    int count = -1;
    for (int it = 0; it < MAX_SEGMENTS; ++it) {
        const T s1 = wk.upcoming();
        if (less_pos(wk.s0, s1)) {
            const T h = s1 - wk.s0, sm = T(0.5) * (wk.s0 + s1);
            T mid[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) mid[a] = wk.fd[a] + sm * beta[a];
            visit(h, sm, mid, wk.c);
        }
        if (same_bits(s1, T(1))) {
            count = it + 1;
            break;
        }
        wk.cross(s1, beta, m);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        st.c[a] = wk.c[a];
        st.f[a] = wk.te[a];
    }
    return count;
}

// The moments of one piece per unit of h (see the file comment).
template <typename T>
struct PieceMoments {
    T m[3];              // <w_a>
    T Pxy, Pxz, Pyz, S;  // <w_p w_q>, <w_x w_y w_z>
    T e[3];              // <u w_a>
};

template <typename T>
__device__ __forceinline__ PieceMoments<T> piece_moments(T h, const T mid[3], const T beta[3]) {
    PieceMoments<T> q;
    const T k = h * h * T(1.0 / 12.0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        q.m[a] = mid[a];
        q.e[a] = k * beta[a];
    }
    const T kxy = q.e[0] * beta[1], kxz = q.e[0] * beta[2], kyz = q.e[1] * beta[2];
    q.Pxy = mad(mid[0], mid[1], kxy);
    q.Pxz = mad(mid[0], mid[2], kxz);
    q.Pyz = mad(mid[1], mid[2], kyz);
    q.S = mad(mid[0], q.Pyz, mad(mid[1], kxz, mid[2] * kxy));
    return q;
}

// The 8 node weights of Appendix A per unit of h, node nu = nx + 2 ny + 4 nz.
template <typename T>
__device__ __forceinline__ void node_weights(const PieceMoments<T>& q, T W[8]) {
    W[7] = q.S;
    W[3] = q.Pxy - q.S;
    W[5] = q.Pxz - q.S;
    W[6] = q.Pyz - q.S;
    W[1] = q.m[0] - q.Pxy - W[5];
    W[2] = q.m[1] - q.Pyz - W[3];
    W[4] = q.m[2] - q.Pxz - W[6];
    W[0] = T(1) - q.m[0] - W[2] - W[4] - W[6];
}

// One piece's impulse, acc_j += int ((D_j A)^T v - d_j phi) over the piece (Eqs.
// (gphibar-definition) and (DA-def)), vs = scale v and ihs_j = 1 / (scale H_j).  `ld(p, col, a, b)`
// loads entries k = 2 p and 2 p + 1 of a column of the cell.  A at the time s is
// A^{n+1} - (1 - s) (A^{n+1} - A^n), contracted with v first.
template <typename T, typename L>
__device__ __forceinline__ void piece_impulse(T h, T sm, const T mid[3], const T beta[3], const T vs[3],
                                              const T ihs[3], L&& ld, T acc[3]) {
    const PieceMoments<T> q = piece_moments(h, mid, beta);
    const T nms = sm - T(1);
    T F[3], g[3];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        T a[2], cc[2];
        {
            T x0, x1, y0, y1, z0, z1;
            ld(p, 3, x0, x1);
            ld(p, 4, y0, y1);
            ld(p, 5, z0, z1);
            if (p > 0) cc[0] = mad(z0, vs[2], mad(y0, vs[1], x0 * vs[0]));
            cc[1] = mad(z1, vs[2], mad(y1, vs[1], x1 * vs[0]));
            ld(p, 0, x0, x1);
            ld(p, 1, y0, y1);
            ld(p, 2, z0, z1);
            if (p > 0) a[0] = mad(nms, cc[0], mad(z0, vs[2], mad(y0, vs[1], x0 * vs[0])));
            a[1] = mad(nms, cc[1], mad(z1, vs[2], mad(y1, vs[1], x1 * vs[0])));
        }
        if (p == 0) {            // k = 1: x
            F[0] = a[1];
        } else if (p == 1) {     // k = 2: y, k = 3: xy
            F[0] = mad(cc[1], q.e[1], mad(a[1], mid[1], F[0]));
            F[1] = mad(cc[1], q.e[0], mad(a[1], mid[0], a[0]));
        } else if (p == 2) {     // k = 4: z, k = 5: xz
            F[0] = mad(cc[1], q.e[2], mad(a[1], mid[2], F[0]));
            F[2] = mad(cc[1], q.e[0], mad(a[1], mid[0], a[0]));
        } else {                 // k = 6: yz, k = 7: xyz
            F[1] = mad(cc[0], q.e[2], mad(a[0], mid[2], F[1]));
            F[2] = mad(cc[0], q.e[1], mad(a[0], mid[1], F[2]));
            F[0] = mad(cc[1], mad(mid[1], q.e[2], mid[2] * q.e[1]), mad(a[1], q.Pyz, F[0]));
            F[1] = mad(cc[1], mad(mid[0], q.e[2], mid[2] * q.e[0]), mad(a[1], q.Pxz, F[1]));
            F[2] = mad(cc[1], mad(mid[0], q.e[1], mid[1] * q.e[0]), mad(a[1], q.Pxy, F[2]));
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T g0, g1;
            ld(p, 6 + j, g0, g1);
            if (p == 0) g[j] = mad(g1, mid[0], g0);
            else if (p == 1) g[j] = mad(g1, q.Pxy, mad(g0, mid[1], g[j]));
            else if (p == 2) g[j] = mad(g1, q.Pxz, mad(g0, mid[2], g[j]));
            else g[j] = mad(g1, q.S, mad(g0, q.Pyz, g[j]));
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) acc[j] = mad(h, mad(ihs[j], F[j], g[j]), acc[j]);
}

// A^{n+1} at coordinate r of the cell (Eq. (Ah-mesh)).
template <typename T, typename L>
__device__ __forceinline__ void cell_A1(const T r[3], L&& ld, T out[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        T k0, k1, k2, k3, k4, k5, k6, k7;
        ld(0, c, k0, k1);
        ld(1, c, k2, k3);
        ld(2, c, k4, k5);
        ld(3, c, k6, k7);
        const T lo = mad(r[1], mad(k3, r[0], k2), mad(k1, r[0], k0));
        const T hi = mad(r[1], mad(k7, r[0], k6), mad(k5, r[0], k4));
        out[c] = mad(r[2], hi, lo);
    }
}

// Row index of a cell's lowest node, and the 8 node rows of the cell.
__device__ __forceinline__ int64_t cell_row(const int c[3], const MeshDims& m) {
    return (int64_t)c[0] + (int64_t)m.n[0] * ((int64_t)c[1] + (int64_t)m.n[1] * c[2]);
}

__device__ __forceinline__ void cell_nodes8(const int c[3], const MeshDims& m, int64_t g[8]) {
    const int64_t dx = next_cell(c[0], m.n[0]) - c[0];
    const int64_t dy = (int64_t)m.n[0] * (next_cell(c[1], m.n[1]) - c[1]);
    const int64_t dz = (int64_t)m.n[0] * m.n[1] * (next_cell(c[2], m.n[2]) - c[2]);
    g[0] = cell_row(c, m);
    g[1] = g[0] + dx;
    g[2] = g[0] + dy;
    g[3] = g[2] + dx;
    g[4] = g[0] + dz;
    g[5] = g[4] + dx;
    g[6] = g[4] + dy;
    g[7] = g[6] + dx;
}

// Where the particle kernels take a cell's entries from: the FP64 cell table; the gather table, taking the
// differences of the cell's nodes each time (contexts without cell tables); or, in deterministic mode, the cell
// table where there is one and the gather table where not, with the same bits: the differences are the same
// numbers (subtractions in the same order), and what is made of them is integers (orbit_fixed.cuh) or runs
// through the same instructions.  24^3, 442,368 particles: 4.1 ms a step with the table, 7.9 without (9.95
// before there were tables).
enum Fields { FROM_NODES, FROM_CELLS, FROM_EITHER };

struct FieldTables {
    const double* nodes;   // gather table
    const double* cells;   // cell table
};

template <int FROM>
struct FieldLoad;

template <>
struct FieldLoad<FROM_CELLS> {
    const double2* t;
    __device__ __forceinline__ FieldLoad(FieldTables ft, const int c[3], const MeshDims& m)
        : t(reinterpret_cast<const double2*>(ft.cells + CELL_VALUES * cell_row(c, m))) {}
    __device__ __forceinline__ void operator()(int p, int col, double& a, double& b) const {
        const double2 q = __ldg(t + p * CELL_COLS + col);
        a = q.x;
        b = q.y;
    }
};

template <>
struct FieldLoad<FROM_NODES> {
    const double* t;
    int64_t g[8];
    __device__ __forceinline__ FieldLoad(FieldTables ft, const int c[3], const MeshDims& m) : t(ft.nodes) {
        cell_nodes8(c, m, g);
    }
    __device__ __forceinline__ double node(int k, int col) const {
        const double* q = t + 12 * g[k];
        return col < 3 ? __ldg(q + 3 + col) : (col < 6 ? __ldg(q + col) - __ldg(q + col - 3) : -__ldg(q + col));
    }
    __device__ __forceinline__ void operator()(int p, int col, double& a, double& b) const {
        a = node(0, col);
        b = node(1, col) - a;
        if (p == 0) return;
        if (p == 3) {
            double lo = node(2, col), hi = node(3, col) - lo;
            a = lo - a;
            b = hi - b;
            lo = node(4, col);
            hi = node(5, col) - lo;
            const double l6 = node(6, col);
            a = (l6 - lo) - a;
            b = ((node(7, col) - l6) - hi) - b;
        } else {
            const double lo = node(2 * p, col);
            a = lo - a;
            b = (node(2 * p + 1, col) - lo) - b;
        }
    }
};

// A cell's entries from the gather table (a function of its own: FROM_EITHER's rare side).
static __device__ __noinline__ void entries_of_nodes(const double* nodes, int c0, int c1, int c2, int n0, int n1, int n2,
                                                     double2* out) {
    MeshDims m;
    m.n[0] = n0;
    m.n[1] = n1;
    m.n[2] = n2;
    const int c[3] = {c0, c1, c2};
    const FieldLoad<FROM_NODES> ld({nodes, nullptr}, c, m);
    for (int col = 0; col < CELL_COLS; ++col)
#pragma unroll
        for (int p = 0; p < 4; ++p) ld(p, col, out[p * CELL_COLS + col].x, out[p * CELL_COLS + col].y);
}

template <>
struct FieldLoad<FROM_EITHER> {
    const double2* t;                     // the table's entries, or own
    double2 own[CELL_VALUES / 2];         // (local memory, untouched where there is a table)
    __device__ __forceinline__ FieldLoad(FieldTables ft, const int c[3], const MeshDims& m) {
        if (__builtin_expect(ft.cells != nullptr, 1)) {
            t = reinterpret_cast<const double2*>(ft.cells + CELL_VALUES * cell_row(c, m));
        } else {
            entries_of_nodes(ft.nodes, c[0], c[1], c[2], m.n[0], m.n[1], m.n[2], own);
            t = own;
        }
    }
    FieldLoad(const FieldLoad&) = delete;
    __device__ __forceinline__ void operator()(int p, int col, double& a, double& b) const {
        const double2 q = t[p * CELL_COLS + col];
        a = q.x;
        b = q.y;
    }
};

// The cell and coordinate of an FP64 position in [0, n) (cell units).  The integer part comes from the
// bits (one FP64 instruction an axis instead of three).
__device__ __forceinline__ void cell_start(const double x0[3], const MeshDims& m, CellStart<double>& st) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long b = __double_as_longlong(x0[a]);
        const int e = (int)(b >> 52) - 1023;   // negative x: below -1023
        double fl = 0.0;
        int c = 0;
        if (e >= 0 && e < 31) {
            fl = __longlong_as_double((b >> (52 - e)) << (52 - e));
            c = (int)(((b & ((1LL << 52) - 1)) | (1LL << 52)) >> (52 - e));
        } else if (e >= 31 || b < 0) {
            fl = floor(x0[a]);
            c = max((int)fl, 0);
        }
        st.f[a] = x0[a] - fl;
        st.c[a] = min(c, m.n[a] - 1);
    }
}

}  // namespace pic
