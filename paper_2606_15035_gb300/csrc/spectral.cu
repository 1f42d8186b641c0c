// Spectral mesh operators (the paper's choice, §3.3) for the PIC step (FP64, sm_103a).
//
// With ops = PIC_OPS_SPECTRAL the first derivative D_a has the Fourier symbol i k_a,
// k_a = 2 pi m_a / L_a, with the Nyquist symbol (2 |m_a| = n_a) set to zero so that D_a stays
// real and skew-adjoint; Delta_h = sum_a D_a D_a has the symbol -|k|^2 and the same 8 null
// modes as the central difference.  The Crank--Nicolson update (§3.2, Eq. (cn-field-update))
// is then diagonal: per mode, with b = dt kappa^2 lambda / 2 and lambda = -|k|^2,
//     [ 1     -dt/2 ] [u1]   [ u0 + dt/2 w0                  ]
//     [ -b      1   ] [w1] = [ w0 + b u0 + dt kappa^2 c src   ],
// solved exactly (no iteration), with src = rho^{n+1/2} (c = sigma1) for (phi, psi) and
// src = J_c^{n+1/2} (c = sigma2) for (A_c, U_c); continuity (Eq. (cn-continuity)) is
// rho^{n+1} = rho^n - dt D . J in the same basis.
//
// Transforms: a batched, mixed-radix (4, 2 and 3) Stockham FFT of complex FP64 lines, up to 16 lines
// per block in shared memory, applied along x, y and z; unnormalised forward transform and
// a 1/N scale on the way back to real space.  Mesh sizes n_a = 2^p 3^q <= 1024.
#include <cmath>
#include <vector>

#include "pic_internal.h"

namespace pic {
namespace {

struct FftStage {
    int R, L, nb, tstep;         // radix, product of the radices before, n / R, n / (L R)
    unsigned mL, mnb;            // multipliers of the divisions by L and nb
};

struct FftAxis {
    int axis, n, nst, lb;        // lb: lines of a block
    int64_t stride;              // element stride of a line along this axis
    unsigned mn, mlb;
    FftStage st[FFT_MAX_STAGES];
    const double2* tw;           // exp(-2 pi i t / n), t = 0 .. n-1
};

// Real fields that a pass reads or writes in place of the complex ones (null: complex).
constexpr int SPEC_FIELDS = 12;
struct RealFields {
    double* f[SPEC_FIELDS] = {};
    double scale = 1.0;
};

unsigned multiplier(int d) { return d <= 1 ? 0u : (unsigned)((((uint64_t)1 << 32) + d - 1) / d); }
// x / d for x < 2^16 by m = ceil(2^32 / d) (d = 1: m = 0)
__device__ __forceinline__ int quot(int x, unsigned m) { return m ? (int)__umulhi((unsigned)x, m) : x; }

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// First element of line l along the axis.
__device__ __forceinline__ int64_t line_base(int axis, int64_t l, const MeshDims& m) {
    if (axis == 0) return l * m.n[0];
    if (axis == 1) return (l % m.n[0]) + (int64_t)m.n[0] * m.n[1] * (l / m.n[0]);
    return l;
}

// In-place 1D transforms of every line of field blockIdx.y along one axis (fields N apart).
// Stockham autosort: stage s of radix R, with L = product of the previous radices, takes
// v_r = x[j + r n/R] (j < n/R, k = j mod L), twiddles v_r by exp(-+2 pi i k r / (L R)),
// applies the radix-R DFT and stores output s at (j div L) L R + k + s L.
// A block transforms `lb` lines that are adjacent in memory (along x one after the other; along y and z
// element by element, so that the loads and stores of a strided axis take lb consecutive values at a
// time).  Shared memory holds the lb lines twice (ping-pong), line j at j n.  The first pass of a forward
// transform reads the real fields, the last of an inverse one writes them.
//
// At small meshes the passes are bound by latency (index divisions, stages, launches): a mesh phase of 15
// fields at 16^3 took 14 launches and 77 us of kernels with separate conversions and radix 2, now 9 and 47;
// a pass at 36^3 19.6 us, now 14.1.
__global__ void k_fft_axis(double2* __restrict__ data, MeshDims m, FftAxis ax, int inverse, RealFields rin,
                           RealFields rout) {
    extern __shared__ double2 sbuf[];
    const int n = ax.n, lb = ax.lb, tot = lb * n;
    const int64_t ngroups = m.ncell / tot;
    double2* field = data + (int64_t)blockIdx.y * m.ncell;
    const double* real_in = rin.f[blockIdx.y];
    double* real_out = rout.f[blockIdx.y];
    const double sgn = inverse ? 1.0 : -1.0;
    const double s3 = sgn * 0.86602540378443864676;   // sin(2 pi / 3) with the transform's sign
    auto tw = [&](int t) {
        double2 w = ax.tw[t];
        if (inverse) w.y = -w.y;
        return w;
    };
    // element t of line j: place in memory (from the first line's start) and in the buffer
    auto place = [&](int e, int& at) {
        if (ax.axis == 0) {
            at = e;
            return (int64_t)e;
        }
        const int t = quot(e, ax.mlb), j = e - t * lb;
        at = j * n + t;
        return j + (int64_t)t * ax.stride;
    };
    for (int64_t gr = blockIdx.x; gr < ngroups; gr += gridDim.x) {
        double2* x = sbuf;
        double2* y = sbuf + tot;
        const int64_t first = line_base(ax.axis, gr * lb, m);
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            int at;
            const int64_t g = first + place(e, at);
            x[at] = real_in ? make_double2(real_in[g], 0.0) : field[g];
        }
        __syncthreads();
        for (int si = 0; si < ax.nst; ++si) {
            const FftStage st = ax.st[si];
            for (int e = threadIdx.x; e < lb * st.nb; e += blockDim.x) {
                const int line = quot(e, st.mnb), j = e - line * st.nb;
                const int jl = quot(j, st.mL), k = j - jl * st.L;
                const double2* in = x + line * n + j;
                double2* out = y + line * n + jl * st.L * st.R + k;
                const double2 v0 = in[0], v1 = cmul(in[st.nb], tw(k * st.tstep));
                if (st.R == 2) {
                    out[0] = cadd(v0, v1);
                    out[st.L] = csub(v0, v1);
                } else if (st.R == 4) {
                    const double2 v2 = cmul(in[2 * st.nb], tw(2 * k * st.tstep));
                    const double2 v3 = cmul(in[3 * st.nb], tw(3 * k * st.tstep));
                    const double2 a = cadd(v0, v2), b = csub(v0, v2), c = cadd(v1, v3), d = csub(v1, v3);
                    const double2 id = make_double2(-sgn * d.y, sgn * d.x);   // +- i d
                    out[0] = cadd(a, c);
                    out[st.L] = cadd(b, id);
                    out[2 * st.L] = csub(a, c);
                    out[3 * st.L] = csub(b, id);
                } else {
                    const double2 v2 = cmul(in[2 * st.nb], tw(2 * k * st.tstep));
                    const double2 sum = cadd(v1, v2), dif = csub(v1, v2);
                    const double2 mid = make_double2(v0.x - 0.5 * sum.x, v0.y - 0.5 * sum.y);
                    out[0] = cadd(v0, sum);
                    out[st.L] = make_double2(mid.x - s3 * dif.y, mid.y + s3 * dif.x);        // + i s3 dif
                    out[2 * st.L] = make_double2(mid.x + s3 * dif.y, mid.y - s3 * dif.x);    // - i s3 dif
                }
            }
            __syncthreads();
            double2* t = x;
            x = y;
            y = t;
        }
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            int at;
            const int64_t g = first + place(e, at);
            if (real_out) real_out[g] = x[at].x * rout.scale;
            else field[g] = x[at];
        }
        __syncthreads();
    }
}

struct SpecParams {
    MeshDims m;
    double kscale[3];   // 2 pi / L_a
    double dt, kappa2, sigma1, sigma2, dV, invN;
};

// Wavenumber of index i on an axis of n nodes (fftfreq order), 0 at the Nyquist index.
__device__ __forceinline__ double kwave(int i, int n, double scale) {
    const int mm = i <= (n - 1) / 2 ? i : i - n;
    return 2 * (mm < 0 ? -mm : mm) == n ? 0.0 : mm * scale;
}

__device__ __forceinline__ void mode_k(const SpecParams& p, int64_t g, double k[3]) {
    const int ix = (int)(g % p.m.n[0]);
    const int64_t t = g / p.m.n[0];
    const int iy = (int)(t % p.m.n[1]), iz = (int)(t / p.m.n[1]);
    k[0] = kwave(ix, p.m.n[0], p.kscale[0]);
    k[1] = kwave(iy, p.m.n[1], p.kscale[1]);
    k[2] = kwave(iz, p.m.n[2], p.kscale[2]);
}

// i k z
__device__ __forceinline__ double2 ik(double k, double2 z) { return make_double2(-k * z.y, k * z.x); }

#define SPEC_LOOP(g, N) for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < (N); g += (int64_t)gridDim.x * blockDim.x)

// Continuity and the CN update per mode.  In: J^ (3), level n: [phi, A (3) | psi, U (3) | rho].
// Out: level n+1 [phi, A | psi, U | rho] and D phi^{n+1/2} (3).
__global__ void k_spec_cn(SpecParams p, const double2* __restrict__ Jh, const double2* __restrict__ S0,
                          double2* __restrict__ S1) {
    const int64_t N = p.m.ncell;
    const double hdt = 0.5 * p.dt;
    SPEC_LOOP(g, N) {
        double k[3];
        mode_k(p, g, k);
        const double lam = -(k[0] * k[0] + k[1] * k[1] + k[2] * k[2]);
        const double b = hdt * p.kappa2 * lam, det = 1.0 - hdt * b, inv = 1.0 / det;
        // x / det by Markstein's method: the quotient by the reciprocal, and one correction from the exact
        // remainder (16 divisions bound the kernel)
        auto over = [&](double x) {
            const double q = x * inv;
            return fma(fma(-q, det, x), inv, q);
        };
        const double2 J[3] = {Jh[g], Jh[N + g], Jh[2 * N + g]};
        double2 divJ = cadd(cadd(ik(k[0], J[0]), ik(k[1], J[1])), ik(k[2], J[2]));
        const double2 r0 = S0[8 * N + g];
        const double2 r1 = make_double2(r0.x - p.dt * divJ.x, r0.y - p.dt * divJ.y);
        S1[8 * N + g] = r1;
        const double2 rh = make_double2(0.5 * (r0.x + r1.x), 0.5 * (r0.y + r1.y));
        double2 phi1 = make_double2(0.0, 0.0);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const double2 u0 = S0[f * N + g], w0 = S0[(4 + f) * N + g];
            const double2 src = f == 0 ? rh : J[f - 1];
            const double cs = p.dt * p.kappa2 * (f == 0 ? p.sigma1 : p.sigma2);
            const double2 q1 = make_double2(u0.x + hdt * w0.x, u0.y + hdt * w0.y);
            const double2 q2 = make_double2(w0.x + b * u0.x + cs * src.x, w0.y + b * u0.y + cs * src.y);
            const double2 u1 = make_double2(over(q1.x + hdt * q2.x), over(q1.y + hdt * q2.y));
            const double2 w1 = make_double2(over(q2.x + b * q1.x), over(q2.y + b * q1.y));
            S1[f * N + g] = u1;
            S1[(4 + f) * N + g] = w1;
            if (f == 0) phi1 = u1;
        }
        const double2 ph = make_double2(0.5 * (phi1.x + S0[g].x), 0.5 * (phi1.y + S0[g].y));
#pragma unroll
        for (int a = 0; a < 3; ++a) S1[(9 + a) * N + g] = ik(k[a], ph);
    }
}

// The CN Helmholtz solve of the central-difference operators by FFT: (I - a Delta_h) x = b, the
// wide Laplacian sum_a (f_{+2} - 2 f + f_{-2}) / (4 H_a^2) having the symbol -sum_a s2_a[m_a],
// s2_a[m] = sin^2(2 pi m / n_a) / H_a^2, so each mode is divided by 1 + a sum_a s2_a[m_a] (>= 1;
// the 1/N of the inverse transform is folded in).
__global__ void k_helm_fft_divide(MeshDims m, const double* __restrict__ s2, double a, double invN,
                                  double2* __restrict__ data, int nf) {
    const int64_t N = m.ncell;
    SPEC_LOOP(g, N) {
        const int ix = (int)(g % m.n[0]);
        const int64_t t = g / m.n[0];
        const int iy = (int)(t % m.n[1]), iz = (int)(t / m.n[1]);
        const double d = invN / (1.0 + a * (s2[ix] + s2[m.n[0] + iy] + s2[m.n[0] + m.n[1] + iz]));
        for (int f = 0; f < nf; ++f) {
            const double2 z = data[f * N + g];
            data[f * N + g] = make_double2(z.x * d, z.y * d);
        }
    }
}

// Gather table per node: A^n (3), A^{n+1} (3), D phi^{n+1/2} (3), U^{n+1/2} (3).
__global__ void k_spec_table(int64_t N, const double* __restrict__ F0, const double* __restrict__ W0,
                             const double* __restrict__ F1, const double* __restrict__ W1,
                             const double* __restrict__ gphi, double* __restrict__ table) {
    SPEC_LOOP(g, N) {
        double* t = table + 12 * g;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            t[c] = F0[(1 + c) * N + g];
            t[3 + c] = F1[(1 + c) * N + g];
            t[6 + c] = gphi[c * N + g];
            t[9 + c] = 0.5 * (W1[(1 + c) * N + g] + W0[(1 + c) * N + g]);
        }
    }
}

// e_J partial sums of the iteration (real space).
__global__ void k_spec_ej(int64_t N, const double* __restrict__ J, const double* __restrict__ Jprev,
                          double* __restrict__ partials) {
    __shared__ double sm[32];
    double num = 0.0, den = 0.0;
    SPEC_LOOP(g, 3 * N) {
        const double j = J[g];
        den += j * j;
        if (Jprev) {
            const double d = j - Jprev[g];
            num += d * d;
        }
    }
    double r = block_sum(num, sm);
    if (threadIdx.x == 0) partials[S_EJ_NUM * MAX_BLOCKS + blockIdx.x] = r;
    r = block_sum(den, sm);
    if (threadIdx.x == 0) partials[S_EJ_DEN * MAX_BLOCKS + blockIdx.x] = r;
}

// Field energy W = dV sum_g (|E|^2 / 2 sigma1 + |B|^2 / 2 sigma2) by Parseval from the
// unnormalised transforms [phi, A | psi, U]: E^ = -i k phi^ - U^, B^ = i k x A^.
__global__ void k_spec_energy(SpecParams p, const double2* __restrict__ S, double* __restrict__ partials, int slot) {
    __shared__ double sm[32];
    const int64_t N = p.m.ncell;
    double e = 0.0;
    SPEC_LOOP(g, N) {
        double k[3];
        mode_k(p, g, k);
        const double2 phi = S[g];
        const double2 A[3] = {S[N + g], S[2 * N + g], S[3 * N + g]};
        double e2 = 0.0, b2 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double2 U = S[(5 + a) * N + g];
            const double2 E = make_double2(k[a] * phi.y - U.x, -k[a] * phi.x - U.y);   // -i k phi - U
            e2 += E.x * E.x + E.y * E.y;
        }
        const double2 Bx = csub(ik(k[1], A[2]), ik(k[2], A[1]));
        const double2 By = csub(ik(k[2], A[0]), ik(k[0], A[2]));
        const double2 Bz = csub(ik(k[0], A[1]), ik(k[1], A[0]));
        b2 = Bx.x * Bx.x + Bx.y * Bx.y + By.x * By.x + By.y * By.y + Bz.x * Bz.x + Bz.y * Bz.y;
        e += (e2 / (2.0 * p.sigma1) + b2 / (2.0 * p.sigma2)) * p.dV * p.invN;
    }
    const double r = block_sum(e, sm);
    if (threadIdx.x == 0) partials[slot * MAX_BLOCKS + blockIdx.x] = r;
}

// Residual transforms of the committed level n+1 (§5.1): gauge G = psi / kappa^2 + D . A,
// Gauss R = D . E - sigma1 rho, continuity C = rho^{n+1} - rho^n + dt D . J.
__global__ void k_spec_resid(SpecParams p, const double2* __restrict__ S1, const double2* __restrict__ S0,
                             const double2* __restrict__ Jh, double2* __restrict__ out) {
    const int64_t N = p.m.ncell;
    SPEC_LOOP(g, N) {
        double k[3];
        mode_k(p, g, k);
        const double2 phi = S1[g], psi = S1[4 * N + g], rho1 = S1[8 * N + g], rho0 = S0[8 * N + g];
        double2 divA = make_double2(0.0, 0.0), divE = make_double2(0.0, 0.0), divJ = make_double2(0.0, 0.0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            divA = cadd(divA, ik(k[a], S1[(1 + a) * N + g]));
            const double2 U = S1[(5 + a) * N + g];
            const double2 E = make_double2(k[a] * phi.y - U.x, -k[a] * phi.x - U.y);
            divE = cadd(divE, ik(k[a], E));
            divJ = cadd(divJ, ik(k[a], Jh[a * N + g]));
        }
        out[g] = make_double2(psi.x / p.kappa2 + divA.x, psi.y / p.kappa2 + divA.y);
        out[N + g] = make_double2(divE.x - p.sigma1 * rho1.x, divE.y - p.sigma1 * rho1.y);
        out[2 * N + g] = make_double2(rho1.x - rho0.x + p.dt * divJ.x, rho1.y - rho0.y + p.dt * divJ.y);
    }
}

// Real-space reductions of the final sweep: mesh work sum_g J . E^{n+1/2} dV with
// E^{n+1/2} = -D phi^{n+1/2} - U^{n+1/2}, and max / sum of squares of the residuals.
__global__ void k_spec_diag(SpecParams p, const double* __restrict__ J, const double* __restrict__ gphi,
                            const double* __restrict__ W0, const double* __restrict__ W1,
                            const double2* __restrict__ resid, double* __restrict__ partials) {
    __shared__ double sm[32];
    const int64_t N = p.m.ncell;
    double mwork = 0.0, gmax = 0.0, gsq = 0.0, rmax = 0.0, rsq = 0.0, cmax = 0.0;
    SPEC_LOOP(g, N) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double Eh = -gphi[a * N + g] - 0.5 * (W1[(1 + a) * N + g] + W0[(1 + a) * N + g]);
            mwork += J[a * N + g] * Eh * p.dV;
        }
        const double G = resid[g].x * p.invN, R = resid[N + g].x * p.invN, Cc = resid[2 * N + g].x * p.invN;
        gmax = fmax(gmax, fabs(G));
        gsq += G * G;
        rmax = fmax(rmax, fabs(R));
        rsq += R * R;
        cmax = fmax(cmax, fabs(Cc));
    }
    const double v[6] = {mwork, gmax, gsq, rmax, rsq, cmax};
    const int slots[6] = {S_MWORK, S_G_MAX, S_G_SQ, S_R_MAX, S_R_SQ, S_CONT_MAX};
    const bool mx[6] = {false, true, false, true, false, true};
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        const double r = mx[t] ? block_max(v[t], sm) : block_sum(v[t], sm);
        if (threadIdx.x == 0) partials[slots[t] * MAX_BLOCKS + blockIdx.x] = r;
    }
}

// phi^ = sigma1 rho^ / |k|^2 away from the null modes (-Delta_h phi = sigma1 rho), 0 on them.
__global__ void k_spec_poisson(SpecParams p, double2* __restrict__ rh) {
    SPEC_LOOP(g, p.m.ncell) {
        double k[3];
        mode_k(p, g, k);
        const double k2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2];
        const double s = k2 > 0.0 ? p.sigma1 / k2 : 0.0;
        rh[g] = make_double2(rh[g].x * s, rh[g].y * s);
    }
}

SpecParams spec_params(const Ctx& c) {
    SpecParams p;
    p.m = c.m;
    for (int a = 0; a < 3; ++a) p.kscale[a] = 2.0 * M_PI / c.cfg.L[a];
    p.dt = c.cfg.dt;
    p.kappa2 = c.cfg.kappa * c.cfg.kappa;
    p.sigma1 = c.cfg.sigma1;
    p.sigma2 = c.cfg.sigma2;
    p.dV = c.dV;
    p.invN = 1.0 / (double)c.m.ncell;
    return p;
}

int spec_blocks(const Ctx& c, int64_t n) {
    int64_t b = (n + THREADS - 1) / THREADS;
    if (b > (int64_t)c.sms * 8) b = (int64_t)c.sms * 8;
    return (int)std::max<int64_t>(b, 1);
}

FftAxis make_axis(const Ctx& c, int a, int nf) {
    FftAxis ax{};
    ax.axis = a;
    ax.n = c.m.n[a];
    ax.stride = a == 0 ? 1 : (a == 1 ? c.m.n[0] : (int64_t)c.m.n[0] * c.m.n[1]);
    ax.tw = c.fft_tw[a];
    // lines per block: as many as keep the two shared copies within 32 KB and divide the run of adjacent
    // lines (all of them along x, the x extent for y, the x-y plane for z), while the blocks fill the SMs
    const int64_t nlines = c.m.ncell / ax.n, run = a == 0 ? nlines : ax.stride;
    ax.lb = 1;
    while (ax.lb < 16 && 2 * (2 * ax.lb) * ax.n <= 2048 && run % (2 * ax.lb) == 0 &&
           (ax.lb < (a == 0 ? 1 : 4) || nf * (nlines / (2 * ax.lb)) >= 2 * c.sms))
        ax.lb *= 2;
    ax.mn = multiplier(ax.n);
    ax.mlb = multiplier(ax.lb);
    for (int s = 0, L = 1; s < c.fft_nst[a]; ++s) {
        FftStage& st = ax.st[ax.nst++];
        st.R = c.fft_radix[a][s];
        if (st.R == 2 && s + 1 < c.fft_nst[a]) {   // (the 3s come first)
            st.R = 4;
            ++s;
        }
        st.L = L;
        st.nb = ax.n / st.R;
        st.tstep = ax.n / (L * st.R);
        st.mL = multiplier(L);
        st.mnb = multiplier(st.nb);
        L *= st.R;
    }
    return ax;
}

// 3D transform of nf contiguous complex fields, in place, or from (forward) or to (inverse) real ones.
void fft3(Ctx& c, double2* data, int nf, bool inverse, const RealFields* real = nullptr) {
    const RealFields none;
    int first = 0, last = 2;
    while (first < 2 && c.m.n[first] == 1) ++first;
    while (last > first && c.m.n[last] == 1) --last;
    for (int a = first; a <= last; ++a) {   // (one pass at least, which converts)
        if (c.m.n[a] == 1 && first != last) continue;
        const FftAxis ax = make_axis(c, a, nf);
        const int threads = std::min(256, std::max(32, ((ax.lb * ax.n / 4 + 31) / 32) * 32));
        const int64_t gx = std::min<int64_t>(c.m.ncell / (ax.lb * ax.n), (int64_t)c.sms * 16);
        dim3 grid((unsigned)gx, (unsigned)nf);
        k_fft_axis<<<grid, threads, 2 * ax.lb * ax.n * sizeof(double2), c.stream>>>(
            data, c.m, ax, inverse ? 1 : 0, !inverse && real && a == first ? *real : none,
            inverse && real && a == last ? *real : none);
        ++c.launches;
    }
}

// The state's fields [phi, A (3) | psi, U (3) | rho | gphi (3)] as real fields (null ones left out at the end).
RealFields state_fields(const Ctx& c, const double* F, const double* W, const double* rho = nullptr,
                        const double* gphi = nullptr) {
    const int64_t N = c.m.ncell;
    RealFields r;
    for (int f = 0; f < 4; ++f) {
        r.f[f] = const_cast<double*>(F) + f * N;
        r.f[4 + f] = const_cast<double*>(W) + f * N;
    }
    r.f[8] = const_cast<double*>(rho);
    for (int f = 0; f < 3 && gphi; ++f) r.f[9 + f] = const_cast<double*>(gphi) + f * N;
    return r;
}

RealFields fields_of(const Ctx& c, const double* x, int nf, double scale = 1.0) {
    RealFields r;
    for (int f = 0; f < nf; ++f) r.f[f] = const_cast<double*>(x) + f * c.m.ncell;
    r.scale = scale;
    return r;
}

}  // namespace

// Mesh sizes of the form 2^p 3^q up to FFT_MAX: the radices, 3s first.
bool fft_factor(int n, int* radix, int& nst) {
    nst = 0;
    if (n < 1 || n > FFT_MAX) return false;
    int r = n;
    while (r % 3 == 0) {
        radix[nst++] = 3;
        r /= 3;
    }
    while (r % 2 == 0) {
        radix[nst++] = 2;
        r /= 2;
    }
    return r == 1 && nst <= FFT_MAX_STAGES;
}

// Twiddles exp(-2 pi i t / n) of each axis, computed on the host in double precision.
void spec_twiddles(int n, std::vector<double2>& tw) {
    tw.resize((size_t)n);
    for (int t = 0; t < n; ++t) tw[t] = make_double2(std::cos(2.0 * M_PI * t / n), -std::sin(2.0 * M_PI * t / n));
}

// Start of a step: transforms of the level-n state [phi, A | psi, U | rho] into spec0.
void launch_spec_begin(Ctx& c) {
    const RealFields in = state_fields(c, c.F0, c.W0, c.rho0);
    fft3(c, c.spec0, 9, false, &in);
}

// The mesh half of an iteration with spectral operators: e_J partials, continuity and the
// exact CN update per mode, level n+1 and D phi^{n+1/2} back in real space, gather table.
void launch_spec_mesh_phase(Ctx& c, const double* Jcur, const double* Jprev) {
    const int64_t N = c.m.ncell;
    const SpecParams p = spec_params(c);
    k_spec_ej<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(N, Jcur, Jprev, c.partials);
    ++c.launches;
    const RealFields J = fields_of(c, Jcur, 3);
    fft3(c, c.specJ, 3, false, &J);
    k_spec_cn<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(p, c.specJ, c.spec0, c.spec1);
    ++c.launches;
    RealFields out = state_fields(c, c.F1, c.W1, c.rho1, c.spec_gphi);
    out.scale = p.invN;
    fft3(c, c.spec1, 12, true, &out);
    k_spec_table<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(N, c.F0, c.W0, c.F1, c.W1, c.spec_gphi, c.table);
    ++c.launches;
}

// Field energy of the state (F, W) into partial slot `slot` (spec1 is used as scratch).
void launch_spec_energy(Ctx& c, const double* F, const double* W, int slot) {
    const RealFields in = state_fields(c, F, W);
    fft3(c, c.spec1, 8, false, &in);
    k_spec_energy<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(spec_params(c), c.spec1, c.partials, slot);
    ++c.launches;
}

// Diagnostics of the final sweep (after launch_spec_mesh_phase with the final current).
void launch_spec_diag(Ctx& c, const double* Jfinal) {
    const int64_t N = c.m.ncell;
    const SpecParams p = spec_params(c);
    // level n+1 in spectral form again (the mesh phase transformed spec1 back), its energy
    const RealFields in = state_fields(c, c.F1, c.W1, c.rho1);
    fft3(c, c.spec1, 9, false, &in);
    k_spec_energy<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(p, c.spec1, c.partials, S_W);
    ++c.launches;
    k_spec_resid<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(p, c.spec1, c.spec0, c.specJ, c.specR);
    ++c.launches;
    fft3(c, c.specR, 3, true);
    k_spec_diag<<<mesh_blocks(c), mesh_threads(c), 0, c.stream>>>(p, Jfinal, c.spec_gphi, c.W0, c.W1, c.specR, c.partials);
    ++c.launches;
}

// (I - a Delta_h) x = b for nf fields with the central-difference Laplacian, exactly per mode
// (c.helm_spec: nf N complex scratch; c.helm_s2: the per-axis symbols).
void launch_helmholtz_fft(Ctx& c, const double* b, double* x, int nf, double a) {
    const int64_t N = c.m.ncell;
    const RealFields in = fields_of(c, b, nf), out = fields_of(c, x, nf);
    fft3(c, c.helm_spec, nf, false, &in);
    k_helm_fft_divide<<<spec_blocks(c, N), THREADS, 0, c.stream>>>(c.m, c.helm_s2, a, 1.0 / (double)N, c.helm_spec,
                                                                   nf);
    ++c.launches;
    fft3(c, c.helm_spec, nf, true, &out);
}

// Initial potential: -Delta_h phi = sigma1 rho, zero on the null modes (§5.4).
void launch_spec_poisson(Ctx& c) {
    const int64_t N = c.m.ncell;
    const RealFields in = fields_of(c, c.rho0, 1), out = fields_of(c, c.F0, 1, 1.0 / (double)N);
    fft3(c, c.specR, 1, false, &in);
    k_spec_poisson<<<spec_blocks(c, N), THREADS, 0, c.stream>>>(spec_params(c), c.specR);
    ++c.launches;
    fft3(c, c.specR, 1, true, &out);
}

}  // namespace pic
