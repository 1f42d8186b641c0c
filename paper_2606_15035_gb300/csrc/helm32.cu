// The Crank--Nicolson Helmholtz solve on meshes of small prime factors: FP64 residuals, FP32 transforms (sm_103a).
//
// (I - a Delta_h) x = b for the four potentials, by iterative refinement: the FP64 stencil residual
// r = b - (I - a Delta_h) x of the warm start, its correction by an FFT solve in FP32 (the operator is
// diagonal there, with the wide Laplacian's symbol -sum_a sin^2(2 pi m_a / n_a) / H_a^2), x += that,
// in FP64.  One correction reduces the error by the FP32 transforms' ~1e-6, so three bring any start
// to the rounding of the FP64 residual, which is what the FP64 transforms with one refinement step
// left (the correction only has to be good to its leading digits).  FP64 transforms are bound by the
// FP64 pipe on this GPU (28 operations a point and axis at 128, of the few hundred that a particle
// has); in FP32 they are bound by L2.
//
// Real fields travel in pairs, f + i g (the symbol is real and even, so the solve keeps them apart),
// each scaled by a power of two near the inverse of its right-hand side's largest value, so that no
// magnitude leaves the FP32 range and neither field of a pair drowns the other.  Five launches a
// correction: residual and x transforms; y; z forward, division, z back; y; x and the addition; or three
// where a plane of y and z fits a block (a launch costs 1.3-3 us of gap here: the static update at 32^3
// took 121.5 us with five, 106.5 with three).
//
// A mesh phase's solves measured against FP64 transforms with one refinement: 128^3 6.5 -> 1.8 ms (the
// residuals 1.0 of it, FP64), 64^3 0.86 -> 0.25 ms, 32^3 0.17 -> 0.07 ms.
#include <algorithm>
#include <cmath>
#include <vector>

#include "pic_internal.h"

namespace pic {
namespace {

constexpr int ELEMS = 2048;   // complex elements of a block's lines
constexpr int PLANE = 4096;   // ... of a block of whole y-z planes (64 KB of shared memory)

struct Stage {
    int R, L, nb, tstep;      // radix, product of the radices before, n / R, n / (L R)
    unsigned mL, mnb;         // multipliers of the divisions by L and nb
};

struct Axis32 {
    int axis, n, nst, lb;     // lb: lines of a block
    int64_t stride;
    unsigned mn, mlb;
    Stage st[FFT_MAX_STAGES];
    const float2* tw;         // exp(-2 pi i t / n)
};

// x / d for x < 2^16 by m = ceil(2^32 / d) (d = 1: m = 0)
__device__ __forceinline__ int quot(int x, unsigned m) { return m ? (int)__umulhi((unsigned)x, m) : x; }

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

template <bool INV>
__device__ __forceinline__ float2 twiddle(float2 v, float2 t) {
    const float ty = INV ? -t.y : t.y;
    return make_float2(v.x * t.x - v.y * ty, v.x * ty + v.y * t.x);
}

// Stockham transforms of the block's lb lines of n elements in x (line j at j n), with y as the other
// buffer; returns the one that holds the result.  Ends with a barrier.
template <bool INV>
__device__ __forceinline__ float2* lines_fft(float2* x, float2* y, const Axis32& ax, int lines) {
    const int n = ax.n;
    for (int s = 0; s < ax.nst; ++s) {
        const Stage st = ax.st[s];
        // a larger prime: a thread sums one output, input r rotated by r (k n / (L R) + q n / R) / n of a turn
        for (int e = threadIdx.x; st.R > 4 && e < lines * n; e += blockDim.x) {
            const int o = quot(e, st.mnb), q = o % st.R, line = o / st.R, j = e - o * st.nb;
            const int jl = quot(j, st.mL), k = j - jl * st.L, step = k * st.tstep + q * st.nb;
            const float2* in = x + line * n + j;
            float2 a = in[0];
            for (int r = 1, t = step; r < st.R; ++r) {
                const float2 v = twiddle<INV>(in[r * st.nb], __ldg(ax.tw + t));
                a = a + v;
                t += step;
                t -= t >= n ? n : 0;
            }
            y[line * n + jl * st.L * st.R + k + q * st.L] = a;
        }
        for (int e = threadIdx.x; st.R <= 4 && e < lines * st.nb; e += blockDim.x) {
            const int line = quot(e, st.mnb), j = e - line * st.nb;
            const int jl = quot(j, st.mL), k = j - jl * st.L;
            const float2* in = x + line * n + j;
            float2* out = y + line * n + jl * st.L * st.R + k;
            const int t = k * st.tstep;
            if (st.R == 4) {
                const float2 a = in[0];
                const float2 b = twiddle<INV>(in[st.nb], __ldg(ax.tw + t));
                const float2 c = twiddle<INV>(in[2 * st.nb], __ldg(ax.tw + 2 * t));
                const float2 d = twiddle<INV>(in[3 * st.nb], __ldg(ax.tw + 3 * t));
                const float2 p = a + c, q = a - c, r = b + d, u = b - d;
                const float2 iu = INV ? make_float2(-u.y, u.x) : make_float2(u.y, -u.x);   // +- i u
                out[0] = p + r;
                out[st.L] = q + iu;
                out[2 * st.L] = p - r;
                out[3 * st.L] = q - iu;
            } else if (st.R == 2) {
                const float2 a = in[0], b = twiddle<INV>(in[st.nb], __ldg(ax.tw + t));
                out[0] = a + b;
                out[st.L] = a - b;
            } else if (st.R == 3) {
                const float s3 = INV ? 0.86602540378f : -0.86602540378f;
                const float2 a = in[0];
                const float2 b = twiddle<INV>(in[st.nb], __ldg(ax.tw + t));
                const float2 c = twiddle<INV>(in[2 * st.nb], __ldg(ax.tw + 2 * t));
                const float2 sum = b + c, dif = b - c;
                const float2 mid = make_float2(a.x - 0.5f * sum.x, a.y - 0.5f * sum.y);
                out[0] = a + sum;
                out[st.L] = make_float2(mid.x - s3 * dif.y, mid.y + s3 * dif.x);
                out[2 * st.L] = make_float2(mid.x + s3 * dif.y, mid.y - s3 * dif.x);
            }
        }
        __syncthreads();
        float2* t = x;
        x = y;
        y = t;
    }
    return x;
}

struct Helm32 {
    MeshDims m;
    double invH[3], a;
    const double* b;          // right-hand sides, 4 N
    double* x;                // iterate, 4 N
    const int* top;           // per field: largest biased exponent of its right-hand side and start
    int up;                   // scale of this correction: 2^up over the right-hand side's
    float2* z;                // 2 N
    const float* s2;          // symbols sin^2 / H^2 of the three axes
    float af, invN;
};

// The power of two that brings field f's residual near one: 2^(1023 + up - top).
__device__ __forceinline__ int scale_exponent(const Helm32& h, int f) {
    return min(max(2046 + h.up - max(__ldg(h.top + f), 80), 1), 2046);
}
__device__ __forceinline__ double pow2(int biased) { return __hiloint2double(biased << 20, 0); }

__device__ __forceinline__ int wrap2(int i, int n) {
    if (i >= n) i -= n;
    if (i >= n) i -= n;
    if (i < 0) i += n;
    if (i < 0) i += n;
    return i;
}

// b - (I - a Delta_h) x of one field at node (ix, iy, iz).
__device__ __forceinline__ double residual(const Helm32& h, const double* __restrict__ f, const double* __restrict__ b,
                                           int ix, int iy, int iz) {
    const int64_t sy = h.m.n[0], sz = (int64_t)h.m.n[0] * h.m.n[1], row = sy * iy + sz * iz, g = row + ix;
    const double c = f[g];
    const double fx = f[row + wrap2(ix + 2, h.m.n[0])] - 2.0 * c + f[row + wrap2(ix - 2, h.m.n[0])];
    const double fy = f[g + sy * (wrap2(iy + 2, h.m.n[1]) - iy)] - 2.0 * c + f[g + sy * (wrap2(iy - 2, h.m.n[1]) - iy)];
    const double fz = f[g + sz * (wrap2(iz + 2, h.m.n[2]) - iz)] - 2.0 * c + f[g + sz * (wrap2(iz - 2, h.m.n[2]) - iz)];
    double s = 0.25 * h.invH[0] * h.invH[0] * fx;
    s += 0.25 * h.invH[1] * h.invH[1] * fy;
    s += 0.25 * h.invH[2] * h.invH[2] * fz;
    return b[g] - (c - h.a * s);
}

// Along x: INV = false, the residuals of fields 2 y and 2 y + 1 (y = blockIdx.y), scaled, and their
// forward transforms; INV = true, the inverse transforms, and x += what they hold.
template <bool INV>
__global__ void __launch_bounds__(256) k_helm_x(Helm32 h, Axis32 ax) {
    extern __shared__ float2 buf[];
    const int n = ax.n, tot = ax.lb * n;
    const int64_t N = h.m.ncell, nlines = N / n;
    const int f = 2 * blockIdx.y;
    float2* z = h.z + blockIdx.y * N;
    double* x0 = h.x + f * N;
    const int e0 = scale_exponent(h, f), e1 = scale_exponent(h, f + 1);
    // a field with a value that is not finite is left out of the transforms, which would hand it on to the
    // other field of the pair, and becomes NaN
    const bool ok0 = __ldg(h.top + f) < 0x7ff, ok1 = __ldg(h.top + f + 1) < 0x7ff;
    for (int64_t gr = blockIdx.x; gr * ax.lb < nlines; gr += gridDim.x) {
        const int64_t l0 = gr * ax.lb;
        const int lines = (int)min((int64_t)ax.lb, nlines - l0), cnt = lines * n;
        if (!INV) {
            const double s0 = pow2(e0), s1 = pow2(e1);
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
                const int j = quot(e, ax.mn), ix = e - j * n;
                const unsigned l = (unsigned)(l0 + j), iz = l / (unsigned)h.m.n[1], iy = l - iz * (unsigned)h.m.n[1];
                buf[e] = make_float2(ok0 ? (float)(s0 * residual(h, x0, h.b + f * N, ix, (int)iy, (int)iz)) : 0.f,
                                     ok1 ? (float)(s1 * residual(h, x0 + N, h.b + (f + 1) * N, ix, (int)iy, (int)iz)) : 0.f);
            }
        } else {
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) buf[e] = z[l0 * n + e];
        }
        __syncthreads();
        const float2* r = lines_fft<INV>(buf, buf + tot, ax, lines);
        if (!INV) {
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) z[l0 * n + e] = r[e];
        } else {
            const double s0 = ok0 ? pow2(2046 - e0) : NAN, s1 = ok1 ? pow2(2046 - e1) : NAN;
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
                const float2 v = r[e];
                x0[l0 * n + e] += s0 * (double)v.x;
                x0[N + l0 * n + e] += s1 * (double)v.y;
            }
        }
        __syncthreads();   // the buffers are rewritten by the next lines
    }
}

// Along y or z, lb lines whose elements are adjacent in memory: y forward or inverse (SOLVE = false),
// or z forward, division by N (1 + a sum s2), z inverse.
template <bool INV, bool SOLVE>
__global__ void __launch_bounds__(256) k_helm_yz(Helm32 h, Axis32 ax) {
    extern __shared__ float2 buf[];
    const int n = ax.n, lb = ax.lb, tot = lb * n;
    const int64_t N = h.m.ncell, plane = (int64_t)h.m.n[0] * h.m.n[1];
    // adjacent lines start within a row (y) or the whole plane (z)
    const int64_t run = SOLVE ? plane : h.m.n[0], groups = (run + lb - 1) / lb, total = groups * (SOLVE ? 1 : h.m.n[2]);
    float2* field = h.z + blockIdx.y * N;
    for (int64_t gr = blockIdx.x; gr < total; gr += gridDim.x) {
        const int64_t outer = gr / groups, first = (gr - outer * groups) * lb;
        const int lines = (int)min((int64_t)lb, run - first);
        float2* z = field + outer * plane + first;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int t = quot(e, ax.mlb), j = e - t * lb;
            if (j < lines) buf[j * n + t] = z[j + (int64_t)t * ax.stride];
        }
        __syncthreads();
        float2* r = lines_fft<INV>(buf, buf + tot, ax, lines);
        if (SOLVE) {
            for (int e = threadIdx.x; e < lines * n; e += blockDim.x) {
                const int j = quot(e, ax.mn), iz = e - j * n;
                const unsigned l = (unsigned)(first + j), iy = l / (unsigned)h.m.n[0], ix = l - iy * (unsigned)h.m.n[0];
                const float s = __ldg(h.s2 + ix) + __ldg(h.s2 + h.m.n[0] + iy) + __ldg(h.s2 + h.m.n[0] + h.m.n[1] + iz);
                const float d = h.invN / (1.f + h.af * s);
                r[e] = make_float2(r[e].x * d, r[e].y * d);
            }
            __syncthreads();
            r = lines_fft<true>(r, r == buf ? buf + tot : buf, ax, lines);
        }
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int t = quot(e, ax.mlb), j = e - t * lb;
            if (j < lines) z[j + (int64_t)t * ax.stride] = r[j * n + t];
        }
        __syncthreads();
    }
}

// k_helm_yz's three passes in one, where a plane of y and z fits a block's shared memory: lb adjacent x of
// field blockIdx.y, y forward, z forward, division, z back, y back.
__global__ void __launch_bounds__(512) k_helm_plane(Helm32 h, Axis32 ay, Axis32 az, int lb) {
    extern __shared__ float2 buf[];
    const int nx = h.m.n[0], ny = ay.n, nz = az.n, plane = ny * nz;
    const int first = blockIdx.x * lb, xs = min(lb, nx - first), cnt = xs * plane;
    float2* z = h.z + blockIdx.y * h.m.ncell + first;
    float2* a = buf;
    float2* b = buf + lb * plane;
    // element (j, iz, iy) of the lines along y at (j nz + iz) ny + iy, of those along z at (j ny + iy) nz + iz
    for (int e = threadIdx.x; e < lb * plane; e += blockDim.x) {
        const int r = e / lb, j = e - r * lb, iz = quot(r, ay.mn), iy = r - iz * ny;
        if (j < xs) a[(j * nz + iz) * ny + iy] = z[j + (int64_t)nx * r];
    }
    __syncthreads();
    float2* r = lines_fft<false>(a, b, ay, xs * nz);
    float2* o = r == a ? b : a;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        const int l = quot(e, ay.mn), iy = e - l * ny, j = quot(l, az.mn), iz = l - j * nz;
        o[(j * ny + iy) * nz + iz] = r[e];
    }
    __syncthreads();
    r = lines_fft<false>(o, r, az, xs * ny);
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        const int l = quot(e, az.mn), iz = e - l * nz, j = quot(l, ay.mn), iy = l - j * ny;
        const float s = __ldg(h.s2 + first + j) + __ldg(h.s2 + nx + iy) + __ldg(h.s2 + nx + ny + iz);
        const float q = h.invN / (1.f + h.af * s);
        r[e] = make_float2(r[e].x * q, r[e].y * q);
    }
    __syncthreads();
    r = lines_fft<true>(r, r == a ? b : a, az, xs * ny);
    o = r == a ? b : a;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        const int l = quot(e, az.mn), iz = e - l * nz, j = quot(l, ay.mn), iy = l - j * ny;
        o[(j * nz + iz) * ny + iy] = r[e];
    }
    __syncthreads();
    r = lines_fft<true>(o, r, ay, xs * nz);
    for (int e = threadIdx.x; e < lb * plane; e += blockDim.x) {
        const int q = e / lb, j = e - q * lb, iz = quot(q, ay.mn), iy = q - iz * ny;
        if (j < xs) z[j + (int64_t)nx * q] = r[(j * nz + iz) * ny + iy];
    }
}

// top[f] = max over field f of the biased exponents of b (top starts at zero).
__global__ void k_exponents(int64_t N, const double* __restrict__ b, int* __restrict__ top) {
    int e = 0;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x)
        e = max(e, (__double2hiint(b[blockIdx.y * N + g]) >> 20) & 0x7ff);
    e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
    if ((threadIdx.x & 31) == 0) atomicMax(top + blockIdx.y, e);
}

unsigned multiplier(int d) { return d <= 1 ? 0u : (unsigned)((((uint64_t)1 << 32) + d - 1) / d); }

Axis32 make_axis32(const HelmPlan& c, int a) {
    Axis32 ax{};
    ax.axis = a;
    ax.n = c.m.n[a];
    ax.stride = a == 0 ? 1 : (a == 1 ? c.m.n[0] : (int64_t)c.m.n[0] * c.m.n[1]);
    ax.tw = c.tw + (a == 0 ? 0 : (a == 1 ? c.m.n[0] : c.m.n[0] + c.m.n[1]));
    const int64_t run = a == 0 ? c.m.ncell / ax.n : (a == 1 ? c.m.n[0] : (int64_t)c.m.n[0] * c.m.n[1]);
    ax.lb = (int)std::max<int64_t>(1, std::min<int64_t>(run, ELEMS / ax.n));
    // few lines: a block for each part of them, so that the launch spreads over the SMs
    const int64_t lines = 2 * c.m.ncell / ax.n;
    while (ax.lb > (a == 0 ? 1 : 4) && lines / ax.lb < c.sms) ax.lb = (ax.lb + 1) / 2;
    ax.mn = multiplier(ax.n);
    ax.mlb = multiplier(ax.lb);
    int L = 1, r = ax.n;
    while (r > 1) {
        Stage& s = ax.st[ax.nst++];
        s.R = r % 4 == 0 ? 4 : 2;
        while (r % s.R) ++s.R;   // a prime from here on
        s.L = L;
        s.nb = ax.n / s.R;
        s.tstep = ax.n / (L * s.R);
        s.mL = multiplier(L);
        s.mnb = multiplier(s.nb);
        L *= s.R;
        r /= s.R;
    }
    return ax;
}

}  // namespace

void helm32_tables(const Ctx& c, std::vector<float2>& tw, std::vector<float>& s2) {
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < c.m.n[a]; ++i) {
            const double t = 2.0 * M_PI * i / c.m.n[a], s = std::sin(t);
            tw.push_back(make_float2((float)std::cos(t), (float)-s));
            s2.push_back((float)(s * s * c.invH[a] * c.invH[a]));
        }
}

// Largest exponents of the four right-hand sides (a solve from zero) into top.
void launch_helm_exponents(Ctx& c, const double* b, int* top) {
    cudaMemsetAsync(top, 0, 4 * sizeof(int), c.stream);
    k_exponents<<<dim3(std::min(mesh_blocks(c), c.sms), 4), THREADS, 0, c.stream>>>(c.m.ncell, b, top);
    ++c.launches;
}

bool setup_helm_kernels() {
    return cudaFuncSetAttribute(k_helm_plane, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                2 * (int)sizeof(float2) * PLANE) == cudaSuccess;
}

bool helm32_factor(int n) {
    if (n < 1 || n > FFT_MAX) return false;
    for (int p = 2; p <= HELM_MAX_RADIX; ++p)
        while (n % p == 0) n /= p;
    return n == 1;
}

int helm32_corrections(double lmax, double to) {
    const double q = 2.5e-7 * std::max(lmax, 2.0);
    if (!(q < 1.0)) return 0;
    const double k = std::ceil(std::log(to) / std::log(q));
    return k > HELM_MAX_CORRECTIONS ? 0 : std::max(1, (int)k);
}

namespace {

// Adjacent x of a block of k_helm_plane, fewer while the blocks do not fill the SMs, and its threads.
int plane_lines(const MeshDims& m, int sms) {
    const int64_t plane = (int64_t)m.n[1] * m.n[2];
    int lb = 4;
    while (lb > 1 && (lb * plane > PLANE || 2 * ((m.n[0] + lb - 1) / lb) < sms / 2)) lb /= 2;
    return lb;
}
int plane_threads(int64_t elements) {
    return (int)std::max<int64_t>(64, std::min<int64_t>(512, (elements / 4 + 31) / 32 * 32));
}

}  // namespace

// Measured on 18 meshes up to 430,784 nodes (8^3 to 127 x 64 x 53, primes to 127 on each axis, sizes to 1024): 17
// us and a share of the nodes, two launches more where y and z go apart, and 0.05 us for each product that
// a thread sums in the stages of larger primes.  Between -10% and +30% of the times.
double helm32_micros(const MeshDims& m, int sms) {
    HelmPlan c{};
    c.m = m;
    c.sms = sms;
    const Axis32 ax[3] = {make_axis32(c, 0), make_axis32(c, 1), make_axis32(c, 2)};
    const int64_t plane = (int64_t)m.n[1] * m.n[2];
    const bool fused = plane <= PLANE;
    double products = 0.0;
    for (int a = 0; a < 3; ++a) {
        const bool in_plane = fused && a > 0;
        const int64_t elements = in_plane ? plane_lines(m, sms) * plane : (int64_t)ax[a].lb * ax[a].n;
        const int threads = in_plane ? plane_threads(elements) : 256;
        for (int s = 0; s < ax[a].nst; ++s)
            if (ax[a].st[s].R > 4) products += 2.0 * (double)((elements + threads - 1) / threads) * ax[a].st[s].R;
    }
    return 17.5 + (double)m.ncell / 2400.0 + 0.05 * products + (fused ? 0.0 : 8.0);
}

int helm32_solve(const HelmPlan& c, const double* b, double* x, const int* top, int corrections, cudaStream_t stream) {
    Helm32 h;
    h.m = c.m;
    for (int a = 0; a < 3; ++a) h.invH[a] = c.invH[a];
    h.a = c.a;
    h.af = (float)c.a;
    h.invN = (float)(1.0 / (double)c.m.ncell);
    h.b = b;
    h.x = x;
    h.top = top;
    h.z = c.z;
    h.s2 = c.s2;
    const Axis32 ax = make_axis32(c, 0), ay = make_axis32(c, 1), az = make_axis32(c, 2);
    auto grid = [&](int64_t groups) { return dim3((unsigned)std::min<int64_t>(groups, (int64_t)c.sms * 16), 2); };
    auto smem = [](const Axis32& q) { return 2 * sizeof(float2) * (size_t)q.lb * q.n; };
    const dim3 gx = grid((c.m.ncell / ax.n + ax.lb - 1) / ax.lb);
    const dim3 gy = grid((int64_t)((c.m.n[0] + ay.lb - 1) / ay.lb) * c.m.n[2]);
    const dim3 gz = grid(((int64_t)c.m.n[0] * c.m.n[1] + az.lb - 1) / az.lb);
    // one launch for y and z where a plane fits (PLANE elements): lb adjacent x a block
    const int64_t plane = (int64_t)ay.n * az.n;
    const bool fused = plane <= PLANE;
    const int lb = plane_lines(c.m, c.sms);
    for (int k = 0; k < corrections; ++k) {
        h.up = 20 * k;   // each correction leaves a residual some 2^20 smaller
        k_helm_x<false><<<gx, 256, smem(ax), stream>>>(h, ax);
        if (fused) {
            k_helm_plane<<<dim3((c.m.n[0] + lb - 1) / lb, 2), plane_threads(lb * plane),
                           2 * sizeof(float2) * lb * plane, stream>>>(h, ay, az, lb);
            k_helm_x<true><<<gx, 256, smem(ax), stream>>>(h, ax);
            continue;
        }
        if (ay.n > 1) k_helm_yz<false, false><<<gy, 256, smem(ay), stream>>>(h, ay);
        k_helm_yz<false, true><<<gz, 256, smem(az), stream>>>(h, az);
        if (ay.n > 1) k_helm_yz<true, false><<<gy, 256, smem(ay), stream>>>(h, ay);
        k_helm_x<true><<<gx, 256, smem(ax), stream>>>(h, ax);
    }
    return corrections * (fused || ay.n <= 1 ? 3 : 5);
}

void launch_helm32(Ctx& c, const double* b, double* x, const int* top, int corrections) {
    HelmPlan p;
    p.m = c.m;
    for (int a = 0; a < 3; ++a) p.invH[a] = c.invH[a];
    p.a = 0.25 * c.cfg.kappa * c.cfg.kappa * c.cfg.dt * c.cfg.dt;
    p.sms = c.sms;
    p.z = c.helm_z;
    p.tw = c.helm_tw;
    p.s2 = c.helm_s2f;
    c.launches += helm32_solve(p, b, x, top, corrections, c.stream);
}

}  // namespace pic
