// pdq_p3m.cu -- P3M electrostatics for the periodic pipe (App. A.2: the
// particle-particle particle-mesh method the paper uses for large samples).
//
// The pipe is periodic along z (period L) and isolated across.  The Coulomb
// kernel d/r^3 is split with a Gaussian screening of width 1/alpha,
//   K_L(d) = d [erf(alpha r)/r^3 - 2 alpha/sqrt(pi) exp(-alpha^2 r^2)/r^2],
//   K_S(d) = d/max(r, d_c)^3 - K_L(d)  (negligible beyond r_cut),
// K_L handled on a mesh, K_S pair by pair:
//   plan:  K_L summed over the z images at every node offset of a mesh that is
//          periodic in z and twice the charge region across (so the FFT's
//          circular convolution is the open one), transformed, divided by the
//          squared TSC window (sinc^3 per axis) and by the transform size;
//   solve: TSC charge assignment (atomics) -> FFT -> product with each kernel
//          component -> inverse FFT -> TSC interpolation; then a cell list
//          (cells >= r_cut/2 x r_cut/4, stable per-cell order, particles copied in
//          cell order) and the direct short-range sum with the minimum image along z.
// FP64 on the mesh (cuFFT does the transforms) and for the short-range pairs of the inner half of r_cut; the outer
// ones, where K_S is below a sixth of 1/r^3, in float-float (pdq_split.cuh).  One sample at a time.
#include <cufft.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "pdq_common.cuh"
#include "pdq_device.cuh"
#include "pdq_split.cuh"

struct pdq_p3m {
    int device;
    double R, L, h, hz, x0, alpha, rc;
    int M, Mx, Nx, Nz, n_img;
    int64_t max_n;
    size_t nreal, ncplx;
    size_t nhalf;               // real nodes of the Mx planes the charges reach
    cufftHandle fwd, lines, inv;     // planes (y, z) real to complex, lines along x, planes back
    bool have_fwd, have_lines, have_inv;
    cufftDoubleComplex* Gh;     // [3][ncplx] influence function
    double* Q;                  // [nhalf] charges
    cufftDoubleComplex* Qh;     // [ncplx]
    cufftDoubleComplex* Ah;     // [ncplx]
    double* A;                  // [3][nhalf] the field's components
    int ncx, ncz;
    int64_t ncells;
    int* cell_count;            // [ncells]
    int* cell_start;            // [ncells + 1]
    int* cell_fill;             // [ncells]
    int* cell_list;             // [max_n]
    double4_32a* sorted64;      // [max_n] live particles in cell order: x, y, z, q
    float4* sorted;             // [3][max_n] the same, split: x, y, z hi and q hi; mid and q lo; lo and the cell's index
    float4* ks_tab;             // short-range factor: near_tab and far_tab, kTabWords
    double* sums;               // [sums_cap][3], for the step driver
    int64_t sums_cap;
};

namespace pdq {
namespace {

struct P3MGeom {
    double R, L, h, hz, x0, alpha, rc, contact;
    int Mx, Nx, Nz, n_img, ncx, ncz;
    const float4* ks_tab;
    SplitGrid grid;             // of the split coordinates
};

// The short-range pairs read K_S's factor 1/r^3 - K_L from polynomials in r^2, in place of the reciprocal square root, K_L
// and their difference; both tables fit shared memory beside the queues.
// Inner pairs, r < r_n: sextics in FP64 on kOct octaves of 64 intervals each that end at the first power of two from
// r_n^2 on.  Through 7 Chebyshev nodes 6.3 (h/(4 r^2))^7 <= 2^-53 of r^-3 remains; where the factor falls off
// faster it is small against 1/r^3, which is what its error matters against.  Closer pairs (below r_n/16, or
// inside the contact distance) take pp_close.
// Outer pairs, r_n = r_cut/2 <= r: quintics on kFar intervals, in float-float down to t^2; t^3 carries 7e-7 of the value,
// so its float leaves 2^-45 of K_S, 2^-48 of 1/r^3.
constexpr int kOct = 8, kNear = 64 * kOct, kFar = 512;
constexpr int kTabWords = 7 * kNear / 2 + 2 * kFar + kFar / 2;      // in float4

struct P3MPart {                // the particles of one sample, current half of the state
    const void* pos;
    const void* vel;
    const double2* xy;
    int64_t o, n;
    int precision;
};

__device__ __forceinline__ bool load_particle(const P3MPart& S, int64_t g, double& x, double& y, double& z,
                                              double& q) {
    if (S.precision == PDQ_FP64) {
        const double4_32a p = ((const double4_32a*)S.pos)[g];
        const double4_32a v = ((const double4_32a*)S.vel)[g];
        x = p.x; y = p.y; z = p.z; q = p.w;
        return v.w > 0.5;
    }
    const float4 p = ((const float4*)S.pos)[g];
    const float4 v = ((const float4*)S.vel)[g];
    const double2 xy = S.xy[g];
    x = xy.x; y = xy.y; z = (double)p.z; q = (double)p.w;
    return v.w > 0.5f;
}

// K_L(d) / |d| factor: erf(ar)/r^3 - 2a/sqrt(pi) e^{-a^2 r^2}/r^2; Taylor series near 0, 1/r^3 far out.
__device__ __forceinline__ double long_factor(double r2, double alpha) {
    const double r = sqrt(r2), ar = alpha * r;
    const double c = 1.1283791670955126;      // 2 / sqrt(pi)
    if (ar < 0.05) {                          // Taylor series where the closed form cancels
        const double u = ar * ar;
        return c * alpha * alpha * alpha * (2.0 / 3.0) * (1.0 - 0.6 * u + (3.0 / 14.0) * u * u);
    }
    const double ir2 = 1.0 / r2, ir3 = ir2 / r;
    if (ar > 6.5) return ir3;                 // erf = 1, the Gaussian below 1e-18
    return erf(ar) * ir3 - c * alpha * exp(-ar * ar) * ir2;
}

__global__ void k_p3m_kernel(const P3MGeom G, double* gx, double* gy, double* gz) {
    const int64_t nreal = (int64_t)G.Nx * G.Nx * G.Nz;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nreal) return;
    const int iz = (int)(idx % G.Nz);
    const int iy = (int)((idx / G.Nz) % G.Nx);
    const int ix = (int)(idx / ((int64_t)G.Nz * G.Nx));
    if (2 * ix == G.Nx || 2 * iy == G.Nx) { gx[idx] = 0.0; gy[idx] = 0.0; gz[idx] = 0.0; return; }
    const double dx = (ix > G.Nx / 2 ? ix - G.Nx : ix) * G.h;
    const double dy = (iy > G.Nx / 2 ? iy - G.Nx : iy) * G.h;
    const double dz0 = (iz > G.Nz / 2 ? iz - G.Nz : iz) * G.hz;
    const double rho2 = dx * dx + dy * dy;
    double sx = 0.0, sy = 0.0, sz = 0.0;
    for (int k = -G.n_img; k <= G.n_img; ++k) {
        const double dz = dz0 - k * G.L;
        const double r2 = rho2 + dz * dz;
        const double f = long_factor(r2, G.alpha);
        sx += f * dx; sy += f * dy; sz += f * dz;
    }
    const double tail = 1.0 / (2.0 * (G.n_img + 0.5) * (G.n_img + 0.5)) / (G.L * G.L * G.L);
    sx += 2.0 * dx * tail;
    sy += 2.0 * dy * tail;
    sz += -4.0 * dz0 * tail;
    if (2 * iz == G.Nz) sz = 0.0;              // half a period: the odd z-component vanishes
    gx[idx] = sx; gy[idx] = sy; gz[idx] = sz;
}

__device__ __forceinline__ double sinc6(double m) {
    if (m == 0.0) return 1.0;
    const double a = kPi * m, s = sin(a) / a;
    const double s3 = s * s * s;
    return s3 * s3;
}

// Divide the kernel transforms by the squared TSC window and the transform size.
__global__ void k_p3m_deconv(const P3MGeom G, cufftDoubleComplex* gh, int64_t ncplx) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ncplx) return;
    const int nzh = G.Nz / 2 + 1;
    const int iz = (int)(idx % nzh);
    const int iy = (int)((idx / nzh) % G.Nx);
    const int ix = (int)(idx / ((int64_t)nzh * G.Nx));
    const double mx = (double)min(ix, G.Nx - ix) / G.Nx, my = (double)min(iy, G.Nx - iy) / G.Nx;
    const double mz = (double)iz / G.Nz;
    const double w = sinc6(mx) * sinc6(my) * sinc6(mz) * ((double)G.Nx * G.Nx * G.Nz);
    for (int c = 0; c < 3; ++c) {
        cufftDoubleComplex& v = gh[c * ncplx + idx];
        v.x /= w;
        v.y /= w;
    }
}

// TSC: nearest node and weights of a coordinate in node units.
__device__ __forceinline__ int tsc(double t, int lo, int hi, double w[3]) {
    int i0 = (int)rint(t);
    const double d = t - i0;
    w[0] = 0.5 * (0.5 - d) * (0.5 - d);
    w[1] = 0.75 - d * d;
    w[2] = 0.5 * (0.5 + d) * (0.5 + d);
    return i0 < lo ? lo : (i0 > hi ? hi : i0);   // particles are inside the pipe; the clamp is a guard
}

__global__ void k_p3m_assign(const P3MGeom G, const P3MPart S, double* Q) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= S.n) return;
    double x, y, z, q;
    if (!load_particle(S, S.o + k, x, y, z, q) || q == 0.0) return;
    double wx[3], wy[3], wz[3];
    const int ix = tsc((x - G.x0) / G.h, 1, G.Mx - 2, wx);
    const int iy = tsc((y - G.x0) / G.h, 1, G.Mx - 2, wy);
    const int iz = tsc(z / G.hz, -1 << 30, 1 << 30, wz);
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            const int64_t rowb = ((int64_t)(ix + a - 1) * G.Nx + (iy + b - 1)) * G.Nz;
            for (int c = 0; c < 3; ++c) {
                int zz = (iz + c - 1) % G.Nz;
                if (zz < 0) zz += G.Nz;
                atomicAdd(&Q[rowb + zz], q * wx[a] * wy[b] * wz[c]);
            }
        }
}

__global__ void k_p3m_mul(const cufftDoubleComplex* __restrict__ Qh, const cufftDoubleComplex* __restrict__ gh,
                          cufftDoubleComplex* __restrict__ Ah, int64_t ncplx) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ncplx) return;
    const cufftDoubleComplex a = Qh[idx], b = gh[idx];
    Ah[idx] = make_cuDoubleComplex(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Long-range sums interpolated with the assignment weights (written, not added).
__global__ void k_p3m_interp(const P3MGeom G, const P3MPart S, const double* __restrict__ A, int64_t nhalf,
                             double* sums) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= S.n) return;
    const int64_t g = S.o + k;
    double x, y, z, q;
    if (!load_particle(S, g, x, y, z, q)) return;
    double wx[3], wy[3], wz[3];
    const int ix = tsc((x - G.x0) / G.h, 1, G.Mx - 2, wx);
    const int iy = tsc((y - G.x0) / G.h, 1, G.Mx - 2, wy);
    const int iz = tsc(z / G.hz, -1 << 30, 1 << 30, wz);
    double s[3] = {0.0, 0.0, 0.0};
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            const int64_t rowb = ((int64_t)(ix + a - 1) * G.Nx + (iy + b - 1)) * G.Nz;
            for (int cc = 0; cc < 3; ++cc) {
                int zz = (iz + cc - 1) % G.Nz;
                if (zz < 0) zz += G.Nz;
                for (int c = 0; c < 3; ++c) s[c] += A[c * nhalf + rowb + zz] * wx[a] * wy[b] * wz[cc];
            }
        }
    for (int c = 0; c < 3; ++c) sums[3 * g + c] = s[c];
}

// Cells are at least r_cut / kReachXY wide across the pipe and r_cut / kReachZ along it, so a particle's
// neighbours lie at most that many cells away.
constexpr int kReachXY = 2, kReachZ = 4;

__device__ __forceinline__ int cell_of(const P3MGeom& G, double x, double y, double z) {
    const double wxy = 2.0 * G.R / G.ncx, wz = G.L / G.ncz;
    int cx = (int)floor((x + G.R) / wxy), cy = (int)floor((y + G.R) / wxy), cz = (int)floor(z / wz);
    cx = cx < 0 ? 0 : (cx >= G.ncx ? G.ncx - 1 : cx);
    cy = cy < 0 ? 0 : (cy >= G.ncx ? G.ncx - 1 : cy);
    cz = cz < 0 ? 0 : (cz >= G.ncz ? G.ncz - 1 : cz);
    return (cx * G.ncx + cy) * G.ncz + cz;
}

__global__ void k_cell_count(const P3MGeom G, const P3MPart S, int* count) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= S.n) return;
    double x, y, z, q;
    if (!load_particle(S, S.o + k, x, y, z, q)) return;
    atomicAdd(&count[cell_of(G, x, y, z)], 1);
}

// Exclusive scan of the cell counts (one CTA of 1024 threads, 8 cells per thread, chunks in order).
__global__ void __launch_bounds__(1024) k_cell_scan(const int* count, int64_t ncells, int* start) {
    constexpr int E = 8;
    __shared__ int warp_sum[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int carry = 0;
    for (int64_t c0 = 0; c0 < ncells; c0 += 1024 * E) {
        const int64_t c = c0 + (int64_t)tid * E;
        int v[E], sum = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = c + e < ncells ? count[c + e] : 0;
            sum += v[e];
        }
        int incl = sum;
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int w = warp_sum[lane];
            int wi = w;
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, wi, d);
                if (lane >= d) wi += t;
            }
            warp_sum[lane] = wi - w;
            if (lane == 31) warp_sum[32] = wi;
        }
        __syncthreads();
        int at = carry + warp_sum[warp] + incl - sum;
        carry += warp_sum[32];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (c + e < ncells) start[c + e] = at;
            at += v[e];
        }
        __syncthreads();
    }
    if (tid == 0) start[ncells] = carry;
}

__global__ void k_cell_fill(const P3MGeom G, const P3MPart S, const int* start, int* fill, int* list) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= S.n) return;
    double x, y, z, q;
    if (!load_particle(S, S.o + k, x, y, z, q)) return;
    const int c = cell_of(G, x, y, z);
    list[start[c] + atomicAdd(&fill[c], 1)] = (int)k;
}

// Each cell's particles in increasing index (the fill order above is not deterministic).
__global__ void k_cell_sort(const int* start, int64_t ncells, int* list) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncells) return;
    const int b = start[c], e = start[c + 1];
    for (int i = b + 1; i < e; ++i) {
        const int v = list[i];
        int j = i - 1;
        while (j >= b && list[j] > v) { list[j + 1] = list[j]; --j; }
        list[j + 1] = v;
    }
}

// Live particles copied in cell order, in FP64 and split into floats.  A particle whose coordinates lie off the split
// grid, or whose charge leaves FP32's range, gets a split charge that is none, and its pairs all run in FP64.
__global__ void k_cell_gather(const P3MGeom G, const P3MPart S, const int* start, int64_t ncells, const int* list,
                              double4_32a* s64, float4* sorted, int64_t stride) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= start[ncells]) return;
    double x, y, z, q;
    load_particle(S, S.o + list[t], x, y, z, q);
    s64[t] = make_double4_32a(x, y, z, q);
    float4 h, m, l;
    split3(G.grid, x, h.x, m.x, l.x);
    split3(G.grid, y, h.y, m.y, l.y);
    split3(G.grid, z, h.z, m.z, l.z);
    const bool fits = fmax(fabs(x), fmax(fabs(y), fabs(z))) <= (double)G.grid.top && (q == 0.0 || (fabs(q) > 1e-15 && fabs(q) < 1e20));
    h.w = fits ? (float)q : NAN;
    m.w = (float)(q - (double)h.w);
    l.w = __int_as_float(cell_of(G, x, y, z));
    sorted[t] = h;
    sorted[stride + t] = m;
    sorted[2 * stride + t] = l;
}

// One thread per interval: the polynomial in t = r^2 - (the interval's lower edge) through N Chebyshev nodes, by divided
// differences over the interval's width h (a power of two, or any), expanded to powers.
template <int N>
__device__ void ks_poly(double alpha, double lower, double h, double p[N]) {
    double x[N], f[N];
    for (int i = 0; i < N; ++i) {
        x[i] = 0.5 - 0.5 * cos(kPi * (2 * i + 1) / (2.0 * N));
        const double r2 = lower + h * x[i], r = sqrt(r2);
        f[i] = erfc(alpha * r) / (r2 * r) + 1.1283791670955126 * alpha * exp(-alpha * alpha * r2) / r2;
    }
    for (int j = 1; j < N; ++j)
        for (int i = N - 1; i >= j; --i) f[i] = (f[i] - f[i - 1]) / (x[i] - x[i - j]);
    p[0] = f[N - 1];
    for (int j = 1; j < N; ++j) p[j] = 0.0;
    for (int i = N - 2; i >= 0; --i) {              // p <- p (t - x_i) + f_i
        for (int j = N - 1; j > 0; --j) p[j] = p[j - 1] - x[i] * p[j];
        p[0] = f[i] - x[i] * p[0];
    }
    double scale = 1.0;
    for (int j = 0; j < N; ++j, scale /= h) p[j] *= scale;
}
__global__ void k_ks_table(double alpha, int e0, double far0, double h_far, float4* tab) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kNear) {
        double p[7];
        const double octave = ldexp(1.0, e0 + k / 64), h = octave / 64.0;
        ks_poly<7>(alpha, octave + h * (k % 64), h, p);
        for (int j = 0; j < 7; ++j) ((double*)tab)[j * kNear + k] = p[j];
    }
    if (k < kFar) {
        double p[6];
        const float lower = (float)(far0 + h_far * k);
        ks_poly<6>(alpha, (double)lower, h_far, p);
        float c[6], l[3];
        for (int j = 0; j < 6; ++j) {
            c[j] = (float)p[j];
            if (j < 3) l[j] = (float)(p[j] - (double)c[j]);
        }
        float4* far = tab + 7 * kNear / 2;
        far[k] = make_float4(c[0], l[0], c[1], l[1]);
        far[kFar + k] = make_float4(c[2], l[2], c[3], c[4]);
        ((float2*)(far + 2 * kFar))[k] = make_float2(c[5], lower);
    }
}

// The particle-independent numbers of the short-range pairs.  Comparisons of positive doubles are made on their
// bits, beside the FP64 pipe.
struct PPConst {
    double L, invL, alpha, dc2;
    long long half_bits, cut_bits;               // L/2, r_cut^2
    long long low_bits, end_bits;                // the near table's range, from d_c^2 at the least
    int base;                                    // its first edge's upper word without the last 14 bits
    float Lh, Lm, Ll;                            // the period, split like a coordinate
    float rch, rcl;                              // r_cut^2
    float far0, kf, far_min;                     // the far table's start, intervals per unit r^2; from d_c^2 at the least
    float Lf, invLf, rc2, rn2;                   // of the screen: the period, the widened r_cut^2, and r_n^2
    float wxy, R;                                // cell width across, pipe radius
};

// 1 / max(r, d_c)^3 - K_L factor at the close pairs: K_L by c alpha^3 sum_m (-1)^m 2 u^m / (m! (2m + 3)), u = (alpha r)^2, to
// m = 17 below u = 1 (where the closed form cancels; the next term is below 2^-56), by the closed form above.
__device__ __forceinline__ double pp_close(const PPConst& K, double r2) {
    const double c = 1.1283791670955126, u = K.alpha * K.alpha * r2, a3 = K.alpha * K.alpha * K.alpha;
    double kl;
    if (u < 1.0) {
        constexpr double inv_fact[18] = {
            1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320, 1.0 / 362880,
            1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0, 1.0 / 87178291200.0,
            1.0 / 1307674368000.0, 1.0 / 20922789888000.0, 1.0 / 355687428096000.0};
        double s = 0.0;
#pragma unroll
        for (int m = 17; m >= 0; --m) s = __fma_rn(s, -u, 2.0 * inv_fact[m] / (2 * m + 3));
        kl = c * a3 * s;
    } else {
        const double x = sqrt(u);
        kl = a3 * (erf(x) / (u * x) - c * exp(-u) / u);
    }
    const double ic = rsqrt(fmax(r2, K.dc2));             // 1 / max(r, d_c)
    return ic * (ic * ic) - kl;
}

// One short-range pair: q_j (d / max(r, d_c)^3 - K_L(d)) when r < r_cut, in FP64 (17 operations).
__device__ __forceinline__ void pp_pair(const PPConst& K, const double* T, const double4_32a& pi, const double4_32a& pj,
                                        double& sx, double& sy, double& sz) {
    const double dx = pi.x - pj.x, dy = pi.y - pj.y;
    double dz = pi.z - pj.z;
    if ((__double_as_longlong(dz) & 0x7fffffffffffffffll) > K.half_bits)      // few pairs: nearest image
        dz = __fma_rn(-K.L, rint(dz * K.invL), dz);
    const double r2 = __fma_rn(dx, dx, __fma_rn(dy, dy, dz * dz));
    const long long bits = __double_as_longlong(r2);
    if ((unsigned long long)bits >= (unsigned long long)K.cut_bits) return;      // NaN too, of either sign
    double f;
    if (bits >= K.low_bits && bits < K.end_bits) {
        const int hi = (int)(bits >> 32);
        const double* p = T + ((hi >> 14) - K.base);
        const double t = r2 - __hiloint2double(hi & ~0x3fff, 0);
        f = p[6 * kNear];
#pragma unroll
        for (int j = 5; j >= 0; --j) f = __fma_rn(f, t, p[j * kNear]);
    } else f = pp_close(K, r2);
    f *= pj.w;
    sx = __fma_rn(f, dx, sx);
    sy = __fma_rn(f, dy, sy);
    sz = __fma_rn(f, dz, sz);
}

// The same for r >= r_n in float-float (~110 FP32 operations), added to the float-float sums s, c; false (and
// nothing added) when the pair is not one for it.
__device__ __forceinline__ bool pp_far(const PPConst& K, const float4* T, const float4 ih, const float4 im,
                                       const float4 il, const float4 jh, const float4 jm, const float4 jl, float s[3],
                                       float c[3]) {
    float D[3], E[3], R, r;
    split_diff(ih.x, im.x, il.x, jh.x, jm.x, jl.x, D[0], E[0]);
    split_diff(ih.y, im.y, il.y, jh.y, jm.y, jl.y, D[1], E[1]);
    const float dz = __fsub_rn(ih.z, jh.z), n = rintf(dz * K.invLf);       // nearest image, n in {-1, 0, 1}
    two_sum(__fmaf_rn(-n, K.Lh, dz), __fmaf_rn(-n, K.Lm, __fsub_rn(im.z, jm.z)), D[2], E[2]);
    E[2] = __fadd_rn(E[2], __fmaf_rn(-n, K.Ll, __fsub_rn(il.z, jl.z)));
    split_norm2(D, E, R, r);
    if (!(R >= K.far_min) || isnan(__fadd_rn(ih.w, jh.w))) return false;
    if (!(__fadd_rn(__fsub_rn(R, K.rch), __fsub_rn(r, K.rcl)) < 0.f)) return true;
    int k = (int)__fmul_rn(__fsub_rn(R, K.far0), K.kf);
    k = k < kFar ? k : kFar - 1;
    const float4 t0 = T[k], t1 = T[kFar + k];
    const float2 t2 = ((const float2*)(T + 2 * kFar))[k];
    float th, te, kl, ke;
    fast_two_sum(__fsub_rn(R, t2.y), r, th, te);
    fast_two_sum(t1.x, __fmul_rn(th, __fmaf_rn(th, __fmaf_rn(th, t2.x, t1.w), t1.z)), kl, ke);
    ke = __fadd_rn(ke, t1.y);
    auto horner = [&](float ch, float cl) {        // (kl, ke) <- (ch, cl) + (th, te) (kl, ke), |ch| above the rest
        const float m = __fmul_rn(th, kl);
        const float me = __fmaf_rn(th, ke, __fmaf_rn(te, kl, __fmaf_rn(th, kl, -m)));
        float e;
        fast_two_sum(ch, m, kl, e);
        ke = __fadd_rn(e, __fadd_rn(cl, me));
    };
    horner(t0.z, t0.w);
    horner(t0.x, t0.y);
    float f, fe;
    split_mul(kl, ke, jh.w, jm.w, f, fe);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float p, e, u;
        split_mul(f, fe, D[a], E[a], p, e);
        two_sum(s[a], p, s[a], u);
        c[a] = __fadd_rn(c[a], __fadd_rn(u, e));
    }
    return true;
}

// Short-range part: q_j (d / max(r, d_c)^3 - K_L(d)) over j != i closer than r_cut, added to sums.
// One warp per particle i (cell order).  Cells are r_cut/2 wide across and r_cut/4 along the pipe
// and a column's cells follow one another, so the candidates are one run of particles (two across the
// period) in each of at most 25 columns; lane c looks column c's runs up, all at once.  The lanes then
// screen 32 candidates at a time on the hi parts (r_cut widened by the coordinates' rounding), the next 32 in flight.
// The survivors go to one of two per-warp queues in shared memory, inner or outer, and every 32 queued pairs are
// evaluated with all lanes busy; the lanes' partial sums are reduced in a fixed order.
// Bound by instruction issue and the FP64 pipe together (~1,500 candidates, ~50 inner pairs of 17 FP64 operations and
// ~360 outer ones of ~130 instructions per particle).  One million particles, mesh 256^3: 8.0 ms; all pairs in FP64 by
// the table 16.5 ms; 42.4 ms in FP64 over the 27 cells of width r_cut with K_L by a cubic table.  Error of the sums
// against extended precision, 2-norm at 100,000 particles: 1.0e-16 (like charges) and 2.2e-16 (both signs), 4.5e-16
// and 7.1e-16 with that table; all pairs in float-float with K_L in quartics left 8e-12 and 7e-11, that K_L to 2^-50
// still 1.6e-15 and 7.6e-15.
constexpr int kPPWarps = 8, kPPShared = 16 * kTabWords + kPPWarps * 128 * 4;
__global__ void __launch_bounds__(32 * kPPWarps, 3) k_p3m_pp(const P3MGeom G, const PPConst K, const P3MPart S,
                                                          const int* start, int64_t ncells, const int* list,
                                                          const double4_32a* __restrict__ s64,
                                                          const float4* __restrict__ sorted, int64_t stride,
                                                          double* sums) {
    extern __shared__ float4 pp_smem[];                    // the tables, then the queues
    for (int k = threadIdx.x; k < kTabWords; k += blockDim.x) pp_smem[k] = G.ks_tab[k];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double* Tn = (const double*)pp_smem;
    const float4* Tf = pp_smem + 7 * kNear / 2;
    int* qw = (int*)(pp_smem + kTabWords) + w * 128;       // inner, outer: 64 entries each
    const int n_live = start[ncells];
    const float rc2f = K.rc2, rn2f = K.rn2, Lf = K.Lf, invLf = K.invLf;
    const float4 *sh = sorted, *sm = sorted + stride, *sl = sorted + 2 * stride;
    const unsigned lt = (1u << lane) - 1u;
    const float wxy = K.wxy, Rf = K.R;
    for (int t = blockIdx.x * kPPWarps + w; t < n_live; t += gridDim.x * kPPWarps) {
        const float4 ih = sh[t], im = sm[t], il = sl[t];
        const double4_32a pi = s64[t];
        // column lane of the 5 x 5 around i: its runs [b0, e0) and, across the period, [b1, e1)
        int b0 = 0, e0 = 0, b1 = 0, e1 = 0;
        {
            const int ci = __float_as_int(il.w);
            const int cz = ci % G.ncz, cy = (ci / G.ncz) % G.ncx, cx = ci / (G.ncz * G.ncx);
            constexpr int kCols = 2 * kReachXY + 1;
            const int a = cx + lane / kCols - kReachXY, b = cy + lane % kCols - kReachXY;
            if (lane < kCols * kCols && a >= 0 && a < G.ncx && b >= 0 && b < G.ncx) {
                // distance across from i to the column (an edge column reaches outward without end)
                const float xl = a == 0 ? -INFINITY : a * wxy - Rf, xh = a == G.ncx - 1 ? INFINITY : (a + 1) * wxy - Rf;
                const float yl = b == 0 ? -INFINITY : b * wxy - Rf, yh = b == G.ncx - 1 ? INFINITY : (b + 1) * wxy - Rf;
                const float ex = fmaxf(0.f, fmaxf(xl - ih.x, ih.x - xh)), ey = fmaxf(0.f, fmaxf(yl - ih.y, ih.y - yh));
                if (ex * ex + ey * ey < rc2f) {
                    const int* st = start + (a * G.ncx + b) * G.ncz;
                    const int zl = cz - kReachZ, zh = cz + kReachZ + 1;          // cells [zl, zh)
                    if (zh - zl >= G.ncz) { b0 = st[0]; e0 = st[G.ncz]; }
                    else {
                        b0 = st[zl > 0 ? zl : 0];
                        e0 = st[zh < G.ncz ? zh : G.ncz];
                        if (zl < 0) { b1 = st[G.ncz + zl]; e1 = st[G.ncz]; }
                        else if (zh > G.ncz) { b1 = st[0]; e1 = st[zh - G.ncz]; }
                    }
                }
            }
        }
        double sx = 0.0, sy = 0.0, sz = 0.0;
        float s[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f};
        int qn[2] = {0, 0};
        auto near = [&](int p) { pp_pair(K, Tn, pi, s64[p], sx, sy, sz); };
        auto far = [&](int p) { if (!pp_far(K, Tf, ih, im, il, sh[p], sm[p], sl[p], s, c)) near(p); };
        const float4 none = make_float4(1e15f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const int bb = half ? b1 : b0, ee = half ? e1 : e0;
            unsigned cols = __ballot_sync(0xffffffffu, bb < ee);
            int p = 0, pe = 0;
            // the next 32 candidates: on in the run, or the first of the next column's
            auto advance = [&]() -> bool {
                p += 32;
                if (p - lane < pe) return true;
                if (!cols) return false;
                const int src = __ffs(cols) - 1;
                cols &= cols - 1;
                p = __shfl_sync(0xffffffffu, bb, src) + lane;
                pe = __shfl_sync(0xffffffffu, ee, src);
                return true;
            };
            bool more = advance();
            float4 fj = more && p < pe && p != t ? sh[p] : none;
            while (more) {
                const int pc = p;
                const float4 fc = fj;
                more = advance();
                fj = more && p < pe && p != t ? sh[p] : none;
                const float ex = ih.x - fc.x, ey = ih.y - fc.y;
                float ez = ih.z - fc.z;
                ez -= Lf * rintf(ez * invLf);
                const float d2 = ex * ex + ey * ey + ez * ez;
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const bool pass = o ? d2 >= rn2f && d2 < rc2f : d2 < rn2f;
                    const unsigned m = __ballot_sync(0xffffffffu, pass);
                    if (pass) qw[64 * o + qn[o] + __popc(m & lt)] = pc;
                    qn[o] += __popc(m);
                }
                __syncwarp();
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    if (qn[o] >= 32) {
                        if (o) far(qw[64 + lane]);
                        else near(qw[lane]);
                        __syncwarp();
                        if (lane < qn[o] - 32) qw[64 * o + lane] = qw[64 * o + 32 + lane];
                        qn[o] -= 32;
                        __syncwarp();
                    }
                }
            }
        }
        if (lane < qn[0]) near(qw[lane]);
        if (lane < qn[1]) far(qw[64 + lane]);
        __syncwarp();
        sx += (double)s[0] + (double)c[0];
        sy += (double)s[1] + (double)c[1];
        sz += (double)s[2] + (double)c[2];
        // half of the components each time the lanes halve (6 adds): x ends in lane 0, y in lane 8, z in lane 16
        const bool up = lane & 16, up2 = lane & 8;
        const double a = (up ? sz : sx) + __shfl_xor_sync(0xffffffffu, up ? sx : sz, 16);
        const double b = (up ? 0.0 : sy) + __shfl_xor_sync(0xffffffffu, up ? sy : 0.0, 16);
        double v = (up2 ? b : a) + __shfl_xor_sync(0xffffffffu, up2 ? a : b, 8);
        for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        if ((lane & 7) == 0 && lane < 24) sums[3 * (S.o + list[t]) + lane / 8] += v;
    }
}

unsigned grid_of(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

int cufft_status(cufftResult r) { return r == CUFFT_SUCCESS ? PDQ_OK : (r == CUFFT_ALLOC_FAILED ? PDQ_ERR_OOM : PDQ_ERR_CUDA); }

P3MGeom geom_of(const pdq_p3m* P, double contact) {
    P3MGeom G;
    G.R = P->R; G.L = P->L; G.h = P->h; G.hz = P->hz; G.x0 = P->x0; G.alpha = P->alpha; G.rc = P->rc;
    G.contact = contact; G.Mx = P->Mx; G.Nx = P->Nx; G.Nz = P->Nz; G.n_img = P->n_img;
    G.ncx = P->ncx; G.ncz = P->ncz;
    G.ks_tab = P->ks_tab;
    G.grid = split_grid(std::max(P->R, P->L));
    return G;
}

long long bits_of(double v) {
    long long b;
    memcpy(&b, &v, sizeof(b));
    return b;
}

// The outer pairs start at r_n: half of r_cut where K_S is small there (alpha r_cut as usual) and its floats keep
// their range, else none are.
double near_end(double alpha, double rc) { return alpha * rc >= 3.0 && rc > 1e-3 && rc < 1e4 ? 0.5 * rc : rc; }
// The near table's first octave is 2^e0, the far table's first edge far0.
int near_start(double alpha, double rc) {
    const double rn = near_end(alpha, rc);
    int e;
    const double m = frexp(rn * rn, &e);            // r_n^2 = m 2^e, 1/2 <= m < 1
    return (m > 0.5 ? e : e - 1) - kOct;
}
double far_start(double alpha, double rc) {
    const double rn = near_end(alpha, rc);
    return (double)(float)(0.98 * rn * rn);
}

PPConst pp_const_of(const P3MGeom& G) {
    PPConst K;
    const int e0 = near_start(G.alpha, G.rc);
    const double first = ldexp(1.0, e0), rc2 = G.rc * G.rc, rn = near_end(G.alpha, G.rc), far0 = far_start(G.alpha, G.rc);
    K.L = G.L; K.invL = 1.0 / G.L; K.alpha = G.alpha;
    K.dc2 = std::max(G.contact * G.contact, 1e-20);       // coincident particles stay finite: 1e-10 wall units
    K.half_bits = bits_of(0.5 * G.L);
    K.cut_bits = bits_of(rc2);
    K.low_bits = bits_of(std::max(K.dc2, first));
    K.end_bits = bits_of(ldexp(1.0, e0 + kOct));
    K.base = (int)(bits_of(first) >> 46);
    split3(G.grid, G.L, K.Lh, K.Lm, K.Ll);
    K.rch = (float)rc2; K.rcl = (float)(rc2 - (double)K.rch);
    K.far0 = (float)far0; K.far_min = (float)std::max(far0, K.dc2); K.kf = (float)(kFar / (rc2 - far0));
    K.Lf = (float)G.L; K.invLf = 1.0f / K.Lf;
    // a hi part is off by half of the grid's 2^-23 max(R, L) (up to twice that), their differences by as much again in
    // FP32: the distances of the screen are off by less than (R + L) 2^-21
    const float rcf = (float)(G.rc + 1e-3 + (G.R + G.L) * 4.76837158203125e-07);
    K.rc2 = rcf * rcf + 1e-3f;
    K.rn2 = rn < G.rc ? (float)(rn * rn) : K.rc2;          // at most rc2: the screen's filler must fail both
    K.wxy = (float)(2.0 * G.R / G.ncx); K.R = (float)G.R;
    return K;
}

void free_plan(pdq_p3m* P) {
    if (!P) return;
    if (P->have_fwd) cufftDestroy(P->fwd);
    if (P->have_lines) cufftDestroy(P->lines);
    if (P->have_inv) cufftDestroy(P->inv);
    cudaFree(P->Gh); cudaFree(P->Q); cudaFree(P->Qh); cudaFree(P->Ah); cudaFree(P->A);
    cudaFree(P->cell_count); cudaFree(P->cell_start); cudaFree(P->cell_fill); cudaFree(P->cell_list);
    cudaFree(P->sorted64); cudaFree(P->sorted); cudaFree(P->ks_tab);
    cudaFree(P->sums);
    delete P;
}

}  // namespace
}  // namespace pdq

using namespace pdq;

extern "C" int pdq_p3m_create(const pdq_field* field, const pdq_p3m_desc* d, int64_t max_particles,
                              pdq_stream_t stream, pdq_p3m** out) {
    if (!field || !d || !out || max_particles < 1 || max_particles > ((int64_t)1 << 31) - 1 || d->M < 4 ||
        d->Nz < 4 || d->alpha < 0 || d->r_cut < 0 || d->n_img < 0)
        return PDQ_ERR_INVALID_ARG;
    *out = nullptr;
    pdq_p3m* P = new pdq_p3m();
    memset(P, 0, sizeof(*P));
    cudaGetDevice(&P->device);
    P->R = field->desc.r_plus;
    P->L = field->desc.l_plus;
    P->M = d->M;
    P->Nz = d->Nz;
    P->h = 2.0 * P->R / P->M;
    P->hz = P->L / P->Nz;
    P->Mx = P->M + 5;
    P->x0 = -P->R - 2.0 * P->h;
    P->Nx = 2 * P->Mx;
    P->alpha = d->alpha > 0 ? d->alpha : 0.5 / P->h;
    P->rc = d->r_cut > 0 ? d->r_cut : 3.3 / P->alpha;
    P->n_img = d->n_img > 0 ? d->n_img : 200;
    P->max_n = max_particles;
    if (!(P->rc < 0.5 * P->L)) { delete P; return PDQ_ERR_INVALID_ARG; }
    P->nreal = (size_t)P->Nx * P->Nx * P->Nz;
    P->nhalf = (size_t)P->Mx * P->Nx * P->Nz;
    P->ncplx = (size_t)P->Nx * P->Nx * (P->Nz / 2 + 1);
    P->ncx = std::max(1, (int)std::min(128.0, floor(2.0 * P->R * kReachXY / P->rc)));
    P->ncz = std::max(1, (int)std::min(512.0, floor(P->L * kReachZ / P->rc)));
    P->ncells = (int64_t)P->ncx * P->ncx * P->ncz;
    cudaStream_t s = (cudaStream_t)stream;
    int rc = PDQ_OK;
    double* Gr = nullptr;
    auto alloc = [&](void** p, size_t bytes) {
        if (rc == PDQ_OK && cudaMalloc(p, bytes) != cudaSuccess) rc = PDQ_ERR_OOM;
    };
    alloc((void**)&P->Gh, 3 * P->ncplx * sizeof(cufftDoubleComplex));
    alloc((void**)&P->Q, P->nhalf * sizeof(double));
    alloc((void**)&P->Qh, P->ncplx * sizeof(cufftDoubleComplex));
    alloc((void**)&P->Ah, P->ncplx * sizeof(cufftDoubleComplex));
    alloc((void**)&P->A, 3 * P->nhalf * sizeof(double));
    alloc((void**)&P->cell_count, P->ncells * sizeof(int));
    alloc((void**)&P->cell_start, (P->ncells + 1) * sizeof(int));
    alloc((void**)&P->cell_fill, P->ncells * sizeof(int));
    alloc((void**)&P->cell_list, P->max_n * sizeof(int));
    alloc((void**)&P->sorted64, P->max_n * sizeof(double4_32a));
    alloc((void**)&P->sorted, 3 * P->max_n * sizeof(float4));
    alloc((void**)&P->ks_tab, kTabWords * sizeof(float4));
    alloc((void**)&Gr, 3 * P->nreal * sizeof(double));
    // The charges reach only Mx of the Nx planes across (the rest is the zero padding of the open
    // convolution) and the field is read on the same Mx: the (y, z) transforms run on those planes alone,
    // the x transforms on all lines.  256^3: 1.75 -> 1.1 ms forward and 1.77 -> 1.1 ms back per component
    // against whole 3-D transforms.
    int n2[2] = {P->Nx, P->Nz}, real2[2] = {P->Nx, P->Nz}, cplx2[2] = {P->Nx, P->Nz / 2 + 1}, n1[1] = {P->Nx};
    const int plane = P->Nx * (P->Nz / 2 + 1);
    if (rc == PDQ_OK) rc = cufft_status(cufftPlanMany(&P->fwd, 2, n2, real2, 1, P->Nx * P->Nz, cplx2, 1, plane, CUFFT_D2Z, P->Mx));
    if (rc == PDQ_OK) P->have_fwd = true;
    if (rc == PDQ_OK) rc = cufft_status(cufftPlanMany(&P->lines, 1, n1, n1, plane, 1, n1, plane, 1, CUFFT_Z2Z, plane));
    if (rc == PDQ_OK) P->have_lines = true;
    if (rc == PDQ_OK) rc = cufft_status(cufftPlanMany(&P->inv, 2, n2, cplx2, 1, plane, real2, 1, P->Nx * P->Nz, CUFFT_Z2D, P->Mx));
    if (rc == PDQ_OK) P->have_inv = true;
    cufftHandle whole = 0;
    bool have_whole = false;
    if (rc == PDQ_OK) rc = cufft_status(cufftPlan3d(&whole, P->Nx, P->Nx, P->Nz, CUFFT_D2Z));
    if (rc == PDQ_OK) have_whole = true;
    if (rc == PDQ_OK) rc = cufft_status(cufftSetStream(whole, s));
    if (rc == PDQ_OK) {
        const P3MGeom G = geom_of(P, 0.0);
        k_p3m_kernel<<<grid_of(P->nreal, 256), 256, 0, s>>>(G, Gr, Gr + P->nreal, Gr + 2 * P->nreal);
        const double far0 = far_start(P->alpha, P->rc);
        k_ks_table<<<grid_of(std::max(kNear, kFar), 128), 128, 0, s>>>(P->alpha, near_start(P->alpha, P->rc), far0,
                                                                       (P->rc * P->rc - far0) / kFar, P->ks_tab);
        for (int c = 0; c < 3 && rc == PDQ_OK; ++c)
            rc = cufft_status(cufftExecD2Z(whole, Gr + c * P->nreal, P->Gh + c * P->ncplx));
        if (rc == PDQ_OK) k_p3m_deconv<<<grid_of(P->ncplx, 256), 256, 0, s>>>(G, P->Gh, (int64_t)P->ncplx);
        if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess) rc = PDQ_ERR_CUDA;
    }
    if (have_whole) cufftDestroy(whole);
    cudaFree(Gr);
    if (rc != PDQ_OK) { free_plan(P); return rc; }
    *out = P;
    return PDQ_OK;
}

extern "C" int pdq_p3m_destroy(pdq_p3m* plan) {
    free_plan(plan);
    return PDQ_OK;
}

extern "C" int pdq_p3m_params(const pdq_p3m* P, double* alpha, double* r_cut, int32_t* n_img, int32_t* nx) {
    if (!P) return PDQ_ERR_INVALID_ARG;
    if (alpha) *alpha = P->alpha;
    if (r_cut) *r_cut = P->rc;
    if (n_img) *n_img = P->n_img;
    if (nx) *nx = P->Nx;
    return PDQ_OK;
}

extern "C" int pdq_p3m_coulomb(pdq_p3m* P, const pdq_phys* phys, const pdq_state* st, double* sums,
                               pdq_stream_t stream) {
    if (!P || !phys || !st || !sums || !st->count || !st->offset || st->n_samples < 1 ||
        (st->cur != 0 && st->cur != 1) || !st->pos[st->cur] || !st->vel[st->cur] ||
        (st->precision != PDQ_FP64 && st->precision != PDQ_MIXED) ||
        (st->precision == PDQ_MIXED && !st->xy[st->cur]))
        return PDQ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (st->n_classes < 1 || st->n_classes > PDQ_MAX_CLASSES) return PDQ_ERR_INVALID_ARG;
    int rc = PDQ_OK;
    const P3MGeom G = geom_of(P, contact_distance(phys, st));
    const PPConst K = pp_const_of(G);
    std::vector<int64_t> off(st->n_samples + 1);
    std::vector<int32_t> cnt(st->n_samples);
    PDQ_CUDA(cudaMemcpyAsync(off.data(), st->offset, off.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    PDQ_CUDA(cudaMemcpyAsync(cnt.data(), st->count, cnt.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    PDQ_CUDA(cudaStreamSynchronize(s));
    for (int k = 0; k < st->n_samples; ++k)
        if (cnt[k] < 0 || cnt[k] > P->max_n) return PDQ_ERR_INVALID_ARG;
    PDQ_CUDA(cudaMemsetAsync(sums, 0, (size_t)st->capacity * 3 * sizeof(double), s));
    PDQ_CUDA(cufftSetStream(P->fwd, s) == CUFFT_SUCCESS ? cudaSuccess : cudaErrorUnknown);
    PDQ_CUDA(cufftSetStream(P->lines, s) == CUFFT_SUCCESS ? cudaSuccess : cudaErrorUnknown);
    PDQ_CUDA(cufftSetStream(P->inv, s) == CUFFT_SUCCESS ? cudaSuccess : cudaErrorUnknown);
    PDQ_CUDA(cudaFuncSetAttribute(k_p3m_pp, cudaFuncAttributeMaxDynamicSharedMemorySize, kPPShared));
    const int h = st->cur;
    for (int k = 0; k < st->n_samples; ++k) {
        if (cnt[k] == 0) continue;
        P3MPart S;
        S.pos = st->pos[h]; S.vel = st->vel[h]; S.xy = (const double2*)st->xy[h];
        S.o = off[k]; S.n = cnt[k]; S.precision = st->precision;
        const unsigned gp = grid_of(S.n, 256);
        // long range: assign, transform, multiply, transform back, interpolate
        PDQ_CUDA(cudaMemsetAsync(P->Q, 0, P->nhalf * sizeof(double), s));
        k_p3m_assign<<<gp, 256, 0, s>>>(G, S, P->Q);
        rc = cufft_status(cufftExecD2Z(P->fwd, P->Q, P->Qh));
        if (rc) return rc;
        const size_t filled = (size_t)P->Mx * P->Nx * (P->Nz / 2 + 1);
        PDQ_CUDA(cudaMemsetAsync(P->Qh + filled, 0, (P->ncplx - filled) * sizeof(cufftDoubleComplex), s));
        rc = cufft_status(cufftExecZ2Z(P->lines, P->Qh, P->Qh, CUFFT_FORWARD));
        if (rc) return rc;
        for (int c = 0; c < 3; ++c) {
            k_p3m_mul<<<grid_of(P->ncplx, 256), 256, 0, s>>>(P->Qh, P->Gh + c * P->ncplx, P->Ah, (int64_t)P->ncplx);
            rc = cufft_status(cufftExecZ2Z(P->lines, P->Ah, P->Ah, CUFFT_INVERSE));
            if (rc) return rc;
            rc = cufft_status(cufftExecZ2D(P->inv, P->Ah, P->A + c * P->nhalf));
            if (rc) return rc;
        }
        k_p3m_interp<<<gp, 256, 0, s>>>(G, S, P->A, (int64_t)P->nhalf, sums);
        // short range: cell list, then the direct sum
        PDQ_CUDA(cudaMemsetAsync(P->cell_count, 0, P->ncells * sizeof(int), s));
        PDQ_CUDA(cudaMemsetAsync(P->cell_fill, 0, P->ncells * sizeof(int), s));
        k_cell_count<<<gp, 256, 0, s>>>(G, S, P->cell_count);
        k_cell_scan<<<1, 1024, 0, s>>>(P->cell_count, P->ncells, P->cell_start);
        k_cell_fill<<<gp, 256, 0, s>>>(G, S, P->cell_start, P->cell_fill, P->cell_list);
        k_cell_sort<<<grid_of(P->ncells, 128), 128, 0, s>>>(P->cell_start, P->ncells, P->cell_list);
        k_cell_gather<<<gp, 256, 0, s>>>(G, S, P->cell_start, P->ncells, P->cell_list, P->sorted64, P->sorted, P->max_n);
        k_p3m_pp<<<(unsigned)std::min<int64_t>(grid_of(S.n, kPPWarps), 16 * 152), 32 * kPPWarps, kPPShared, s>>>(
            G, K, S, P->cell_start, P->ncells, P->cell_list, P->sorted64, P->sorted, P->max_n, sums);
    }
    PDQ_CUDA(cudaGetLastError());
    return PDQ_OK;
}

extern "C" int pdq_step_particles_p3m(const pdq_field* field, const pdq_phys* phys, pdq_state* st,
                                      const pdq_sample_params* params, const pdq_step_cfg* cfg, int64_t n_steps,
                                      pdq_tally* tally, pdq_p3m* P, void* workspace, size_t workspace_bytes,
                                      pdq_stream_t stream) {
    if (!P || !cfg || !st || n_steps < 0 || cfg->use_graph || (cfg->forces & PDQ_F_CONTACT))
        return PDQ_ERR_INVALID_ARG;
    if (st->capacity > P->sums_cap) {
        cudaFree(P->sums);
        P->sums = nullptr;
        P->sums_cap = 0;
        if (cudaMalloc(&P->sums, (size_t)std::max<int64_t>(st->capacity, 1) * 3 * sizeof(double)) != cudaSuccess)
            return PDQ_ERR_OOM;
        P->sums_cap = st->capacity;
    }
    pdq_step_cfg c1 = *cfg;
    c1.compact_every = 0;
    c1.variant = 0;
    for (int64_t k = 0; k < n_steps; ++k) {
        int rc = PDQ_OK;
        if (cfg->forces & PDQ_F_COULOMB) {
            rc = pdq_p3m_coulomb(P, phys, st, P->sums, stream);
            if (rc) return rc;
        }
        rc = step_impl(field, phys, st, params, &c1, 1, tally, workspace, workspace_bytes, stream,
                       (cfg->forces & PDQ_F_COULOMB) ? P->sums : nullptr, false);
        if (rc) return rc;
        if (cfg->compact_every > 0 && st->step % cfg->compact_every == 0 && k + 1 < n_steps) {
            rc = compact_state(st, (cudaStream_t)stream);
            if (rc) return rc;
        }
    }
    return PDQ_OK;
}
