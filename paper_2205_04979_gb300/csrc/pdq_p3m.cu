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
// FP64 on the mesh (cuFFT does the transforms), float-float for the short-range pairs
// (pdq_split.cuh).  One sample at a time.
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
    float4* sorted;             // [3][max_n] live particles in cell order, split: x, y, z hi and q hi; mid and q lo;
                                // lo and the cell's index
    float4* lf_tab;             // [2][kTab] K_L factor by quartics on kTab intervals of u = (alpha r)^2 < (alpha r_cut)^2
    double* sums;               // [sums_cap][3], for the step driver
    int64_t sums_cap;
};

namespace pdq {
namespace {

struct P3MGeom {
    double R, L, h, hz, x0, alpha, rc, contact;
    int Mx, Nx, Nz, n_img, ncx, ncz;
    const float4* lf_tab;
    SplitGrid grid;             // of the split coordinates
};

// The short-range pairs read the long-range factor from quartics in u = (alpha r)^2, one per interval
// of a table (through 5 Chebyshev nodes each: relative interpolation error ~2e-15 at alpha r_cut = 3.3),
// instead of erf and exp.  1,024 intervals of 32 B fit shared memory beside the pair queues.
constexpr int kTab = 1024;

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

// Live particles copied in cell order, their coordinates and charge split into floats.
__global__ void k_cell_gather(const P3MGeom G, const P3MPart S, const int* start, int64_t ncells, const int* list,
                              float4* sorted, int64_t stride) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= start[ncells]) return;
    double x, y, z, q;
    load_particle(S, S.o + list[t], x, y, z, q);
    float4 h, m, l;
    split3(G.grid, x, h.x, m.x, l.x);
    split3(G.grid, y, h.y, m.y, l.y);
    split3(G.grid, z, h.z, m.z, l.z);
    h.w = (float)q;
    m.w = (float)(q - (double)h.w);
    l.w = __int_as_float(cell_of(G, x, y, z));
    sorted[t] = h;
    sorted[stride + t] = m;
    sorted[2 * stride + t] = l;
}

// K_L factor at u = (alpha r)^2: c alpha^3 sum_m (-1)^m 2 u^m / (m! (2m + 3)) below u = 1 (where the
// closed form cancels), the closed form above.
__device__ __forceinline__ double long_factor_u(double u, double alpha) {
    const double c = 1.1283791670955126, a3 = alpha * alpha * alpha;
    if (u < 1.0) {
        double s = 0.0, t = 1.0;                    // t = (-u)^m / m!
        for (int m = 0; m < 24; ++m) {
            s += 2.0 * t / (2 * m + 3);
            t *= -u / (m + 1);
        }
        return c * a3 * s;
    }
    const double x = sqrt(u);
    return a3 * (erf(x) / (u * x) - c * exp(-u) / u);
}

// One thread per interval: the quartic in t = position inside the interval (0..1) through the five
// Chebyshev nodes, by divided differences expanded to powers; the two leading coefficients as
// float-floats.
__global__ void k_lf_table(double alpha, double umax, float4* tab) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kTab) return;
    double x[5], f[5];
    for (int i = 0; i < 5; ++i) {
        x[i] = 0.5 - 0.5 * cos(kPi * (2 * i + 1) / 10.0);
        f[i] = long_factor_u(umax * (k + x[i]) / kTab, alpha);
    }
    for (int j = 1; j < 5; ++j)
        for (int i = 4; i >= j; --i) f[i] = (f[i] - f[i - 1]) / (x[i] - x[i - j]);
    double p[5] = {f[4], 0.0, 0.0, 0.0, 0.0};
    for (int i = 3; i >= 0; --i) {                  // p <- p (t - x_i) + f_i
        for (int j = 4; j > 0; --j) p[j] = p[j - 1] - x[i] * p[j];
        p[0] = f[i] - x[i] * p[0];
    }
    const float c0 = (float)p[0], c1 = (float)p[1];
    tab[k] = make_float4(c0, (float)(p[0] - (double)c0), c1, (float)(p[1] - (double)c1));
    tab[kTab + k] = make_float4((float)p[2], (float)p[3], (float)p[4], 0.f);
}

// The particle-independent floats of the pair arithmetic.
struct PPConst {
    float Lh, Lm, Ll;            // the period, split like a coordinate
    float rch, rcl, dch, dcl;    // r_cut^2 and d_c^2
    float kh, kl;                // table intervals per unit r^2
    float L, invL, rc2;          // of the screen: the period and (r_cut + 1e-3)^2 + 1e-3
    float wxy, R;                // cell width across, pipe radius
};

// One short-range pair: q_j (d / max(r, d_c)^3 - K_L(d)) when r < r_cut, in float-float (~145 FP32
// operations); added to the float-float sums s, c.
__device__ __forceinline__ void pp_pair(const PPConst& K, const float4* T, const float4 ih, const float4 im,
                                        const float4 il, const float4 jh, const float4 jm, const float4 jl, float s[3],
                                        float c[3]) {
    float D[3], E[3], R, r;
    split_diff(ih.x, im.x, il.x, jh.x, jm.x, jl.x, D[0], E[0]);
    split_diff(ih.y, im.y, il.y, jh.y, jm.y, jl.y, D[1], E[1]);
    const float dz = __fsub_rn(ih.z, jh.z), n = rintf(dz * K.invL);        // nearest image, n in {-1, 0, 1}
    two_sum(__fmaf_rn(-n, K.Lh, dz), __fmaf_rn(-n, K.Lm, __fsub_rn(im.z, jm.z)), D[2], E[2]);
    E[2] = __fadd_rn(E[2], __fmaf_rn(-n, K.Ll, __fsub_rn(il.z, jl.z)));
    split_norm2(D, E, R, r);
    if (!(__fadd_rn(__fsub_rn(R, K.rch), __fsub_rn(r, K.rcl)) < 0.f)) return;
    // K_L factor: interval and position inside it, then the quartic with its last steps in float-float
    float X, Xe;
    split_mul(R, r, K.kh, K.kl, X, Xe);
    int k = (int)X;
    k = k < kTab ? k : kTab - 1;
    const float th = __fsub_rn(X, (float)k);
    const float4 t0 = T[k], t1 = T[kTab + k];
    const float v = __fmaf_rn(th, __fmaf_rn(th, __fmaf_rn(th, t1.z, t1.y), t1.x), t0.w);    // c1 lo and the rest
    const float m = __fmul_rn(th, t0.z);
    float kl, ke;
    fast_two_sum(t0.x, m, kl, ke);
    ke = __fadd_rn(__fadd_rn(ke, t0.y),
                   __fmaf_rn(th, v, __fmaf_rn(Xe, t0.z, __fmaf_rn(th, t0.z, -m))));
    const bool clamp = __fadd_rn(__fsub_rn(R, K.dch), __fsub_rn(r, K.dcl)) < 0.f;
    float w, we, g, ge;
    split_inv_cube(clamp ? K.dch : R, clamp ? K.dcl : r, w, we);
    two_sum(w, -kl, g, ge);
    ge = __fadd_rn(ge, __fsub_rn(we, ke));
    float f, fe;
    split_mul(g, ge, jh.w, jm.w, f, fe);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float p, e, u;
        split_mul(f, fe, D[a], E[a], p, e);
        two_sum(s[a], p, s[a], u);
        c[a] = __fadd_rn(c[a], __fadd_rn(u, e));
    }
}

// Short-range part: q_j (d / max(r, d_c)^3 - K_L(d)) over j != i closer than r_cut, added to sums.
// One warp per particle i (cell order).  Cells are r_cut/2 wide across and r_cut/4 along the pipe
// and a column's cells follow one another, so the candidates are one run of particles (two across the
// period) in each of at most 25 columns; lane c looks column c's runs up, all at once.  The lanes then
// screen 32 candidates at a time on the hi parts (r^2 < (r_cut + 1e-3)^2 + 1e-3), the next 32 in
// flight, the survivors go to a per-warp queue in shared memory, and every 32 queued pairs are
// evaluated with all lanes busy; the lanes' partial sums (about a dozen pairs each) are reduced in a
// fixed order.
// Bound by instruction issue (screening ~1,500 candidates and ~410 pairs of ~190 instructions per
// particle).  One million particles, mesh 256^3: 5.4 ms (5.9 ms with PPConst worked out per thread: its FP64 was
// repeated where registers ran short, pipe 53 % busy, now 8 %; 6.8 ms at 3 CTAs and 80 registers, 7.5 ms with the cell
// index recomputed in FP64 by every lane); 42.4 ms in FP64 with the Hermite table in
// global memory (FP64 pipe 87 % busy), 13.6 ms in float-float over the 27 cells of width r_cut.
constexpr int kPPWarps = 8;
__global__ void __launch_bounds__(32 * kPPWarps, 4) k_p3m_pp(const P3MGeom G, const PPConst K, const P3MPart S,
                                                          const int* start, int64_t ncells, const int* list,
                                                          const float4* __restrict__ sorted, int64_t stride,
                                                          double* sums) {
    __shared__ float4 T[2 * kTab];
    __shared__ int queue[kPPWarps][64];
    for (int k = threadIdx.x; k < 2 * kTab; k += blockDim.x) T[k] = G.lf_tab[k];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int* qw = queue[w];
    const int n_live = start[ncells];
    const float rc2f = K.rc2, Lf = K.L, invLf = K.invL;
    const unsigned lt = (1u << lane) - 1u;
    const float4 *sh = sorted, *sm = sorted + stride, *sl = sorted + 2 * stride;
    const float wxy = K.wxy, Rf = K.R;
    for (int t = blockIdx.x * kPPWarps + w; t < n_live; t += gridDim.x * kPPWarps) {
        const float4 ih = sh[t], im = sm[t], il = sl[t];
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
        float s[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f};
        int qn = 0;
        auto pair = [&](int p) { pp_pair(K, T, ih, im, il, sh[p], sm[p], sl[p], s, c); };
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
                const bool pass = ex * ex + ey * ey + ez * ez < rc2f;
                const unsigned m = __ballot_sync(0xffffffffu, pass);
                if (pass) qw[qn + __popc(m & lt)] = pc;
                qn += __popc(m);
                __syncwarp();
                if (qn >= 32) {
                    pair(qw[lane]);
                    __syncwarp();
                    if (lane < qn - 32) qw[lane] = qw[32 + lane];
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
        if (lane < qn) pair(qw[lane]);
        __syncwarp();
        for (int d = 16; d > 0; d >>= 1) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float os = __shfl_xor_sync(0xffffffffu, s[a], d), oc = __shfl_xor_sync(0xffffffffu, c[a], d);
                float u;
                two_sum(s[a], os, s[a], u);
                c[a] = __fadd_rn(__fadd_rn(c[a], oc), u);
            }
        }
        if (lane < 3) {      // lane a adds component a
            const float sa = lane == 0 ? s[0] : lane == 1 ? s[1] : s[2], ca = lane == 0 ? c[0] : lane == 1 ? c[1] : c[2];
            sums[3 * (S.o + list[t]) + lane] += (double)sa + (double)ca;
        }
    }
}

unsigned grid_of(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

int cufft_status(cufftResult r) { return r == CUFFT_SUCCESS ? PDQ_OK : (r == CUFFT_ALLOC_FAILED ? PDQ_ERR_OOM : PDQ_ERR_CUDA); }

P3MGeom geom_of(const pdq_p3m* P, double contact) {
    P3MGeom G;
    G.R = P->R; G.L = P->L; G.h = P->h; G.hz = P->hz; G.x0 = P->x0; G.alpha = P->alpha; G.rc = P->rc;
    G.contact = contact; G.Mx = P->Mx; G.Nx = P->Nx; G.Nz = P->Nz; G.n_img = P->n_img;
    G.ncx = P->ncx; G.ncz = P->ncz;
    G.lf_tab = P->lf_tab;
    G.grid = split_grid(std::max(P->R, P->L));
    return G;
}

PPConst pp_const_of(const P3MGeom& G) {
    // (the floor keeps d_c^-3 inside FP32's range; it is 1e-10 wall units)
    const double rc2 = G.rc * G.rc, dc2 = std::max(G.contact * G.contact, 1e-20), kk = kTab / rc2;
    const float rcf = (float)G.rc + 1e-3f;
    PPConst K;
    split3(G.grid, G.L, K.Lh, K.Lm, K.Ll);
    K.rch = (float)rc2; K.rcl = (float)(rc2 - (double)K.rch);
    K.dch = (float)dc2; K.dcl = (float)(dc2 - (double)K.dch);
    K.kh = (float)kk; K.kl = (float)(kk - (double)K.kh);
    K.L = (float)G.L; K.invL = 1.0f / K.L;
    K.rc2 = rcf * rcf + 1e-3f;
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
    cudaFree(P->sorted); cudaFree(P->lf_tab);
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
    alloc((void**)&P->sorted, 3 * P->max_n * sizeof(float4));
    alloc((void**)&P->lf_tab, 2 * kTab * sizeof(float4));
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
        k_lf_table<<<grid_of(kTab, 128), 128, 0, s>>>(P->alpha, P->alpha * P->alpha * P->rc * P->rc, P->lf_tab);
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
        k_cell_gather<<<gp, 256, 0, s>>>(G, S, P->cell_start, P->ncells, P->cell_list, P->sorted, P->max_n);
        k_p3m_pp<<<(unsigned)std::min<int64_t>(grid_of(S.n, kPPWarps), 16 * 152), 32 * kPPWarps, 0, s>>>(
            G, K, S, P->cell_start, P->ncells, P->cell_list, P->sorted, P->max_n, sums);
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
