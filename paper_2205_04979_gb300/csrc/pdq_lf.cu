// pdq_lf.cu -- the 1-D Eulerian low-fidelity deposition model of App. B,
// batched over (sample, size class) items.
//
// Per item the model is two ODEs in the wall distance y of the particle
// centre (wall units; V = mean wall-normal particle velocity, < 0 toward the
// wall; rho = particle density over its value on the axis):
//   momentum   d/dy(V^2/2 + R v_f'^2 + Phi) = -V/tau_1     (Eq. mom_modified,
//              Phi the potentials of F_elec and F_vdw, R v_f'^2 the
//              turbophoretic term),
//   continuity J = -(D_B + eps) rho' + rho V = const, V_dep+ = -J, with the
//              kinetic wall condition J = rho_w K(V_w) at contact y = d/2.
// The closures App. B cites but does not print: v_f'^2 = (theta, z) variance
// of the synthetic field's radial velocity, R = T_L/(T_L + tau_p),
// eps = v_f'^2 T_L, tau_1 = tau_p, D_B = k_B T tau_p/m_p, isothermal gas,
// M_r = -V_w/(sqrt(2) sigma) with sigma^2 = R v_f'^2 + k_B T/m_p at contact.
//
// Layout: CTAs per class in one wave, their warps walking runs of 32 (FP64) or
// 64 samples (FP32, two per thread).  A CTA first writes the class's per-cell table into shared memory (differences
// of the turbophoretic term and of the two potential shapes, dy/tau and dy/D
// across each cell: 40 B per cell, in FP32 each value twice); then each thread
// marches its samples from the axis (V = 0) to the wall.  At every cell it solves the implicit momentum step
//   V_k^2/2 - a V_k = c,  a = dy/tau,  c = V_{k+1}^2/2 + dw + dPhi,
// taking the root V_k <= 0 in the cancellation-free form -2c/(a + sqrt(a^2+2c))
// (V_k = 0 where c < 0), and composes the exact cell solution of the flux
// equation with V and D at their cell means (exponential fitting):
//   rho_{k+1} = E_k rho_k - J G_k,  E_k = e^{a'}, G_k = (e^{a'} - 1)/V_m,
//   a' = V_m dy/D_m,
// inward as rho_axis = P rho_k - J Q (P <- P E_k, Q <- Q + P G_k), so nothing
// per node is stored.  At the wall J = rho_w K and rho_axis = 1 give
// V_dep+ = -K/(P - K Q).  PDQ_FP64 marches in FP64 (bound by the FP64 pipe);
// PDQ_MIXED marches in FP32 with the wall condition and the final ratio in
// FP64.  Either way the ~2,000 cells per item are tiny next to one
// high-fidelity sample.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "pdq_device.cuh"
#include "pdq_lf_math.cuh"

namespace pdq {

constexpr double kBoltzmann = 1.380649e-23;   // J/K
constexpr int kLfThreads = 512, kLfThreads64 = 256;   // threads per CTA of the FP32 and the FP64 march

struct LfClass {
    double tau;       // tau_p+ = tau_1+
    double y_w;       // contact distance d+/2
    double resp;      // R = T_L/(T_L + tau_p)
    double d_b;       // D_B / nu
    double thermal;   // k_B T / (m u*^2)
    double ce;        // Phi_elec+ = -ce xi^2 / y+
    double cv;        // Phi_vdw+ = -cv zeta psi(gap+)
};

struct LfArgs {
    LfClass cls[PDQ_MAX_CLASSES];
    int32_t C, n_y, n_r;
    int64_t S;
    double R, beta, tanh_beta, stretch, em1_stretch, t_lagr, cut;
    const double* var;                    // [n_r], at the field's radial nodes
    const pdq_sample_params* params;      // [S]
    double* vdep;                         // [S][C]
};

// Fluid variance at wall distance y: linear in the stretched radial coordinate
// s = atanh(r tanh(beta)/R)/beta between the field's nodes s_i = i/(n_r - 1).
__device__ __forceinline__ double lf_var_at(const LfArgs& A, double y) {
    const double r = A.R - y;
    const double s = atanh(r * A.tanh_beta / A.R) / A.beta;
    const double t = s * (double)(A.n_r - 1);
    int i = (int)floor(t);
    i = i > A.n_r - 2 ? A.n_r - 2 : i;
    i = i < 0 ? 0 : i;
    const double f = t - (double)i;
    return (1.0 - f) * A.var[i] + f * A.var[i + 1];
}

// vdW potential shape: psi = 1/gap beyond the cutoff, linear inside it (force held constant).
__device__ __forceinline__ double lf_psi(double gap, double cut) {
    return gap >= cut ? 1.0 / gap : 2.0 / cut - gap / (cut * cut);
}

struct LfNode {
    double y, w, D, inv_y, psi;
};

__device__ __forceinline__ LfNode lf_node(const LfArgs& A, const LfClass& K, int k) {
    LfNode n;
    const double s = (double)k / (double)(A.n_y - 1);
    n.y = K.y_w + (A.R - K.y_w) * expm1(A.stretch * s) / A.em1_stretch;
    const double v = lf_var_at(A, n.y);
    n.w = K.resp * v;
    n.D = K.d_b + v * A.t_lagr;
    n.inv_y = 1.0 / n.y;
    n.psi = lf_psi(n.y - K.y_w, A.cut);
    return n;
}

// One cell of the class table: differences of R v_f'^2 and of the two potential
// shapes across the cell and dy/tau (the cell's dy/D_m sits in a second array).  T:
// double, or f2 with the FP32 value in both halves, as the packed march reads it.
template <typename T>
struct __align__(16) LfCell {
    T dw, de, dv, a;
};
__device__ __forceinline__ void lf_put(double& t, double v) { t = v; }
__device__ __forceinline__ void lf_put(f2& t, double v) { t = f2_dup((float)v); }

// The class's cell table into shared memory, each node evaluated once: chunks of blockDim nodes staged
// in s_node (the last one carried over), a cell from each neighbouring pair.
template <typename T>
__device__ __forceinline__ void lf_table(const LfArgs& A, const LfClass& K, LfCell<T>* cell, T* t_h, LfNode* s_node,
                                         double* s_sigma) {
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int c0 = 0; c0 < A.n_y; c0 += nt) {
        const int k = c0 + tid;                        // node k; cell k - 1 lies between nodes k - 1 and k
        if (k < A.n_y) s_node[tid + 1] = lf_node(A, K, k);
        __syncthreads();
        if (k < A.n_y && k > 0) {
            const LfNode lo = s_node[tid], hi = s_node[tid + 1];
            const double dy = hi.y - lo.y;
            LfCell<T> e;
            lf_put(e.dw, hi.w - lo.w);
            lf_put(e.de, hi.inv_y - lo.inv_y);
            lf_put(e.dv, hi.psi - lo.psi);
            lf_put(e.a, dy / K.tau);
            cell[k - 1] = e;
            lf_put(t_h[k - 1], dy / (0.5 * (lo.D + hi.D)));
        }
        if (k == 0) *s_sigma = sqrt(K.resp * lf_var_at(A, s_node[1].y) + K.thermal);
        __syncthreads();
        if (tid == 0) s_node[0] = s_node[nt];
        __syncthreads();
    }
}

// kinetic wall condition: one-way flux of a Gaussian velocity (mean V_w, sd sigma), FP64
__device__ __forceinline__ double lf_result(double v_w, double sg, double P, double Q) {
    const double u = -v_w;
    const double M = u / (1.4142135623730951 * sg);
    const double Kw = -(0.5 * u * (1.0 + erf(M)) + sg * exp(-M * M) * 0.3989422804014327);
    return -Kw / (P - Kw * Q);
}

// The march in FP64, one sample per thread.  Bound by the FP64 pipe, so the root of the momentum equation and
// (e^x - 1)/x come from the hardware's 20-bit estimates and series of their own (pdq_lf_math.cuh) in place of the
// library's square root, divisions and expm1.  65,536 samples x 10 classes: 109 ms (157 ms with
// the library's functions), 42 FP64 operations per cell (61), pipe 83 % busy; error against 64 bits 8.7e-16 to
// 9.7e-16 (8.8e-16 to 1.3e-15).
constexpr int kLfStride = 32;   // cells between two looks at P

__global__ void __launch_bounds__(kLfThreads64) k_lf_vdep64(const LfArgs A) {
    extern __shared__ __align__(16) unsigned char lf_smem[];
    const int c = blockIdx.y;
    const LfClass K = A.cls[c];
    const int ncell = A.n_y - 1;
    LfCell<double>* cell = reinterpret_cast<LfCell<double>*>(lf_smem);
    double* t_h = reinterpret_cast<double*>(cell + ncell);
    __shared__ LfNode s_node[kLfThreads64 + 1];
    __shared__ double s_sigma;
    lf_table(A, K, cell, t_h, s_node, &s_sigma);
    const double sg = s_sigma;
    // the class's samples by runs of 32, dealt out over the CTAs first and the warps then, so that the last,
    // partial round leaves every SM the same work
    const int64_t nrun = (A.S + 31) / 32;
    for (int64_t b = (threadIdx.x >> 5) * (int64_t)gridDim.x + blockIdx.x; b < nrun;
         b += (int64_t)(kLfThreads64 / 32) * gridDim.x) {
        const int64_t s = b * 32 + (threadIdx.x & 31);
        const pdq_sample_params sp = A.params[s < A.S ? s : A.S - 1];      // past the end: a copy, not stored
        const double ae = -K.ce * sp.xi * sp.xi, av = -K.cv * sp.zeta;
        double v = 0.0, P = 1.0, Q = 0.0;   // v at node k + 1 (the axis: 0)
        // momentum: implicit drag, root <= 0 of V^2/2 - a V = c
        auto momentum = [&](const LfCell<double>& e) {
            const double c2 = __fma_rn(0.5 * v, v, e.dw) + __fma_rn(ae, e.de, av * e.dv);
            return c2 > 0.0 ? -lf_root(e.a, c2) : 0.0;
        };
        for (int k1 = ncell; k1 > 0;) {
            const int k0 = k1 > kLfStride ? k1 - kLfStride : 0;
            if (__all_sync(0xffffffffu, P == 0.0)) {
                // the flux solution is complete (P and every further P G vanish): momentum alone
                for (int k = k1 - 1; k >= k0; --k) v = momentum(cell[k]);
            } else {
                for (int k = k1 - 1; k >= k0; --k) {
                    const double h = t_h[k], vi = momentum(cell[k]);
                    // continuity: exact cell solution with the cell-mean V and D
                    double E;
                    const double phi = lf_phi64((0.5 * (vi + v)) * h, &E);
                    Q = __fma_rn(P, h * phi, Q);
                    P *= E;
                    v = vi;
                }
            }
            k1 = k0;
        }
        if (s < A.S) A.vdep[s * A.C + c] = lf_result(v, sg, P, Q);
    }
}

// The approximate division without its fix-up for denormal divisors.
__device__ __forceinline__ float lf_div_ftz(float a, float b) {
    float q;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(q) : "f"(a), "f"(b));
    return q;
}

// The march in FP32 (PDQ_MIXED), two samples per thread as packed f32x2: the cell table and the march
// in FP32 (root by x rsqrt(x) and an approximate division; Q summed with Kahan compensation), the wall
// condition and the final ratio in FP64.  Per item and cell 26 FMA-pipe operations issue as 13 packed
// instructions, beside two table loads per pair of items and the scalar square roots and divisions.
// (e^x - 1)/x is its Taylor polynomial below |x| = 0.5 (terms to x^8/9!, truncation < 1e-9 relative), the
// approximate exponential beyond (E - 1 then stays below -0.39, so its relative rounding does not grow).
// 262,144 samples x 10 classes: 6.25 ms, bit for bit the results of the scalar march (10.1 ms, bound by
// issue); 8.0 ms with the table in single floats, 256-thread CTAs and the denormal fix-ups.
__global__ void __launch_bounds__(kLfThreads) k_lf_vdep32(const LfArgs A) {
    extern __shared__ __align__(16) unsigned char lf_smem[];
    const int c = blockIdx.y;
    const LfClass K = A.cls[c];
    const int ncell = A.n_y - 1;
    LfCell<f2>* cell = reinterpret_cast<LfCell<f2>*>(lf_smem);
    f2* t_h = reinterpret_cast<f2*>(cell + ncell);
    __shared__ LfNode s_node[kLfThreads + 1];
    __shared__ double s_sigma;
    lf_table(A, K, cell, t_h, s_node, &s_sigma);
    const double sg = s_sigma;
    const int64_t nrun = (A.S + 63) / 64;         // runs of 64 samples, dealt out as in the FP64 march
    const f2 half = f2_pack(0.5f, 0.5f);
    for (int64_t b = (threadIdx.x >> 5) * (int64_t)gridDim.x + blockIdx.x; b < nrun;
         b += (int64_t)(kLfThreads / 32) * gridDim.x) {
        const int64_t s0 = b * 64 + (threadIdx.x & 31), s1 = s0 + 32;
        const pdq_sample_params p0 = A.params[s0 < A.S ? s0 : A.S - 1], p1 = A.params[s1 < A.S ? s1 : A.S - 1];
        const f2 ae = f2_pack((float)(-K.ce * p0.xi * p0.xi), (float)(-K.ce * p1.xi * p1.xi));
        const f2 av = f2_pack((float)(-K.cv * p0.zeta), (float)(-K.cv * p1.zeta));
        f2 V = 0ull, P = f2_pack(1.f, 1.f), Q = 0ull, NC = 0ull;      // NC: minus the compensation of Q
        // momentum: implicit drag, root <= 0 of V^2/2 - a V = c
        auto momentum = [&](const LfCell<f2>& e) -> f2 {
            const f2 c2 = f2_add(f2_fma(f2_mul(half, V), V, e.dw), f2_fma(ae, e.de, f2_mul(av, e.dv)));
            const f2 cc = f2_add(c2, c2), x = f2_fma(e.a, e.a, cc);
            float ca, cb, xa, xb, da, db;
            f2_unpack(cc, ca, cb);
            f2_unpack(x, xa, xb);
            f2_unpack(f2_fma(x, f2_pack(rsqrt_ftz(xa), rsqrt_ftz(xb)), e.a), da, db);
            return f2_pack(ca > 0.f ? lf_div_ftz(-ca, da) : 0.f, cb > 0.f ? lf_div_ftz(-cb, db) : 0.f);
        };
        for (int k1 = ncell; k1 > 0;) {
            const int k0 = k1 > kLfStride ? k1 - kLfStride : 0;
            float Pa, Pb;
            f2_unpack(P, Pa, Pb);
            if (__all_sync(0xffffffffu, Pa == 0.f && Pb == 0.f)) {
                // the flux solution is complete (P and every further P G vanish): momentum alone
                for (int k = k1 - 1; k >= k0; --k) V = momentum(cell[k]);
            } else {
                for (int k = k1 - 1; k >= k0; --k) {
                    const f2 h = t_h[k], Vi = momentum(cell[k]);
                    // continuity: exact cell solution with the cell-mean V and D
                    const f2 am = f2_mul(f2_mul(half, f2_add(Vi, V)), h);      // <= 0
                    f2 p = f2_dup(2.7557319e-6f);                              // 1/9!
                    p = f2_fma(p, am, f2_dup(2.4801587e-5f));
                    p = f2_fma(p, am, f2_dup(1.9841270e-4f));
                    p = f2_fma(p, am, f2_dup(1.3888889e-3f));
                    p = f2_fma(p, am, f2_dup(8.3333333e-3f));
                    p = f2_fma(p, am, f2_dup(4.1666667e-2f));
                    p = f2_fma(p, am, f2_dup(1.6666667e-1f));
                    p = f2_fma(p, am, f2_dup(0.5f));
                    p = f2_fma(p, am, f2_dup(1.0f));
                    f2 E = f2_fma(am, p, f2_dup(1.0f));
                    float ma, mb;
                    f2_unpack(am, ma, mb);
                    if (!(ma > -0.5f && mb > -0.5f)) {
                        float ea, eb, pa, pb;
                        f2_unpack(E, ea, eb);
                        f2_unpack(p, pa, pb);
                        if (!(ma > -0.5f)) { ea = __expf(ma); pa = lf_div_ftz(ea - 1.0f, ma); }
                        if (!(mb > -0.5f)) { eb = __expf(mb); pb = lf_div_ftz(eb - 1.0f, mb); }
                        E = f2_pack(ea, eb);
                        p = f2_pack(pa, pb);
                    }
                    const f2 y = f2_fma(P, f2_mul(h, p), NC), t = f2_add(Q, y);
                    NC = f2_sub(y, f2_sub(t, Q));
                    Q = t;
                    P = f2_mul(P, E);
                    V = Vi;
                }
            }
            k1 = k0;
        }
        float va, vb, Pa, Pb, Qa, Qb, na, nb;
        f2_unpack(V, va, vb);
        f2_unpack(P, Pa, Pb);
        f2_unpack(Q, Qa, Qb);
        f2_unpack(NC, na, nb);
        if (s0 < A.S) A.vdep[s0 * A.C + c] = lf_result((double)va, sg, (double)Pa, (double)Qa + (double)na);
        if (s1 < A.S) A.vdep[s1 * A.C + c] = lf_result((double)vb, sg, (double)Pb, (double)Qb + (double)nb);
    }
}

// Population variance over (theta, z) of u_r = cos(theta) u_x + sin(theta) u_y
// at radial node blockIdx.x, two passes (mean, then centred squares), fixed
// reduction order.
__global__ void __launch_bounds__(256) k_lf_variance(const double4_32a* __restrict__ g, int n_r, int n_th, int n_z,
                                                     double* __restrict__ var) {
    const int i = blockIdx.x;
    const int64_t n = (int64_t)n_th * n_z;
    __shared__ double red[256];
    double mean = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        double acc = 0.0;
        for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
            const int j = (int)(t % n_th);
            const double4_32a u = g[t * n_r + i];
            double sn, cs;
            sincos(2.0 * kPi * j / n_th, &sn, &cs);
            const double ur = cs * u.x + sn * u.y;
            const double e = pass == 0 ? ur : ur - mean;
            acc += pass == 0 ? e : e * e;
        }
        red[threadIdx.x] = acc;
        __syncthreads();
        for (int h = blockDim.x / 2; h > 0; h >>= 1) {
            if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
            __syncthreads();
        }
        const double tot = red[0] / (double)n;
        __syncthreads();
        if (pass == 0) mean = tot;
        else if (threadIdx.x == 0) var[i] = tot;
    }
}

}  // namespace pdq

using namespace pdq;

extern "C" void pdq_lf_desc_default(pdq_lf_desc* out) {
    if (!out) return;
    memset(out, 0, sizeof(*out));
    out->n_y = 2048;
    out->precision = PDQ_FP64;
    out->stretch = 8.0;
    out->t_lagr = 10.0;
    out->temperature = 293.15;
    out->vdw_cutoff = 1e-12;
}

extern "C" int pdq_lf_fluid_variance(const pdq_field* field, double* var, pdq_stream_t stream) {
    if (!field || !var) return PDQ_ERR_INVALID_ARG;
    const pdq_field_desc& d = field->desc;
    k_lf_variance<<<d.n_r, 256, 0, (cudaStream_t)stream>>>(field->grid64, d.n_r, d.n_th, d.n_z, var);
    PDQ_CUDA(cudaGetLastError());
    return PDQ_OK;
}

static size_t lf_shared_bytes(int32_t n_y, size_t elem) { return (size_t)5 * (size_t)(n_y - 1) * elem; }

// One wave: as many CTAs per class as fit on the GPU at once (its SMs times the
// resident CTAs per SM, divided among the classes), each building its class's
// table once and walking its share of the runs of `per` samples (a warp's).  Few
// samples spread a run to a CTA over as many SMs.
static int launch_lf(void (*kernel)(LfArgs), int threads, int per, size_t elem, const LfArgs& A, pdq_stream_t stream) {
    const size_t smem = lf_shared_bytes(A.n_y, elem);
    PDQ_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int dev = 0, sms = 0, per_sm = 0;
    PDQ_CUDA(cudaGetDevice(&dev));
    PDQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PDQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
    const int64_t nblk = (A.S + per - 1) / per;
    int64_t gx = (int64_t)(sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1) / A.C;
    if (gx < 1) gx = 1;
    // one CTA per SM while its warps take all the runs: a second one builds a table of its own on the same FP64 pipe
    // (FP32, 2,048 nodes, 2,500 samples of 10 classes: 396 us, 494 us with two; one march per class and SM 377 us)
    const int64_t one = std::max<int64_t>(1, sms / A.C);
    if (nblk <= one * (threads / 32)) gx = std::min(gx, one);
    if (gx > nblk) gx = nblk;
    const dim3 grid((unsigned)gx, (unsigned)A.C);
    kernel<<<grid, threads, smem, (cudaStream_t)stream>>>(A);
    PDQ_CUDA(cudaGetLastError());
    return PDQ_OK;
}

extern "C" int pdq_lf_vdep(const pdq_field* field, const pdq_phys* phys, const pdq_lf_desc* lf, const double* var,
                           int32_t n_classes, const double* st_plus, int64_t n_samples,
                           const pdq_sample_params* params, double* vdep, pdq_stream_t stream) {
    if (!field || !phys || !lf || !var || !st_plus || n_samples < 0) return PDQ_ERR_INVALID_ARG;
    if (n_classes < 1 || n_classes > PDQ_MAX_CLASSES) return PDQ_ERR_INVALID_ARG;
    if (lf->n_y < 3 || lf->n_y > PDQ_LF_MAX_NODES) return PDQ_ERR_INVALID_ARG;
    if (lf->precision != PDQ_FP64 && lf->precision != PDQ_MIXED) return PDQ_ERR_INVALID_ARG;
    if (!(lf->stretch > 0.0) || !(lf->stretch <= 700.0) || !(lf->t_lagr > 0.0) || !(lf->temperature > 0.0) ||
        !(lf->vdw_cutoff > 0.0))
        return PDQ_ERR_INVALID_ARG;
    if (field->desc.n_r < 2) return PDQ_ERR_INVALID_ARG;
    if (fabs(field->desc.r_plus - phys->re_tau) > 1e-9 * phys->re_tau) return PDQ_ERR_INVALID_ARG;
    if (n_samples == 0) return PDQ_OK;
    if (!params || !vdep) return PDQ_ERR_INVALID_ARG;
    const double ustar = phys->re_tau * phys->nu / phys->radius;
    const double ell = phys->nu / ustar;
    const double tauf = phys->nu / (ustar * ustar);
    const double acc = phys->nu / (ustar * ustar * ustar);
    LfArgs A;
    memset(&A, 0, sizeof(A));
    for (int c = 0; c < n_classes; ++c) {
        const double tau = st_plus[c];
        if (!(tau > 0.0)) return PDQ_ERR_INVALID_ARG;
        // tau_p = rho_p d^2/(18 rho_f nu), tau_p+ = tau_p/tau_f (Sec. 2.1)
        const double d = sqrt(18.0 * phys->rho_f * phys->nu * tau * tauf / phys->rho_p);
        const double m = phys->rho_p * kPi * d * d * d / 6.0;
        const double q1 = phys->q_unit * (d * 1e6) * (d * 1e6);     // q_max of the class
        LfClass& K = A.cls[c];
        K.tau = tau;
        K.y_w = 0.5 * d / ell;
        if (!(K.y_w < field->desc.r_plus)) return PDQ_ERR_INVALID_ARG;
        K.resp = lf->t_lagr / (lf->t_lagr + tau);
        K.d_b = kBoltzmann * lf->temperature * (tau * tauf) / m / phys->nu;
        K.thermal = kBoltzmann * lf->temperature / m / (ustar * ustar);
        // F_elec = -3 q^2/(8 pi^2 eps0 rho_p d^3 y^2), F_vdw = -A d/(12 m gap^2) per unit mass (App. B)
        K.ce = 3.0 * q1 * q1 / (8.0 * kPi * kPi * phys->eps0 * phys->rho_p * d * d * d) * acc / (ell * ell);
        K.cv = phys->hamaker0 * d / (12.0 * m) * acc / (ell * ell);
    }
    A.C = n_classes;
    A.n_y = lf->n_y;
    A.n_r = field->desc.n_r;
    A.S = n_samples;
    A.R = field->desc.r_plus;
    A.beta = field->desc.beta;
    A.tanh_beta = tanh(field->desc.beta);
    A.stretch = lf->stretch;
    A.em1_stretch = expm1(lf->stretch);
    A.t_lagr = lf->t_lagr;
    A.cut = lf->vdw_cutoff / ell;
    A.var = var;
    A.params = params;
    A.vdep = vdep;
    if (lf->precision == PDQ_FP64) return launch_lf(k_lf_vdep64, kLfThreads64, 32, sizeof(double), A, stream);
    return launch_lf(k_lf_vdep32, kLfThreads, 64, sizeof(f2), A, stream);
}
