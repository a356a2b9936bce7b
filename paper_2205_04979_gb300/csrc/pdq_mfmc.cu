// pdq_mfmc.cu -- multi-fidelity Monte Carlo allocation and Sobol' estimators
// (Sec. 3 of the paper): FP64 pick-freeze sums and estimators on the device,
// percentiles on the host.
//
// Model i's evaluations are laid out as y_i[g][col][c]: group g (a shared
// sample sequence, nested across models), column 0 = f(x), 1 = f(x'),
// 2 + j = f(z^(j)) with z^(j) = x' except input j from x, class/output c.
// For every model i and both prefix lengths m_{i-1} and m_i, one cluster of CTAs
// reduces, per output c, the sums
//   S1 = sum f(x), S2 = sum f(x)^2, R1 = sum f(x'), R2 = sum f(x')^2,
//   P_j = sum f(x) f(z^(j)), Q_j = sum (f(x') - f(z^(j)))^2,
// in a fixed order (deterministic).  Bootstrap replicate b >= 1 replaces group
// position t by an index drawn from word = Philox4x32-10 counter (t, b, 0, 2),
// key = seed, resampled within its nesting block: position t in
// [m_{l-1}, m_l) maps to m_{l-1} + ((word (m_l - m_{l-1})) >> 32); model i
// reads positions t < m_i, so it only touches its own evaluations and the
// nesting of the samples is kept.
#include <cooperative_groups.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "pdq_common.cuh"

namespace pdq {

constexpr int kMaxInputs = 16;

struct SumArgs {
    const double* y[8];     // per model, device [n_i][d+2][C]
    int64_t m[8];           // nested counts
    int32_t k, d, C;
    int32_t outs;           // outputs per cluster, at most kSumOutputs
    uint2 key;
    double* sums;           // [1+B][k][2][C][4+2d]
};

// One cluster of CTAs per (block of outputs, model, replicate): thread (t, c) of the cluster takes
// the group positions t, t + T, ... of output c, so that a warp's reads of a group are runs of the table
// (one output per CTA read a 32-byte sector for each 8-byte value, and drew every position's index again
// for each output).  The sums up to m_{i-1} (prefix 0) are taken on the way to m_i.  Each CTA adds its
// threads' sums in a fixed tree, the first CTA of the cluster adds the CTAs' in rank order: the
// result does not depend on the schedule.  Bound by the FP64 pipe, 13 operations per position and
// output at d = 3; D: the number of inputs (0: any, from A.d), so that the accumulators stay in registers.
// A study of 834 and 16,570 groups, 10 outputs, 200 replicates: 1.11 ms; 1.39 ms before.
// A thread adds its positions in runs of kRun, and the last adds keep what they round off: with few rows a thread's chain
// is up to ten times as long as with a CTA per output, and the variance and the total indices were 20 to 30 % further
// from extended precision (834 and 16,570 groups, 10 outputs, 40 seeds, rms: 2.3e-15 and 3.3e-15; 2.0e-15 and 2.6e-15
// with a CTA per output; 1.4e-15 and 1.9e-15 now).
constexpr int kSumThreads = 256, kSumOutputs = 32, kRun = 32;

// s + err = a + b exactly (Knuth's two-sum).
__device__ __forceinline__ double add_exactly(double a, double b, double& err) {
    const double s = a + b, bb = s - a;
    err = (a - (s - bb)) + (b - bb);
    return s;
}

template <int D>
__global__ void __launch_bounds__(kSumThreads) k_mfmc_sums(const SumArgs A) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int kMaxD = D ? D : kMaxInputs, kSums = 4 + 2 * kMaxD;
    __shared__ double red[8][kSumThreads];
    __shared__ double total[D ? kSums : 1][kSumThreads];
    __shared__ double part[kSums][kSumOutputs];
    const int d = D ? D : A.d, C = A.C, ncol = d + 2, nq = 4 + 2 * d;
    const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), c0 = (int)(blockIdx.x / ctas) * A.outs;
    const int i = blockIdx.y, b = blockIdx.z;         // model; 0 = the sample itself, >= 1 bootstrap
    const int nc = C - c0 < A.outs ? C - c0 : A.outs, T = kSumThreads / nc;
    const int tid = threadIdx.x, cc = tid % nc, tt = tid / nc;
    const bool active = tt < T;                       // the threads past T whole rows of outputs idle
    const double* __restrict__ y = A.y[i];
    // acc: a thread's run of kRun positions; total (its own slots; registers when the number of inputs is general): the runs before
    double acc[kSums], reg[D ? 1 : kSums];
#pragma unroll
    for (int q = 0; q < kSums; ++q) {
        acc[q] = 0.0;
        if constexpr (D) total[q][tid] = 0.0;
        else reg[q] = 0.0;
    }
    auto flush = [&]() {
#pragma unroll
        for (int q = 0; q < kSums; ++q) {
            if constexpr (D) total[q][tid] += acc[q];
            else reg[q] += acc[q];
            acc[q] = 0.0;
        }
    };
    int run = 0;
    int64_t t = (int64_t)rank * T + tt;
    for (int p = i > 0 ? 0 : 1; p < 2; ++p) {
        const int64_t m = p ? A.m[i] : A.m[i - 1];
        if (active) {
            for (; t < m; t += (int64_t)ctas * T) {
                int64_t g = t;
                if (b > 0) {
                    // block-wise resampling: position t in [m_{l-1}, m_l) draws from the same block,
                    // so every index stays below m_i for the positions model i reads
                    int l = 0;
                    while (t >= A.m[l]) ++l;
                    const int64_t lo = l > 0 ? A.m[l - 1] : 0;
                    const uint4 w = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)b, 0u, 2u), A.key);
                    g = lo + (int64_t)(((uint64_t)w.x * (uint64_t)(A.m[l] - lo)) >> 32);
                }
                const double* row = y + g * ncol * C + c0 + cc;
                const double fx = row[0], fxp = row[C];
                acc[0] += fx; acc[1] += fx * fx; acc[2] += fxp; acc[3] += fxp * fxp;
#pragma unroll
                for (int j = 0; j < kMaxD; ++j) {
                    if (j < d) {
                        const double fz = row[(int64_t)(2 + j) * C];
                        acc[4 + j] += fx * fz;
                        const double e = fxp - fz;
                        acc[4 + kMaxD + j] += e * e;
                    }
                }
                if (++run == kRun) {
                    flush();
                    run = 0;
                }
            }
        }
        flush();
        // the rows of threads fold in a fixed tree, 8 sums at a time, the last four rows with what their adds round off (a
        // chain of T FP64 adds by one thread per output took 20 us a sum at one output)
#pragma unroll
        for (int q0 = 0; q0 < kSums; q0 += 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (q0 + e < kSums) {
                    if constexpr (D) red[e][tid] = total[q0 + e][tid];
                    else red[e][tid] = reg[q0 + e];
                }
            }
            __syncthreads();
            int n = T;
            while (n > 4) {
                const int half = (n + 1) / 2, fold = (n - half) * nc;
                for (int u = tid; u < 8 * fold; u += kSumThreads) {
                    const int e = u / fold, r = u - e * fold;
                    red[e][r] += red[e][half * nc + r];
                }
                __syncthreads();
                n = half;
            }
            for (int u = tid; u < 8 * nc; u += kSumThreads) {
                const int e = u / nc, c = u - e * nc;
                if (q0 + e >= kSums) continue;
                double v = red[e][c], off = 0.0, err;
                for (int r = 1; r < n; ++r) {
                    v = add_exactly(v, red[e][r * nc + c], err);
                    off += err;
                }
                part[q0 + e][c] = v + off;
            }
            __syncthreads();
        }
        cluster.sync();
        if (rank == 0) {
            double* out = A.sums + ((((int64_t)b * A.k + i) * 2 + p) * C + c0) * nq;
            for (int u = tid; u < nc * nq; u += kSumThreads) {
                const int c = u / nq, q = u % nq;
                const int qs = q < 4 + d ? q : 4 + kMaxD + (q - 4 - d);
                double v = 0.0, off = 0.0, err;
                for (int r = 0; r < ctas; ++r) {
                    v = add_exactly(v, cluster.map_shared_rank(&part[0][0], r)[qs * kSumOutputs + c], err);
                    off += err;
                }
                out[(int64_t)c * nq + q] = v + off;
            }
        }
        cluster.sync();                               // part is read before it is written again, or the CTA ends
    }
}

template <int D>
static int launch_sums_d(const SumArgs& A, int ctas, int n_boot, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)((A.C + A.outs - 1) / A.outs * ctas), (unsigned)A.k, (unsigned)(1 + n_boot));
    cfg.blockDim = dim3(kSumThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof(attr));
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ctas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    PDQ_CUDA(cudaLaunchKernelEx(&cfg, k_mfmc_sums<D>, A));
    return PDQ_OK;
}

// A cluster takes all outputs (up to 32) with one CTA; while the clusters of a model are too few to give every SM
// 8 CTAs, and a thread keeps 12 positions of the longest model, the cluster grows to 8 CTAs and then
// takes fewer outputs, at the price of partly used sectors.  No replicates, 40,000 groups, 10 outputs: 0.10 ms
// (0.45 ms with 4 CTAs for all outputs, 0.30 ms with a CTA per output).  While SMs are idle an output more or less
// costs a CTA nothing, so there a thread keeps only 2 positions: the few CTAs' FP64 pipes are the bound
// (no replicates, 600 groups, 3 inputs, 10 outputs: 66 to 72 us a call; 79 us without this, 71 us with a CTA per
// output).
static int launch_sums(SumArgs A, int n_boot, int sms, cudaStream_t s) {
    int ctas = 1;
    A.outs = A.C < kSumOutputs ? A.C : kSumOutputs;
    const auto few = [&] { return (int64_t)((A.C + A.outs - 1) / A.outs) * (1 + n_boot) * ctas < 8 * (int64_t)sms; };
    const auto keeps = [&](int outs, int n, int positions) {
        return A.m[A.k - 1] >= (int64_t)positions * n * (kSumThreads / outs);
    };
    const auto idle = [&] { return (int64_t)((A.C + A.outs - 1) / A.outs) * (1 + n_boot) * ctas * A.k < sms; };
    while (ctas < 8 && few() && keeps(A.outs, 2 * ctas, 12)) ctas *= 2;
    while (A.outs > 1 && few() && keeps((A.outs + 1) / 2, ctas, 12)) A.outs = (A.outs + 1) / 2;
    while (A.outs > 1 && idle() && keeps((A.outs + 1) / 2, ctas, 2)) A.outs = (A.outs + 1) / 2;
    switch (A.d) {
        case 1: return launch_sums_d<1>(A, ctas, n_boot, s);
        case 2: return launch_sums_d<2>(A, ctas, n_boot, s);
        case 3: return launch_sums_d<3>(A, ctas, n_boot, s);
        case 4: return launch_sums_d<4>(A, ctas, n_boot, s);
        default: return launch_sums_d<0>(A, ctas, n_boot, s);
    }
}

struct AssembleArgs {
    double alpha[8];
    int64_t m[8];
    int32_t k, d, C, reps;
    double* sums;
};
// Mean, variance and the indices of input j of one (replicate, output) from its sums, into the slot of model 0's
// prefix 0, which has none: [2 + 2d] doubles (mean, var, s_main [d], s_total [d]).
__host__ __device__ inline void assemble(const AssembleArgs& A, double* rep, int c, int j) {
    const int nq = 4 + 2 * A.d;
    double mean = 0.0, var = 0.0, Vj = 0.0, Tj = 0.0;
    for (int i = 0; i < A.k; ++i) {
        for (int p = 1; p >= (i > 0 ? 0 : 1); --p) {
            const double mm = (double)(p ? A.m[i] : A.m[i - 1]);
            const double* s = rep + (((int64_t)i * 2 + p) * A.C + c) * nq;
            const double E = s[0] / mm, Ep = s[2] / mm;
            const double V = (s[1] - mm * E * E) / (mm - 1.0), Vp = (s[3] - mm * Ep * Ep) / (mm - 1.0);
            // term sign/weight: model 1 enters once; model i >= 2 as alpha_i (y_{m_i} - y_{m_{i-1}})
            const double wgt = i == 0 ? 1.0 : (p ? A.alpha[i] : -A.alpha[i]);
            mean += wgt * E;
            var += wgt * V;
            // Owen's main-effect estimator and Jansen's total-effect estimator (Sec. 3.3)
            Vj += wgt * (2.0 * mm / (2.0 * mm - 1.0) *
                         (s[4 + j] / mm - 0.25 * (E + Ep) * (E + Ep) + (V + Vp) / (4.0 * mm)));
            Tj += wgt * (s[4 + A.d + j] / (2.0 * mm));
        }
    }
    double* out = rep + (int64_t)c * nq;
    if (j == 0) { out[0] = mean; out[1] = var; }
    out[2 + j] = Vj / var;
    out[2 + A.d + j] = Tj / var;
}
// One thread per (replicate, output, input).
__global__ void k_mfmc_assemble(const AssembleArgs A) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, b = u / ((int64_t)A.C * A.d);
    if (b < A.reps) assemble(A, A.sums + b * A.k * 2 * A.C * (4 + 2 * A.d), (int)(u / A.d % A.C), (int)(u % A.d));
}

}  // namespace pdq

using namespace pdq;

extern "C" int pdq_mfmc_allocate(int32_t k, const double* rho, const double* sigma, const double* w, double budget,
                                 int32_t d_inputs, int64_t* m_out, double* alpha_out, double* m_real_out,
                                 double* gamma_out) {
    if (k < 1 || k > 8 || !rho || !sigma || !w || !m_out || !alpha_out || !(budget > 0) || d_inputs < 0)
        return PDQ_ERR_INVALID_ARG;
    for (int i = 0; i < k; ++i)
        if (!(sigma[i] > 0) || !(w[i] > 0) || !(fabs(rho[i]) <= 1.0)) return PDQ_ERR_INVALID_ARG;
    // rho_{1,1} = 1; rho_{1,k+1} taken as 0.
    std::vector<double> r2(k + 1, 0.0);
    for (int i = 0; i < k; ++i) r2[i] = i == 0 ? 1.0 : rho[i] * rho[i];
    for (int i = 1; i < k; ++i)
        if (!(r2[i] < r2[i - 1])) return PDQ_ERR_PRECOND;                    // models sorted by correlation
    // Eq. (mf-precond): w_{i-1}/w_i > (rho_{i-1}^2 - rho_i^2)/(rho_i^2 - rho_{i+1}^2), i = 2..k
    for (int i = 1; i < k; ++i) {
        const double lhs = w[i - 1] / w[i];
        const double rhs = (r2[i - 1] - r2[i]) / (r2[i] - r2[i + 1]);
        if (!(lhs > rhs)) return PDQ_ERR_PRECOND;
    }
    const double p = d_inputs > 0 ? budget / (d_inputs + 2) : budget;   // effective budget for Sobol' (d+2 runs)
    std::vector<double> r(k);
    double wr = 0.0;
    for (int i = 0; i < k; ++i) {
        // Eq. (opt2): r_i = sqrt(w_1 (rho_i^2 - rho_{i+1}^2) / (w_i (1 - rho_2^2)))
        r[i] = sqrt(w[0] * (r2[i] - r2[i + 1]) / (w[i] * (1.0 - r2[1])));
        wr += w[i] * r[i];
    }
    const double m1 = p / wr;                                             // m_1 = p / (w^T r)
    for (int i = 0; i < k; ++i) {
        const double mi = m1 * r[i];                                      // Eq. (opt3)
        if (m_real_out) m_real_out[i] = mi;
        m_out[i] = (int64_t)floor(mi);
        if (i > 0 && m_out[i] < m_out[i - 1]) m_out[i] = m_out[i - 1];
        alpha_out[i] = i == 0 ? 1.0 : rho[i] * sigma[0] / sigma[i];        // Eq. (opt1)
    }
    if (gamma_out) {
        // MSE of the MFMC mean with the real-valued optimum, relative to MC with the same budget:
        // MSE = sigma_1^2/m_1 + sum_i (1/m_{i-1} - 1/m_i)(alpha_i^2 sigma_i^2 - 2 alpha_i rho_i sigma_1 sigma_i)
        double mse = sigma[0] * sigma[0] / m1;
        for (int i = 1; i < k; ++i) {
            const double a = alpha_out[i];
            mse += (1.0 / (m1 * r[i - 1]) - 1.0 / (m1 * r[i])) *
                   (a * a * sigma[i] * sigma[i] - 2.0 * a * rho[i] * sigma[0] * sigma[i]);
        }
        *gamma_out = mse / (sigma[0] * sigma[0] * w[0] / p);
    }
    return PDQ_OK;
}

extern "C" int pdq_mfmc_workspace_size(int32_t k, int32_t d, int32_t C, int32_t n_boot, size_t* bytes) {
    if (!bytes || k < 1 || k > 8 || d < 1 || d > kMaxInputs || C < 1 || n_boot < 0) return PDQ_ERR_INVALID_ARG;
    *bytes = sizeof(double) * (size_t)(1 + n_boot) * k * 2 * C * (4 + 2 * d);
    return PDQ_OK;
}

extern "C" int pdq_mfmc_sobol(int32_t k, const double* const* y, const int64_t* m, const double* alpha, int32_t d,
                              int32_t C, int32_t n_boot, uint64_t seed, double* mean, double* var, double* s_main,
                              double* s_total, double* s_main_ci, double* s_total_ci, void* workspace,
                              size_t workspace_bytes, pdq_stream_t stream) {
    size_t need = 0;
    int rc = pdq_mfmc_workspace_size(k, d, C, n_boot, &need);
    if (rc) return rc;
    if (!y || !m || !alpha || !mean || !var || !s_main || !s_total) return PDQ_ERR_INVALID_ARG;
    if (n_boot > 0 && (!s_main_ci || !s_total_ci)) return PDQ_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < need) return PDQ_ERR_WORKSPACE;
    for (int i = 0; i < k; ++i) {
        if (!y[i] || m[i] < 2 || (i > 0 && m[i] < m[i - 1])) return PDQ_ERR_INVALID_ARG;
    }
    if ((uint64_t)m[k - 1] > 0xffffffffull) return PDQ_ERR_INVALID_ARG;
    SumArgs A;
    memset(&A, 0, sizeof(A));
    for (int i = 0; i < k; ++i) { A.y[i] = y[i]; A.m[i] = m[i]; }
    A.k = k; A.d = d; A.C = C;
    A.key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    A.sums = (double*)workspace;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 1;
    PDQ_CUDA(cudaGetDevice(&dev));
    PDQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    rc = launch_sums(A, n_boot, sms, s);
    if (rc) return rc;
    AssembleArgs B;
    memset(&B, 0, sizeof(B));
    for (int i = 0; i < k; ++i) { B.alpha[i] = alpha[i]; B.m[i] = m[i]; }
    B.k = k; B.d = d; B.C = C; B.reps = 1 + n_boot; B.sums = A.sums;
    // Each replicate's estimates are the first C rows of its sums.  A few are put together on the host, which
    // takes less than a kernel's launch.
    const size_t nq = 4 + 2 * (size_t)d, row = (size_t)C * nq, per_rep = (size_t)k * 2 * row;
    std::vector<double> h;
    if (n_boot == 0) {
        h.resize(per_rep);
        PDQ_CUDA(cudaMemcpyAsync(h.data(), workspace, per_rep * sizeof(double), cudaMemcpyDeviceToHost, s));
        PDQ_CUDA(cudaStreamSynchronize(s));
        for (int c = 0; c < C; ++c)
            for (int j = 0; j < d; ++j) assemble(B, h.data(), c, j);
    } else {
        h.resize(row * (size_t)(1 + n_boot));
        k_mfmc_assemble<<<(unsigned)(((int64_t)B.reps * C * d + 63) / 64), 64, 0, s>>>(B);
        PDQ_CUDA(cudaGetLastError());
        PDQ_CUDA(cudaMemcpy2DAsync(h.data(), row * sizeof(double), workspace, per_rep * sizeof(double),
                                   row * sizeof(double), (size_t)(1 + n_boot), cudaMemcpyDeviceToHost, s));
        PDQ_CUDA(cudaStreamSynchronize(s));
    }
    for (int c = 0; c < C; ++c) {
        const double* e = h.data() + (size_t)c * nq;
        mean[c] = e[0];
        var[c] = e[1];
        for (int j = 0; j < d; ++j) { s_main[(size_t)j * C + c] = e[2 + j]; s_total[(size_t)j * C + c] = e[2 + d + j]; }
    }
    if (n_boot > 0) {
        // percentile interval: the replicate values of ranks round(0.025 (B-1)) and round(0.975 (B-1))
        const int lo = (int)lround(0.025 * (n_boot - 1)), hi = (int)lround(0.975 * (n_boot - 1));
        std::vector<double> v(n_boot);
        const auto less = [](double a, double b) { return a < b || (b != b && a == a); };      // NaN last
        for (int which = 0; which < 2; ++which) {
            for (int j = 0; j < d; ++j) {
                for (int c = 0; c < C; ++c) {
                    for (int b = 0; b < n_boot; ++b) v[b] = h[row * (size_t)(1 + b) + (size_t)c * nq + 2 + which * d + j];
                    double* ci = (which ? s_total_ci : s_main_ci) + 2 * ((size_t)j * C + c);
                    std::nth_element(v.begin(), v.begin() + lo, v.end(), less);
                    ci[0] = v[lo];
                    std::nth_element(v.begin() + lo, v.begin() + hi, v.end(), less);
                    ci[1] = v[hi];
                }
            }
        }
    }
    return PDQ_OK;
}

// ---------------------------------------------------------------------------
// Derivative-based global sensitivity (DGSM) bounds on the total Sobol'
// indices (Sobol' & Kucherenko): for inputs uniform on [a_j, b_j],
//   s_j^t <= (b_j - a_j)^2 nu_j / (pi^2 Var f),  nu_j = E[(df/dx_j)^2],
// from S samples of the gradient.  One CTA per (output c, input j) reduces
// sum (df/dx_j)^2; one CTA per output computes the sample variance (two
// passes, divisor S - 1); fixed-order reductions.
// ---------------------------------------------------------------------------
namespace pdq {
__device__ __forceinline__ double block_sum_256(double v, double* red) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(256) k_dgsm(const double* __restrict__ grad, const double* __restrict__ y, int S,
                                              int C, int d, double* __restrict__ out /*[d+1][C]*/) {
    __shared__ double red[256];
    const int c = blockIdx.x, j = blockIdx.y;   // j == d: variance of y
    if (j < d) {
        double acc = 0.0;
        for (int s = threadIdx.x; s < S; s += blockDim.x) {
            const double gv = grad[((int64_t)s * C + c) * d + j];
            acc += gv * gv;
        }
        const double tot = block_sum_256(acc, red);
        if (threadIdx.x == 0) out[(int64_t)j * C + c] = tot / S;
    } else {
        double acc = 0.0;
        for (int s = threadIdx.x; s < S; s += blockDim.x) acc += y[(int64_t)s * C + c];
        const double mu = block_sum_256(acc, red) / S;
        double acc2 = 0.0;
        for (int s = threadIdx.x; s < S; s += blockDim.x) {
            const double e = y[(int64_t)s * C + c] - mu;
            acc2 += e * e;
        }
        const double tot = block_sum_256(acc2, red);
        if (threadIdx.x == 0) out[(int64_t)d * C + c] = tot / (S - 1);
    }
}
}  // namespace pdq

extern "C" int pdq_dgsm_workspace_size(int32_t C, int32_t d, size_t* bytes) {
    if (C < 1 || d < 1 || d > 64 || !bytes) return PDQ_ERR_INVALID_ARG;
    *bytes = sizeof(double) * (size_t)(d + 1) * (size_t)C;
    return PDQ_OK;
}

extern "C" int pdq_dgsm_bounds(int32_t S, int32_t C, int32_t d, const double* grad, const double* y,
                               const double* width, double* nu, double* bound, void* workspace,
                               size_t workspace_bytes, pdq_stream_t stream) {
    if (S < 2 || C < 1 || d < 1 || d > 64 || !grad || !y || !width || !nu || !bound) return PDQ_ERR_INVALID_ARG;
    size_t need = 0;
    pdq_dgsm_workspace_size(C, d, &need);
    if (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 7)) return PDQ_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    double* dev = (double*)workspace;   // (d+1) x C results: nu per input, then Var f
    k_dgsm<<<dim3(C, d + 1), 256, 0, s>>>(grad, y, S, C, d, dev);
    std::vector<double> h((size_t)(d + 1) * C);
    PDQ_CUDA(cudaGetLastError());
    PDQ_CUDA(cudaMemcpyAsync(h.data(), dev, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s));
    PDQ_CUDA(cudaStreamSynchronize(s));
    const double pi2 = kPi * kPi;
    for (int j = 0; j < d; ++j)
        for (int c = 0; c < C; ++c) {
            const double n = h[(size_t)j * C + c], var = h[(size_t)d * C + c];
            nu[(size_t)j * C + c] = n;
            bound[(size_t)j * C + c] = var > 0 ? width[j] * width[j] * n / (pi2 * var) : NAN;
        }
    return PDQ_OK;
}
