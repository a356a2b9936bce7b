// The FP64 helpers of csrc/ beside CUDA's functions, for tests/test_gpu_math64.py (compiled there).
#include "pdq_lf_math.cuh"

using namespace pdq;

// out[k][2 n]: k = 0 rsqrt_seed, 1 rcp_seed, 2 lf_root(a, x), 3 lf_phi64(-x), 4 its E; ours, then CUDA's.
__global__ void k_math(const double* xs, const double* as, int n, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = xs[i], a = as[i];
    double E;
    auto put = [&](int k, double ours, double cuda) {
        out[(int64_t)(2 * k) * n + i] = ours;
        out[(int64_t)(2 * k + 1) * n + i] = cuda;
    };
    put(0, rsqrt_seed(x), 1.0 / sqrt(x));
    put(1, rcp_seed(x), 1.0 / x);
    put(2, lf_root(a, x), (x + x) / (a + sqrt(fma(a, a, x + x))));
    put(3, lf_phi64(-x, &E), expm1(-x) / -x);
    put(4, E, exp(-x));
}

extern "C" int check_math(const double* xs, const double* as, int n, double* out) {
    k_math<<<(n + 255) / 256, 256>>>(xs, as, n, out);
    return (int)cudaGetLastError();
}
