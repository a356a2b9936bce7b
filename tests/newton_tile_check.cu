// newton_tile over given cuts, for tests/test_gpu_newton_tile.py (compiled there).
#include "pdq_newton.cuh"

using namespace pdq;

struct TileArgs {
    const float4* pos;
    float4* acc;
    int n;
    float L, c2;
};

template <int NT, int U, bool CUT>
__global__ void __launch_bounds__(NT) k_tile(const TileArgs A) {
    const float4* pos = A.pos;
    const auto load = [pos](int64_t g) { return pos[g]; };
    newton_tile<NT, U, CUT>(load, (int64_t)blockIdx.x * NT * U, A.n, A.L, 1.0f / A.L, A.c2, A.acc, blockIdx.y, gridDim.y);
}

template <int NT, int U>
static void launch(const TileArgs& A, int parts) {
    const dim3 grid((A.n + NT * U - 1) / (NT * U), parts);
    if (parts > 1) k_tile<NT, U, true><<<grid, NT>>>(A);
    else k_tile<NT, U, false><<<grid, NT>>>(A);
}

// Coulomb sums of one sample of n particles, tiles of NT U, each over `parts` CTAs.
extern "C" int check_tile(const float4* pos, float4* acc, int n, int NT, int U, int parts, float L, float c2) {
    const TileArgs A{pos, acc, n, L, c2};
    if (NT == 64 && U == 4) launch<64, 4>(A, parts);
    else if (NT == 64 && U == 8) launch<64, 8>(A, parts);
    else if (NT == 64 && U == 12) launch<64, 12>(A, parts);
    else if (NT == 128 && U == 4) launch<128, 4>(A, parts);
    else if (NT == 128 && U == 8) launch<128, 8>(A, parts);
    else if (NT == 128 && U == 12) launch<128, 12>(A, parts);
    else return -1;
    return (int)cudaGetLastError();
}

// newton_cut's answer.
extern "C" void check_cut(int64_t capacity, int64_t samples, int NT, int64_t slots, int u_max, int* U, int* parts) {
    const NewtonCut c = newton_cut(capacity, samples, NT, slots, u_max);
    *U = c.U;
    *parts = c.parts;
}
