// pdq_split.cuh -- pair arithmetic on unevaluated sums of floats (float-float, T. J. Dekker 1971,
// D. E. Knuth's two-sum), for the FP64 pair sums whose work would otherwise sit on the FP64 pipe.
// GB300 issues 2 FP64 operations per clock and SM against 128 FP32 ones, so a pair at ~140 FP32
// operations costs a tenth of one at ~35 FP64 operations.
//
// A coordinate is cut into three floats on fixed grids, hi + mid + lo (all 53 bits), so the
// differences of the hi and of the mid parts are exact; a separation is then a float-float (D, E)
// and everything after it carries ~47 bits (a pair's term is off by 2^-47.6 of it, rms).
#pragma once

#include "pdq_device.cuh"

namespace pdq {

// a + b = s + e exactly, |a| >= |b| or a = 0 (fast), or any a, b.
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// The grids of the coordinate parts: hi a multiple of g, mid a multiple of g 2^-23; magic = 1.5 * 2^52 g
// rounds a double to a multiple of g.  g = 2^-23 times a power of two above every coordinate.
struct SplitGrid {
    double magic_hi, magic_mid;
    float top, g;
};
inline SplitGrid split_grid(double extent) {
    double top = 1.0;
    while (top < extent) top *= 2.0;
    while (top > 2.0 * extent) top *= 0.5;
    const double g = top * 1.1920928955078125e-07;                    // 2^-23
    return SplitGrid{6755399441055744.0 * g, 6755399441055744.0 * g * 1.1920928955078125e-07, (float)top, (float)g};
}
// hi + mid + lo = x; off the grid's range (|x| > top) the parts still sum to x.
__host__ __device__ __forceinline__ void split3(const SplitGrid& G, double x, float& hi, float& mid, float& lo) {
    // sums only, so no contraction can change them
    hi = (float)((x + G.magic_hi) - G.magic_hi);
    const double r = x - (double)hi;
    mid = (float)((r + G.magic_mid) - G.magic_mid);
    lo = (float)(r - (double)mid);
}

// Separation (D, E) of two split coordinates.  The hi parts' difference is 0 or at least g, the mid
// parts' at most g, so the fast sum is exact.
__device__ __forceinline__ void split_diff(float ah, float am, float al, float bh, float bm, float bl, float& D,
                                           float& E) {
    const float dh = __fsub_rn(ah, bh), dm = __fsub_rn(am, bm), dl = __fsub_rn(al, bl);
    fast_two_sum(dh, dm, D, E);
    E = __fadd_rn(E, dl);
}

// (R, r) = dx^2 + dy^2 + dz^2.
__device__ __forceinline__ void split_norm2(const float D[3], const float E[3], float& R, float& r) {
    float p[3], e[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = __fmul_rn(D[k], D[k]);
        e[k] = __fmaf_rn(D[k], __fadd_rn(E[k], E[k]), __fmaf_rn(E[k], E[k], __fmaf_rn(D[k], D[k], -p[k])));
    }
    float s, t1, t2;
    two_sum(p[0], p[1], s, t1);
    two_sum(s, p[2], R, t2);
    r = __fadd_rn(__fadd_rn(__fadd_rn(e[0], e[1]), __fadd_rn(e[2], t1)), t2);
}

// (w, v) = (R + r)^(-3/2): the hardware estimate y of R^(-1/2) is off by a few 2^-23, so with
// 1 - (R + r) y^2 = a + b (a exact, b its float remainder) y^3 (1 + 3/2 (a + b) + 15/8 (a + b)^2)
// leaves a relative 2^-63.
__device__ __forceinline__ void split_inv_cube(float R, float r, float& w, float& v) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(R));
    const float q = __fmul_rn(y, y), qe = __fmaf_rn(y, y, -q);
    const float p = __fmul_rn(R, q), pe = __fmaf_rn(R, q, -p);
    const float a = __fsub_rn(1.0f, p);
    const float b = __fmaf_rn(-r, q, __fmaf_rn(-R, qe, -pe));
    const float ab = __fadd_rn(a, b);
    const float ch = __fmul_rn(1.5f, a), cl = __fmaf_rn(1.875f, __fmul_rn(ab, ab), __fmul_rn(1.5f, b));
    const float c = __fmul_rn(y, q), ce = __fmaf_rn(y, qe, __fmaf_rn(y, q, -c));
    w = __fmaf_rn(ch, c, c);
    const float rem = __fmaf_rn(ch, c, -__fsub_rn(w, c));
    v = __fadd_rn(rem, __fmaf_rn(c, cl, __fmaf_rn(ce, __fadd_rn(ch, cl), ce)));
}

// (p, e) = (a, b) * (c, d).
__device__ __forceinline__ void split_mul(float a, float b, float c, float d, float& p, float& e) {
    p = __fmul_rn(a, c);
    e = __fmaf_rn(a, d, __fmaf_rn(b, c, __fmaf_rn(b, d, __fmaf_rn(a, c, -p))));
}

// The same on two pairs at a time (f32x2), for one j against two i-particles.
__device__ __forceinline__ f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ void two_sum(f2 a, f2 b, f2& s, f2& e) {
    const f2 t = f2_add(a, b), bb = f2_sub(t, a);
    e = f2_add(f2_sub(a, f2_sub(t, bb)), f2_sub(b, bb));
    s = t;
}
__device__ __forceinline__ void split_diff(f2 ah, f2 am, f2 al, f2 bh, f2 bm, f2 bl, f2& D, f2& E) {
    const f2 dh = f2_sub(ah, bh), dm = f2_sub(am, bm);
    D = f2_add(dh, dm);
    E = f2_add(f2_sub(dm, f2_sub(D, dh)), f2_sub(al, bl));
}
__device__ __forceinline__ void split_mul(f2 a, f2 b, f2 c, f2 d, f2& p, f2& e) {
    p = f2_mul(a, c);
    e = f2_fma(a, d, f2_fma(b, c, f2_fma(b, d, f2_fma(a, c, f2_neg(p)))));
}
// (w, v) = (D + E)^2 summed over the components, to the power -3/2.
__device__ __forceinline__ void split_inv_cube_norm(const f2 D[3], const f2 E[3], f2& w, f2& v) {
    f2 p[3], e[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = f2_mul(D[k], D[k]);
        e[k] = f2_fma(D[k], f2_add(E[k], E[k]), f2_fma(E[k], E[k], f2_fma(D[k], D[k], f2_neg(p[k]))));
    }
    f2 s, t1, t2, R;
    two_sum(p[0], p[1], s, t1);
    two_sum(s, p[2], R, t2);
    const f2 r = f2_add(f2_add(f2_add(e[0], e[1]), f2_add(e[2], t1)), t2);
    float Ra, Rb;
    f2_unpack(R, Ra, Rb);
    const f2 y = f2_pack(rsqrt_ftz(Ra), rsqrt_ftz(Rb));
    const f2 q = f2_mul(y, y), qe = f2_fma(y, y, f2_neg(q));
    const f2 m = f2_mul(R, q);
    // 1 - (R + r) y^2 = a - u
    const f2 a = f2_sub(f2_dup(1.0f), m);
    const f2 u = f2_fma(r, q, f2_fma(R, qe, f2_fma(R, q, f2_neg(m))));
    const f2 ab = f2_sub(a, u);
    const f2 ch = f2_mul(f2_dup(1.5f), a);
    const f2 cl = f2_fma(f2_dup(1.875f), f2_mul(ab, ab), f2_mul(f2_dup(-1.5f), u));
    const f2 c = f2_mul(y, q), ce = f2_fma(y, qe, f2_fma(y, q, f2_neg(c)));
    w = f2_fma(ch, c, c);
    v = f2_add(f2_fma(ch, c, f2_sub(c, w)), f2_fma(c, cl, f2_fma(ce, f2_add(ch, cl), ce)));
}

}  // namespace pdq
