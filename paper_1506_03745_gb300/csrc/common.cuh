// Device helpers shared by the kernels of libpgb (no host state).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pgb_rules.h"

namespace pgb {

#define PGB_FOUR_PI 12.566370614359172953850573533118

// Quadrature rules passed to kernels by value (Section 3.1): far rule (K
// points), fine rule (19 points) and the edge rule of the self integral.
struct Rules {
    int K, Kn, ne;
    double mu[7][3], w[7];
    double mun[37][3], wn[37];  // close-by rule: 19 or 37 points
    double ex[12], ew[12];
};

Rules make_rules(int K, int Kn, int ne);

// Unfused IEEE double arithmetic: the tree decisions (Morton cells, box
// centres, acceptance tests) are evaluated operation by operation so that they
// are reproducible on any IEEE machine.
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ void rigid(const double* P, const double* v, double* out) {
    // out = ((R0 v0 + R1 v1) + R2 v2) + t, each row, no fused products
    for (int a = 0; a < 3; ++a)
        out[a] = dadd(dadd(dadd(dmul(P[3 * a + 0], v[0]), dmul(P[3 * a + 1], v[1])), dmul(P[3 * a + 2], v[2])), P[9 + a]);
}

// A long thin panel, whose points are summed one by one (treecode.cuh,
// point_sums): its farthest vertex lies more than sqrt(2 area) from the centroid.
// 0.88 of sqrt(area) on an equilateral triangle and 1.05 on a right isosceles
// one; sqrt(2) from an aspect ratio (longest edge over the height on it) of 2.3
// with the apex over one end to 4 over the middle.  Meshes of spheres, smooth
// molecules and boxes have none; where there are some, they cost what every
// panel did before the sums went panel by panel.  g: the squared distances of
// the vertices.
__host__ __device__ __forceinline__ bool is_sliver(const double (&g)[3], double area) {
    return g[0] > 2.0 * area || g[1] > 2.0 * area || g[2] > 2.0 * area;
}

// FP64 reciprocal square root to FP64 rounding: the SFU's estimate from the
// upper half of x (relative error d below 2^-20) refined by one step of
// Halley's iteration, y <- y + y e (1/2 + 3/8 e) with e = 1 - x y^2, which
// leaves about (5/2) d^3.  Five FP64 operations; two steps of Newton's iteration
// on the FP32 estimate take eight and two conversions.  x = 0 gives a
// non-finite value; callers mask it.
__device__ __forceinline__ double rsqrt_halley(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Coefficients (ln 2)^k / k! of the Taylor series of 2^f = e^{f ln 2}.
constexpr double PGB_LN2 = 0.69314718055994530941723212145818;
template <int K>
struct Exp2Coef {
    static constexpr double v = Exp2Coef<K - 1>::v * PGB_LN2 / K;
};
template <>
struct Exp2Coef<0> {
    static constexpr double v = 1.0;
};

// 2^(i / 32), rounded from 60 digits
static __device__ const double kExp2Frac[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0,
};

// FP64 2^t for t <= 1020.  32 t = n + 32 f with n = rint(32 t), found by adding
// and removing 1.5 * 2^47 (the sum rounds to a 32nd, whose low word is n),
// |f| <= 1/64; 2^f from its Taylor series to degree 5 (remainder below
// (ln 2 / 64)^6 / 6! < 3e-15 relative), times 2^((n mod 32) / 32) from a table
// (256 bytes, two lines of L1) with n / 32 added to its exponent field.
// Results from 2^-1020 down are returned as 0 (t beyond -1020 by more than
// 2^-11, which its upper word tells).  Nine FP64 operations; the series to
// degree 11 without a table takes fourteen.
__device__ __forceinline__ double exp2_table(double t) {
    const double magic = 211106232532992.0;  // 1.5 * 2^47
    const double s = t + magic;
    const int n = __double2loint(s);
    const double f = t - (s - magic);
    double p = Exp2Coef<5>::v;
    p = fma(p, f, Exp2Coef<4>::v);
    p = fma(p, f, Exp2Coef<3>::v);
    p = fma(p, f, Exp2Coef<2>::v);
    p = fma(p, f, Exp2Coef<1>::v);
    p = fma(p, f, 1.0);
    const double u = __ldg(kExp2Frac + (n & 31));
    const double y = p * __hiloint2double(__double2hiint(u) + (int)((unsigned)(n >> 5) << 20), __double2loint(u));
    return (unsigned)__double2hiint(t) > 0xC08FE000u ? 0.0 : y;  // by the upper word
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide reduction helpers (blockDim.x multiple of 32, <= 1024).
template <typename T>
__device__ T block_sum(T v, T* sh) {
    v = warp_sum(v);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? sh[threadIdx.x] : T(0);
    if (w == 0) v = warp_sum(v);
    __syncthreads();
    return v;  // valid in thread 0
}

// y = H(0:k,0:k)^{-1} g(0:k), upper triangular, column-major with ld, k at
// most BACK_THREADS, by one block of as many threads: column by column from the
// last, thread r holds row r and eight columns are in flight.  One thread's
// chain of dependent loads took 0.3 ms for 80 columns.
#define BACK_THREADS 256
__device__ __forceinline__ void backsolve(const double* __restrict__ H, int ld, const double* __restrict__ g, int k,
                                          double* __restrict__ y) {
    __shared__ double yi[2];
    const int r = threadIdx.x;
    double s = r < k ? g[r] : 0.0;
    const double d = r < k ? H[(int64_t)r * ld + r] : 0.0;
    double x[8], nx[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int i = k - 1 - u;
        nx[u] = i > r ? H[(int64_t)i * ld + r] : 0.0;
    }
    for (int i0 = k - 1; i0 >= 0; i0 -= 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            x[u] = nx[u];
            const int i = i0 - 8 - u;
            nx[u] = i > r ? H[(int64_t)i * ld + r] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 - u;
            if (i >= 0) {  // block-uniform
                if (r == i) {
                    s = d != 0 ? s / d : 0.0;
                    yi[u & 1] = s;
                    y[i] = s;
                }
                __syncthreads();
                if (r < i) s -= x[u] * yi[u & 1];
            }
        }
    }
}

}  // namespace pgb
